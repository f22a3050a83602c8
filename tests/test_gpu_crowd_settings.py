"""Block size of the recursions of full launches, from the environment: parity with the
FP64 oracle at each, and a smaller block that shows in the order of the additions.  Two
frames carry boundary priors."""
import numpy as np
import pytest

import oracle
from parity import check_app, check_ll
from paper_1802_08483_gb300 import mapdec, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1802_08483_gb300 import build
    build.build()
    mapdec.load()
    oracle.build()


def test_block_size_from_the_environment(monkeypatch):
    monkeypatch.setenv("MAPDEC_CHAIN_CLUSTER", "0")
    frames = [synth.stream_frame(np.random.default_rng(41), 8, 6, 150, 2, 40, 0.03, 0.03, 0.01,
                                 6, 7, 3.0),
              synth.stream_frame(np.random.default_rng(42), 4, 6, 100, 2, 90, 0.04, 0.02, 0.01,
                                 9, 4, 4.0),
              synth.make_frame(np.random.default_rng(43), 8, 6, 120, 2, 60, 0.03, 0.03, 0.01,
                               dirichlet=True)]
    out = {}
    for threads in (None, 128, 256, 512):
        if threads:
            monkeypatch.setenv("MAPDEC_CHAIN_THREADS", str(threads))
        b = mapdec.Batch(frames, flags=mapdec.MAPDEC_BATCH_GRAPH)
        rx, pr = b.concat_inputs()
        st, app, ll = b.decode(rx, pr)
        assert st == 0
        out[threads] = (app.copy(), ll.copy())
        for k, (fr, a) in enumerate(zip(frames, b.split(app))):
            ref, _, ll_ref = oracle.decode_ext(
                fr.codebook, fr.N, fr.Pi, fr.Pd, fr.Ps, fr.I, fr.xmax, fr.rx,
                priors=fr.priors_or_uniform(), kappa=2.0,
                drift_start=getattr(fr, "drift_start", None),
                drift_end=getattr(fr, "drift_end", None))
            check_app(a, ref, what=f"frame {k}, {threads} threads")
            check_ll(ll[k], ll_ref, what=f"frame {k}, {threads} threads")
        b.close()
    assert np.array_equal(out[None][0], out[256][0])
    assert not np.array_equal(out[128][0], out[256][0])
