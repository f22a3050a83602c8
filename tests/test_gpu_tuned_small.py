"""Small batches (fewer recursions than SMs) with a tuning table: parity with the FP64
oracle, and recursions that do not depend on the table, whose shared-memory budget and
stages are those of full launches' recursions."""
import os

import numpy as np
import pytest

import oracle
from parity import check_app, check_ll
from paper_1802_08483_gb300 import mapdec, synth, tune

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
    yield
    mapdec.mapdec_tune_clear()


def test_committed_table_on_a_small_batch():
    mapdec.mapdec_tune_clear()
    tune.load(os.path.join(os.path.dirname(tune.__file__), "tuning", "gb300_mixed4096.json"))
    rng = np.random.default_rng(15)
    frames = [synth.make_frame(rng, q, n, 90, I, 40, 0.03, 0.03, 0.01, dirichlet=True)
              for q, n, I in ((2, 4, 2), (8, 6, 2), (16, 10, 2), (32, 8, 2), (64, 12, 2))]
    b = mapdec.Batch(frames, flags=mapdec.MAPDEC_BATCH_GRAPH)
    rx, pr = b.concat_inputs()
    st, app, ll = b.decode(rx, pr)
    mapdec.mapdec_tune_clear()
    assert st == 0
    for fr, a, l in zip(frames, b.split(app), ll):
        ref, ll_ref = oracle.decode(fr.codebook, fr.N, fr.Pi, fr.Pd, fr.Ps, fr.I, fr.xmax, fr.rx,
                                    priors=fr.priors, kappa=2.0)
        check_app(a, ref, what=f"n={fr.n}")
        check_ll(l, ll_ref, what=f"n={fr.n}")
    b.close()


def _recursion_ms(frames):
    b = mapdec.Batch(frames, flags=mapdec.MAPDEC_BATCH_GRAPH | mapdec.MAPDEC_BATCH_TIMING)
    rx, pr = b.concat_inputs()
    best = float("inf")
    for _ in range(10):
        st, _, _ = b.decode(rx, pr)
        assert st == 0
        best = min(best, float(mapdec.mapdec_batch_phase_ms(b.b)[2]))
    b.close()
    return best


def test_recursion_time_of_a_tuned_small_batch():
    """A row of 171 states does not fit 52 KB in one staged chunk."""
    mapdec.mapdec_tune_clear()
    rng = np.random.default_rng(16)
    frames = [synth.make_frame(rng, 16, 10, 300, 2, 85, 0.01, 0.01, 0.005, dirichlet=True)
              for _ in range(64)]
    plain = _recursion_ms(frames)
    mapdec.mapdec_tune_set(16, 10, 2, {"chain_budget_kb": 52, "chain_stages": 2,
                                       "chain_threads": 128})
    tuned = _recursion_ms(frames)
    mapdec.mapdec_tune_clear()
    assert tuned <= 1.2 * plain, (tuned, plain)
