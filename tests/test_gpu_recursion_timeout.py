"""A copy of the transition sums that is never issued (test hook), on every split of the
recursions: the first one of every block, or a later one of a cluster's last block only,
at each place in a run of four steps.  Every block gives up at the same step: the call
returns the status, and the next decode on the device is right."""
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


NARROW, WIDE = (8, 6, 110, 2, 33), (8, 6, 90, 2, 349)  # q, n, N, I, xmax


@pytest.mark.parametrize("copy", [0, 3, 70, 71, 72, 73])
@pytest.mark.parametrize("cluster, shape", [(0, NARROW), (1, NARROW), (1, WIDE), (2, WIDE),
                                            (4, WIDE), (8, WIDE)])
def test_copy_that_never_lands(monkeypatch, cluster, shape, copy):
    q, n, N, I, xmax = shape
    fr = synth.make_frame(np.random.default_rng(5), q, n, N, I, xmax, 0.03, 0.03, 0.01,
                          dirichlet=True)
    monkeypatch.setenv("MAPDEC_CHAIN_CLUSTER", str(cluster))
    monkeypatch.setenv("MAPDEC_TEST_STALL_CHAIN", str(copy + 1))
    b = mapdec.Batch([fr], flags=mapdec.MAPDEC_BATCH_GRAPH)
    for _ in range(2):
        st, _, _ = b.decode(fr.rx, fr.priors.reshape(-1))
        assert st == mapdec.MAPDEC_ERR_TIMEOUT
    b.close()
    monkeypatch.delenv("MAPDEC_TEST_STALL_CHAIN")
    b = mapdec.Batch([fr], flags=mapdec.MAPDEC_BATCH_GRAPH)
    st, app, ll = b.decode(fr.rx, fr.priors.reshape(-1))
    b.close()
    assert st == 0
    ref, ll_ref = oracle.decode(fr.codebook, N, fr.Pi, fr.Pd, fr.Ps, I, xmax, fr.rx,
                                priors=fr.priors, kappa=2.0)
    check_app(app.reshape(N, q), ref)
    check_ll(ll[0], ll_ref)
