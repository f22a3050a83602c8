"""The recursion kernel's splits: CTAs per recursion (a cluster), chunks of
states per step, and copies in flight, at the sizes where they can go wrong:
fewer states than a cluster has blocks (CTAs that own none), blocks no longer
than the band halo, a state count that no split divides, a single state, chunks of
more lane groups than virtual warps, and a row that is scaled at once because a step shrank it below the lagged scaling's
range.  Against the FP64 oracle, with the parity tolerances of every decode."""
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


# q, n, N, I, xmax
SHAPES = [(4, 4, 30, 2, 0), (5, 7, 40, 1, 3), (8, 6, 50, 2, 33), (16, 10, 40, 2, 79),
          (12, 12, 24, 3, 64), (4, 15, 20, 3, 40), (8, 6, 12, 2, 349)]


@pytest.mark.parametrize("cluster", [0, 1, 2, 4, 8])
@pytest.mark.parametrize("shape", SHAPES)
def test_cluster_split(monkeypatch, cluster, shape):
    q, n, N, I, xmax = shape
    monkeypatch.setenv("MAPDEC_CHAIN_CLUSTER", str(cluster))
    rng = np.random.default_rng(1000 + n * N)
    p = 0.05 if xmax > 3 else 0.002
    fr = synth.make_frame(rng, q, n, N, I, xmax, p, p, 0.01, dirichlet=True)
    ref, ll_ref = oracle.decode(fr.codebook, N, p, p, 0.01, I, xmax, fr.rx, priors=fr.priors,
                                kappa=2.0)
    for cd in (None, "32"):
        if cd:
            monkeypatch.setenv("MAPDEC_CHAIN_CD", cd)
            monkeypatch.setenv("MAPDEC_CHAIN_STAGES", "3")
        b = mapdec.Batch([fr], flags=mapdec.MAPDEC_BATCH_GRAPH)
        st, app, ll = b.decode(fr.rx, fr.priors.reshape(-1))
        assert st == 0
        check_app(app.reshape(N, q), ref, what=f"cluster {cluster} chunk {cd}")
        check_ll(ll[0], ll_ref, what=f"cluster {cluster} chunk {cd}")
        b.close()


@pytest.mark.parametrize("xmax", [1300, 6000])
def test_long_rows(xmax):
    """Rows too long for four buffers of them, and for the latency kernel at all."""
    q, n, N, I = 2, 4, 8, 1
    fr = synth.make_frame(np.random.default_rng(xmax), q, n, N, I, xmax, 0.05, 0.05, 0.01,
                          dirichlet=True)
    ref, ll_ref = oracle.decode(fr.codebook, N, 0.05, 0.05, 0.01, I, xmax, fr.rx,
                                priors=fr.priors, kappa=2.0)
    b = mapdec.Batch([fr], flags=mapdec.MAPDEC_BATCH_GRAPH)
    st, app, ll = b.decode(fr.rx, fr.priors.reshape(-1))
    b.close()
    assert st == 0
    check_app(app.reshape(N, q), ref)
    check_ll(ll[0], ll_ref)


@pytest.mark.parametrize("cluster", [1, 4])
def test_rows_scaled_at_once(monkeypatch, cluster):
    """Priors that give the sent symbol 2^-40 in three symbols running: each step
    shrinks the row by about that, past the lagged scaling's range."""
    monkeypatch.setenv("MAPDEC_CHAIN_CLUSTER", str(cluster))
    q, n, N, I, xmax = 8, 8, 40, 2, 40
    rng = np.random.default_rng(77)
    fr = synth.make_frame(rng, q, n, N, I, xmax, 0.01, 0.01, 0.002, dirichlet=False)
    pr = np.full((N, q), 1.0 / q, np.float32)
    for i in (10, 11, 12, 25):
        pr[i] = 2.0 ** -40
    ref, ll_ref = oracle.decode(fr.codebook, N, 0.01, 0.01, 0.002, I, xmax, fr.rx, priors=pr,
                                kappa=2.0)
    b = mapdec.Batch([fr], flags=mapdec.MAPDEC_BATCH_GRAPH)
    st, app, ll = b.decode(fr.rx, pr.reshape(-1))
    assert st == 0
    check_app(app.reshape(N, q), ref)
    check_ll(ll[0], ll_ref)
    b.close()
