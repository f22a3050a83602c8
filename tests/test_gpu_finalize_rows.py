"""Partial rows of a symbol in the finalize kernel, which loads four at a time: counts
just below, at and above a multiple of four (tiles of one and two positions, one to a
super-tile), for decodes and gradients.  Against the FP64 oracle, with the parity
tolerances."""
import numpy as np
import pytest

import oracle
from parity import check_app, check_grad, check_ll
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


# 2 xmax + 1 rows a symbol with tiles of one position, xmax + 1 (or one more) with two
@pytest.mark.parametrize("grad", [False, True])
@pytest.mark.parametrize("tile, xmax", [(1, 1), (1, 2), (1, 3), (1, 4), (2, 3), (2, 4), (2, 7)])
def test_rows_around_a_multiple_of_four(monkeypatch, tile, xmax, grad):
    monkeypatch.setenv("MAPDEC_FORCE_P", str(tile))
    monkeypatch.setenv("MAPDEC_FORCE_NSUB", "1")
    q, n, N, I = 9, 5, 21, 1
    fr = synth.make_frame(np.random.default_rng(60 + xmax), q, n, N, I, xmax, 0.004, 0.004, 0.01,
                          dirichlet=True)
    b = mapdec.Batch([fr], flags=mapdec.MAPDEC_BATCH_GRAPH |
                     (mapdec.MAPDEC_BATCH_GRAD if grad else 0))
    pr = fr.priors.reshape(-1)
    st, app, ll = b.decode(fr.rx, pr)
    assert st == 0
    ref, ll_ref = oracle.decode(fr.codebook, N, fr.Pi, fr.Pd, fr.Ps, I, xmax, fr.rx,
                                priors=fr.priors, kappa=2.0)
    check_app(app.reshape(N, q), ref)
    check_ll(ll[0], ll_ref)
    if grad:
        stg, dchan, _, _ = b.loglik_grad(fr.rx, pr)
        assert stg == 0
        check_grad(dchan[0], oracle.loglik_grad(fr.codebook, N, fr.Pi, fr.Pd, fr.Ps, I, xmax, fr.rx,
                                                priors=fr.priors.astype(np.float64), kappa=2.0)[1])
    b.close()
