"""The shared reductions at their edges, against the FP64 oracle with the parity
tolerances of every decode: the finalize kernel's groups of eight symbols and its
register slices of 32 codewords, and the per-symbol forward producer's
halving sums over the lanes of a group."""
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


# symbols around the groups of 8 and the chunk of 16, codewords around 32, 64
@pytest.mark.parametrize("N,q,n", [(1, 2, 3), (7, 31, 6), (8, 32, 6), (9, 33, 7), (15, 64, 8),
                                   (17, 65, 8), (33, 5, 5)])
def test_finalize_edges(N, q, n):
    rng = np.random.default_rng(40 + N)
    fr = synth.make_frame(rng, q, n, N, 2, 9, 0.04, 0.04, 0.01, dirichlet=True)
    ref, ext_ref, ll_ref = oracle.decode_ext(fr.codebook, N, 0.04, 0.04, 0.01, 2, 9, fr.rx,
                                             priors=fr.priors, kappa=2.0)
    b = mapdec.Batch([fr], flags=mapdec.MAPDEC_BATCH_EXTRINSIC)
    st, app, ext, ll = b.decode_ext(fr.rx, fr.priors.reshape(-1))
    b.close()
    assert st == 0
    check_app(app.reshape(N, q), ref)
    check_app(ext.reshape(N, q), ext_ref)
    check_ll(ll[0], ll_ref)
    g = mapdec.Batch([fr], flags=mapdec.MAPDEC_BATCH_GRAD)
    st, dchan, _, _ = g.loglik_grad(fr.rx, fr.priors.reshape(-1))
    g.close()
    assert st == 0
    check_grad(dchan[0], oracle.loglik_grad(fr.codebook, N, 0.04, 0.04, 0.01, 2, 9, fr.rx,
                                            priors=fr.priors)[1])


# compiled lattices of long codewords, and run-time ones past them
@pytest.mark.parametrize("n,I", [(13, 1), (14, 1), (15, 1), (13, 2), (15, 2), (13, 3), (14, 3),
                                 (15, 3), (16, 2), (20, 1)])
def test_long_codewords(n, I):
    N, q, xmax = 14, 6, 18
    fr = synth.make_frame(np.random.default_rng(n * I), q, n, N, I, xmax, 0.03, 0.03, 0.01,
                          dirichlet=True)
    ref, ll_ref = oracle.decode(fr.codebook, N, 0.03, 0.03, 0.01, I, xmax, fr.rx,
                                priors=fr.priors, kappa=2.0)
    b = mapdec.Batch([fr], flags=mapdec.MAPDEC_BATCH_GRAPH)
    st, app, ll = b.decode(fr.rx, fr.priors.reshape(-1))
    b.close()
    assert st == 0
    check_app(app.reshape(N, q), ref)
    check_ll(ll[0], ll_ref)


# lone frames whose tiles are cut to one round of lattices: q that divides the
# 256 threads or not, one that fills a round alone
@pytest.mark.parametrize("q,n", [(3, 4), (48, 6), (64, 7), (256, 9)])
def test_short_tiles(q, n):
    N, xmax = 25, 20
    fr = synth.make_frame(np.random.default_rng(q), q, n, N, 2, xmax, 0.04, 0.04, 0.01, dirichlet=True)
    ref, ll_ref = oracle.decode(fr.codebook, N, 0.04, 0.04, 0.01, 2, xmax, fr.rx, priors=fr.priors,
                                kappa=2.0)
    dec = mapdec.Decoder.for_frame(fr)
    app, ll = dec.decode(fr.rx, fr.priors)
    llg, dchan, _ = dec.loglik_grad(fr.rx, fr.priors)
    dec.close()
    check_app(app, ref)
    check_ll(ll, ll_ref)
    check_ll(llg, ll_ref)
    check_grad(dchan, oracle.loglik_grad(fr.codebook, N, 0.04, 0.04, 0.01, 2, xmax, fr.rx,
                                         priors=fr.priors)[1])


def test_many_supertiles_per_symbol():
    """A lone frame's super-tiles are short: a symbol's window spans more than the
    32 partial rows that finalize looks up at a time."""
    N, q, n, I, xmax = 30, 64, 6, 3, 230
    fr = synth.make_frame(np.random.default_rng(5), q, n, N, I, xmax, 0.05, 0.05, 0.01,
                          dirichlet=True)
    ref, ll_ref = oracle.decode(fr.codebook, N, 0.05, 0.05, 0.01, I, xmax, fr.rx,
                                priors=fr.priors, kappa=2.0)
    b = mapdec.Batch([fr], flags=mapdec.MAPDEC_BATCH_GRAPH)
    st, app, ll = b.decode(fr.rx, fr.priors.reshape(-1))
    b.close()
    assert st == 0
    check_app(app.reshape(N, q), ref)
    check_ll(ll[0], ll_ref)


# lanes per group 2, 2, 4, 8, 16, 32, 32; lengths below, at and above the group's lanes
@pytest.mark.parametrize("q,n,I", [(2, 4, 1), (3, 3, 2), (5, 5, 2), (9, 4, 3), (17, 5, 3),
                                   (33, 6, 1), (40, 12, 3)])
def test_per_symbol_forward_sums(q, n, I):
    N, xmax = 12, 14
    fr = synth.per_symbol_frame(np.random.default_rng(q * n), q, n, N, I, xmax, 0.04, 0.04, 0.01)
    ref, _, ll_ref = oracle.decode_ext(fr.codebook, N, 0.04, 0.04, 0.01, I, xmax, fr.rx,
                                       priors=fr.priors, kappa=2.0)
    b = mapdec.Batch([fr], flags=mapdec.MAPDEC_BATCH_GRAPH)
    st, app, ll = b.decode(fr.rx, fr.priors.reshape(-1))
    b.close()
    assert st == 0
    check_app(app.reshape(N, q), ref)
    check_ll(ll[0], ll_ref)
