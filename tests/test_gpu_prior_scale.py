"""Prior rows of any positive sum, used as given: symbols whose row sums to 2^44 or to
2^-100, one alone and several running, at every place in a run of rows between two sums,
on every split of the recursions, in one piece and from checkpoints, with the kernels of
decodes and of gradients.  Row scales do not change the APPs, and every row of the
recursions stays within FP32 when it is scaled at its own step (2^44 or 2^-100 times a
step's 2^+-20 at most).  Against the FP64 oracle, with the parity tolerances."""
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


def _frame(scales, xmax=40, N=140):
    fr = synth.make_frame(np.random.default_rng(78), 8, 10, N, 2, xmax, 0.01, 0.01, 0.002,
                          dirichlet=True)
    pr = fr.priors.copy()
    for i, e in scales.items():
        pr[i] *= np.float32(2.0 ** e)
    return fr, pr


UP = {i: 44 for i in (66, 67, 68, 70, 71, 72, 73, 74, 90, 97, 103, 120)}
DOWN = {i: -100 for i in (67, 72, 73, 75, 81, 90, 91, 92, 93, 94, 104)}
MIXED = {**{i: 44 for i in (68, 69, 74, 99)}, **{i: -100 for i in (70, 75, 76, 100)}}
ALL = {i: 30 for i in range(140)}


@pytest.mark.parametrize("cluster", [None, 0, 1, 2, 8])
@pytest.mark.parametrize("scales", [UP, DOWN, MIXED, ALL], ids=["up", "down", "mixed", "all"])
def test_row_sums(monkeypatch, cluster, scales):
    if cluster is not None:
        monkeypatch.setenv("MAPDEC_CHAIN_CLUSTER", str(cluster))
    fr, pr = _frame(scales)
    ref, ll_ref = oracle.decode(fr.codebook, fr.N, fr.Pi, fr.Pd, fr.Ps, fr.I, fr.xmax, fr.rx,
                                priors=pr.astype(np.float64), kappa=2.0)
    b = mapdec.Batch([fr], flags=mapdec.MAPDEC_BATCH_GRAPH)
    for _ in range(2):
        st, app, ll = b.decode(fr.rx, pr.reshape(-1))
        assert st == 0
        check_app(app.reshape(fr.N, fr.q), ref)
        check_ll(ll[0], ll_ref)
    b.close()


@pytest.mark.parametrize("cluster", [1, 4])
@pytest.mark.parametrize("K", [None, 31])
def test_row_sums_checkpoints_gradients(monkeypatch, cluster, K):
    monkeypatch.setenv("MAPDEC_CHAIN_CLUSTER", str(cluster))
    flags = mapdec.MAPDEC_BATCH_GRAPH | mapdec.MAPDEC_BATCH_GRAD
    if K:
        monkeypatch.setenv("MAPDEC_SEG_K", str(K))
        flags |= mapdec.MAPDEC_BATCH_SEGMENTED
    cases = [_frame(UP, 150), _frame(DOWN, 150), _frame({}, 150)]
    frames = [fr for fr, _ in cases]
    b = mapdec.Batch(frames, flags=flags)
    rx, _ = b.concat_inputs()
    pr = np.concatenate([p.reshape(-1) for _, p in cases])
    st, app, ll = b.decode(rx, pr)
    apps = [a.copy() for a in b.split(app)]
    stg, dchan, _, llg = b.loglik_grad(rx, pr)
    b.close()
    assert (st, stg) == (0, 0)
    for k, (fr, p) in enumerate(cases):
        ref, ll_ref = oracle.decode(fr.codebook, fr.N, fr.Pi, fr.Pd, fr.Ps, fr.I, fr.xmax, fr.rx,
                                    priors=p.astype(np.float64), kappa=2.0)
        check_app(apps[k], ref, what=f"frame {k}")
        check_ll(ll[k], ll_ref, what=f"frame {k}")
        check_ll(llg[k], ll_ref, what=f"frame {k}")
        _, dchan_ref, _ = oracle.loglik_grad(fr.codebook, fr.N, fr.Pi, fr.Pd, fr.Ps, fr.I, fr.xmax,
                                             fr.rx, priors=p.astype(np.float64), kappa=2.0)
        check_grad(dchan[k], dchan_ref, what=f"frame {k}")
