"""The recursion kernel past its settling phase (64 steps), where up to four rows are
built between two sums: every split of the work (several frames' rows wide and
narrow, clusters, staged chunks), checkpoints with recorded and replayed tilts,
boundary priors and gradients on clusters, launches per code length side by side.
MAPDEC_CHAIN_CLUSTER = 0 is the kernel of launches with more recursions than SMs.
Against the FP64 oracle, with the parity tolerances of every decode."""
import numpy as np
import pytest

import oracle
from parity import check_app, check_grad, check_grad_priors, check_ll
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


# q, n, N, I, xmax: one lane group; a warp per virtual warp; a warp per lane group;
# more groups than warps
SHAPES = [(5, 7, 100, 1, 3), (8, 6, 110, 2, 33), (4, 4, 130, 1, 150), (8, 6, 90, 2, 349)]


@pytest.mark.parametrize("cluster", [0, 1, 2, 4, 8])
@pytest.mark.parametrize("shape", SHAPES)
def test_runs_of_rows(monkeypatch, cluster, shape):
    q, n, N, I, xmax = shape
    monkeypatch.setenv("MAPDEC_CHAIN_CLUSTER", str(cluster))
    p = 0.05 if xmax > 3 else 0.002
    fr = synth.make_frame(np.random.default_rng(7 + n * N), q, n, N, I, xmax, p, p, 0.01,
                          dirichlet=True)
    ref, ll_ref = oracle.decode(fr.codebook, N, p, p, 0.01, I, xmax, fr.rx, priors=fr.priors,
                                kappa=2.0)
    for cd in (None, "32"):
        if cd:
            monkeypatch.setenv("MAPDEC_CHAIN_CD", cd)
            monkeypatch.setenv("MAPDEC_CHAIN_STAGES", "3")
        b = mapdec.Batch([fr], flags=mapdec.MAPDEC_BATCH_GRAPH)
        st, app, ll = b.decode(fr.rx, fr.priors.reshape(-1))
        b.close()
        assert st == 0
        check_app(app.reshape(N, q), ref, what=f"cluster {cluster} chunk {cd}")
        check_ll(ll[0], ll_ref, what=f"cluster {cluster} chunk {cd}")


@pytest.mark.parametrize("cluster", [0, 1, 2, 8])
@pytest.mark.parametrize("K", [None, 29, 90])
def test_priors_checkpoints_gradients(monkeypatch, cluster, K):
    """Boundary priors, extrinsic outputs and gradients, in one piece and from
    checkpoints (K = 29: a run of rows ends at a segment's edge; 90: in one)."""
    monkeypatch.setenv("MAPDEC_CHAIN_CLUSTER", str(cluster))
    flags = mapdec.MAPDEC_BATCH_GRAPH
    if K:
        monkeypatch.setenv("MAPDEC_SEG_K", str(K))
        flags |= mapdec.MAPDEC_BATCH_SEGMENTED
    frames = [synth.stream_frame(np.random.default_rng(31), 8, 6, 150, 2, 60, 0.03, 0.03, 0.01,
                                 6, 7, 3.0),
              synth.stream_frame(np.random.default_rng(32), 4, 6, 100, 2, 170, 0.04, 0.02, 0.01,
                                 9, 4, 4.0),
              synth.make_frame(np.random.default_rng(33), 8, 6, 120, 2, 90, 0.03, 0.03, 0.01,
                               dirichlet=True)]
    b = mapdec.Batch(frames, flags=flags | mapdec.MAPDEC_BATCH_EXTRINSIC)
    rx, pr = b.concat_inputs()
    st, app, ext, ll = b.decode_ext(rx, pr)
    apps, exts = [a.copy() for a in b.split(app)], [a.copy() for a in b.split(ext)]
    b.close()
    g = mapdec.Batch(frames, flags=flags | mapdec.MAPDEC_BATCH_GRAD)
    stg, dchan, dpri, llg = g.loglik_grad(rx, pr)
    dpris = [a.copy() for a in g.split(dpri)]
    g.close()
    assert st == 0 and stg == 0
    for k, fr in enumerate(frames):
        what = f"frame {k}"
        edges = dict(drift_start=getattr(fr, "drift_start", None),
                     drift_end=getattr(fr, "drift_end", None))
        pri = fr.priors_or_uniform()
        ref, ext_ref, ll_ref = oracle.decode_ext(fr.codebook, fr.N, fr.Pi, fr.Pd, fr.Ps, fr.I,
                                                 fr.xmax, fr.rx, priors=pri, kappa=2.0, **edges)
        check_app(apps[k], ref, what=what)
        check_app(exts[k], ext_ref, what=what + " extrinsic")
        check_ll(ll[k], ll_ref, what=what)
        check_ll(llg[k], ll_ref, what=what)
        _, dchan_ref, dpri_ref = oracle.loglik_grad(
            fr.codebook, fr.N, fr.Pi, fr.Pd, fr.Ps, fr.I, fr.xmax, fr.rx,
            priors=pri.astype(np.float64), kappa=2.0, **edges)
        check_grad(dchan[k], dchan_ref, what=what + " channel")
        check_grad_priors(dpris[k], dpri_ref, pri, what=what + " priors")


# codes of a batch: up to six lengths run side by side, more in one general launch
@pytest.mark.parametrize("codes", [((4, 1), (6, 2), (5, 3)),
                                   ((4, 1), (6, 2), (5, 3), (7, 1), (8, 1), (9, 1), (10, 1), (3, 2))])
def test_launches_per_code_length(codes):
    rng = np.random.default_rng(90)
    frames = [synth.make_frame(rng, 8, n, 90, I, 24, 0.03, 0.03, 0.01, dirichlet=True)
              for n, I in codes]
    b = mapdec.Batch(frames, flags=mapdec.MAPDEC_BATCH_GRAPH)
    rx, pr = b.concat_inputs()
    st, app, ll = b.decode(rx, pr)
    assert st == 0
    for fr, a, l in zip(frames, b.split(app), ll):
        ref, ll_ref = oracle.decode(fr.codebook, fr.N, fr.Pi, fr.Pd, fr.Ps, fr.I, fr.xmax, fr.rx,
                                    priors=fr.priors, kappa=2.0)
        check_app(a, ref, what=f"n={fr.n} I={fr.I}")
        check_ll(l, ll_ref, what=f"n={fr.n} I={fr.I}")
    b.close()
