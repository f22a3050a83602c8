"""Decoding with a batch planned for gradients: one batch serves mapdec_batch_decode,
_decode_ext and _loglik_grad in any order, whatever its producers' launches look
like.  Tiles of one position make enough of them that a CTA of the APP producer
takes several (two here), the layout in which the partial sums of a decode and of a
gradient call have to agree.  Against the FP64 oracle, with the parity tolerances
of every decode."""
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


# frames, N: about 360 and 145 tiles a frame and launch, more than 16 per SM in all
@pytest.mark.parametrize("segmented,count,N", [(False, 8, 60), (True, 20, 45)])
@pytest.mark.parametrize("tile", [1, 0])
def test_decode_between_gradients(monkeypatch, segmented, count, N, tile):
    if tile:
        monkeypatch.setenv("MAPDEC_FORCE_P", str(tile))
    if segmented:
        monkeypatch.setenv("MAPDEC_SEG_K", "20")
    rng = np.random.default_rng(2024)
    frames = [synth.make_frame(rng, 16, 6, N, 2, 12, 0.03, 0.03, 0.01, dirichlet=True)
              for _ in range(count)]
    flags = mapdec.MAPDEC_BATCH_GRAPH | mapdec.MAPDEC_BATCH_GRAD | mapdec.MAPDEC_BATCH_EXTRINSIC
    b = mapdec.Batch(frames, flags=flags | (mapdec.MAPDEC_BATCH_SEGMENTED if segmented else 0))
    rx, pr = b.concat_inputs()
    st, app, ext, ll = b.decode_ext(rx, pr)
    apps, exts = [a.copy() for a in b.split(app)], [a.copy() for a in b.split(ext)]
    st2, dchan, _, llg = b.loglik_grad(rx, pr)
    st3, app2, ll2 = b.decode(rx, pr)
    assert (st, st2, st3) == (0, 0, 0)
    assert np.array_equal(np.concatenate([a.ravel() for a in apps]), np.asarray(app2).ravel())
    assert np.array_equal(ll, ll2)
    b.close()
    for k in (0, 1, count // 2, count - 1):
        fr = frames[k]
        what = f"frame {k}"
        ref, ext_ref, ll_ref = oracle.decode_ext(fr.codebook, fr.N, fr.Pi, fr.Pd, fr.Ps, fr.I,
                                                 fr.xmax, fr.rx, priors=fr.priors, kappa=2.0)
        check_app(apps[k], ref, what=what)
        check_app(exts[k], ext_ref, what=what + " extrinsic")
        check_ll(ll[k], ll_ref, what=what)
        check_ll(llg[k], ll_ref, what=what)
        check_grad(dchan[k], oracle.loglik_grad(fr.codebook, fr.N, fr.Pi, fr.Pd, fr.Ps, fr.I,
                                                fr.xmax, fr.rx, priors=fr.priors)[1], what=what)
