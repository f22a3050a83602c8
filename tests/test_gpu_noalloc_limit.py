"""Allocation-free decode near the limit of its arena: frames whose scratch fits with the
planner's tiles but not with the short ones that fill the GPU, against mapdec_decode with
the parity tolerances; and one past the limit."""
import numpy as np
import pytest

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


def _noalloc(fr, priors):
    import torch
    rx = torch.from_numpy(np.ascontiguousarray(fr.rx)).cuda()
    pr = None if priors is None else torch.from_numpy(np.ascontiguousarray(priors)).cuda()
    app = torch.full((fr.N, fr.q), float("nan"), dtype=torch.float32, device="cuda")
    ll = torch.full((1,), float("nan"), dtype=torch.float64, device="cuda")
    st = mapdec.mapdec_decode_noalloc(fr, rx, pr, app, ll)
    return st, app.cpu().numpy(), float(ll.cpu()[0])


# q, n, N, I, xmax: 31.1, 24.4 and 29.7 MiB with the planner's tiles; 36.6, 40.2 and 34.0
# with the shortest
@pytest.mark.parametrize("shape", [(64, 8, 660, 2, 220), (64, 6, 460, 1, 440), (32, 8, 360, 2, 396)])
@pytest.mark.parametrize("uniform", [False, True])
def test_frames_near_the_limit(shape, uniform):
    q, n, N, I, xmax = shape
    fr = synth.make_frame(np.random.default_rng(N), q, n, N, I, xmax, 0.03, 0.03, 0.005,
                          dirichlet=not uniform)
    pri = None if uniform else fr.priors
    dec = mapdec.Decoder.for_frame(fr)
    app_ref, ll_ref = dec.decode(fr.rx, pri)
    dec.close()
    st, app, ll = _noalloc(fr, pri)
    assert st == mapdec.MAPDEC_OK, mapdec.mapdec_strerror(st)
    check_app(app, app_ref)
    check_ll(ll, ll_ref)


def test_frame_past_the_limit():
    """Transition sums alone: 800 x 441 x 25 floats, 33.6 MiB."""
    fr = synth.make_frame(np.random.default_rng(1), 64, 8, 800, 2, 220, 0.03, 0.03, 0.005,
                          dirichlet=False)
    st, _, _ = _noalloc(fr, None)
    assert st == mapdec.MAPDEC_ERR_TOO_LARGE
