"""Scratch of short tiles against the budget: a batch that fits its budget in one wave
with the planner's tiles runs in one wave; gradient batches that fill the GPU with the
planned super-tiles keep one row of partial sums for each.  Against the FP64 oracle or
the same batch without a limit, with the parity tolerances of every decode."""
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


def _check_gradients(b, frames, rx, pr, which):
    st, dchan, dpri, ll = b.loglik_grad(rx, pr)
    assert st == 0
    dpris = b.split(dpri)
    for k in which:
        fr = frames[k]
        ll_ref, dchan_ref, dpri_ref = oracle.loglik_grad(
            fr.codebook, fr.N, fr.Pi, fr.Pd, fr.Ps, fr.I, fr.xmax, fr.rx,
            priors=fr.priors.astype(np.float64), kappa=2.0)
        check_ll(ll[k], ll_ref, what=f"frame {k}")
        check_grad(dchan[k], dchan_ref, what=f"frame {k}")
        check_grad_priors(dpris[k], dpri_ref, fr.priors, what=f"frame {k}")


@pytest.mark.parametrize("segmented", [False, True])
def test_full_launch_of_planned_supertiles(monkeypatch, segmented):
    """Tiles of one position, two to a super-tile: more than 16 tiles per SM."""
    monkeypatch.setenv("MAPDEC_FORCE_P", "1")
    monkeypatch.setenv("MAPDEC_FORCE_NSUB", "2")
    count, N = (20, 45) if segmented else (8, 61)
    flags = mapdec.MAPDEC_BATCH_GRAPH | mapdec.MAPDEC_BATCH_GRAD
    if segmented:
        monkeypatch.setenv("MAPDEC_SEG_K", "20")
        flags |= mapdec.MAPDEC_BATCH_SEGMENTED
    rng = np.random.default_rng(2025)
    frames = [synth.make_frame(rng, 15, 6, N, 2, 12, 0.03, 0.03, 0.01, dirichlet=True)
              for _ in range(count)]
    b = mapdec.Batch(frames, flags=flags)
    rx, pr = b.concat_inputs()
    which = (0, 3, count - 1)
    _check_gradients(b, frames, rx, pr, which)
    st, app, ll = b.decode(rx, pr)
    assert st == 0
    for k in which:
        fr = frames[k]
        ref, _ = oracle.decode(fr.codebook, N, fr.Pi, fr.Pd, fr.Ps, fr.I, fr.xmax, fr.rx,
                               priors=fr.priors, kappa=2.0)
        check_app(b.split(app)[k], ref, what=f"frame {k}")
    b.close()


def test_gradient_budget():
    """About 32 KB of scratch a symbol with the planned super-tiles, 60 with a row of
    partial sums per tile of two positions."""
    N, count = 50, 16
    rng = np.random.default_rng(2026)
    frames = [synth.make_frame(rng, 64, 12, N, 2, 100, 0.03, 0.03, 0.01, dirichlet=True)
              for _ in range(count)]
    flags = mapdec.MAPDEC_BATCH_GRAPH | mapdec.MAPDEC_BATCH_GRAD
    for kb in (45, 120):
        b = mapdec.Batch(frames, flags=flags, mem_budget_bytes=kb * 1024 * N * count)
        assert mapdec.mapdec_batch_num_waves(b.b) == 1
        rx, pr = b.concat_inputs()
        _check_gradients(b, frames, rx, pr, (0, count - 1))
        b.close()


def test_decode_budget():
    """24.4 MiB a frame with the planner's tiles, up to 40 with the short ones."""
    rng = np.random.default_rng(2027)
    frames = [synth.make_frame(rng, 64, 6, 460, 1, 440, 0.03, 0.03, 0.01, dirichlet=True)
              for _ in range(2)]
    out = []
    for mib in (52, 0):
        b = mapdec.Batch(frames, flags=mapdec.MAPDEC_BATCH_GRAPH, mem_budget_bytes=mib << 20)
        assert mapdec.mapdec_batch_num_waves(b.b) == 1
        rx, pr = b.concat_inputs()
        st, app, ll = b.decode(rx, pr)
        assert st == 0
        out.append((app.copy(), ll.copy()))
        b.close()
    check_app(out[0][0], out[1][0])
    for x, y in zip(out[0][1], out[1][1]):
        check_ll(x, y)
