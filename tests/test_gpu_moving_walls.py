"""Diffuse walls that slide in their own plane (GPU): a channel turned by 45
degrees, moving along its walls with (U, U).  At the velocities along a wall
(v_x = v_y, a diagonal of the velocity grid) w.S is zero up to its rounding, so
every kernel has to take the same side of the sign, and no value may come from
memory that nothing wrote: the workspace holds NaN bytes before the mesh is set.
One physical step with one inner iteration from a uniform state (interior faces
then have equal sides, whichever the rounding picks) against the FP64 oracle,
within the parity bounds of the step (1e-11 FP64, 1e-5 FP32 of the largest
value)."""
import os

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from oracle.run import Run  # noqa: E402
from paper_2604_09984_gb300 import ugks as U  # noqa: E402
from paper_2604_09984_gb300 import workloads as wl  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    if not os.path.exists(U.LIB_PATH):
        import __graft_entry__
        __graft_entry__.build()
    U.load()


def sliding_channel(ni, nj, nv, speed, dt):
    case = wl.channel(ni=ni, nj=nj, nv=nv, vmax=6.0, n_inner=1, noise=0.0)
    b = case.blocks[0]
    x, y = b.x_ref[..., 0].copy(), b.x_ref[..., 1].copy()
    b.x_ref = np.stack([x - y, x + y], axis=-1)
    b.wall_T = (0.0, 0.0, 1.2, 0.9)

    def motion(t):
        return np.array([[1.0, 0.0, 0.0, 1.0, speed * t, speed * t]])

    case.motion, case.dt = motion, dt
    return case


@pytest.mark.parametrize("prec", [U.FP64, U.FP32])
@pytest.mark.parametrize("ni,nj,nv,speed,dt", [(24, 8, 24, 0.2, 0.01), (24, 8, 24, 0.3, 0.02),
                                               (64, 8, 32, 0.3, 0.02), (17, 9, 13, 0.2, 1.0 / 64)])
def test_sliding_walls_match_oracle(monkeypatch, prec, ni, nj, nv, speed, dt):
    case = sliding_channel(ni, nj, nv, speed, dt)
    empty = torch.empty

    def nan_bytes(*a, **k):
        t = empty(*a, **k)
        return t.fill_(255) if t.dtype == torch.uint8 else t

    monkeypatch.setattr(torch, "empty", nan_bytes)
    s = U.Solver(case, prec)
    monkeypatch.undo()
    assert bool((s.ws[-16:] == 255).all())
    ref = Run(case)
    s.advance()
    ref.step()
    tol = 1e-11 if prec == U.FP64 else 1e-5
    W = s.moments()[0]
    f = s.get_state()[0].cpu().numpy()
    assert np.isfinite(f).all()
    assert np.abs(W - ref.state.W).max() <= tol * np.abs(ref.state.W).max()
    assert np.abs(f - ref.state.f).max() <= tol * np.abs(ref.state.f).max()
