"""Macro LU-SGS sweep (GPU) at the edges of its launch shapes: rows around one
band, several bands, the limits of the four-lane and eight-band shapes and the
tallest ones, two to five columns, periodic rows (including two cells that
share two faces) and walls on all sides; one physical step with two inner
iterations against the FP64 oracle, within the parity bounds of the step
(1e-11 FP64, 1e-5 FP32 of the largest value)."""
import os

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from oracle.run import Run  # noqa: E402
from paper_2604_09984_gb300 import ugks as U  # noqa: E402
from paper_2604_09984_gb300 import workloads as wl  # noqa: E402

SHAPES = [(2, 2, True), (5, 31, False), (3, 33, True), (2, 65, False), (3, 128, True), (4, 129, False),
          (3, 257, True), (2, 300, False)]


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    if not os.path.exists(U.LIB_PATH):
        import __graft_entry__
        __graft_entry__.build()
    U.load()


@pytest.mark.parametrize("prec", [U.FP64, U.FP32])
@pytest.mark.parametrize("ni,nj,periodic", SHAPES)
def test_step_matches_oracle_at_sweep_edges(prec, ni, nj, periodic):
    case = wl.channel(ni=ni, nj=nj, nv=6, n_inner=2)
    if not periodic:
        b = case.blocks[0]
        b.periodic_i, b.bc, b.wall_T = False, (wl.BC_WALL,) * 4, (1.0, 1.1, 1.0, 1.0)
    prim = wl.random_prim(case, 5, amp_rho=0.05, amp_u=0.05, amp_T=0.05)
    s = U.Solver(case, prec, prim=prim)
    ref = Run(case, prim=prim)
    s.advance()
    ref.step()
    W, q, st, wall = s.moments()
    tol = 1e-11 if prec == U.FP64 else 1e-5
    assert np.abs(W - ref.state.W).max() <= tol * np.abs(ref.state.W).max()
    f = s.get_state()[0].cpu().numpy()
    assert np.abs(f - ref.state.f).max() <= tol * np.abs(ref.state.f).max()
