"""Micro LU-SGS sweeps (GPU) at the edges of their launch shapes: one band, a
row less and a row more than a band, the limits of the shapes of one, two and
four rows a group and the tallest one, two and three columns (fewer than the
groups of a warp), periodic rows and walls on all sides, velocity counts that
fill no lane, group or padding; one physical step with two inner iterations
against the FP64 oracle, within the parity bounds of the step (1e-11 FP64,
1e-5 FP32, 2e-2 with f stored in bf16, of the largest value)."""
import os

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from oracle.run import Run  # noqa: E402
from paper_2604_09984_gb300 import ugks as U  # noqa: E402
from paper_2604_09984_gb300 import workloads as wl  # noqa: E402

SHAPES = [(2, 3, 5, True), (3, 8, 7, True), (9, 9, 5, False), (17, 15, 5, True), (3, 17, 5, False), (2, 128, 5, True),
          (3, 129, 5, False), (2, 256, 5, False), (3, 257, 5, True), (2, 510, 5, False)]


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    if not os.path.exists(U.LIB_PATH):
        import __graft_entry__
        __graft_entry__.build()
    U.load()


@pytest.mark.parametrize("prec", [U.FP64, U.FP32, U.BF16F])
@pytest.mark.parametrize("ni,nj,nv,periodic", SHAPES)
def test_step_matches_oracle_at_sweep_edges(prec, ni, nj, nv, periodic):
    case = wl.channel(ni=ni, nj=nj, nv=nv, n_inner=2)
    if not periodic:
        b = case.blocks[0]
        b.periodic_i, b.bc, b.wall_T = False, (wl.BC_WALL,) * 4, (1.0, 1.1, 1.0, 1.0)
    prim = wl.random_prim(case, 7, amp_rho=0.05, amp_u=0.05, amp_T=0.05)
    s = U.Solver(case, prec, prim=prim)
    ref = Run(case, prim=prim)
    s.advance()
    ref.step()
    tol = {U.FP64: 1e-11, U.FP32: 1e-5, U.BF16F: 2e-2}[prec]
    W = s.moments()[0]
    assert np.abs(W - ref.state.W).max() <= tol * np.abs(ref.state.W).max()
    f = s.get_state()[0].cpu().numpy()
    assert np.abs(f - ref.state.f).max() <= tol * np.abs(ref.state.f).max()
