"""Face reduction, face coefficients and flux (GPU) at the edges of their tiles
and velocity splits: meshes of one tile and a row or column more or less than a
tile, velocity counts whose rows are whole, ragged or shorter than a chunk (the
joint and the separable Maxwellian), and many more splits than a velocity row
has chunks; one physical step with two inner iterations against the FP64
oracle, within the parity bounds of the step (1e-11 FP64, 1e-5 FP32 of the
largest value)."""
import os

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from oracle.run import Run  # noqa: E402
from paper_2604_09984_gb300 import ugks as U  # noqa: E402
from paper_2604_09984_gb300 import workloads as wl  # noqa: E402

SHAPES = [(16, 8, 16, True), (17, 9, 17, False), (15, 7, 33, True), (33, 3, 32, False), (2, 17, 21, True),
          (32, 16, 7, False)]


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    if not os.path.exists(U.LIB_PATH):
        import __graft_entry__
        __graft_entry__.build()
    U.load()


@pytest.mark.parametrize("prec", [U.FP64, U.FP32])
@pytest.mark.parametrize("ni,nj,nv,periodic", SHAPES)
def test_step_matches_oracle_at_face_edges(prec, ni, nj, nv, periodic):
    case = wl.channel(ni=ni, nj=nj, nv=nv, n_inner=2)
    if not periodic:
        b = case.blocks[0]
        b.periodic_i, b.bc, b.wall_T = False, (wl.BC_WALL, wl.BC_OUTFLOW, wl.BC_WALL, wl.BC_WALL), (1.0, 0.0, 1.1, 1.0)
    prim = wl.random_prim(case, 3, amp_rho=0.05, amp_u=0.05, amp_T=0.05)
    s = U.Solver(case, prec, prim=prim)
    ref = Run(case, prim=prim)
    s.advance()
    ref.step()
    tol = 1e-11 if prec == U.FP64 else 1e-5
    W = s.moments()[0]
    assert np.abs(W - ref.state.W).max() <= tol * np.abs(ref.state.W).max()
    f = s.get_state()[0].cpu().numpy()
    assert np.abs(f - ref.state.f).max() <= tol * np.abs(ref.state.f).max()
