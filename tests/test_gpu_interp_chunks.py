"""Receptor interpolation (GPU) at the edges of its velocity chunks: fewer
velocities than a chunk's first half, one chunk and a part of the next, two and a
part; one physical step of an overset pair against the FP64 oracle, within the
parity bounds of the step (1e-11 FP64, 1e-5 FP32 of the largest value)."""
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


@pytest.mark.parametrize("prec", [U.FP64, U.FP32])
@pytest.mark.parametrize("nv", [13, 23, 33])
def test_overset_step_matches_oracle(prec, nv):
    case = wl.mems(nbi=48, nbj=24, noi=32, noj=12, nv=nv, stretch=1.15, n_inner=2)
    prim = wl.random_prim(case, 13, amp_rho=0.05, amp_u=0.05, amp_T=0.05)
    s = U.Solver(case, prec, prim=prim)
    ref = Run(case, prim)
    s.advance()
    ref.step()
    tol = 1e-11 if prec == U.FP64 else 1e-5
    f, W, _ = s.get_state()
    f = f.cpu().numpy()
    field = ref.status == 0
    assert np.array_equal(s.moments()[2], ref.status)
    assert np.abs(W[field] - ref.state.W[field]).max() <= tol * np.abs(ref.state.W[field]).max()
    assert np.abs(f[field] - ref.state.f[field]).max() <= tol * np.abs(ref.state.f[field]).max()
