"""Kernels whose tables outgrow their memory (GPU): Step 7 in FP64 with more columns
and rows than its table of exponentials holds (256; one exponential a velocity
then), against the FP64 oracle within 1e-11 of the largest value, and the node
classification with more wall segments than its CTAs stage in shared memory (3072;
read from global memory then), whose connectivity equals the oracle's bit for
bit."""
import os

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from oracle import mesh, overset  # noqa: E402
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


@pytest.mark.parametrize("nvx,nvy", [(240, 16), (240, 17), (9, 250)])
def test_moments_of_long_velocity_rows(nvx, nvy):
    case = wl.channel(ni=5, nj=3, nv=nvy, n_inner=2)
    case.nvx = nvx
    prim = wl.random_prim(case, 19, amp_rho=0.05, amp_u=0.05, amp_T=0.05)
    s = U.Solver(case, U.FP64, prim=prim)
    ref = Run(case, prim=prim)
    s.advance()
    ref.step()
    W, q = s.moments()[:2]
    for got, want in ((s.get_state()[0].cpu().numpy(), ref.state.f), (W, ref.state.W), (q, ref.state.q)):
        assert np.abs(got - want).max() <= 1e-11 * np.abs(want).max()


def test_assembly_with_many_wall_segments():
    case = wl.mems(nbi=60, nbj=30, noi=2960, noj=12, nv=5, stretch=1.15, n_inner=1)
    assert 2960 + 2 * (60 + 30) > 48 * 1024 // 16
    s = U.Solver(case, U.FP64)
    topo = mesh.Topology(case.blocks)
    conn = overset.connect(topo, case.nodes_at(0.0))
    assert np.array_equal(s.connectivity()[0], conn.status)
    t = 0.1
    conn = overset.connect(topo, case.nodes_at(t), conn.status)
    s.move_mesh(t)
    s.overset_connect()
    st, dn, w = s.connectivity()
    assert np.array_equal(st, conn.status)
    assert np.array_equal(dn[conn.receptors], conn.donors)
    assert np.array_equal(w[conn.receptors].view(np.int64), conn.weights.view(np.int64))
