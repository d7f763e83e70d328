"""Overset assembly (GPU) bit for bit against the oracle (status, donor stencils,
IDW weights): fewer bins than one chunk of their scan and several chunks, O-grids
stretched towards the wall (a hundred candidate cells in a bin) and uniform
ones, two and three zones with bodies, at several positions of the bodies."""
import os

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from oracle import mesh, overset  # noqa: E402
from paper_2604_09984_gb300 import ugks as U  # noqa: E402
from paper_2604_09984_gb300 import workloads as wl  # noqa: E402

CASES = {
    "mems_768_bins": (lambda: wl.mems(nbi=48, nbj=24, noi=32, noj=12, nv=4, stretch=1.15, n_inner=1), 0.3),
    "mems_stretched": (lambda: wl.mems(nbi=72, nbj=36, noi=64, noj=24, nv=4, stretch=1.25, n_inner=1), 0.3),
    "mems_3000_bins": (lambda: wl.mems(nbi=96, nbj=48, noi=64, noj=20, nv=4, stretch=1.05, n_inner=1), 0.3),
    "three_zones": (lambda: wl.tsto(nbi=80, nbj=40, noi=24, noj=10, nv=4, n_inner=1), 0.02),
}


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    if not os.path.exists(U.LIB_PATH):
        import __graft_entry__
        __graft_entry__.build()
    U.load()


@pytest.mark.parametrize("name", sorted(CASES))
def test_assembly_matches_oracle_bit_for_bit(name):
    make, step = CASES[name]
    case = make()
    s = U.Solver(case, U.FP64)
    topo = mesh.Topology(case.blocks)
    conn = overset.connect(topo, case.nodes_at(0.0))
    assert np.array_equal(s.connectivity()[0], conn.status)
    for n in range(1, 4):
        prev = conn.status
        t = n * (step / case.meta["freq"] if "freq" in case.meta else step)
        s.move_mesh(t)
        conn = overset.connect(topo, case.nodes_at(t), prev)
        if conn.n_orphan:
            with pytest.raises(U.UgksError):
                s.overset_connect()
            break
        stats = s.overset_connect()
        st, dn, w = s.connectivity()
        assert np.array_equal(st, conn.status)
        assert np.array_equal(dn[conn.receptors], conn.donors)
        assert np.array_equal(w[conn.receptors].view(np.int64), conn.weights.view(np.int64))
        assert stats["n_fresh"] == conn.fresh.size
