"""Micro sweeps (GPU): the shapes a large workload takes (whole lines of a cell a
warp, bands of 8, 16 and 32 rows), each forced on a small one at the edges of its
bands and velocity groups.  The order of every sum is the sweep's own, so the
state after a step equals the default shape's bit for bit (FP32), and bf16
storage of f likewise."""
import os

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from paper_2604_09984_gb300 import ugks as U  # noqa: E402
from paper_2604_09984_gb300 import workloads as wl  # noqa: E402

SHAPES = [(2, 3, 5, True), (5, 8, 7, True), (3, 9, 5, False), (17, 17, 6, True), (9, 33, 5, False), (3, 128, 5, True),
          (2, 250, 5, False)]


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    if not os.path.exists(U.LIB_PATH):
        import __graft_entry__
        __graft_entry__.build()
    U.load()


def _state(ni, nj, nv, periodic, prec):
    case = wl.channel(ni=ni, nj=nj, nv=nv, n_inner=2)
    if not periodic:
        b = case.blocks[0]
        b.periodic_i, b.bc, b.wall_T = False, (wl.BC_WALL,) * 4, (1.0, 1.1, 1.0, 1.0)
    s = U.Solver(case, prec, prim=wl.random_prim(case, 7, amp_rho=0.05, amp_u=0.05, amp_T=0.05))
    s.advance()
    f, W, q = s.get_state()
    return f.cpu().numpy(), np.asarray(W), np.asarray(q)


@pytest.mark.parametrize("prec", [U.FP32, U.BF16F])
@pytest.mark.parametrize("ni,nj,nv,periodic", SHAPES)
def test_every_shape_gives_the_same_bits(monkeypatch, prec, ni, nj, nv, periodic):
    monkeypatch.delenv("UGKS_SWEEP_SHAPE", raising=False)
    ref = _state(ni, nj, nv, periodic, prec)
    assert np.isfinite(ref[0]).all()
    for shape in range(6):
        monkeypatch.setenv("UGKS_SWEEP_SHAPE", str(shape))
        got = _state(ni, nj, nv, periodic, prec)
        for a, b in zip(got, ref):
            assert np.array_equal(a, b), shape
