"""ugks_eval_flux writes D wherever FP64 values may lie (GPU): into a buffer on a
16-byte boundary and into one 8 bytes past it, the same bits, and nothing beyond
its ends; odd and even velocity counts, the separable (16 columns) and the joint
Maxwellian, a velocity grid with a ragged last chunk."""
import ctypes
import os

import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

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


@pytest.mark.parametrize("prec", [U.FP32, U.BF16F, U.FP64])
@pytest.mark.parametrize("ni,nj,nv", [(9, 7, 5), (16, 8, 16), (11, 9, 18)])
def test_flux_divergence_into_any_buffer(prec, ni, nj, nv):
    case = wl.channel(ni=ni, nj=nj, nv=nv)
    s = U.Solver(case, prec, prim=wl.random_prim(case, 5, amp_rho=0.05, amp_u=0.05, amp_T=0.05))
    s.move_mesh(case.dt)
    n = 2 * s.nc * s.nv
    got = []
    for off in (0, 1):
        buf = torch.full((n + 4,), 7.0, dtype=torch.float64, device=s.device)
        D = buf[off:off + n]
        assert D.data_ptr() % 16 == 8 * off
        r = s.lib.ugks_eval_flux(s.ctx, ctypes.c_void_p(D.data_ptr()), None)
        assert r == U.OK
        assert bool((buf[:off] == 7.0).all()) and bool((buf[off + n:] == 7.0).all())
        got.append(D.clone())
    assert bool(got[0].abs().max() > 0.0)
    assert torch.equal(got[0], got[1])
