"""Micro residual (GPU, FP32 paths): one pass (UGKS_RESIDUAL_ONE_PASS=1, the form of
large velocity grids and of batches) and two (the form of these small meshes) form
it with the same operations in the same order, so the state after a step is the
same, bit for bit; velocity counts that are odd, fill a CTA's share or leave a
ragged one, a single block and overset blocks, with and without the first
iteration's level-n term alone.  The switch shows in the launches: one less an
iteration."""
import os

import numpy as np
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


CASES = {
    "odd": lambda n: wl.channel(ni=9, nj=7, nv=7, n_inner=n),
    "share": lambda n: wl.channel(ni=12, nj=8, nv=32, n_inner=n),
    "ragged": lambda n: wl.channel(ni=6, nj=5, nv=23, n_inner=n),
    "overset": lambda n: wl.mems(nbi=48, nbj=24, noi=32, noj=12, nv=8, stretch=1.15, n_inner=n),
}


@pytest.mark.parametrize("prec", [U.FP32, U.BF16F])
@pytest.mark.parametrize("n_inner", [1, 3])
@pytest.mark.parametrize("name", sorted(CASES))
def test_one_pass_equals_two(monkeypatch, name, n_inner, prec):
    case = CASES[name](n_inner)
    prim = wl.random_prim(case, 11, amp_rho=0.05, amp_u=0.05, amp_T=0.05)
    out = []
    for one in (False, True):
        if one:
            monkeypatch.setenv("UGKS_RESIDUAL_ONE_PASS", "1")
        else:
            monkeypatch.delenv("UGKS_RESIDUAL_ONE_PASS", raising=False)
        s = U.Solver(case, prec, prim=prim)
        s.set_graphs(False)
        n0 = s.launch_count()
        s.advance()
        n1 = s.launch_count()
        W, q = s.moments()[:2]
        out.append((n1 - n0, s.get_state()[0].cpu().numpy(), W, q))
    assert out[0][0] - out[1][0] == n_inner
    assert np.isfinite(out[0][1]).all()
    for a, b in zip(out[0][1:], out[1][1:]):
        assert np.array_equal(a, b)
