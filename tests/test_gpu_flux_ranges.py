"""Flux pass (GPU, FP32, velocity rows that are no multiple of 16): the form
that walks two ranges of columns in turn, which large arrays take, forced on small
meshes (UGKS_FLUX_PAIR); rows of one range, of an even and of an odd number of
ranges, with a whole and with a ragged last one, and more CTAs a tile than
velocity rows.  One physical step of two inner iterations: against the form of one
range after the other within 1e-6 of the largest value (each sum has the same terms
in the same order; the exponent -lam c^2, up to 18 here, may round by one more, 1e-6
of a Maxwellian that has fallen to e^-18 there), and against the FP64 oracle
within the parity bound of the step, 1e-5."""
import os

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from oracle.run import Run  # noqa: E402
from paper_2604_09984_gb300 import ugks as U  # noqa: E402
from paper_2604_09984_gb300 import workloads as wl  # noqa: E402

# cells, velocity columns and rows
SIZES = [(17, 9, 7, 7), (16, 8, 12, 13), (9, 17, 17, 17), (12, 10, 24, 18), (11, 9, 33, 33), (9, 7, 70, 6)]


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    if not os.path.exists(U.LIB_PATH):
        import __graft_entry__
        __graft_entry__.build()
    U.load()


@pytest.mark.parametrize("ni,nj,nvx,nvy", SIZES)
def test_ranges_in_turn_match(monkeypatch, ni, nj, nvx, nvy):
    case = wl.channel(ni=ni, nj=nj, nv=nvy, n_inner=2)
    case.nvx = nvx
    prim = wl.random_prim(case, 13, amp_rho=0.05, amp_u=0.05, amp_T=0.05)
    out = []
    for pair in ("0", "1"):
        monkeypatch.setenv("UGKS_FLUX_PAIR", pair)
        s = U.Solver(case, U.FP32, prim=prim)
        s.advance()
        out.append((s.get_state()[0].cpu().numpy(), s.moments()[0]))
    assert np.isfinite(out[0][0]).all()
    for a, b in zip(*out):
        assert np.abs(a - b).max() <= 1e-6 * np.abs(a).max()
    ref = Run(case, prim=prim)
    ref.step()
    for got, want in zip(out[1], (ref.state.f, ref.state.W)):
        assert np.abs(got - want).max() <= 1e-5 * np.abs(want).max()
