"""ugks_idw_interpolate_static with many velocities and few receptors (GPU): the
same sums as on the host on both sides of the line between its two forms (8192
velocities), within 1e-14 of the largest value (five products), and a call whose
time follows the values it moves: 262,000 velocities of one receptor against
about as many values as 500 receptors of 511 velocities.  The second call takes
some 10 us on the device, the first 18; a form whose CTAs take four velocities
each took 172, so the bound of six times leaves three on either side."""
import ctypes
import os

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from paper_2604_09984_gb300 import ugks as U  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    if not os.path.exists(U.LIB_PATH):
        import __graft_entry__
        __graft_entry__.build()
    U.load()


def _p(t):
    return ctypes.c_void_p(t.data_ptr())


def _inputs(nc, nv, nrec):
    rng = np.random.default_rng(nv + nrec)
    a = [rng.standard_normal(s) for s in ((nc, nv, 2), (nc, 4), (nc, 2))]
    rec = rng.permutation(nc)[:nrec].astype(np.int32)
    dn = rng.integers(0, nc, (nrec, 5)).astype(np.int32)
    w = rng.random((nrec, 5))
    dev = torch.device("cuda")
    return a, rec, dn, w, [torch.as_tensor(x, device=dev) for x in (*a, rec, dn, w)]


def _call(t, nc, nv, nrec):
    return U.load().ugks_idw_interpolate_static(_p(t[0]), _p(t[1]), _p(t[2]), nc, nv, _p(t[3]), nrec, _p(t[4]), _p(t[5]),
                                                ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))


@pytest.mark.parametrize("nc,nv,nrec", [(90, 8191, 31), (90, 8192, 31), (90, 8193, 31), (12, 60001, 4), (7, 262000, 1)])
def test_many_velocities_match_host_sums(nc, nv, nrec):
    a, rec, dn, w, t = _inputs(nc, nv, nrec)
    assert _call(t, nc, nv, nrec) == U.OK
    torch.cuda.synchronize()
    for got, x in zip(t, a):
        ref = x.copy()
        ref[rec] = np.einsum("rm,rm...->r...", w, x[dn])
        assert np.abs(got.cpu().numpy() - ref).max() <= 1e-14 * np.abs(ref).max()


def test_time_follows_the_values_moved():
    def device_time(nc, nv, nrec):
        t = _inputs(nc, nv, nrec)[-1]
        e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
        best = 1e30
        for _ in range(6):
            e[0].record()
            for _ in range(50):
                assert _call(t, nc, nv, nrec) == U.OK
            e[1].record()
            e[1].synchronize()
            best = min(best, e[0].elapsed_time(e[1]))
        return best
    assert device_time(7, 262000, 1) < 6.0 * device_time(1200, 511, 500)
