"""ugks_idw_interpolate_static at the edges of its two forms: velocity counts
that fill no chunk of a CTA or one value more, the most receptors whose values
fit in a CTA's shared memory and one more (two passes through the scratch),
receptors that are each other's donors, arrays off a 16-byte
boundary, orphan rows, donors outside the mesh,
with and without W and q; against the sums on the host within 1e-14 of the
largest value (five products and, where weights are renormalised, a division:
some ten roundings of 1.1e-16)."""
import ctypes
import os

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from paper_2604_09984_gb300 import ugks as U  # noqa: E402

SIZES = [(50, 1, 1), (50, 3, 40), (60, 2, 33), (700, 511, 100), (700, 512, 100), (2000, 515, 300), (700, 513, 507),
         (3000, 144, 512), (3000, 144, 513)]


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    if not os.path.exists(U.LIB_PATH):
        import __graft_entry__
        __graft_entry__.build()
    U.load()


def _p(t):
    return ctypes.c_void_p(t.data_ptr()) if t is not None else None


@pytest.mark.parametrize("aligned", [True, False])
@pytest.mark.parametrize("moments", [True, False])
@pytest.mark.parametrize("nc,nv,nrec", SIZES)
def test_interpolation_matches_host_sums(nc, nv, nrec, moments, aligned):
    rng = np.random.default_rng(nc + nv + nrec)
    f, W, q = rng.standard_normal((nc, nv, 2)), rng.standard_normal((nc, 4)), rng.standard_normal((nc, 2))
    rec = rng.permutation(nc)[:nrec].astype(np.int32)
    dn = rng.integers(-1, nc + 2, (nrec, 5)).astype(np.int32)      # -1 unused, nc and nc + 1 outside
    dn[rng.random(nrec) < 0.05, 0] = -1                            # orphans
    w = rng.random((nrec, 5))
    valid = (dn >= 0) & (dn < nc)
    wv = np.where(valid, w, 0.0)
    tot = wv.sum(1)
    bad = ((dn != -1) & ~valid).any(1) & (tot != 0)
    wv[bad] /= tot[bad, None]
    ids = np.where(valid, dn, 0)
    do = (dn[:, 0] >= 0) & (tot != 0)
    ref = [a.copy() for a in (f, W, q)]
    for r, a in zip(ref, (f, W, q)):
        r[rec[do]] = np.einsum("rm,rm...->r...", wv, a[ids])[do]
    dev = torch.device("cuda")
    t = []
    for a in (f, W, q):      # on a 16-byte boundary, or 8 bytes past one
        buf = torch.empty(a.size + 2, dtype=torch.float64, device=dev)
        v = buf[0 if aligned else 1:][:a.size].view(a.shape)
        t.append(v.copy_(torch.as_tensor(a)))
    args = [torch.as_tensor(a, device=dev) for a in (rec, dn, w)]
    r = U.load().ugks_idw_interpolate_static(_p(t[0]), _p(t[1] if moments else None), _p(t[2] if moments else None),
                                             nc, nv, _p(args[0]), nrec, _p(args[1]), _p(args[2]),
                                             ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert r == U.OK
    torch.cuda.synchronize()
    if not moments:
        ref[1:] = W, q
    for got, want in zip(t, ref):
        assert np.abs(got.cpu().numpy() - want).max() <= 1e-14 * np.abs(want).max()
