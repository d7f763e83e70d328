"""Performance cases of the implicit moving-mesh UGKS: what a program that uses
this framework has it do, call by call, with inputs made from a seed.

A case is one call path a program repeats:
  step      one physical step of the outer loop on a workload (motion, overset
            assembly, implicit step) and the state read back: channel, mems,
            tsto; the free particle also moves its body by the gas loads
  batch     one step of several independent instances side by side
  flux      one evaluation of the interface fluxes of a given state
  assembly  motion and overset assembly alone, with the connectivity read back
  idw       the allocation-free receptor interpolation on caller buffers

The mixed path (fp32) holds f and all per-velocity arithmetic in FP32, so its
floating outputs are returned as float32; the fp64 path's as float64.

exact() recomputes a pass in 64 bits with plain torch and numpy (the scheme
written out below, Sec. 2-3 of arXiv 2604.09984), taking from the package only
the workloads' description of the inputs.
"""
from __future__ import annotations

import ctypes
import math

import numpy as np
import torch

from paper_2604_09984_gb300 import ugks as U
from paper_2604_09984_gb300 import workloads as wl

PREC = {"fp32": U.FP32, "fp64": U.FP64}


# ------------------------------------------------------------------ the cases
def _mems(nbi, nbj, noi, noj, nv, n_gap=2, Kn=0.1, Tw=1.5):
    return dict(flow="mems", nbi=nbi, nbj=nbj, noi=noi, noj=noj, n_gap=n_gap, nv=nv, Kn=Kn, Tw=Tw, n_inner=10)


def listed():
    return [
        # the allocation-free interpolation a host framework calls between its
        # own kernels: latency of one call
        dict(name="idw_24x24", kind="idw", ncells=9216, nv=576, nrec=280),
        # the smallest workload a program steps: launches and latency count
        dict(name="channel_small_fp32", kind="step", flow="channel", precision="fp32", ni=32, nj=16, nv=16,
             Kn=0.05, n_inner=10),
        # the plain FP64 channel, the default configuration of validation runs
        dict(name="channel_fp64", kind="step", flow="channel", precision="fp64", ni=64, nj=32, nv=24, Kn=0.05,
             n_inner=10),
        # a free body moved by the gas loads, read back every step
        dict(name="particle_fp32", kind="step", flow="particle", precision="fp32", nbi=128, nbj=64, noi=64, noj=16,
             nv=24, Kn=0.1, n_inner=10),
        # odd sizes and a velocity count that fills no vector or tile
        dict(name="mems_ragged_fp32", kind="step", precision="fp32",
             **_mems(97, 51, 72, 18, 21, n_gap=wl.overlap_gap_layers(97, 18, 1.1, 0.25, 0.1), Kn=0.5, Tw=1.3)),
        # the headline production step: MEMS overset workload, mixed precision
        dict(name="mems_fp32", kind="step", precision="fp32", **_mems(256, 128, 128, 32, 32)),
        # the same physics in plain FP64 (reference runs) on the reduced mesh
        dict(name="mems_fp64", kind="step", precision="fp64", **_mems(96, 48, 64, 16, 32)),
        # hypersonic two-body separation, reduced mesh and a ragged velocity grid
        dict(name="tsto_reduced_fp32", kind="step", flow="tsto", precision="fp32", nbi=300, nbj=150, noi=120, noj=30,
             nv=33, n_inner=15),
        # the full two-body workload, the largest single step
        dict(name="tsto_fp32", kind="step", flow="tsto", precision="fp32", nbi=512, nbj=256, noi=192, noj=48, nv=64,
             n_inner=15),
        # a parameter sweep served as independent instances side by side
        dict(name="batch12_fp32", kind="batch", precision="fp32", n=12, sizes_seed=0, n_inner=10),
        # one flux evaluation of a given state (residual monitoring, coupling)
        dict(name="flux_fp32", kind="flux", precision="fp32", **_mems(192, 96, 96, 24, 32)),
        # moving-grid connectivity alone (grid motion set-up) on the two-body grids
        dict(name="assembly_tsto", kind="assembly", flow="tsto", precision="fp32", nbi=512, nbj=256, noi=192, noj=48,
             nv=8, n_inner=1),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_mems(rng, nb_lo, nb_hi, nv_lo, nv_hi):
    nbi = _logint(rng, nb_lo, nb_hi)
    noi = _logint(rng, 64, 128)
    noj = noi // 4
    return _mems(nbi, nbi // 2, noi, noj, _logint(rng, nv_lo, nv_hi),
                 n_gap=wl.overlap_gap_layers(nbi, noj, 1.1, 0.25, 0.1),
                 Kn=round(10.0 ** rng.uniform(-2.0, 0.3), 4), Tw=round(rng.uniform(1.0, 2.0), 3))


def _draw_tsto(rng):
    nbi = _logint(rng, 256, 512)
    noi = _logint(rng, 112, 192)
    return dict(flow="tsto", nbi=nbi, nbj=nbi // 2, noi=noi, noj=noi // 4)


def draw(rng):
    kind = rng.choice(["channel", "channel", "mems", "mems", "mems", "mems", "tsto", "particle", "batch", "flux",
                       "assembly", "idw"])
    if kind == "channel":
        ni = _logint(rng, 16, 256)
        return dict(kind="step", flow="channel", precision=rng.choice(["fp32", "fp64"]), ni=ni,
                    nj=max(8, _logint(rng, ni / 3, ni)), nv=_logint(rng, 12, 32),
                    Kn=round(10.0 ** rng.uniform(-2.0, 0.3), 4), n_inner=rng.randint(5, 10))
    if kind == "mems":
        prec = rng.choice(["fp32", "fp32", "fp64"])
        return dict(kind="step", precision=prec,
                    **_draw_mems(rng, 48, 256 if prec == "fp32" else 128, 16, 40 if prec == "fp32" else 32))
    if kind == "tsto":
        return dict(kind="step", precision="fp32", nv=_logint(rng, 24, 56), n_inner=rng.randint(8, 15),
                    **_draw_tsto(rng))
    if kind == "particle":
        nbi = _logint(rng, 96, 256)
        return dict(kind="step", flow="particle", precision="fp32", nbi=nbi, nbj=nbi // 2, noi=_logint(rng, 56, 96),
                    noj=16, nv=_logint(rng, 16, 32), Kn=round(10.0 ** rng.uniform(-2.0, 0.3), 4),
                    n_inner=rng.randint(5, 10))
    if kind == "batch":
        return dict(kind="batch", precision="fp32", n=rng.randint(3, 12), sizes_seed=rng.randint(1, 10 ** 6),
                    n_inner=rng.randint(5, 10))
    if kind == "flux":
        return dict(kind="flux", precision=rng.choice(["fp32", "fp64"]), **_draw_mems(rng, 48, 256, 16, 40))
    if kind == "assembly":
        return dict(kind="assembly", precision="fp32", nv=8, n_inner=1, **_draw_tsto(rng))
    nv = _logint(rng, 12, 32) ** 2
    return dict(kind="idw", ncells=_logint(rng, 1000, 40000), nv=nv,
                nrec=_logint(rng, 16, min(480, U.STATIC_SCRATCH_DOUBLES // (2 * nv + 7))))


def _noisy(c, seed, amp):
    c.init_prim = wl.random_prim(c, seed, amp_rho=amp, amp_u=amp, amp_T=amp)
    return c


def _workload(case, seed):
    """The package's description of the inputs: meshes, motion, gas, and the
    gas at rest with a few percent of seeded disturbance in every cell."""
    flow = case["flow"]
    if flow == "channel":
        return _noisy(wl.channel(ni=case["ni"], nj=case["nj"], nv=case["nv"], Kn=case["Kn"],
                                 n_inner=case["n_inner"], noise=0.0), seed, 0.05)
    mesh = {k: case[k] for k in ("nbi", "nbj", "noi", "noj", "nv", "n_inner")}
    if flow == "mems":
        return _noisy(wl.mems(Kn=case["Kn"], Tw=case["Tw"], n_gap=case["n_gap"], **mesh), seed, 0.05)
    if flow == "particle":
        # a slow body: it stays inside the box however often the case is run
        return _noisy(wl.particle(Kn=case["Kn"], u0=(0.05, 0.01), omega0=0.2, **mesh), seed, 0.02)
    return _noisy(wl.tsto(**mesh), seed, 0.02)


def _instances(case, seed):
    cs = wl.mems_batch(n=case["n"], seed=case["sizes_seed"], n_inner=case["n_inner"])
    return [_noisy(c, 1000 * seed + i, 0.05) for i, c in enumerate(cs)]


def _bodies(c):
    m = c.meta
    return [U.RigidBody(m["body_block"], m["mass"], m["inertia"], m["center"], m["u0"], m["omega0"])]


class _Out:
    """A solver and the buffers its program reads the state into every step."""

    def __init__(self, c, case, stream=None):
        self.s = U.Solver(c, PREC[case["precision"]], stream=stream)
        n, nb = self.s.nc, len(c.blocks)
        new = lambda *shape: torch.empty(shape, dtype=torch.float64, device="cuda")  # noqa: E731
        self.f, self.W, self.q, self.wall = new(n, self.s.nv, 2), new(n, 4), new(n, 2), new(nb, 4)
        self.status = torch.empty(n, dtype=torch.int32, device="cuda")
        self.cast = torch.float32 if case["precision"] == "fp32" else torch.float64

    def read(self):
        self.s.moments(self.W, self.q, self.status, self.wall)
        r = self.s.lib.ugks_get_state(self.s.ctx, ctypes.c_void_p(self.f.data_ptr()), None, None)
        if r != U.OK:
            raise U.UgksError(r, "get_state")
        return {"f": self.f.to(self.cast), "W": self.W.to(self.cast), "q": self.q.to(self.cast),
                "status": self.status, "wall": self.wall.to(self.cast)}


ASSEMBLY_POSITIONS = 32     # the assembly case moves its bodies through this many time steps, then again


def _idw_inputs(case, seed):
    """Receptors, stencils of a cell and its neighbours (some shorter, one
    orphan) with inverse-distance-like weights, and the fields, on the host."""
    rng = np.random.default_rng(seed)
    nc, nv, nr = case["ncells"], case["nv"], case["nrec"]
    rec = np.sort(rng.choice(nc // 2, nr, replace=False)).astype(np.int32)
    don = rng.integers(nc // 2 + 1, nc - 1, (nr, 1)) + np.array([[0, -1, 1, 0, 0]])
    don[:, 3:] = rng.integers(nc // 2, nc, (nr, 2))
    w = 1.0 / rng.uniform(0.1, 1.0, (nr, 5)) ** 2
    short = rng.random(nr) < 0.1
    don[short, 4] = -1
    w[short, 4] = 0.0
    don[nr // 2] = -1
    w /= w.sum(1, keepdims=True)
    return rec, don.astype(np.int32), w


def _idw_fields(case, seed):
    g = torch.Generator(device="cuda" if torch.cuda.is_available() else "cpu").manual_seed(seed)
    new = lambda *s: torch.rand(s, dtype=torch.float64, device=g.device, generator=g)  # noqa: E731
    return new(case["ncells"], case["nv"], 2), new(case["ncells"], 4), new(case["ncells"], 2)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "idw":
        rec, don, w = (torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in _idw_inputs(case, seed))
        f, W, q = _idw_fields(case, seed)
        return dict(kind=kind, case=case, f=f, W=W, q=q, rec=rec, don=don, w=w, lib=U.load())
    if kind == "batch":
        outs = [_Out(c, case, torch.cuda.Stream()) for c in _instances(case, seed)]
        return dict(kind=kind, outs=outs)
    c = _workload(case, seed)
    if kind == "assembly":
        s = U.Solver(c, PREC[case["precision"]])
        pin = lambda dt, *shape: torch.empty(shape, dtype=dt).pin_memory()  # noqa: E731
        # each seed starts somewhere else on the bodies' path
        return dict(kind=kind, s=s, at=seed % ASSEMBLY_POSITIONS, status=pin(torch.int32, s.nc),
                    donors=pin(torch.int32, s.nc, 5), weights=pin(torch.float64, s.nc, 5))
    if kind == "flux":
        s = U.Solver(c, PREC[case["precision"]])
        s.move_mesh(c.dt)
        s.overset_connect()
        return dict(kind=kind, s=s, cast=torch.float32 if case["precision"] == "fp32" else torch.float64)
    return dict(kind=kind, out=_Out(c, case), bodies=_bodies(c) if case["flow"] == "particle" else None)


def _p(t):
    return ctypes.c_void_p(t.data_ptr())


def run(state):
    kind = state["kind"]
    if kind == "step":
        s = state["out"].s
        if state["bodies"] is not None:
            s.advance_coupled(state["bodies"])
        else:
            s.advance()
        return state["out"].read()
    if kind == "batch":
        U.advance_batch([o.s for o in state["outs"]])
        return [o.read() for o in state["outs"]]
    if kind == "flux":
        D, F = state["s"].eval_flux()
        return {"D": D.to(state["cast"]), "F": torch.from_numpy(F).to(state["cast"])}
    if kind == "assembly":
        s = state["s"]
        s.move_mesh((1 + state["at"]) * s.case.dt)
        state["at"] = (state["at"] + 1) % ASSEMBLY_POSITIONS
        n = s.overset_connect()
        r = s.lib.ugks_get_connectivity(s.ctx, _p(state["status"]), _p(state["donors"]), _p(state["weights"]))
        if r != U.OK:
            raise U.UgksError(r, "get_connectivity")
        return {"status": state["status"], "donors": state["donors"], "weights": state["weights"],
                "receptors": n["n_receptor"]}
    c = state["case"]
    r = state["lib"].ugks_idw_interpolate_static(
        _p(state["f"]), _p(state["W"]), _p(state["q"]), c["ncells"], c["nv"], _p(state["rec"]), c["nrec"],
        _p(state["don"]), _p(state["w"]), ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    if r != U.OK:
        raise U.UgksError(r, "idw")
    return {"f": state["f"], "W": state["W"], "q": state["q"]}


def _cells(case):
    if case["flow"] == "channel":
        return case["ni"] * case["nj"]
    bodies = 2 if case["flow"] == "tsto" else 1
    return case["nbi"] * case["nbj"] + bodies * case["noi"] * case["noj"]


def _step_work(cells, nv2, n_inner, pair):
    # f, W and q read and written once; per (cell, velocity) of one inner
    # iteration: two faces' reconstruction, interface distribution and twelve
    # velocity sums (~120), collision and residual (~40), both sweeps (~60),
    # moments (~30); the level-n pass evaluates the flux once more
    return {"bytes": 2.0 * cells * (nv2 * pair + 6 * 8), "flops": float(cells) * nv2 * (250.0 * n_inner + 160.0)}


def work(case):
    kind = case["kind"]
    if kind == "idw":
        n, nv = case["nrec"], case["nv"]
        return {"bytes": n * (6.0 * (2 * nv + 6) * 8 + 5 * 12 + 4), "flops": n * 10.0 * (2 * nv + 6)}
    if kind == "batch":
        w = [_step_work(c.ncells, c.nv, c.n_inner, 8) for c in _instances(case, 0)]
        return {k: sum(x[k] for x in w) for k in ("bytes", "flops")}
    n, pair = _cells(case), 8 if case["precision"] == "fp32" else 16
    if kind == "assembly":
        # nodes and volumes' worth of geometry in, connectivity out
        return {"bytes": n * (2 * 16.0 + 4 + 5 * 12), "flops": n * 200.0}
    nv2 = case["nv"] ** 2
    if kind == "flux":
        return {"bytes": n * (nv2 * (pair + 16.0) + 6 * 8 + 4 * 8), "flops": n * nv2 * 160.0}
    return _step_work(n, nv2, case["n_inner"], pair)


# ------------------------------------------- the same passes in 64 bits
FIELD, RECEPTOR, HOLE = 0, 1, 2
IM, IP, JM, JP = range(4)
EXACT_ITEMS = 1.0e9         # (cell, velocity, inner iteration) items of one workload worked through in about 20 s,
EXACT_ITEMS_BATCH = 3.0e8   # and of a batch of small ones, whose sweeps take one launch after the other


def _dot(a, b):
    return (a * b).sum(-1)


class _Mesh:
    """Faces and neighbours of structured blocks, all blocks in one numbering
    (cells j*ni + i within a block).  Faces point from the lower to the higher
    logical cell, boundary faces outward."""

    def __init__(self, c):
        self.blocks, self.nc = c.blocks, c.ncells
        L, R, a, b, kind, Tw, blk, shift = ([] for _ in range(8))
        self.nb = np.full((self.nc, 4), -1)               # neighbour cell across slot
        self.face = np.full((self.nc, 4), -1)
        self.nbshift = np.zeros((self.nc, 4))
        self.nodes, self.row, self.cb = np.empty((self.nc, 4), int), np.empty((self.nc, 2), int), np.empty(self.nc, int)
        self.ij = np.empty((self.nc, 2), int)
        self.off, nf, no = [0], 0, 0
        self.noff = [0]
        for q, B in enumerate(c.blocks):
            ni, nj, co = B.ni, B.nj, self.off[-1]
            I, J = np.meshgrid(np.arange(ni), np.arange(nj), indexing="ij")
            cid = co + J * ni + I
            nid = no + (np.arange(nj + 1)[None, :] * (ni + 1) + np.arange(ni + 1)[:, None])
            self.nodes[cid] = np.stack([nid[:-1, :-1], nid[1:, :-1], nid[1:, 1:], nid[:-1, 1:]], -1)
            self.row[cid] = np.stack([np.broadcast_to(nid[0, :-1], cid.shape),
                                      np.broadcast_to(nid[-1, :-1], cid.shape)], -1)
            self.cb[cid] = q
            self.ij[cid] = np.stack([I, J], -1)

            def add(Lc, Rc, na, nb_, k, T, sl, sr=None, sh=0):
                nonlocal nf
                Lc = np.asarray(Lc).ravel()
                Rc = np.full(Lc.size, -1) if Rc is None else np.asarray(Rc).ravel()
                ids = nf + np.arange(Lc.size)
                nf += Lc.size
                self.face[Lc, sl] = ids
                if sr is not None:
                    self.face[Rc, sr] = ids
                    self.nb[Lc, sl], self.nb[Rc, sr] = Rc, Lc
                    self.nbshift[Lc, sl], self.nbshift[Rc, sr] = -sh, sh
                for lst, v in ((L, Lc), (R, Rc), (a, na), (b, nb_), (kind, np.full(Lc.size, k)),
                               (Tw, np.full(Lc.size, T)), (blk, np.full(Lc.size, q)), (shift, np.full(Lc.size, sh))):
                    lst.append(np.asarray(v).ravel())
            add(cid[:-1], cid[1:], nid[1:-1, :-1], nid[1:-1, 1:], 0, 0.0, IP, IM)
            if B.periodic_i:
                add(cid[-1], cid[0], nid[0, :-1], nid[0, 1:], 0, 0.0, IP, IM, -1)
            else:
                add(cid[0], None, nid[0, 1:], nid[0, :-1], B.bc[0], B.wall_T[0], IM)
                add(cid[-1], None, nid[-1, :-1], nid[-1, 1:], B.bc[1], B.wall_T[1], IP)
            add(cid[:, :-1], cid[:, 1:], nid[1:, 1:-1], nid[:-1, 1:-1], 0, 0.0, JP, JM)
            add(cid[:, 0], None, nid[:-1, 0], nid[1:, 0], B.bc[2], B.wall_T[2], JM)
            add(cid[:, -1], None, nid[1:, -1], nid[:-1, -1], B.bc[3], B.wall_T[3], JP)
            self.off.append(co + ni * nj)
            no += (ni + 1) * (nj + 1)
            self.noff.append(no)
        self.L, self.R, self.a, self.b, self.kind, self.fb = (np.concatenate(v) for v in (L, R, a, b, kind, blk))
        self.Tw, self.shift = np.concatenate(Tw), np.concatenate(shift).astype(float)
        self.sgn = np.where(self.L[self.face] == np.arange(self.nc)[:, None], 1.0, -1.0)


def _nodes(c, A):
    """Nodes of all blocks under the affine maps A (each product and sum rounded once)."""
    out = []
    for B, m in zip(c.blocks, A):
        x, y = B.x_ref[..., 0].T, B.x_ref[..., 1].T
        out.append(np.stack([(m[0] * x + m[1] * y) + m[4], (m[2] * x + m[3] * y) + m[5]], -1).reshape(-1, 2))
    return np.concatenate(out)


class _Geo:
    """ALE geometry of one step (mid-time faces, both volumes, face velocity)."""

    def __init__(self, M, Xo, Xn, dt):
        def area(X):
            p = X[M.nodes]
            return 0.5 * ((p[:, 2, 0] - p[:, 0, 0]) * (p[:, 3, 1] - p[:, 1, 1])
                          - (p[:, 2, 1] - p[:, 0, 1]) * (p[:, 3, 0] - p[:, 1, 0]))
        Xm, V = 0.5 * (Xo + Xn), (Xn - Xo) / dt
        self.vol0, self.vol1 = area(Xo), area(Xn)
        self.xc = Xm[M.nodes].mean(1)
        self.period = Xm[M.row[:, 1]] - Xm[M.row[:, 0]]
        e = Xm[M.b] - Xm[M.a]
        self.Sn = np.stack([e[:, 1], -e[:, 0]], -1)
        self.S = np.hypot(e[:, 0], e[:, 1])
        self.n = self.Sn / self.S[:, None]
        self.xf = 0.5 * (Xm[M.a] + Xm[M.b])
        self.Uf = 0.5 * (V[M.a] + V[M.b])
        self.SUn = _dot(self.Uf, self.Sn)


def _prim(W, Keff):
    rho = W[..., 0]
    u, v = W[..., 1] / rho, W[..., 2] / rho
    e = W[..., 3] - 0.5 * rho * (u * u + v * v)
    return rho, u, v, (2.0 + Keff) * rho / (4.0 * e)


def _vanleer(a, b):
    p = a * b
    return torch.where(p > 0, 2.0 * p / torch.where(p > 0, a + b, torch.ones_like(p)), torch.zeros_like(p))


def _slope(g, dW, Keff):
    """Coefficients a of g (a.Psi) whose moments are dW (Gaussian moments)."""
    rho, u, v, lam = g
    N = 2.0 + Keff
    d = dW / rho[:, None]
    b2, b3 = 2 * lam * (d[:, 1] - u * d[:, 0]), 2 * lam * (d[:, 2] - v * d[:, 0])
    a4 = 8 * lam ** 2 / N * (d[:, 3] - 0.5 * (u * u + v * v) * d[:, 0] - (u * b2 + v * b3) / (2 * lam)
                             - N * d[:, 0] / (4 * lam))
    b1 = d[:, 0] - a4 * N / (4 * lam)
    a2, a3 = b2 - a4 * u, b3 - a4 * v
    return torch.stack([b1 - a2 * u - a3 * v - 0.5 * a4 * (u * u + v * v), a2, a3, a4], -1)


def _time_slope(g, ax, ay, Uf, Keff):
    """Compatibility of the moving frame: int Psi (ax.Psi wx + ay.Psi wy + A.Psi) g = 0,
    the moments by Gauss-Hermite quadrature (exact for these degrees)."""
    rho, u, v, lam = g
    s, w = np.polynomial.hermite.hermgauss(5)
    s, w = (torch.as_tensor(x, device=rho.device) for x in (s, w))
    r = 1.0 / torch.sqrt(lam)
    x = (u[:, None, None] + s[:, None] * r[:, None, None]).expand(-1, 5, 5)
    y = (v[:, None, None] + s[None, :] * r[:, None, None]).expand(-1, 5, 5)
    wt = (w[:, None] * w[None, :]) / math.pi
    z1 = (Keff / (2 * lam))[:, None, None]
    z2 = (Keff * (Keff + 2.0) / (4 * lam * lam))[:, None, None]
    one = torch.ones_like(x)
    psi = [(one, 0 * one), (x, 0 * one), (y, 0 * one), (0.5 * (x * x + y * y), 0.5 * one)]
    p0, p1 = 0, 0
    for c, rel in ((ax, x - Uf[:, 0, None, None]), (ay, y - Uf[:, 1, None, None])):
        p0 = p0 + rel * sum(c[:, m, None, None] * psi[m][0] for m in range(4))
        p1 = p1 + rel * sum(c[:, m, None, None] * psi[m][1] for m in range(4))
    rhs = [-rho * (wt * (p0 * a + (p0 * b + p1 * a) * z1 + p1 * b * z2)).sum((-2, -1)) for a, b in psi]
    return _slope(g, torch.stack(rhs, -1), Keff)


def _time_integrals(dts, tau):
    """Integrals over dts of c1..c5 of the integral solution, closed forms for
    dts/tau >= 1 and their power series below."""
    x = dts / tau
    E, em = torch.exp(-x), -torch.expm1(-x)
    big = [tau * em, tau * (dts + tau) * E - tau ** 2, dts - tau * em, -tau * dts * (1 + E) + 2 * tau ** 2 * em,
           0.5 * dts ** 2 - tau * dts + tau ** 2 * em]
    xs, s = torch.clamp(x, max=1.0), [0.0] * 4
    for m in range(1, 40):
        t = (-1.0) ** (m + 1) / math.factorial(m)
        s[0] = s[0] + t * xs ** (m - 1)
        if m >= 2:
            s[1] = s[1] + t * (m - 1) * xs ** (m - 2)
        if m >= 3:
            s[2] = s[2] + t * (2 - m) * xs ** (m - 2)
            s[3] = s[3] + t * xs ** (m - 2)
    small = [dts * s[0], dts ** 2 * s[1], dts - dts * s[0], dts ** 2 * s[2], dts ** 2 * s[3]]
    return [torch.where(x < 1.0, a, b) for a, b in zip(small, big)]


class _Ref:
    """One workload in 64 bits: state f (cell, velocity, 2), W, q on `dev`."""

    def __init__(self, c):
        self.c, self.M = c, _Mesh(c)
        self.dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
        self.Keff, self.K, self.Pr = 1.0 + c.K, float(c.K), c.Pr
        ux, uy = (np.array([lo + (hi - lo) * i / (n - 1) for i in range(n)])
                  for lo, hi, n in ((c.vbox[0], c.vbox[1], c.nvx), (c.vbox[2], c.vbox[3], c.nvy)))
        wx, wy = (np.full(n, (hi - lo) / (n - 1)) for lo, hi, n in ((c.vbox[0], c.vbox[1], c.nvx),
                                                                   (c.vbox[2], c.vbox[3], c.nvy)))
        for w in (wx, wy):
            w[0] *= 0.5
            w[-1] *= 0.5
        self.vx, self.vy, self.w = self.t(np.tile(ux, c.nvy)), self.t(np.repeat(uy, c.nvx)), self.t(np.outer(wy, wx).ravel())
        r, u, v, T = c.farfield
        self.Winf = np.array([r, r * u, r * v, 0.5 * r * (u * u + v * v) + (2 + self.Keff) * r * T / 2])
        p = self.t(c.init_prim)
        lam = 1.0 / (2.0 * p[:, 3])
        self.f = self.maxwell((p[:, 0], p[:, 1], p[:, 2], lam))
        self.W = torch.stack([p[:, 0], p[:, 0] * p[:, 1], p[:, 0] * p[:, 2],
                              0.5 * p[:, 0] * (p[:, 1] ** 2 + p[:, 2] ** 2) + (2 + self.Keff) * p[:, 0] * p[:, 3] / 2], -1)
        self.q = self.heat(self.f, p[:, 1], p[:, 2])
        self.nb, self.face, self.sgn = self.t(self.M.nb), self.t(self.M.face), self.t(self.M.sgn)
        self.Xo = _nodes(c, c.motion(0.0))
        self.status = np.zeros(self.M.nc, int)
        self.con = None
        if len(c.blocks) > 1:
            self.status = _connect(self.M, self.Xo, self.dev)[0]

    def t(self, x):
        return torch.as_tensor(np.ascontiguousarray(x), device=self.dev)

    def maxwell(self, g):
        rho, u, v, lam = (a[..., None] for a in g)
        H = rho * lam / math.pi * torch.exp(-lam * ((self.vx - u) ** 2 + (self.vy - v) ** 2))
        return torch.stack([H, self.Keff / (2 * lam) * H], -1)

    def shakhov(self, g, q):
        """The Maxwellian with its heat-flux correction, reduced."""
        G = self.maxwell(g)
        rho, u, v, lam = (a[..., None] for a in g)
        cx, cy = self.vx - u, self.vy - v
        k = 4 * (1 - self.Pr) * lam ** 2 / (5 * rho) * (cx * q[..., 0, None] + cy * q[..., 1, None]) * G[..., 0]
        c2 = 2 * lam * (cx * cx + cy * cy)
        return G + torch.stack([k * (c2 - 4), k * ((c2 - 2) * self.Keff - 2 * self.K) / (2 * lam)], -1)

    def moments(self, f):
        h, b, w = f[..., 0], f[..., 1], self.w
        return torch.stack([(w * h).sum(-1), (w * self.vx * h).sum(-1), (w * self.vy * h).sum(-1),
                            (0.5 * w * ((self.vx ** 2 + self.vy ** 2) * h + b)).sum(-1)], -1)

    def heat(self, f, u, v):
        cx, cy = self.vx - u[:, None], self.vy - v[:, None]
        e = self.w * ((cx * cx + cy * cy) * f[..., 0] + f[..., 1])
        return 0.5 * torch.stack([(cx * e).sum(-1), (cy * e).sum(-1)], -1)

    def tau(self, g):
        T = 1.0 / (2.0 * g[3])
        return self.c.mu_ref * T ** self.c.omega / (g[0] * T)

    def move(self, Xn, dt):
        M, self.dt = self.M, dt
        G = self.G = _Geo(M, self.Xo, Xn, dt)
        if len(self.c.blocks) > 1:
            self.con = _connect(M, Xn, self.dev, self.status)
            self.status = self.con[0]
        st, nc = self.status, M.nc
        self.field = st == FIELD
        # dts: the outward sum is convex in v, so its maximum is at a corner of the velocity box
        out = np.zeros(nc)
        for vx in self.c.vbox[:2]:
            for vy in self.c.vbox[2:]:
                wS = vx * G.Sn[:, 0] + vy * G.Sn[:, 1] - G.SUn
                out = np.maximum(out, np.maximum(M.sgn * wS[M.face], 0.0).sum(1))
        self.dts = self.c.cfl_s * G.vol1 / out
        # slope cases and inverse Jacobians of the limited differences
        self.has, d = [], []
        for m, p in ((IM, IP), (JM, JP)):
            has, pos = [], []
            for s in (m, p):
                nb, fc = M.nb[:, s], M.face[:, s]
                ghost = (nb < 0) & np.isin(M.kind[fc], (wl.BC_FARFIELD, wl.BC_OUTFLOW))
                mir = G.xc + 2.0 * _dot(G.xf[fc] - G.xc, G.n[fc])[:, None] * G.n[fc]
                pos.append(np.where((nb >= 0)[:, None], G.xc[nb] + M.nbshift[:, s, None] * G.period, mir))
                has.append(((nb >= 0) & (st[nb] != HOLE)) | ghost)
            g = G.xf[M.face[:, p]] - G.xf[M.face[:, m]]
            g = np.where((has[0] & has[1])[:, None], 0.5 * (pos[1] - pos[0]), g)
            g = np.where((has[1] & ~has[0])[:, None], pos[1] - G.xc, g)
            g = np.where((has[0] & ~has[1])[:, None], G.xc - pos[0], g)
            self.has.append([self.t(h) for h in has])
            d.append(g)
        det = d[0][:, 0] * d[1][:, 1] - d[0][:, 1] * d[1][:, 0]
        self.J = self.t(np.stack([d[1][:, 1], -d[0][:, 1], -d[1][:, 0], d[0][:, 0]], -1) / det[:, None])
        need = (self.field[M.L] | ((M.R >= 0) & self.field[M.R])) & (M.kind != wl.BC_OVERSET)
        self.two = np.nonzero(need & (M.kind != wl.BC_WALL))[0]
        self.walls = np.nonzero(need & (M.kind == wl.BC_WALL))[0]
        self.Sn, self.SUn = self.t(G.Sn), self.t(G.SUn)

    def wS(self, F):
        return self.Sn[F, 0, None] * self.vx + self.Sn[F, 1, None] * self.vy - self.SUn[F, None]

    def grad(self, phi, ghost):
        """Limited gradient of a cell field (cell, ...): (cell, ..., 2)."""
        ex = (slice(None),) + (None,) * (phi.dim() - 1)
        s = []
        for a, (m, p) in enumerate(((IM, IP), (JM, JP))):
            v = []
            for sl in (m, p):
                nb = self.nb[:, sl]
                x = phi[nb.clamp(min=0)]
                edge = torch.nonzero(nb < 0)[:, 0]
                if edge.numel():
                    x[edge] = ghost(self.face[edge, sl])
                v.append(x)
            hm, hp = (h[ex] for h in self.has[a])
            lo, hi = phi - v[0], v[1] - phi
            z = torch.zeros_like(lo)
            s.append(torch.where(hm & hp, _vanleer(lo, hi), torch.where(hp, hi, torch.where(hm, lo, z))))
        J = [self.J[:, k][ex] for k in range(4)]
        return torch.stack([J[0] * s[0] + J[1] * s[1], J[2] * s[0] + J[3] * s[1]], -1)

    def interface(self, F, ff, gup, W0, gW, q0, dts):
        """int_0^dts of the interface distribution (integral solution)."""
        Uf = self.t(self.G.Uf)[F]
        g = _prim(W0, self.Keff)
        ax, ay = _slope(g, gW[..., 0], self.Keff), _slope(g, gW[..., 1], self.Keff)
        A = _time_slope(g, ax, ay, Uf, self.Keff)
        q = [x[:, None, None] for x in _time_integrals(dts, self.tau(g))]
        G = self.maxwell(g)
        v2 = 0.5 * (self.vx ** 2 + self.vy ** 2)
        lam = g[3][:, None]

        def times(a):
            base = a[:, 0, None] + a[:, 1, None] * self.vx + a[:, 2, None] * self.vy + a[:, 3, None] * v2
            return torch.stack([base + a[:, 3, None] * self.Keff / (4 * lam),
                                base + a[:, 3, None] * (self.Keff + 2) / (4 * lam)], -1) * G
        wx, wy = (self.vx - Uf[:, 0, None])[..., None], (self.vy - Uf[:, 1, None])[..., None]
        return (q[0] * ff + q[1] * (wx * gup[..., 0] + wy * gup[..., 1]) + q[2] * self.shakhov(g, q0)
                + q[3] * (wx * times(ax) + wy * times(ay)) + q[4] * times(A))

    def flux(self):
        """D (cell, velocity, 2) and the loads of the blocks' walls."""
        M, G, t = self.M, self.G, self.t
        gW = self.W[t(M.L)].clone()
        gW[t(M.kind == wl.BC_FARFIELD)] = t(self.Winf)
        none = t(~np.isin(M.kind, (wl.BC_FARFIELD, wl.BC_OUTFLOW)))
        ghost_f = lambda F: torch.where(none[F][:, None, None], 0.0, self.maxwell(_prim(gW[F], self.Keff)))  # noqa: E731
        gf, dW = self.grad(self.f, ghost_f), self.grad(self.W, lambda F: gW[F])
        dts, xc, xf, n = t(self.dts), t(G.xc), t(G.xf), t(G.n)
        L, R, sh, per = t(M.L), t(M.R), t(M.shift), t(G.period)
        D = torch.zeros_like(self.f)
        loads = torch.zeros(len(self.c.blocks), 4, dtype=torch.float64, device=self.dev)
        step = max(64, (1 << 24) // self.vx.numel())
        at = lambda dx, g: torch.einsum("nd,n...d->n...", dx, g)  # noqa: E731
        for lo in range(0, self.two.size, step):
            F = t(self.two[lo:lo + step])
            l, inner = L[F], R[F] >= 0
            r = R[F].clamp(min=0)
            e1, e2, e3 = inner[:, None], inner[:, None, None], inner[:, None, None, None]
            xL = xc[l] + sh[F, None] * per[l]
            xR = torch.where(e1, xc[r], xL + 2.0 * _dot(xf[F] - xL, n[F])[:, None] * n[F])
            fL = self.f[l] + at(xf[F] - xL, gf[l])
            fR = torch.where(e2, self.f[r] + at(xf[F] - xR, gf[r]), ghost_f(F))
            w = self.wS(F)[..., None]
            pick = lambda a, b, s: torch.where(s > 0, a, torch.where(s < 0, b, 0.5 * (a + b)))  # noqa: E731
            ff = pick(fL, fR, w)
            gup = pick(gf[l], torch.where(e3, gf[r], 0.0), w[..., None])
            dL, dR = dW[l], torch.where(e2, dW[r], 0.0)
            jump = torch.where(e1, self.W[r], gW[F]) - self.W[l]
            avg, tv = 0.5 * (dL + dR), xR - xL
            gr = avg + (jump - at(tv, avg))[..., None] * (tv / _dot(tv, tv)[:, None])[:, None, :]
            q0 = 0.5 * (self.q[l] + torch.where(e1, self.q[r], 0.0))
            ds = torch.where(inner, torch.minimum(dts[l], dts[r]), dts[l])
            SF = w / ds[:, None, None] * self.interface(F, ff, gup, self.moments(ff), gr, q0, ds)
            D.index_add_(0, l, SF)
            D.index_add_(0, r[inner], SF[inner], alpha=-1)
        if self.walls.size:
            F = t(self.walls)
            c = L[F]
            dx, ds = xf[F] - xc[c], dts[c]
            I = self.interface(F, self.f[c] + at(dx, gf[c]), gf[c], self.W[c] + at(dx, dW[c]), dW[c], self.q[c], ds)
            w, lw, Uf = self.wS(F), 1.0 / (2.0 * t(M.Tw)[F]), t(G.Uf)[F]
            Hw = self.maxwell((torch.ones_like(lw), Uf[:, 0], Uf[:, 1], lw))
            into = (w > 0)[..., None]
            I = torch.where(into, I / ds[:, None, None], 0.0)
            rho = -(self.w * w * I[..., 0]).sum(-1) / (self.w * w * torch.where(into, 0.0, Hw)[..., 0]).sum(-1)
            SF = w[..., None] * torch.where(into, I, rho[:, None, None] * Hw)
            D.index_add_(0, c, SF)
            loads.index_add_(0, t(M.fb)[F], self.moments(SF))
        return D, loads

    def interpolate(self, cells, donors, weights):
        ok = donors[:, 0] >= 0
        cells, d, w = self.t(cells[ok]), self.t(donors[ok]), self.t(np.where(donors[ok] < 0, 0.0, weights[ok]))
        for x in (self.f, self.W, self.q):
            x[cells] = sum(w[(slice(None), m) + (None,) * (x.dim() - 1)] * x[d[:, m].clamp(min=0)] for m in range(5))

    def diagonals(self):
        """Field cells by i + j, all blocks together: within one, no cell is
        another's lower or upper neighbour."""
        key = self.M.ij.sum(1)
        order = np.nonzero(self.field)[0]
        order = order[np.argsort(key[order], kind="stable")]
        return np.split(order, np.nonzero(np.diff(key[order]))[0] + 1)

    def coupled(self, cells, forward):
        """(cell, slot) neighbours a lexicographic sweep has passed: lower
        (forward) or higher cell indices among the field cells."""
        nb = self.M.nb[cells]
        return (nb >= 0) & self.field[nb] & ((nb < cells[:, None]) if forward else (nb > cells[:, None]))

    def macro(self, W, R, diag, Gam):
        """LU-SGS of the macroscopic increment (Euler-flux variation)."""
        M, G, Keff = self.M, self.G, self.Keff

        def euler(W, n, un):
            rho, u, v, lam = _prim(W, Keff)
            p, vn = rho / (2 * lam), u * n[..., 0] + v * n[..., 1]
            return np.stack([rho * (vn - un), W[..., 1] * (vn - un) + p * n[..., 0],
                             W[..., 2] * (vn - un) + p * n[..., 1], W[..., 3] * (vn - un) + p * vn], -1)
        d = np.zeros_like(R)
        for forward in (True, False):
            for cells in self.lines if forward else reversed(self.lines):
                on, fc, nb = self.coupled(cells, forward), M.face[cells], M.nb[cells]
                n, un = M.sgn[cells, :, None] * G.n[fc], M.sgn[cells] * G.SUn[fc] / G.S[fc]
                x = d[nb]
                c = 0.25 * G.S[fc][..., None] * (euler(W[nb] + x, n, un) - euler(W[nb], n, un) - Gam[fc][..., None] * x)
                c = np.where(on[..., None], c, 0.0).sum(1)
                d[cells] = (R[cells] - c) / diag[cells, None] if forward else d[cells] - c / diag[cells, None]
        return d

    def micro(self, rhs, base):
        """LU-SGS of the distribution (upwind flux variation)."""
        d, t = torch.zeros_like(rhs), self.t
        for forward in (True, False):
            for cells in self.lines if forward else reversed(self.lines):
                on = self.coupled(cells, forward)
                use = [s for s in range(4) if on[:, s].any()]
                C = t(cells)
                w = 0.5 * self.sgn[C][..., None] * self.wS(self.face[C].reshape(-1)).reshape(C.numel(), 4, -1)
                diag = (base[C, None] + w.clamp(min=0).sum(1))[..., None]
                acc = 0.0
                for s in use:
                    acc = acc + (w[:, s].clamp(max=0) * t(on[:, s])[:, None])[..., None] * d[self.nb[C, s].clamp(min=0)]
                d[C] = (rhs[C] - acc) / diag if forward else d[C] - acc / diag
        return d

    def step(self, n_inner):
        """Implicit step n -> n+1 after move() (Steps 1-8)."""
        M, G, t, idt = self.M, self.G, self.t, 1.0 / self.dt
        v0, v1 = t(G.vol0), t(G.vol1)
        e = lambda x: x[:, None, None]  # noqa: E731
        self.lines = self.diagonals()
        if self.con is not None:
            _, rec, don, wgt, fresh, fdon, fwgt, _ = self.con
            self.interpolate(fresh, fdon, fwgt)
            self.interpolate(rec, don, wgt)
        idtp = self.c.cfl_s / (self.c.cfl_pseudo * self.dts)
        field = t(self.field)
        D, loads = self.flux()
        g = _prim(self.W, self.Keff)
        Tf = e(v0 * idt) * self.f + 0.5 * (e(v0 / self.tau(g)) * (self.shakhov(g, self.q) - self.f) - D)
        TW = (v0 * idt)[:, None] * self.W - 0.5 * self.moments(D)
        for it in range(n_inner):
            if it:
                if self.con is not None:
                    self.interpolate(rec, don, wgt)
                D, loads = self.flux()
            R = (TW - (v1 * idt)[:, None] * self.W - 0.5 * self.moments(D)).cpu().numpy()
            W = self.W.cpu().numpy()
            mean = np.where((M.R >= 0)[:, None], 0.5 * (W[M.L] + W[M.R]), W[M.L])
            _, u, v, lam = _prim(mean, self.Keff)
            gam = (4.0 + self.Keff) / (2.0 + self.Keff)
            Gam = np.abs(u * G.n[:, 0] + v * G.n[:, 1] - G.SUn / G.S) + np.sqrt(gam / (2 * lam))
            diag = G.vol1 * (idtp + idt) + 0.25 * (G.S * Gam)[M.face].sum(1)
            Wp = t(W + self.macro(W, R, diag, Gam))
            g = _prim(Wp, self.Keff)
            it2 = 0.5 / self.tau(g)
            rhs = Tf - e(v1 * idt) * self.f + e(v1 * it2) * (self.shakhov(g, self.q) - self.f) - 0.5 * D
            df = self.micro(rhs, v1 * (t(idtp) + idt + it2))
            self.f = torch.where(field[:, None, None], self.f + df, self.f)
            Wn, qn = Wp + self.moments(self.f - self.maxwell(g)), self.heat(self.f, g[1], g[2])
            self.W = torch.where(field[:, None], Wn, self.W)
            self.q = torch.where(field[:, None], qn, self.q)
        return {"f": self.f, "W": self.W, "q": self.q, "status": None, "wall": loads}


def _first_inside(p, quads, allowed):
    """Lowest allowed quad (counter-clockwise, edges included) holding each point, -1 if none."""
    res = torch.full((p.shape[0],), -1, dtype=torch.int64, device=p.device)
    idx = torch.nonzero(allowed)[:, 0]
    if not idx.numel():
        return res
    Q = quads[idx]
    box = [Q[..., k].min(1).values for k in (0, 1)] + [Q[..., k].max(1).values for k in (0, 1)]
    for lo in range(0, p.shape[0], 2048):
        x, y = p[lo:lo + 2048, 0, None], p[lo:lo + 2048, 1, None]
        i, k = torch.nonzero((x >= box[0]) & (x <= box[2]) & (y >= box[1]) & (y <= box[3]), as_tuple=True)
        ok = torch.ones(i.numel(), dtype=torch.bool, device=p.device)
        for e in range(4):
            a, b = Q[k, e], Q[k, (e + 1) % 4]
            l = (b[:, 0] - a[:, 0]) * (p[lo + i, 1] - a[:, 1])
            r = (b[:, 1] - a[:, 1]) * (p[lo + i, 0] - a[:, 0])
            ok &= (l - r) >= 0
        best = torch.full((x.shape[0],), idx.numel(), dtype=torch.int64, device=p.device)
        best.scatter_reduce_(0, i[ok], k[ok], "amin")
        hit = best < idx.numel()
        res[lo:lo + 2048][hit] = idx[best[hit]]
    return res


def _connect(M, X, dev, prev=None):
    """Overset assembly: status, receptors with stencils and weights, fresh
    cells with theirs, cells without a donor (every product and sum rounded once)."""
    Xt = torch.as_tensor(X, device=dev)
    quads = Xt[torch.as_tensor(M.nodes, device=dev)]
    nb_ = len(M.blocks)
    zone = [slice(M.off[b], M.off[b + 1]) for b in range(nb_)]

    def layer(b, n):
        B, ij = M.blocks[b], M.ij[zone[b]]
        m = np.zeros(len(ij), bool)
        for s, v in enumerate((ij[:, 0], B.ni - 1 - ij[:, 0], ij[:, 1], B.nj - 1 - ij[:, 1])):
            if B.bc[s] == wl.BC_OVERSET:
                m |= v < n
        return m

    def wall2(b, p):
        F = np.nonzero((M.fb == b) & (M.kind == wl.BC_WALL))[0]
        best = torch.full((p.shape[0],), math.inf, dtype=torch.float64, device=dev)
        B, nodes = M.blocks[b], M.noff[b] + np.arange(M.noff[b + 1] - M.noff[b]).reshape(-1, M.blocks[b].ni + 1)
        ends = []
        for s, line in enumerate((nodes[:, 0], nodes[:, -1], nodes[0], nodes[-1])):
            if B.bc[s] == wl.BC_WALL:
                ends += list(zip(line[:-1], line[1:]))
        assert len(ends) == F.size
        for a, c in ends:
            (ax, ay), (bx, by) = X[a], X[c]
            ex, ey = bx - ax, by - ay
            px, py = p[:, 0] - ax, p[:, 1] - ay
            t = ((px * ex + py * ey) / (ex * ex + ey * ey)).clamp(0.0, 1.0)
            dx, dy = px - t * ex, py - t * ey
            best = torch.minimum(best, dx * dx + dy * dy)
        return best

    active = np.ones(len(X), bool)
    for z in range(nb_):
        p = Xt[M.noff[z]:M.noff[z + 1]]
        off = torch.zeros(p.shape[0], dtype=torch.bool, device=dev)
        for b in range(nb_):
            if b == z:
                continue
            B = M.blocks[b]
            if B.periodic_i and B.bc[2] == wl.BC_WALL:         # inside the body?
                ring, ins = X[M.noff[b]:M.noff[b] + B.ni], torch.zeros_like(off)
                for i in range(B.ni):
                    (ax, ay), (bx, by) = ring[i], ring[(i + 1) % B.ni]
                    cross = (ay > p[:, 1]) != (by > p[:, 1])
                    if ay != by:
                        ins ^= cross & (p[:, 0] < ax + (p[:, 1] - ay) * (bx - ax) / (by - ay))
                off |= ins
            core = torch.as_tensor(~layer(b, B.n_fringe + B.n_gap), device=dev)
            hit = torch.nonzero(_first_inside(p, quads[zone[b]], core) >= 0)[:, 0]
            if hit.numel():
                db, dz = wall2(b, p[hit]), wall2(z, p[hit])
                off[hit] |= (db < dz) | ((db == dz) & (B.priority > M.blocks[z].priority))
        active[M.noff[z]:M.noff[z + 1]] = ~off.cpu().numpy()
    na = active[M.nodes].sum(1)
    fringe = np.concatenate([layer(b, M.blocks[b].n_fringe) for b in range(nb_)])
    status = np.where(na == 0, HOLE, np.where((na < 4) | fringe, RECEPTOR, FIELD))
    seed = na < 4
    status[(status == FIELD) & ((M.nb >= 0) & seed[M.nb]).any(1)] = RECEPTOR
    xn = 0.25 * ((X[M.nodes[:, 0]] + X[M.nodes[:, 1]]) + (X[M.nodes[:, 2]] + X[M.nodes[:, 3]]))

    def donors(cells):
        don, wgt = np.full((cells.size, 5), -1), np.zeros((cells.size, 5))
        found = np.full(cells.size, -1)
        for cls in (FIELD, RECEPTOR):
            for b in sorted(range(nb_), key=lambda b: (-M.blocks[b].priority, b)):
                todo = np.nonzero((found < 0) & (M.cb[cells] != b))[0]
                if todo.size:
                    k = _first_inside(torch.as_tensor(xn[cells[todo]], device=dev), quads[zone[b]],
                                      torch.as_tensor(status[zone[b]] == cls, device=dev)).cpu().numpy()
                    found[todo] = np.where(k >= 0, M.off[b] + k, -1)
        for r in np.nonzero(found >= 0)[0]:
            st = [found[r]] + [n for n in M.nb[found[r]] if n >= 0 and status[n] != HOLE]
            d = xn[cells[r]] - xn[st]
            d2 = d[:, 0] * d[:, 0] + d[:, 1] * d[:, 1]
            don[r, :len(st)] = st
            if (d2 == 0).any():
                wgt[r, np.argmax(d2 == 0)] = 1.0
                continue
            inv, tot = 1.0 / d2, 0.0
            for v in inv:
                tot = tot + v
            wgt[r, :len(st)] = inv / tot
        return don, wgt, int((found < 0).sum())

    rec = np.nonzero(status == RECEPTOR)[0]
    fresh = np.zeros(0, int) if prev is None else np.nonzero((prev == HOLE) & (status == FIELD))[0]
    rd, rw, n1 = donors(rec)
    fd, fw, n2 = donors(fresh)
    return status, rec, rd, rw, fresh, fd, fw, n1 + n2


def exact(case, seed):
    kind = case["kind"]
    if kind == "idw":
        rec, don, w = _idw_inputs(case, seed)
        f, W, q = _idw_fields(case, seed)
        ok = don[:, 0] >= 0
        R, d = (torch.as_tensor(x[ok].astype(np.int64), device=f.device) for x in (rec, don))
        wt = torch.as_tensor(np.where(don[ok] < 0, 0.0, w[ok]), device=f.device)
        for x in (f, W, q):
            x[R] = sum(wt[(slice(None), m) + (None,) * (x.dim() - 1)] * x[d[:, m].clamp(min=0)] for m in range(5))
        return {"f": f, "W": W, "q": q}
    if kind == "batch":
        cs = _instances(case, seed)
        if sum(c.ncells * c.nv for c in cs) * case["n_inner"] > EXACT_ITEMS_BATCH:
            return None
        out = []
        for c in cs:
            r = _Ref(c)
            r.move(_nodes(c, c.motion(c.dt)), c.dt)
            out.append(r.step(c.n_inner))
        return out
    if kind != "assembly" and _cells(case) * case["nv"] ** 2 * (case["n_inner"] if kind == "step" else 2) > EXACT_ITEMS:
        return None
    c = _workload(case, seed)
    if kind == "assembly":
        M, dev = _Mesh(c), torch.device("cuda" if torch.cuda.is_available() else "cpu")
        before = _connect(M, _nodes(c, c.motion(0.0)), dev)[0]
        st, rec, rd, rw, fresh, fd, fw, _ = _connect(M, _nodes(c, c.motion((1 + seed % ASSEMBLY_POSITIONS) * c.dt)),
                                                     dev, before)
        don, wgt = np.full((M.nc, 5), -1, np.int32), np.zeros((M.nc, 5))
        don[rec], wgt[rec], don[fresh], wgt[fresh] = rd, rw, fd, fw
        return {"status": st.astype(np.int32), "donors": don, "weights": wgt, "receptors": int(rec.size)}
    r = _Ref(c)
    A = np.array(c.motion(c.dt), dtype=np.float64)
    if case.get("flow") == "particle":         # first step: no gas load yet, the body drifts and spins
        m = c.meta
        a, (cx, cy) = c.dt * m["omega0"], m["center"]
        co, si = math.cos(a), math.sin(a)
        A[m["body_block"]] = [co, -si, si, co, cx + c.dt * m["u0"][0] - (co * cx - si * cy),
                              cy + c.dt * m["u0"][1] - (si * cx + co * cy)]
    r.move(_nodes(c, A), c.dt)
    if kind == "flux":
        if r.con is not None:
            r.interpolate(*r.con[1:4])
        D, _ = r.flux()
        F = r.moments(D)
        D[r.t(~r.field)] = 0.0
        return {"D": D, "F": F}
    return r.step(c.n_inner)
