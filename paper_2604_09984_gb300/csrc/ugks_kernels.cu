// ugks_kernels.cu -- CUDA kernels of the implicit UGKS step (arXiv 2604.09984
// Sec. 2.2 Steps 1-8) on moving structured blocks, and the mesh-motion /
// geometry kernels (Sec. 3 Step 1).  Launch wrappers at the end are the only
// symbols used by the host orchestration (ugks_api.cu).
#include <cstdlib>
#include <cstring>
#include "ugks_internal.cuh"
#include "ugks_launch.h"

namespace ugks {

// ------------------------------------------------------------- geometry
// x = (m00 x0 + m01 y0) + b0, y = (m10 x0 + m11 y0) + b1 without contraction
// (bit-identical to the FP64 reference evaluation).
__global__ void k_move_nodes(Dev d) {
  int n = blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= d.nn) return;
  const double *a = d.affine + 6 * d.node_block[n];
  double x = d.X_ref[2 * n], y = d.X_ref[2 * n + 1];
  d.X_new[2 * n] = __dadd_rn(__dadd_rn(__dmul_rn(a[0], x), __dmul_rn(a[1], y)), a[4]);
  d.X_new[2 * n + 1] = __dadd_rn(__dadd_rn(__dmul_rn(a[2], x), __dmul_rn(a[3], y)), a[5]);
}

__device__ __forceinline__ double shoelace(const double *X, const int *nd) {
  double x1 = X[2 * nd[0]], y1 = X[2 * nd[0] + 1], x2 = X[2 * nd[1]], y2 = X[2 * nd[1] + 1];
  double x3 = X[2 * nd[2]], y3 = X[2 * nd[2] + 1], x4 = X[2 * nd[3]], y4 = X[2 * nd[3] + 1];
  return 0.5 * __dsub_rn(__dmul_rn(x3 - x1, y4 - y2), __dmul_rn(y3 - y1, x4 - x2));
}

// Cell volumes at both levels (shoelace), mid-time and new vertex centres,
// period vector of the cell's row.
__device__ __forceinline__ void cell_geom(const Dev &d, int c) {
  const int *nd = d.cell_nodes + 4 * c;
  double vo = shoelace(d.X_old, nd), vn = shoelace(d.X_new, nd);
  d.vol_old[c] = vo;
  d.vol_new[c] = vn;
  if (!(vn > 0.0) || !(vo > 0.0)) atomicOr(d.err, EF_GEOMETRY);
  for (int m = 0; m < 2; ++m) {
    double pm[4], pn[4];
    for (int v = 0; v < 4; ++v) {
      pm[v] = 0.5 * (d.X_old[2 * nd[v] + m] + d.X_new[2 * nd[v] + m]);
      pn[v] = d.X_new[2 * nd[v] + m];
    }
    d.xc[2 * c + m] = 0.25 * ((pm[0] + pm[1]) + (pm[2] + pm[3]));
    d.xc_new[2 * c + m] = 0.25 * ((pn[0] + pn[1]) + (pn[2] + pn[3]));
    int r0 = d.cell_row[2 * c], r1 = d.cell_row[2 * c + 1];
    double a = 0.5 * (d.X_old[2 * r0 + m] + d.X_new[2 * r0 + m]);
    double b = 0.5 * (d.X_old[2 * r1 + m] + d.X_new[2 * r1 + m]);
    d.period[2 * c + m] = b - a;
  }
}

// Mid-time face vector S n (L -> R / outward), centre, face velocity (mean
// node velocity) and S U.n.
template <typename T> __device__ __forceinline__ void face_geom(const Dev &d, int f) {
  int a = d.face_a[f], b = d.face_b[f];
  double ax = 0.5 * (d.X_old[2 * a] + d.X_new[2 * a]), ay = 0.5 * (d.X_old[2 * a + 1] + d.X_new[2 * a + 1]);
  double bx = 0.5 * (d.X_old[2 * b] + d.X_new[2 * b]), by = 0.5 * (d.X_old[2 * b + 1] + d.X_new[2 * b + 1]);
  double ex = bx - ax, ey = by - ay;
  const double S = sqrt(ex * ex + ey * ey), iS = 1.0 / S, idt = 1.0 / d.dt;
  d.Sn[2 * f] = ey;
  d.Sn[2 * f + 1] = -ex;
  d.S[f] = S;
  d.nrm[2 * f] = ey * iS;
  d.nrm[2 * f + 1] = -ex * iS;
  d.xf[2 * f] = 0.5 * (ax + bx);
  d.xf[2 * f + 1] = 0.5 * (ay + by);
  double ufx = 0.5 * ((d.X_new[2 * a] - d.X_old[2 * a]) + (d.X_new[2 * b] - d.X_old[2 * b])) * idt;
  double ufy = 0.5 * ((d.X_new[2 * a + 1] - d.X_old[2 * a + 1]) + (d.X_new[2 * b + 1] - d.X_old[2 * b + 1])) * idt;
  d.Uf[2 * f] = ufx;
  d.Uf[2 * f + 1] = ufy;
  const double sun = ufx * ey + ufy * (-ex);
  d.SUn[f] = sun;
  d.Un[f] = sun * iS;
  T *g = reinterpret_cast<T *>(d.fgeo) + (size_t)NFG * f;
  g[FG_SNX] = (T)ey;
  g[FG_SNY] = (T)(-ex);
  g[FG_SUN] = (T)sun;
  g[FG_UFX] = (T)ufx;
  g[FG_UFY] = (T)ufy;
}

// Both in one launch (they share nothing): the first CTAs take the faces.  The
// FP64 pipe bounds them (one division and a square root a face), on small
// meshes the launches.
constexpr int GEO_THREADS = 128;
template <typename T> __global__ void __launch_bounds__(GEO_THREADS) k_geom(Dev d, int face_blocks) {
  if ((int)blockIdx.x < face_blocks) {
    const int f = blockIdx.x * GEO_THREADS + threadIdx.x;
    if (f < d.nf) face_geom<T>(d, f);
  } else {
    const int c = ((int)blockIdx.x - face_blocks) * GEO_THREADS + threadIdx.x;
    if (c < d.nc) cell_geom(d, c);
  }
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  return v;
}

// Lane-local sum in the arithmetic type: plain for FP64, Neumaier-compensated
// for FP32 (the mixed path keeps velocity sums accurate to a few FP32 ulps
// before the FP64 warp reduction).
template <typename T> struct Acc {
  T s = T(0);
  __device__ __forceinline__ void add(T x) { s += x; }
  __device__ __forceinline__ double get() const { return (double)s; }
};
template <> struct Acc<float> {
  float s = 0.f, c = 0.f;
  __device__ __forceinline__ void add(float x) {
    float t = s + x;
    c += (fabsf(s) >= fabsf(x)) ? (s - t) + x : (x - t) + s;
    s = t;
  }
  __device__ __forceinline__ double get() const { return (double)s + (double)c; }
};

// Warp total of per-lane accumulators.  FP32: the (sum, compensation) pairs
// are combined in FP32 with an error-free sum at every butterfly level (no
// FP64 arithmetic on the way); FP64: plain FP64 butterfly.
__device__ __forceinline__ double warp_total(const Acc<double> &a) {
  double v = a.s;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
// FP32: the total rounded once to FP32 (relative error ~ulp of the total;
// the compensation only has to stop the error growing with the term count).
__device__ __forceinline__ float warp_total(const Acc<float> &a) {
  float s = a.s, c = a.c;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    float os = __shfl_xor_sync(0xffffffffu, s, o), oc = __shfl_xor_sync(0xffffffffu, c, o);
    float t = s + os, bb = t - s;
    float e = (s - (t - bb)) + (os - bb);
    s = t;
    c = c + oc + e;
  }
  return s + c;
}


// Reading R3: dts_i = cfl_s Omega_i^{n+1} / max_k sum_faces S max(w_out, 0).
// The sum is a convex piecewise-linear function of v, so over the tensor
// velocity grid its maximum is attained at one of the four corners of the
// velocity box (which are grid points): only those are evaluated.
__device__ __forceinline__ void cell_dts(const Dev &d, int c) {
  const double vx0 = d.vbox[0], vx1 = d.vbox[1], vy0 = d.vbox[2], vy1 = d.vbox[3];
  // (positive parts by the sign bit, off the FP64 pipe)
  auto pos = [](double x) { return __double2hiint(x) >= 0 ? x : 0.0; };
  double s00 = 0.0, s01 = 0.0, s10 = 0.0, s11 = 0.0;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int f = d.cell_faces[4 * c + q];
    const bool in = d.cell_sgn[4 * c + q] < 0;
    const double2 n = *reinterpret_cast<const double2 *>(d.Sn + 2 * (size_t)f);
    const double u = d.SUn[f], nx = in ? -n.x : n.x, ny = in ? -n.y : n.y, un = in ? -u : u;
    const double x0 = vx0 * nx, x1 = vx1 * nx, y0 = vy0 * ny - un, y1 = vy1 * ny - un;
    s00 += pos(x0 + y0);
    s01 += pos(x0 + y1);
    s10 += pos(x1 + y0);
    s11 += pos(x1 + y1);
  }
  const double m = fmax(fmax(s00, s01), fmax(s10, s11));
  const double dts = d.cfl_s * d.vol_new[c] / m;
  d.dts[c] = dts;
  d.idtau[c] = d.cfl_s / (d.cfl_pseudo * dts);
}

// Per-step geometry records in the arithmetic type: per face (S n, S U.n,
// U_f, vectors from the L image / R centres to the face centre), per cell
// half the outward (S n, S U.n) of its four faces for the sweeps.
// The face's part without cell centres comes from the face geometry, so that a
// cell takes it in the arithmetic type (conversions pass the FP64 pipe; a half
// and a sign commute with the rounding).
template <typename T> __device__ __forceinline__ void face_record(const Dev &d, int f) {
  int L = d.face_L[f], R = d.face_R[f];
  T *g = reinterpret_cast<T *>(d.fgeo) + (size_t)NFG * f;
  double sh = (double)d.face_shiftL[f];
  g[FG_DXLX] = (T)(d.xf[2 * f] - (d.xc[2 * L] + sh * d.period[2 * L]));
  g[FG_DXLY] = (T)(d.xf[2 * f + 1] - (d.xc[2 * L + 1] + sh * d.period[2 * L + 1]));
  g[FG_DXRX] = R >= 0 ? (T)(d.xf[2 * f] - d.xc[2 * R]) : T(0);
  g[FG_DXRY] = R >= 0 ? (T)(d.xf[2 * f + 1] - d.xc[2 * R + 1]) : T(0);
}
template <typename T> __device__ __forceinline__ void cell_record(const Dev &d, int c) {
  T *r = reinterpret_cast<T *>(d.srec) + (size_t)NSR * c;
#pragma unroll
  for (int s = 0; s < 4; ++s) {
    const T *g = reinterpret_cast<const T *>(d.fgeo) + (size_t)NFG * d.cell_faces[4 * c + s];
    const T h = d.cell_sgn[4 * c + s] < 0 ? T(-0.5) : T(0.5);
    r[sr_at(0, s)] = h * g[FG_SNX];
    r[sr_at(1, s)] = h * g[FG_SNY];
    r[sr_at(2, s)] = h * g[FG_SUN];
  }
}
// the records and the time steps of the cells in one launch
template <typename T> __global__ void __launch_bounds__(GEO_THREADS) k_geo_records(Dev d, int face_blocks) {
  if ((int)blockIdx.x < face_blocks) {
    const int f = blockIdx.x * GEO_THREADS + threadIdx.x;
    if (f < d.nf) face_record<T>(d, f);
  } else {
    const int c = ((int)blockIdx.x - face_blocks) * GEO_THREADS + threadIdx.x;
    if (c >= d.nc) return;
    cell_dts(d, c);
    cell_record<T>(d, c);
  }
}

// Slope case and inverse Jacobian per cell (reading R1); depends on the
// geometry and on which neighbours are holes.
__global__ void k_slope_geo(Dev d) {
  int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= d.nc) return;
  double g[2][2];
  int flags = 0;
  double xcx = d.xc[2 * c], xcy = d.xc[2 * c + 1];
  for (int dir = 0; dir < 2; ++dir) {
    bool has[2];
    double px[2], py[2];
    for (int side = 0; side < 2; ++side) {
      int s = 2 * dir + side;
      int kind = d.nb_kind[4 * c + s], id = d.nb_id[4 * c + s];
      has[side] = false;
      px[side] = py[side] = 0.0;
      if (kind == NB_CELL) {
        double sh = (double)d.nb_shift[4 * c + s];
        px[side] = d.xc[2 * id] + sh * d.period[2 * c];
        py[side] = d.xc[2 * id + 1] + sh * d.period[2 * c + 1];
        has[side] = d.status[id] != ST_HOLE;
      } else if (kind == NB_GHOST) {
        double nx = d.nrm[2 * id], ny = d.nrm[2 * id + 1];
        double dd = (d.xf[2 * id] - xcx) * nx + (d.xf[2 * id + 1] - xcy) * ny;
        px[side] = xcx + 2.0 * dd * nx;
        py[side] = xcy + 2.0 * dd * ny;
        has[side] = true;
      }
    }
    int cs;
    if (has[0] && has[1]) {
      cs = SL_BOTH;
      g[dir][0] = 0.5 * (px[1] - px[0]);
      g[dir][1] = 0.5 * (py[1] - py[0]);
    } else if (has[1]) {
      cs = SL_P;
      g[dir][0] = px[1] - xcx;
      g[dir][1] = py[1] - xcy;
    } else if (has[0]) {
      cs = SL_M;
      g[dir][0] = xcx - px[0];
      g[dir][1] = xcy - py[0];
    } else {
      cs = SL_NONE;
      int fm = d.cell_faces[4 * c + 2 * dir], fp = d.cell_faces[4 * c + 2 * dir + 1];
      g[dir][0] = d.xf[2 * fp] - d.xf[2 * fm];
      g[dir][1] = d.xf[2 * fp + 1] - d.xf[2 * fm + 1];
    }
    flags |= cs << (2 * dir);
  }
  double a11 = g[0][0], a12 = g[0][1], a21 = g[1][0], a22 = g[1][1];
  const double idet = 1.0 / (a11 * a22 - a12 * a21);
  d.slope_flags[c] = flags;
  // sweep mask: bit 0 solved cell, bit 1+s: neighbour across face slot s is solved
  int mask = d.status[c] == ST_FIELD ? 1 : 0;
  for (int s = 0; s < 4; ++s) {
    int f = d.cell_faces[4 * c + s];
    int nb = d.cell_sgn[4 * c + s] > 0 ? d.face_R[f] : d.face_L[f];
    if (nb >= 0 && d.status[nb] == ST_FIELD) mask |= 2 << s;
  }
  d.cmask[c] = mask;
  const double j0 = a22 * idet, j1 = -a12 * idet, j2 = -a21 * idet, j3 = a11 * idet;
  reinterpret_cast<double2 *>(d.jinv + 4 * c)[0] = make_double2(j0, j1);
  reinterpret_cast<double2 *>(d.jinv + 4 * c)[1] = make_double2(j2, j3);
  d.jinvf[c] = make_float4((float)j0, (float)j1, (float)j2, (float)j3);
}

// Ghost states of far-field / outflow faces (reading R6).
__global__ void k_ghost(Dev d) {
  int f = blockIdx.x * blockDim.x + threadIdx.x;
  if (f >= d.nf) return;
  int kind = d.face_kind[f];
  for (int m = 0; m < 4; ++m) {
    double v = 0.0;
    if (kind == BC_FARFIELD) v = d.Winf[m];
    else if (kind == BC_OUTFLOW) v = d.W[4 * d.face_L[f] + m];
    d.ghostW[4 * f + m] = v;
  }
}

// Limited gradient of the conservative W per cell (reading R1).  Bound by the
// latency of its loads: a thread per cell and component, and CTAs of 64 threads
// so that a small mesh spreads over the SMs (512 cells: 12.8 us -> 5.4 us; 36864
// cells 15.3 -> 13.6).
constexpr int GW_THREADS = 64;
__global__ void __launch_bounds__(GW_THREADS) k_gradW(Dev d) {
  int t = blockIdx.x * blockDim.x + threadIdx.x;
  int c = t >> 2, m = t & 3;
  if (c >= d.nc) return;
  int fl = d.slope_flags[c];
  const int4 kind = *reinterpret_cast<const int4 *>(d.nb_kind + 4 * c);
  const int4 id = *reinterpret_cast<const int4 *>(d.nb_id + 4 * c);
  const double2 j0 = *reinterpret_cast<const double2 *>(d.jinv + 4 * c);
  const double2 j1 = *reinterpret_cast<const double2 *>(d.jinv + 4 * c + 2);
  double wc = d.W[4 * c + m];
  auto value = [&](int k, int i) { return k == NB_CELL ? d.W[4 * i + m] : k == NB_GHOST ? d.ghostW[4 * i + m] : 0.0; };
  const double v0 = value(kind.x, id.x), v1 = value(kind.y, id.y), v2 = value(kind.z, id.z), v3 = value(kind.w, id.w);
  auto slope = [&](int cs, double lo, double hi) {
    if (cs == SL_BOTH) return vanleer<double>(wc - lo, hi - wc);
    return cs == SL_P ? hi - wc : cs == SL_M ? wc - lo : 0.0;
  };
  const double s0 = slope(fl & 3, v0, v1), s1 = slope((fl >> 2) & 3, v2, v3);
  double2 g;
  g.x = j0.x * s0 + j0.y * s1;
  g.y = j1.x * s0 + j1.y * s1;
  *reinterpret_cast<double2 *>(d.gradW + 8 * c + 2 * m) = g;
}

__device__ __forceinline__ bool face_needed(const Dev &d, int f) {
  int L = d.face_L[f], R = d.face_R[f];
  return d.status[L] == ST_FIELD || (R >= 0 && d.status[R] == ST_FIELD);
}

// Face coefficients, scalar part: g0 parameters and slopes (reading R2), time
// integrals over dts (Eq. fullSolution averaged as in Sec. 2.2), wall
// temperature parameter, Gamma; all in FP64 (per face, not per velocity), the
// mixed path rounds the finished record once to FP32 for its velocity loops.
//
// Bound by the FP64 pipe (some 15 cycles a warp instruction and SM; 500 such
// instructions a face) and, on small meshes, by the latency of one face's chain.
// So a CTA takes only FSC = 32 faces (a small mesh reaches every SM), one warp
// does the face state, slopes and time integrals, a second one the geometry and
// Gamma; with the reduction's parts to fold (small meshes), four warps take the
// sums among them and a third one the time integrals.  The records are collected in shared memory and written as lines.
// 1056 faces with 8 parts to fold: 44.1 us -> 18.2 us (128 faces a CTA, one
// thread a face before); 74112 faces: 113 -> 95 (a fifth fewer FP64
// instructions: one division for p / rho, two sums for the integrals).
constexpr int FSC = 32;
template <typename T, bool FOLD> __global__ void __launch_bounds__(FOLD ? 128 : 64) k_face_scalar(Dev d) {
  constexpr int ROW = FP_IH + 1;
  __shared__ T rec[FSC * ROW];
  __shared__ double W0f[4][FSC];
  __shared__ bool live[FSC];
  const int lane = threadIdx.x & 31, wrp = threadIdx.x >> 5;
  const int f0 = blockIdx.x * FSC, fid = f0 + lane;
  const int kind = fid < d.nf ? d.face_kind[fid] : BC_OVERSET;
  const bool need = kind != BC_OVERSET && face_needed(d, fid);
  const bool wall = kind == BC_WALL;
  const int L = need ? d.face_L[fid] : 0, R = need ? d.face_R[fid] : -1;
  T *PT = rec + lane * ROW;
  if (wrp == 0) live[lane] = need;
  if (FOLD) {                  // the reduction's CTAs left their parts: added here in order
    if (need) {
      const T *p = reinterpret_cast<const T *>(d.fpart) + 2 * (size_t)fid;
#pragma unroll
      for (int j = 0; j < NFS / 4; ++j) {
        const int m = wrp + 4 * j;
        T h = T(0), l = T(0);
        for (int s = 0; s < d.nsplit; ++s) {
          const typename Vec2<T>::type q =
              *reinterpret_cast<const typename Vec2<T>::type *>(p + 2 * ((size_t)s * NFS + m) * d.nf);
          face_sum_add(h, l, q.x, q.y);
        }
        const double v = face_sum_value(h, l);
        d.fsum[(size_t)NFS * fid + m] = v;
        if (j == 0) W0f[m][lane] = v;
      }
    }
    __syncthreads();
  }
  static_assert(FS_W0 == 0 && NFS == 12, "the first sums are the face state");
  // face state: of a wall extrapolated from its cell
  auto face_state = [&](double *W0) {
    if (wall) {
      double dx = d.xf[2 * fid] - d.xc[2 * L], dy = d.xf[2 * fid + 1] - d.xc[2 * L + 1];
      for (int m = 0; m < 4; ++m) W0[m] = d.W[4 * L + m] + (dx * d.gradW[8 * L + 2 * m] + dy * d.gradW[8 * L + 2 * m + 1]);
    } else {
      for (int m = 0; m < 4; ++m) W0[m] = FOLD ? W0f[m][lane] : d.fsum[(size_t)NFS * fid + m];
    }
  };
  auto integrals = [&](const Prim &p0) {
    double qi[5];
    const double dts = R >= 0 ? fmin(d.dts[L], d.dts[R]) : d.dts[L];
    time_integrals(dts, collision_time(p0.rho, p0.lam, d.mu_ref, d.omega), qi);
    const double idts = 1.0 / dts;
    for (int m = 0; m < 5; ++m) PT[FP_Q1 + m] = (T)(qi[m] * idts);
    *reinterpret_cast<double2 *>(d.fq12 + 2 * (size_t)fid) = make_double2(qi[0] * idts, qi[1] * idts);
  };
  if (need && wrp == 0) {
    double W0[4], gx[4], gy[4];
    const double ufx = d.Uf[2 * fid], ufy = d.Uf[2 * fid + 1];
    face_state(W0);
    if (wall) {
      for (int m = 0; m < 4; ++m) {
        gx[m] = d.gradW[8 * L + 2 * m];
        gy[m] = d.gradW[8 * L + 2 * m + 1];
      }
    } else {
      double sh = (double)d.face_shiftL[fid];
      double xLx = d.xc[2 * L] + sh * d.period[2 * L], xLy = d.xc[2 * L + 1] + sh * d.period[2 * L + 1];
      double xRx, xRy, WL[4], WR[4], dL[8], dR[8];
      for (int m = 0; m < 4; ++m) WL[m] = d.W[4 * L + m];
      for (int m = 0; m < 8; ++m) dL[m] = d.gradW[8 * L + m];
      if (R >= 0) {
        xRx = d.xc[2 * R];
        xRy = d.xc[2 * R + 1];
        for (int m = 0; m < 4; ++m) WR[m] = d.W[4 * R + m];
        for (int m = 0; m < 8; ++m) dR[m] = d.gradW[8 * R + m];
      } else {
        double nx = d.nrm[2 * fid], ny = d.nrm[2 * fid + 1];
        double dd = (d.xf[2 * fid] - xLx) * nx + (d.xf[2 * fid + 1] - xLy) * ny;
        xRx = xLx + 2.0 * dd * nx;
        xRy = xLy + 2.0 * dd * ny;
        for (int m = 0; m < 4; ++m) WR[m] = d.ghostW[4 * fid + m];
        for (int m = 0; m < 8; ++m) dR[m] = 0.0;
      }
      double tx = xRx - xLx, ty = xRy - xLy, it2 = 1.0 / (tx * tx + ty * ty);
      double ex = tx * it2, ey = ty * it2;
      for (int m = 0; m < 4; ++m) {
        double avx = 0.5 * (dL[2 * m] + dR[2 * m]), avy = 0.5 * (dL[2 * m + 1] + dR[2 * m + 1]);
        double jump = (WR[m] - WL[m]) - (avx * tx + avy * ty);
        gx[m] = avx + jump * ex;
        gy[m] = avy + jump * ey;
      }
    }
    Prim p0 = primitive(W0, d.Keff);
    const SlopeInv<double> inv = slope_inv<double>(p0, d.Keff);
    double ax[4], ay[4], At[4];
    micro_slope_r<double>(p0, d.Keff, inv, gx, ax);
    micro_slope_r<double>(p0, d.Keff, inv, gy, ay);
    time_slope_r<double>(p0, d.Keff, inv, ax, ay, gx, gy, ufx, ufy, At);
    PT[FP_RHO] = (T)p0.rho; PT[FP_UX] = (T)p0.ux; PT[FP_UY] = (T)p0.uy; PT[FP_LAM] = (T)p0.lam;
    for (int m = 0; m < 4; ++m) { PT[FP_AX + m] = (T)ax[m]; PT[FP_AY + m] = (T)ay[m]; PT[FP_AT + m] = (T)At[m]; }
    PT[FP_PREF] = (T)(0.8 * (1.0 - d.Pr) * p0.lam * p0.lam * inv.irho);
    PT[FP_HPRE] = (T)(p0.rho * p0.lam * M_1_PI);
    PT[FP_IL] = (T)inv.il;
    PT[FP_EH] = (T)(0.5 * d.Keff * inv.il);
    PT[FP_EB] = (T)(0.5 * (d.Keff + 2.0) * inv.il);
    if (!FOLD) integrals(p0);
  }
  if (FOLD && need && wrp == 2) {
    double W0[4];
    face_state(W0);
    integrals(primitive(W0, d.Keff));
  }
  if (need && wrp == 1) {
    const double nx = d.nrm[2 * fid], ny = d.nrm[2 * fid + 1], sun = d.SUn[fid];
    const double fx = d.xf[2 * fid], fy = d.xf[2 * fid + 1], sh = (double)d.face_shiftL[fid];
    const double half = wall ? 1.0 : 0.5;
    PT[FP_QX] = (T)(R >= 0 ? 0.5 * (d.q[2 * L] + d.q[2 * R]) : half * d.q[2 * L]);
    PT[FP_QY] = (T)(R >= 0 ? 0.5 * (d.q[2 * L + 1] + d.q[2 * R + 1]) : half * d.q[2 * L + 1]);
    PT[FP_UFX] = (T)d.Uf[2 * fid]; PT[FP_UFY] = (T)d.Uf[2 * fid + 1];
    PT[FP_LAMW] = wall ? (T)(1.0 / (2.0 * d.face_Tw[fid])) : T(0);
    PT[FP_RHOW] = T(0);
    PT[FP_SNX] = (T)d.Sn[2 * fid];
    PT[FP_SNY] = (T)d.Sn[2 * fid + 1];
    PT[FP_SUN] = (T)sun;
    PT[FP_DXLX] = (T)(fx - (d.xc[2 * L] + sh * d.period[2 * L]));
    PT[FP_DXLY] = (T)(fy - (d.xc[2 * L + 1] + sh * d.period[2 * L + 1]));
    PT[FP_DXRX] = (R >= 0) ? (T)(fx - d.xc[2 * R]) : T(0);
    PT[FP_DXRY] = (R >= 0) ? (T)(fy - d.xc[2 * R + 1]) : T(0);
    PT[FP_EB + 1] = T(0);
    // Gamma from the mean of the two cells' W (boundary: the cell):
    // |u.n - U.n| + sqrt(gamma p / rho), p / rho = (gamma - 1) e
    double W[4];
    for (int m = 0; m < 4; ++m) W[m] = (R >= 0) ? 0.5 * (d.W[4 * L + m] + d.W[4 * R + m]) : d.W[4 * L + m];
    const double ir = 1.0 / W[0], ux = W[1] * ir, uy = W[2] * ir;
    const double e = W[3] * ir - 0.5 * (ux * ux + uy * uy);
    d.gam[fid] = fabs(ux * nx + uy * ny - d.Un[fid]) + sqrt(d.c2fac * e);
  }
  __syncthreads();
  // rows of the record up to the coefficients of the pass below
  T *out = reinterpret_cast<T *>(d.fparT) + (size_t)f0 * NFP;
  for (int t = threadIdx.x; t < FSC * FP_IH; t += blockDim.x) {
    const int r = t / FP_IH, m = t - r * FP_IH;
    if (live[r]) out[(size_t)r * NFP + m] = rec[r * ROW + m];
  }
}

// Face coefficients, velocity part: the g-part of the macro flux by a sum over
// the discrete velocities, the wall density rho_w (Eq. maxWalldes) and the
// total S-weighted macro flux (Eq. macroscopicFlux).  Equilibrium part of the macro flux of an interior face (the velocity sum
// of w wS Psi (q3 (g + g+) + q4 g (a.w Psi) + q5 g (A Psi)) in reduced form,
// Eqs. fullSolution / macroscopicFlux) through the tensor structure of the
// velocity grid: every term is g = HPRE Ex(cx) Ey(cy) (c = v - U0) times a
// polynomial of degree <= 6 in (cx, cy), so the 2D sum is exactly (up to
// rounding) sum_ab coef_ab Mx_a My_b with the 1D moments
// Mx_a = sum_ix wx cx^a Ex(cx), My_b likewise: O(nvx + nvy) work per face
// instead of O(nvx nvy).
// 1D grids of the separable sums in the arithmetic type
template <typename R> struct Grid1;
template <> struct Grid1<float> {
  __device__ static float vx(const Dev &d, int i) { return d.vxf[i]; }
  __device__ static float vy(const Dev &d, int i) { return d.vy1f[i]; }
  __device__ static float wx(const Dev &d, int i) { return d.wx1f[i]; }
  __device__ static float wy(const Dev &d, int i) { return d.wy1f[i]; }
  __device__ static float ex(float x) { return __expf(x); }
};
template <> struct Grid1<double> {
  __device__ static double vx(const Dev &d, int i) { return d.vx1[i]; }
  __device__ static double vy(const Dev &d, int i) { return d.vy1[i]; }
  __device__ static double wx(const Dev &d, int i) { return d.wx1[i]; }
  __device__ static double wy(const Dev &d, int i) { return d.wy1[i]; }
  __device__ static double ex(double x) { return exp(x); }
};

// 1D moments: lane = index in the face's GS-lane group, a = 0..6 (mx) and b =
// 0..6 (my); every lane of the warp takes part in the shuffles
template <typename R, int GS>
__device__ __forceinline__ void face_moments(const Dev &d, R ux, R uy, R lam, int lane, R *mx, R *my) {
  typedef Grid1<R> G;
#pragma unroll
  for (int a = 0; a < 7; ++a) { mx[a] = R(0); my[a] = R(0); }
  for (int ix = lane; ix < d.nvx; ix += GS) {
    R cx = G::vx(d, ix) - ux;
    R e = G::wx(d, ix) * G::ex(-lam * cx * cx), p = e;
#pragma unroll
    for (int a = 0; a < 7; ++a) { mx[a] += p; p *= cx; }
  }
  for (int iy = lane; iy < d.nvy; iy += GS) {     // the whole grid (also when sharded)
    R cy = G::vy(d, iy) - uy;
    R e = G::wy(d, iy) * G::ex(-lam * cy * cy), p = e;
#pragma unroll
    for (int a = 0; a < 7; ++a) { my[a] += p; p *= cy; }
  }
#pragma unroll
  for (int o = GS / 2; o > 0; o >>= 1)
#pragma unroll
    for (int a = 0; a < 7; ++a) {
      mx[a] += __shfl_xor_sync(0xffffffffu, mx[a], o);
      my[a] += __shfl_xor_sync(0xffffffffu, my[a], o);
    }
}

// the four sums from the moments and the interface cubics
template <typename R>
__device__ __forceinline__ void face_eq_flux(const R *P, const Poly2<3, R> &ih, const Poly2<3, R> &ib, const R *mx,
                                             const R *my, R out[4]) {
  R ux = P[FP_UX], uy = P[FP_UY], snx = P[FP_SNX], sny = P[FP_SNY], sun = P[FP_SUN];
  Poly2<1, R> vxp = p2_lin<R>(ux, R(1), R(0)), vyp = p2_lin<R>(uy, R(0), R(1));
  Poly2<2, R> v2 = p2_axpby(R(1), p2_mul(vxp, vxp), R(1), p2_mul(vyp, vyp));
  Poly2<1, R> ws = p2_lin<R>(snx * ux + sny * uy - sun, snx, sny);
  Poly2<4, R> m0 = p2_mul(ws, ih);
  R hpre = P[FP_HPRE];
  out[0] = hpre * p2_sum(m0, mx, my);
  out[1] = hpre * p2_sum(p2_mul(m0, vxp), mx, my);
  out[2] = hpre * p2_sum(p2_mul(m0, vyp), mx, my);
  Poly2<5, R> e3 = p2_axpby(R(0.5), ib, R(0.5), p2_mul(v2, ih));
  out[3] = hpre * p2_sum(p2_mul(ws, e3), mx, my);
}

// Face coefficients, velocity part, in one launch: its first CTAs take the
// walls (a longer job per face), the others every other face (two launches one
// after the other: 16.7 us, one: 9.1, 1056 faces, 64 of them walls; 74112
// faces: 63 -> 55).
//
// Wall faces (`list`, n of them): FCW warps per face split the velocities,
// their warp totals meet in shared memory (summed in warp order).
constexpr int FCW = 4, FC_THREADS = 256;
template <typename T> __device__ __forceinline__ void wall_coef(const Dev &d, const int *list, int n) {
  __shared__ double part[FC_THREADS / 32][9];
  int wg = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  int w = wg / FCW, sub = wg - (wg / FCW) * FCW;
  int lane = threadIdx.x & 31, wl = threadIdx.x >> 5;
  bool in = w < n;
  int fid = in ? list[w] : 0;
  int kind = in ? d.face_kind[fid] : BC_OVERSET;
  bool act = in && kind != BC_OVERSET && face_needed(d, fid);
  if (in && !act && sub == 0) {
    if (lane < 4) d.fflux[4 * fid + lane] = 0.0;
    if (lane == 0) d.gam[fid] = 0.0;
  }
  bool wall = kind == BC_WALL;
  Acc<T> ags[4], ars[4], aden;
  if (act) {
    T *PT = reinterpret_cast<T *>(d.fparT) + (size_t)NFP * fid;
    __align__(16) T parT[NFP];
    load_rec<T, NFP>(PT, parT);
    T snx, sny, sun;
    if (sizeof(T) == 4) { snx = parT[FP_SNX]; sny = parT[FP_SNY]; sun = parT[FP_SUN]; }
    else { snx = (T)d.Sn[2 * fid]; sny = (T)d.Sn[2 * fid + 1]; sun = (T)d.SUn[fid]; }
    T tufx = parT[FP_UFX], tufy = parT[FP_UFY], tlamw = parT[FP_LAMW], tK = (T)d.Keff;
    V2<T> zero = {T(0), T(0)};
    // the equilibrium and reflected parts depend on no f: the whole grid
    // (also on a sharded context, so every shard gets the same totals)
    for (int k = sub * 32 + lane; k < d.nv_all; k += 32 * FCW) {
      T vx = dvxa<T>(d, k), vy = dvya<T>(d, k), w = dwa<T>(d, k);
      T wS = vx * snx + vy * sny - sun;
      T v2 = T(0.5) * (vx * vx + vy * vy);
      T cw = w * wS;
      if (!wall || wS > T(0)) {
        V2<T> I = interface_integral<T>(parT, vx, vy, zero, zero, tK, (T)d.Kint, (T)d.Pr);
        ags[0].add(cw * I.h); ags[1].add(cw * vx * I.h); ags[2].add(cw * vy * I.h);
        ags[3].add(cw * (v2 * I.h + T(0.5) * I.b));
      } else {
        T cx = vx - tufx, cy = vy - tufy;
        T Hw = (tlamw * T(M_1_PI)) * r_exp<T>(-tlamw * (cx * cx + cy * cy));
        T Bw = tK / (T(2) * tlamw) * Hw;
        aden.add(cw * Hw);
        ars[0].add(cw * Hw); ars[1].add(cw * vx * Hw); ars[2].add(cw * vy * Hw);
        ars[3].add(cw * (v2 * Hw + T(0.5) * Bw));
      }
    }
  }
  double tot[9];
  for (int m = 0; m < 4; ++m) { tot[m] = to_double(warp_total(ags[m])); tot[4 + m] = to_double(warp_total(ars[m])); }
  tot[8] = to_double(warp_total(aden));
  if (lane == 0)
    for (int m = 0; m < 9; ++m) part[wl][m] = tot[m];
  __syncthreads();
  if (act && sub == 0 && lane == 0) {
    double acc[9];
    for (int m = 0; m < 9; ++m) {
      acc[m] = part[wl][m];
      for (int j = 1; j < FCW; ++j) acc[m] += part[wl + j][m];
    }
    const double *P = d.fq12 + 2 * (size_t)fid;
    T *PT = reinterpret_cast<T *>(d.fparT) + (size_t)NFP * fid;
    const double *fs = d.fsum + NFS * fid;
    double F[4];
    for (int m = 0; m < 4; ++m)
      F[m] = P[0] * fs[FS_FF + m] + P[1] * fs[FS_WG + m] + acc[m];
    if (wall) {
      double rhow = -F[0] / acc[8];
      PT[FP_RHOW] = (T)rhow;
      for (int m = 0; m < 4; ++m) F[m] += rhow * acc[4 + m];
    }
    {
      __align__(16) T pr[NFP];
      load_rec<T, NFP>(PT, pr);
      Poly2<3, T> ih, ib;
      interface_polys<T>(pr, (T)d.Keff, (T)d.Kint, ih, ib);
      store_polys<T>(PT, ih, ib);
    }
    for (int m = 0; m < 4; ++m) d.fflux[4 * fid + m] = F[m];
  }
}

// The non-wall faces: the equilibrium part of the macro flux from 1D velocity
// moments (exact separable rewrite of the tensor-grid sum), the cubics of the
// interface distribution for the flux pass; faces outside the field get zero
// flux.  FCG lanes a face take the moments, then one warp a face per lane: the
// products of polynomials are the larger part, and eight lanes that each made
// them for their face spent eight times the instructions (FP64 96x48 + 64x16
// cells: 243 us -> 178 with the walls; FP32 256x128 + 128x32: 55 -> 49).
// block: index among their CTAs.
constexpr int FCG = 8;
template <typename T> __device__ __forceinline__ void sep_coef(const Dev &d, int block) {
  constexpr int FPB = FC_THREADS / FCG;          // faces of a CTA, the lanes of a warp
  static_assert(FPB == 32, "one warp finishes the CTA's faces");
  __shared__ T mom[FPB][15];
  const int f0 = block * FPB;
  {
    const int r = threadIdx.x / FCG, sub = threadIdx.x % FCG, fid = f0 + r;
    const bool in = fid < d.nf;
    const int kind = in ? d.face_kind[fid] : BC_OVERSET;
    const bool act = in && kind != BC_OVERSET && kind != BC_WALL && face_needed(d, fid);
    T mx[7], my[7], ux = T(0), uy = T(0), lam = T(0);
    if (act) {
      const T *P = reinterpret_cast<const T *>(d.fparT) + (size_t)NFP * fid;
      ux = P[FP_UX]; uy = P[FP_UY]; lam = P[FP_LAM];
    }
    if (__any_sync(0xffffffffu, act)) {
      face_moments<T, FCG>(d, ux, uy, lam, sub, mx, my);
      if (sub == 0)
#pragma unroll
        for (int a = 0; a < 7; ++a) { mom[r][a] = mx[a]; mom[r][7 + a] = my[a]; }
    }
  }
  __syncthreads();
  if (threadIdx.x >= 32) return;
  const int fid = f0 + threadIdx.x;
  if (fid >= d.nf) return;
  const int kind = d.face_kind[fid];
  double2 *F = reinterpret_cast<double2 *>(d.fflux + 4 * (size_t)fid);
  if (kind == BC_OVERSET || !face_needed(d, fid)) {
    F[0] = F[1] = make_double2(0.0, 0.0);
    d.gam[fid] = 0.0;
    return;
  }
  if (kind == BC_WALL) return;
  T *PT = reinterpret_cast<T *>(d.fparT) + (size_t)NFP * fid;
  __align__(16) T P[FP_IH];
  load_rec<T, FP_IH>(PT, P);
  Poly2<3, T> ih, ib;
  interface_polys<T>(P, (T)d.Keff, (T)d.Kint, ih, ib);
  T o[4];
  face_eq_flux<T>(P, ih, ib, mom[threadIdx.x], mom[threadIdx.x] + 7, o);
  __align__(16) T poly[20];
#pragma unroll
  for (int m = 0; m < 10; ++m) { poly[m] = ih.c[m]; poly[10 + m] = ib.c[m]; }
#pragma unroll
  for (int m = 0; m < 20 * (int)sizeof(T) / 16; ++m)
    reinterpret_cast<float4 *>(PT + FP_IH)[m] = reinterpret_cast<const float4 *>(poly)[m];
  const double2 q = *reinterpret_cast<const double2 *>(d.fq12 + 2 * (size_t)fid);
  const double *fs = d.fsum + NFS * (size_t)fid;
  double v[4];
#pragma unroll
  for (int m = 0; m < 4; ++m) v[m] = q.x * fs[FS_FF + m] + q.y * fs[FS_WG + m] + to_double(o[m]);
  F[0] = make_double2(v[0], v[1]);
  F[1] = make_double2(v[2], v[3]);
}

template <typename T> __global__ void __launch_bounds__(FC_THREADS, sizeof(T) == 4 ? 2 : 1) k_face_coef(Dev d, int wall_blocks) {
  if ((int)blockIdx.x < wall_blocks) wall_coef<T>(d, d.wall_faces, d.nwall);
  else sep_coef<T>(d, (int)blockIdx.x - wall_blocks);
}

// Per-cell sum of the S-weighted macro fluxes (Eq. macroscopicFlux summed
// over the faces); with level_n also the extensive level-n macro term
// TW = Omega^n W^n / dt - F^n / 2 (reading R4).  (The inner iterations sum it
// while they gather the macro sweep's records.)
__global__ void k_cell_macro(Dev d, int level_n) {
  int t = blockIdx.x * blockDim.x + threadIdx.x;
  int c = t >> 2, m = t & 3;
  if (c >= d.nc) return;
  const double F = cell_flux_sum(d, c, m);
  d.Fc[t] = F;
  if (level_n) d.TW[t] = d.vol_old[c] / d.stepc[0] * d.W[t] - 0.5 * F;
}

// Shakhov record in the arithmetic type from W and q (level n).
template <typename T> __global__ void k_cell_params(Dev d) {
  int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= d.nc) return;
  Prim p = primitive(d.W + 4 * c, d.Keff);
  double o[NCP];
  o[CP_RHO] = p.rho; o[CP_UX] = p.ux; o[CP_UY] = p.uy; o[CP_LAM] = p.lam;
  o[CP_QX] = d.q[2 * c]; o[CP_QY] = d.q[2 * c + 1];
  o[CP_ITAU] = 1.0 / collision_time(p.rho, p.lam, d.mu_ref, d.omega);
  write_shrec<T>(d, o, d.vol_old[c], reinterpret_cast<T *>(d.shn) + (size_t)NSH * c);
}

// Step 7 (one warp per cell): W^{s+1} = W' + sum V Psi (f^{s+1} - g(W')),
// heat flux about V' (reading R7); flags non-physical states.
//
// FP32: streaming f.  FP64: its pipe (some 15 cycles a warp instruction and
// SM), so the exponential of g (thirty of them) splits into a factor per column
// and one per row, tabulated first by the warp, and the sums share their
// products (40 -> 21 a velocity; 96x48 + 64x16 cells, 1024 velocities: 454 -> 272
// us).  A velocity grid of more than MOM_TAB columns and rows keeps one
// exponential a velocity.
constexpr int MOM_THREADS = 64, MOM_TAB = 256;
template <typename T, int FB> __global__ void k_moments(Dev d) {
  int c = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  int lane = threadIdx.x & 31;
  if (c >= d.nc) return;
  if (d.status[c] != ST_FIELD) return;
  const T *sr = reinterpret_cast<const T *>(d.shp) + (size_t)NSH * c;
  T hpre = sr[SH_HPRE], ux = sr[SH_UX], uy = sr[SH_UY], lam = sr[SH_LAM];
  T bfac = (T)d.Keff * sr[SH_IL];
  Acc<T> a[6];
  typedef typename Vec2<T>::type T2;
  constexpr int NB = 4;                     // loads of a lane in flight per batch
  constexpr bool SEP = sizeof(T) == 8;
  __shared__ T tab[SEP ? MOM_THREADS / 32 : 1][SEP ? MOM_TAB : 1];
  const int rows = SEP ? d.nv / d.nvx : 0;
  const bool sep = SEP && d.nvx + rows <= MOM_TAB;
  if (sep) {
    T *ex = tab[(threadIdx.x >> 5) % (SEP ? MOM_THREADS / 32 : 1)], *ey = ex + d.nvx;
    for (int i = lane; i < d.nvx + rows; i += 32) {
      const T u = i < d.nvx ? dvx<T>(d, i) - ux : dvy<T>(d, (i - d.nvx) * d.nvx) - uy;
      ex[i] = (i < d.nvx ? hpre : T(1)) * r_exp<T>(-lam * u * u);
    }
    __syncwarp();
    for (int kb = lane; kb < d.nv; kb += 32 * NB) {
      T2 fb[NB];
#pragma unroll
      for (int u = 0; u < NB; ++u) {
        int k = kb + 32 * u;
        fb[u] = k < d.nv ? ldF<T, FB>(d, (size_t)c * d.nvp + k) : T2{T(0), T(0)};
      }
      T p[6] = {T(0), T(0), T(0), T(0), T(0), T(0)};
#pragma unroll
      for (int u = 0; u < NB; ++u) {
        const int k = kb + 32 * u;
        if (k >= d.nv) break;
        const int iy = k / d.nvx, ix = k - iy * d.nvx;
        const T vx = dvx<T>(d, k), vy = dvy<T>(d, k), w = dw<T>(d, k), hw = T(0.5) * w;
        const T h = fb[u].x, b = fb[u].y, H = ex[ix] * ey[iy];
        const T wd = w * (h - H);
        p[0] += wd;
        p[1] += vx * wd;
        p[2] += vy * wd;
        p[3] += T(0.5) * (vx * vx + vy * vy) * wd + hw * (b - bfac * H);
        const T cx = vx - ux, cy = vy - uy;
        const T e = hw * ((cx * cx + cy * cy) * h + b);
        p[4] += cx * e;
        p[5] += cy * e;
      }
#pragma unroll
      for (int m = 0; m < 6; ++m) a[m].add(p[m]);
    }
  }
  for (int kb = sep ? d.nv : lane; kb < d.nv; kb += 32 * NB) {
    T2 fb[NB];
#pragma unroll
    for (int u = 0; u < NB; ++u) {
      int k = kb + 32 * u;
      fb[u] = k < d.nv ? ldF<T, FB>(d, (size_t)c * d.nvp + k) : T2{T(0), T(0)};
    }
    // the batch's terms are summed plainly, the batch sums compensated
    T p[6] = {T(0), T(0), T(0), T(0), T(0), T(0)};
#pragma unroll
    for (int u = 0; u < NB; ++u) {
      int k = kb + 32 * u;
      if (k >= d.nv) break;
      T2 fv = fb[u];
      T vx = dvx<T>(d, k), vy = dvy<T>(d, k), w = dw<T>(d, k);
      V2<T> g = maxwellian_pre<T>(hpre, ux, uy, lam, bfac, vx, vy);
      T h = fv.x, b = fv.y;
      T dh = h - g.h, db = b - g.b;
      T v2 = T(0.5) * (vx * vx + vy * vy);
      p[0] += w * dh;
      p[1] += w * vx * dh;
      p[2] += w * vy * dh;
      p[3] += w * (v2 * dh + T(0.5) * db);
      T cx = vx - ux, cy = vy - uy;
      T e = (cx * cx + cy * cy) * h + b;
      p[4] += T(0.5) * w * cx * e;
      p[5] += T(0.5) * w * cy * e;
    }
#pragma unroll
    for (int m = 0; m < 6; ++m) a[m].add(p[m]);
  }
  // lane m < 6 stores component m (W' + sum for W, the sum for q); lane 0
  // then checks the new state for rho > 0 and a positive internal energy
  // (2 rho (rho E) - |rho V|^2 > 0), i.e. rho and lambda positive and finite
  auto tot = [&](int m) { return to_double(warp_total(a[m])); };
  double t0 = tot(0), t1 = tot(1), t2 = tot(2), t3 = tot(3), t4 = tot(4), t5 = tot(5);
  double mine = lane == 0 ? t0 : lane == 1 ? t1 : lane == 2 ? t2 : lane == 3 ? t3 : lane == 4 ? t4 : t5;
  if (d.shard) {        // this shard's sums; k_moments_finish completes them after the exchange
    if (lane < 6) d.msum[6 * c + lane] = mine;
    return;
  }
  double wn = 0.0;
  if (lane < 4) {
    wn = d.Wp[4 * c + lane] + mine;
    d.W[4 * c + lane] = wn;
  } else if (lane < 6) {
    d.q[2 * c + lane - 4] = mine;
  }
  double w0 = __shfl_sync(0xffffffffu, wn, 0), w1 = __shfl_sync(0xffffffffu, wn, 1);
  double w2 = __shfl_sync(0xffffffffu, wn, 2), w3 = __shfl_sync(0xffffffffu, wn, 3);
  if (lane == 0) {
    double ei2 = 2.0 * w0 * w3 - (w1 * w1 + w2 * w2);
    if (!(w0 > 0.0) || !(ei2 > 0.0) || !isfinite(w0) || !isfinite(ei2))
      atomicOr(d.err, EF_NONPHYSICAL);
  }
}

// Step 7 of a sharded step after the exchange: msum holds the sums over the
// whole velocity grid; W = W' + the fix, q the heat flux, checked as above.
__global__ void k_moments_finish(Dev d) {
  int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= d.nc || d.status[c] != ST_FIELD) return;
  const double *m = d.msum + 6 * (size_t)c;
  double w[4];
  for (int i = 0; i < 4; ++i) {
    w[i] = d.Wp[4 * c + i] + m[i];
    d.W[4 * c + i] = w[i];
  }
  d.q[2 * c] = m[4];
  d.q[2 * c + 1] = m[5];
  double ei2 = 2.0 * w[0] * w[3] - (w[1] * w[1] + w[2] * w[2]);
  if (!(w[0] > 0.0) || !(ei2 > 0.0) || !isfinite(w[0]) || !isfinite(ei2)) atomicOr(d.err, EF_NONPHYSICAL);
}

// Initial state: f = reduced Maxwellian of the primitive field, W, and q from f.
template <typename T> __global__ void k_init_state(Dev d, const double *prim) {
  int c = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  int lane = threadIdx.x & 31;
  if (c >= d.nc) return;
  double rho = prim[4 * c], ux = prim[4 * c + 1], uy = prim[4 * c + 2], T0 = prim[4 * c + 3];
  double lam = 1.0 / (2.0 * T0);
  for (int k = lane; k < d.nvp; k += 32) {
    if (k >= d.nv) { stF<T>(d, (size_t)c * d.nvp + k, T(0), T(0)); continue; }
    V2<double> g = maxwellian<double>(rho, ux, uy, lam, d.vx[k], d.vy[k], (double)d.Keff);
    stF<T>(d, (size_t)c * d.nvp + k, (T)g.h, (T)g.b);
  }
  // q from the stored values over the whole grid (a shard recomputes the
  // other shards' Maxwellian values, so no exchange is needed)
  double qx = 0, qy = 0;
  for (int k = lane; k < d.nv_all; k += 32) {
    V2<double> g = maxwellian<double>(rho, ux, uy, lam, d.vxa[k], d.vya[k], (double)d.Keff);
    T h = (T)g.h, b = (T)g.b;
    double cx = d.vxa[k] - ux, cy = d.vya[k] - uy;
    double e = (cx * cx + cy * cy) * (double)h + (double)b;
    qx += 0.5 * d.wa[k] * cx * e;
    qy += 0.5 * d.wa[k] * cy * e;
  }
  qx = warp_sum(qx);
  qy = warp_sum(qy);
  if (lane == 0) {
    double W[4];
    conservative(rho, ux, uy, lam, d.Keff, W);
    for (int m = 0; m < 4; ++m) d.W[4 * c + m] = W[m];
    d.q[2 * c] = qx;
    d.q[2 * c + 1] = qy;
  }
}

// Sum of S * wall macro flux per block: one CTA per block, a strided partial
// sum per thread and a fixed-shape tree, so the order (and the result) is
// the same on every call.  It walks the list of wall faces: over all faces (74240
// of the 256x128 + 128x32 mesh) the loads of one CTA took 190 us, over its wall
// faces under 10.
constexpr int WL_THREADS = 256;
__global__ void __launch_bounds__(WL_THREADS) k_wall_loads(Dev d) {
  __shared__ double part[4][WL_THREADS];
  int b = blockIdx.x;
  double s[4] = {0, 0, 0, 0};
  for (int i = threadIdx.x; i < d.nwall; i += WL_THREADS) {
    const int f = d.wall_faces[i];
    if (d.face_block[f] != b) continue;
    for (int m = 0; m < 4; ++m) s[m] += d.fflux[4 * f + m];
  }
  for (int m = 0; m < 4; ++m) part[m][threadIdx.x] = s[m];
  __syncthreads();
  for (int w = WL_THREADS / 2; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w)
      for (int m = 0; m < 4; ++m) part[m][threadIdx.x] += part[m][threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x < 4) d.wall_loads[4 * b + threadIdx.x] = part[threadIdx.x][0];
}

// Torque about the point ctr[b] of each block's wall force: sum over its
// wall faces of (x_f - ctr) x (S F_x, S F_y) of the last flux evaluation
// (mid-time face centres), same fixed reduction shape as k_wall_loads.
__global__ void __launch_bounds__(WL_THREADS) k_wall_torque(Dev d, const double *ctr, double *out) {
  __shared__ double part[WL_THREADS];
  int b = blockIdx.x;
  double cx = ctr[2 * b], cy = ctr[2 * b + 1], s = 0.0;
  for (int i = threadIdx.x; i < d.nwall; i += WL_THREADS) {
    const int f = d.wall_faces[i];
    if (d.face_block[f] != b) continue;
    double rx = d.xf[2 * f] - cx, ry = d.xf[2 * f + 1] - cy;
    s += rx * d.fflux[4 * f + 2] - ry * d.fflux[4 * f + 1];
  }
  part[threadIdx.x] = s;
  __syncthreads();
  for (int w = WL_THREADS / 2; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w) part[threadIdx.x] += part[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) out[b] = part[0];
}

// Copy f between the storage type and FP64 (get/set state).
template <typename T> __global__ void k_f_to_double(Dev d, double *out) {
  size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  size_t n = (size_t)d.nc * d.nv;
  if (t >= n) return;
  int c = (int)(t / d.nv), k = (int)(t % d.nv);
  auto v = ldF<T>(d, (size_t)c * d.nvp + k);
  out[2 * t] = (double)v.x;
  out[2 * t + 1] = (double)v.y;
}
template <typename T> __global__ void k_f_from_double(Dev d, const double *in) {
  size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  size_t n = (size_t)d.nc * d.nv;
  if (t >= n) return;
  int c = (int)(t / d.nv), k = (int)(t % d.nv);
  stF<T>(d, (size_t)c * d.nvp + k, (T)in[2 * t], (T)in[2 * t + 1]);
}

// ------------------------------------------------------- launch wrappers
static inline int nblk(size_t n, int b) { return (int)((n + b - 1) / b); }

// ---------------------------------------------------------------- metrics
// Per-block sums in a fixed order (each thread strides over its items, then
// a shared-memory tree), finished by one block in the same way: the metrics
// are the same bits on every run of a given mesh and launch shape.
__device__ __forceinline__ void met_block_sum(double *sh, double v, double *out) {
  sh[threadIdx.x] = v;
  __syncthreads();
  for (int h = MET_THREADS / 2; h > 0; h >>= 1) {
    if (threadIdx.x < h) sh[threadIdx.x] += sh[threadIdx.x + h];
    __syncthreads();
  }
  if (threadIdx.x == 0) *out = sh[0];
  __syncthreads();
}

// |R|^2 of Step 4: R = T_W - Omega^{n+1} W / dt - F / 2 (the right-hand side
// of the macro LU-SGS, before W changes in this iteration)
__global__ void __launch_bounds__(MET_THREADS) k_met_macro(Dev d) {
  __shared__ double sh[MET_THREADS];
  double idt = 1.0 / d.stepc[0], acc = 0.0;
  for (int c = blockIdx.x * MET_THREADS + threadIdx.x; c < d.nc; c += MET_BLOCKS * MET_THREADS) {
    if (!(d.cmask[c] & 1)) continue;
    double vol = d.vol_new[c];
    for (int m = 0; m < 4; ++m) {
      double r = d.TW[4 * c + m] - vol * idt * d.W[4 * c + m] - 0.5 * d.Fc[4 * c + m];
      acc += r * r;
    }
  }
  met_block_sum(sh, acc, d.mpart + MET_R2 * MET_BLOCKS + blockIdx.x);
}

// |r|^2 of Step 5 over the solved cells and this context's velocities
template <typename T> __global__ void __launch_bounds__(MET_THREADS) k_met_micro(Dev d) {
  __shared__ double sh[MET_THREADS];
  double acc = 0.0;
  size_t n = (size_t)d.nc * d.nvp;
  for (size_t t = (size_t)blockIdx.x * MET_THREADS + threadIdx.x; t < n; t += (size_t)MET_BLOCKS * MET_THREADS) {
    int c = (int)(t / d.nvp), k = (int)(t - (size_t)c * d.nvp);
    if (k >= d.nv || !(d.cmask[c] & 1)) continue;
    typename Vec2<T>::type r = ldf<T>(d.dfs, t);
    acc += (double)r.x * (double)r.x + (double)r.y * (double)r.y;
  }
  met_block_sum(sh, acc, d.mpart + MET_RMICRO2 * MET_BLOCKS + blockIdx.x);
}

// |W^{s+1} - W'|^2 (Step 7) and the totals of Omega^{n+1} W over the field
__global__ void __launch_bounds__(MET_THREADS) k_met_fix(Dev d) {
  __shared__ double sh[MET_THREADS];
  double acc[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
  for (int c = blockIdx.x * MET_THREADS + threadIdx.x; c < d.nc; c += MET_BLOCKS * MET_THREADS) {
    if (d.status[c] != ST_FIELD) continue;
    double vol = d.vol_new[c];
    for (int m = 0; m < 4; ++m) {
      double w = d.W[4 * c + m], e = w - d.Wp[4 * c + m];
      acc[0] += e * e;
      acc[1 + m] += vol * w;
    }
  }
  for (int q = 0; q < 5; ++q) met_block_sum(sh, acc[q], d.mpart + (MET_FIX2 + q) * MET_BLOCKS + blockIdx.x);
}

__global__ void __launch_bounds__(MET_THREADS) k_met_final(Dev d) {
  __shared__ double sh[MET_THREADS];
  for (int q = 0; q < MET_NQ; ++q) {
    double acc = 0.0;
    for (int b = threadIdx.x; b < MET_BLOCKS; b += MET_THREADS) acc += d.mpart[q * MET_BLOCKS + b];
    met_block_sum(sh, acc, d.mout + q);
  }
}

void launch_metrics(const Dev &d, cudaStream_t s, int stage, int fp32) {
  if (stage == 0) k_met_macro<<<MET_BLOCKS, MET_THREADS, 0, s>>>(d);
  else if (stage == 1) {
    if (fp32) k_met_micro<float><<<MET_BLOCKS, MET_THREADS, 0, s>>>(d);
    else k_met_micro<double><<<MET_BLOCKS, MET_THREADS, 0, s>>>(d);
  } else {
    k_met_fix<<<MET_BLOCKS, MET_THREADS, 0, s>>>(d);
    k_met_final<<<1, MET_THREADS, 0, s>>>(d);
  }
}

void launch_move_nodes(const Dev &d, cudaStream_t s) { k_move_nodes<<<nblk(d.nn, 256), 256, 0, s>>>(d); }

// Small host->device uploads (motion maps, search-bin boxes) travel as kernel
// arguments: the bytes are captured when the launch is issued, so the upload
// neither waits on the stream nor needs pinned staging, and it can be
// captured in a graph.
struct UploadBlob {
  unsigned char b[2048];
};
__global__ void k_upload(unsigned char *dst, UploadBlob blob, int n) {
  for (int i = threadIdx.x; i < n; i += blockDim.x) dst[i] = blob.b[i];
}
int launch_upload(void *dst, const void *src, size_t n, cudaStream_t s) {
  const unsigned char *p = static_cast<const unsigned char *>(src);
  unsigned char *q = static_cast<unsigned char *>(dst);
  int launches = 0;
  while (n > 0) {
    size_t m = n < sizeof(UploadBlob) ? n : sizeof(UploadBlob);
    UploadBlob blob;
    memcpy(blob.b, p, m);
    k_upload<<<1, 256, 0, s>>>(q, blob, (int)m);
    p += m;
    q += m;
    n -= m;
    ++launches;
  }
  return launches;
}
void launch_geometry(const Dev &d, cudaStream_t s, int fp32) {
  const int faces = nblk(d.nf, GEO_THREADS), grid = faces + nblk(d.nc, GEO_THREADS);
  if (fp32) k_geom<float><<<grid, GEO_THREADS, 0, s>>>(d, faces);
  else k_geom<double><<<grid, GEO_THREADS, 0, s>>>(d, faces);
  if (fp32) k_geo_records<float><<<grid, GEO_THREADS, 0, s>>>(d, faces);
  else k_geo_records<double><<<grid, GEO_THREADS, 0, s>>>(d, faces);
}
void launch_slope_geo(const Dev &d, cudaStream_t s) { k_slope_geo<<<nblk(d.nc, 128), 128, 0, s>>>(d); }

void launch_ghost_gradW(const Dev &d, cudaStream_t s) {
  k_ghost<<<nblk(d.nf, 256), 256, 0, s>>>(d);
  launch_gradW(d, s);
}
void launch_gradW(const Dev &d, cudaStream_t s) {
  k_gradW<<<nblk(4 * (size_t)d.nc, GW_THREADS), GW_THREADS, 0, s>>>(d);
}
template <typename T> static void face_coef(const Dev &d, cudaStream_t s) {
  if (d.nsplit > 1) k_face_scalar<T, true><<<nblk(d.nf, FSC), 128, 0, s>>>(d);
  else k_face_scalar<T, false><<<nblk(d.nf, FSC), 64, 0, s>>>(d);
  const int walls = nblk((size_t)d.nwall * 32 * FCW, FC_THREADS);
  k_face_coef<T><<<walls + nblk((size_t)d.nf * FCG, FC_THREADS), FC_THREADS, 0, s>>>(d, walls);
}
void launch_face_coef(const Dev &d, cudaStream_t s, int fp32) {
  if (fp32) face_coef<float>(d, s);
  else face_coef<double>(d, s);
}
void launch_cell_macro(const Dev &d, cudaStream_t s, int level_n) {
  k_cell_macro<<<nblk(4 * (size_t)d.nc, 128), 128, 0, s>>>(d, level_n);
}
void launch_cell_params(const Dev &d, cudaStream_t s, int fp32) {
  if (fp32) k_cell_params<float><<<nblk(d.nc, 32), 32, 0, s>>>(d);
  else k_cell_params<double><<<nblk(d.nc, 32), 32, 0, s>>>(d);
}
void launch_moments_finish(const Dev &d, cudaStream_t s) { k_moments_finish<<<nblk(d.nc, 256), 256, 0, s>>>(d); }
// Two cells (warps) a CTA: small CTAs fit beside the velocity reduction's
// two CTAs an SM, with which this Step 7 runs concurrently.
void launch_moments(const Dev &d, cudaStream_t s, int fp32) {
  int g = nblk((size_t)d.nc * 32, MOM_THREADS);
  if (fp32 && d.fbf) k_moments<float, 1><<<g, MOM_THREADS, 0, s>>>(d);
  else if (fp32) k_moments<float, 0><<<g, MOM_THREADS, 0, s>>>(d);
  else k_moments<double, 0><<<g, MOM_THREADS, 0, s>>>(d);
}
void launch_init_state(const Dev &d, cudaStream_t s, const double *prim, int fp32) {
  if (fp32) k_init_state<float><<<nblk((size_t)d.nc * 32, 256), 256, 0, s>>>(d, prim);
  else k_init_state<double><<<nblk((size_t)d.nc * 32, 256), 256, 0, s>>>(d, prim);
}
void launch_wall_loads(const Dev &d, cudaStream_t s) { k_wall_loads<<<d.nblocks, WL_THREADS, 0, s>>>(d); }
void launch_wall_torque(const Dev &d, cudaStream_t s, const double *ctr, double *out) {
  k_wall_torque<<<d.nblocks, WL_THREADS, 0, s>>>(d, ctr, out);
}
void launch_f_convert(const Dev &d, cudaStream_t s, double *out, const double *in, int fp32) {
  size_t n = (size_t)d.nc * d.nv;
  if (out) {
    if (fp32) k_f_to_double<float><<<nblk(n, 256), 256, 0, s>>>(d, out);
    else k_f_to_double<double><<<nblk(n, 256), 256, 0, s>>>(d, out);
  } else {
    if (fp32) k_f_from_double<float><<<nblk(n, 256), 256, 0, s>>>(d, in);
    else k_f_from_double<double><<<nblk(n, 256), 256, 0, s>>>(d, in);
  }
}

}  // namespace ugks
