// ugks_internal.cuh -- device-side context of libugks and what its kernels
// share: record layouts, loads and stores of f in its storage type, pairs in
// packed instructions, asynchronous copies, the error-free sums of the velocity
// reductions, and the polynomials of the interface equilibrium (Eq.
// fullSolution).
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>
#include "ugks_math.cuh"

namespace ugks {

enum { BC_NONE = 0, BC_WALL = 1, BC_FARFIELD = 2, BC_OUTFLOW = 3, BC_OVERSET = 4 };
enum { ST_FIELD = 0, ST_RECEPTOR = 1, ST_HOLE = 2 };
enum { NB_CELL = 0, NB_GHOST = 1, NB_NONE = 2 };
// slope case per logical direction: none, only minus side, only plus side, both
enum { SL_NONE = 0, SL_M = 1, SL_P = 2, SL_BOTH = 3 };
// face sums of the velocity-reduction pass
enum { FS_W0 = 0, FS_FF = 4, FS_WG = 8, NFS = 12 };
// error flags
enum { EF_GEOMETRY = 1, EF_NONPHYSICAL = 2, EF_BINS = 4, EF_TIMEOUT = 8, EF_ORPHAN = 16, EF_CAPACITY = 32 };

template <typename T> struct Vec2;
template <> struct Vec2<double> { typedef double2 type; };
template <> struct Vec2<float> { typedef float2 type; };

// Everything a kernel needs: sizes, constants and borrowed device pointers
// into the caller's workspace.  Passed by value.
struct Dev {
  int nc, nf, nn, nv, nvp, nblocks;
  int Keff, Kint;
  double Pr, omega, mu_ref, cfl_s, cfl_pseudo;
  double c2fac;              // gamma (gamma - 1): square of the sound speed over the internal energy
  double Winf[4];
  double dt, idt;            // physical step and its inverse
  float idt_f;
  // velocity space (double and float copies), length nvp (padding weight 0)
  const double *vx, *vy, *w;
  const float *vxf, *vyf, *wf;
  int nvx, nvy;              // tensor grid: k = iy nvx + ix, w_k = wy1(iy) wx1(ix); nvy of the whole grid
  const float *wx1f, *wy1f;  // 1D trapezoid weights (whole grid)
  const float *vy1f;         // 1D y nodes of the whole grid
  const double *vx1, *vy1, *wx1, *wy1;   // 1D nodes and trapezoid weights of the whole grid (FP64)
  // velocity sharding: this context holds the rows iy0 <= iy < iy0 + nv / nvx
  // of the grid; the arrays above (vx, vy, w and copies) are its own rows, the
  // ones below the whole grid (the same arrays when not sharded)
  int shard, iy0, nv_all;
  const double *vxa, *vya, *wa;
  const float *vxaf, *vyaf, *waf;
  double *msum;              // nc*6: partial moment sums of a sharded step (W fix 4, q 2)
  // static topology
  const int *cell_nodes;     // nc*4
  const int *cell_faces;     // nc*4 (IM, IP, JM, JP)
  const int8_t *cell_sgn;    // nc*4, +1 if the cell is the face's L side
  const int *nb_kind;        // nc*4
  const int *nb_id;          // nc*4 cell id or ghost face id
  const int8_t *nb_shift;    // nc*4 period multiplier
  const int *cell_row;       // nc*2 node ids (0,j), (ni,j)
  const int *cell_block;     // nc
  const int *node_block;     // nn
  const int *face_L, *face_R, *face_a, *face_b, *face_kind, *face_block;
  const int8_t *face_shiftL;
  const double *face_Tw;
  // per-step geometry
  const double *X_ref;
  double *X_old, *X_new;     // nn*2
  float2 *Xf;                // nn: X_new rounded to nearest float (overset filters)
  float4 *cbb;               // nc: cell bounding box at t^{n+1}, rounded outward
  double *vol_old, *vol_new; // nc
  double *xc, *xc_new;       // nc*2
  double *period;            // nc*2
  double *dts;               // nc
  double *idtau;             // nc 1 / pseudo-time step = cfl_s / (cfl_pseudo dts)
  double *Sn, *S, *nrm, *xf, *Uf, *SUn, *Un;   // nf*2 / nf
  int *slope_flags;          // nc: 2 bits per direction (i: bits 0-1, j: 2-3)
  int *cmask;                // nc: bit 0 solved cell, bit 1+s solved neighbour across slot s
  double *jinv;              // nc*4 inverse of [[x_xi, y_xi],[x_eta, y_eta]]
  float4 *jinvf;             // nc: the same in FP32
  void *fgeo;                // nf*NFG face geometry record (arithmetic type)
  void *srec;                // nc*NSR sweep record (layout at NSR)
  int *mrec_off;             // nblocks+1: first macro-sweep record of each block (padded diagonals x rows)
  int mpad;                  // diagonals of padding on both sides of a block's macro-sweep records
  double vbox[4];            // velocity box (vx_min, vx_max, vy_min, vy_max)
  double *affine;            // nblocks*6
  // state
  void *f;                   // nc*nvp (h, b) pairs in the storage type
  double *W, *q;             // nc*4, nc*2
  int *status;               // nc
  // work
  void *Tn, *dfs;            // nc*nvp pairs: level-n term, forward-sweep result
  void *Dbuf;                // nc*nvp pairs: flux divergence of the inner iteration
  void *fval;                // ntiles*nvp*NSLOT 4-vectors: upwind face value (h, b) and w.grad f (h, b) of the face pass
  const double *stepc;       // [4]: dt, 1/dt, (float)(1/dt) as a float, of the pending step, on the device (the step's
                             // kernels read it there, so a captured step graph stays valid when dt changes)
  double *TW;                // nc*4 extensive level-n macro term
  double *Fc;                // nc*4 macro flux divergence of the last flux
  void *mrec;                // macro-sweep records (arithmetic type, layout in ugks_macro.cu)
  double *Wp;                // nc*4 macro predictor W'
  void *shp, *shn;           // nc*NSH Shakhov records in the arithmetic type (predictor / level n)
  double *gradW;             // nc*8
  double *ghostW;            // nf*4
  double *fsum;              // nf*NFS
  void *fpart;               // nsplit*NFS*nf (sum, error) pairs of the face reduction's CTAs (nsplit > 1)
  int nsplit;                // CTAs that share a tile's velocity chunks in the face kernels
  int flux_pair;             // FP32 flux pass, joint form: two ranges of columns in turn
  double *fq12;              // nf*2 time integrals q1 / dts, q2 / dts of the faces
  void *fparT;               // nf*NFP in the arithmetic type
  double *fflux;             // nf*4 S * macro flux (L -> R / outward)
  double *gam;               // nf spectral radius Gamma
  double *wall_loads;        // nblocks*4
  double *torque_io;         // nblocks*3: torque centres (2 per block), torques
  int *wall_faces;           // ids of the wall faces, ascending
  int nwall;
  // overset
  int *node_active;          // nn
  int *cls;                  // nc scratch classification
  int *donors;               // nc*5
  double *dwgt;              // nc*5
  int fbf;                   // f stored as bf16 pairs (FP32 arithmetic)
  int *rec_list;             // receptor cells, ascending (compacted on the device)
  int *fresh_list;           // cells uncovered by the motion, ascending
  int *conn_cnt;             // 8 counters: receptors, fresh, field, hole, orphans
  int4 *conn_chunk;          // per 1024-cell chunk: receptors, fresh, field, other
  int cap_interp;            // capacity of the lists' interpolation staging
  void *itmp;                // interpolation staging: cap_interp*nvp pairs
  double *itmpW;             // ... *6 doubles
  int *wall_seg;             // segments: node id pairs, grouped per block
  float4 *segf;              // float endpoints of each wall segment (assembly filters)
  int nseg;
  int *wall_seg_off;         // nblocks+1
  int *body_ring;            // body polygon node ids, grouped per block
  int *body_ring_off;        // nblocks+1
  float4 *body_bb;           // nblocks: outward-rounded float box of the body polygon
  float4 *bin_bb;            // per block: box of its bins, rounded outward
  const int *cell_off;       // nblocks+1 (device copy)
  const int *node_off;       // nblocks+1
  const int *blk_info;       // nblocks*8: ni, nj, periodic, priority, n_fringe, n_gap, bc-overset mask, body?
  // overset search bins (per block uniform grid, CSR of cell ids)
  double *bin_geo;           // nblocks*4: x0, y0, 1/hx, 1/hy
  int *bin_dim;              // nblocks*3: nbx, nby, first bin
  int *bin_cnt, *bin_start;  // nbins, nbins+1
  int *bin_items;            // bin_cap
  int2 *bin_rng;             // nc: a cell's first and last bin, x | y << 16
  int *node_todo;            // nn: nodes of the second classification pass
  int *node_todo_n;          // their count
  int nbins, bin_cap;
  const int *tiles;          // ntiles*3: block, i0, j0 of the 8x8 cell tiles
  int ntiles;
  int *err;                  // error flags
  int wait_polls;            // bounded waits (sweeps): polls before giving up (EF_TIMEOUT)
  double *mpart;             // MET_NQ*MET_BLOCKS per-block partial sums of the step metrics
  double *mout;              // MET_NQ step metrics of the last metered step
};

// Step metrics (sums over the solved cells, fixed-order reductions):
// squared norms of the macro residual R and the micro residual r of the last
// inner iteration, of the Step-7 moment fix W^{s+1} - W', and the totals of
// Omega^{n+1} W.
enum { MET_R2 = 0, MET_RMICRO2 = 1, MET_FIX2 = 2, MET_TOT = 3, MET_NQ = 7 };
constexpr int MET_BLOCKS = 304, MET_THREADS = 256;

// Polls of a bounded wait before it gives up.
constexpr int kWaitPolls = 1 << 21;

// face geometry record / per-cell sweep record
enum { FG_SNX = 0, FG_SNY, FG_SUN, FG_UFX, FG_UFY, FG_DXLX, FG_DXLY, FG_DXRX, FG_DXRY, NFG = 12 };
// sweep record: half the outward S n_x, S n_y, S U.n of the four face slots,
// the i and the j faces in pairs ((n_x i-low, i-high), (n_y ..), (U.n ..), then j),
// and the micro-sweep diagonal base at SR_DBASE, zero for a cell that is not
// solved; 16 values so a record is a whole number of 16-byte chunks
enum { SR_DBASE = 12, NSR = 16 };
__host__ __device__ constexpr int sr_at(int comp, int slot) { return 6 * (slot >> 1) + 2 * comp + (slot & 1); }

// per-cell parameter record (from W' or W^n)
enum { CP_RHO = 0, CP_UX, CP_UY, CP_LAM, CP_QX, CP_QY, CP_ITAU, CP_DBASE, NCP = 8 };

// float -> double on the integer pipes, from the IEEE 754 layouts (sign;
// exponent rebiased by 1023 - 127; 23-bit fraction shifted into the 52-bit
// one): exact for normal numbers, zero and subnormals give signed zero,
// infinities and NaNs are kept.  The FP64 pipe of this GPU retires a warp
// instruction in tens of cycles, so per-face and per-cell conversions go
// through here.
__device__ __forceinline__ double f2d_bits(float x) {
  unsigned u = __float_as_uint(x);
  unsigned sign = u & 0x80000000u, e = (u >> 23) & 0xffu, m = u & 0x7fffffu;
  unsigned hi, lo;
  if (e == 0u) { hi = sign; lo = 0u; }
  else if (e == 0xffu) { hi = sign | 0x7ff00000u | (m >> 3); lo = (m & 7u) << 29; }
  else { hi = sign | ((e + 896u) << 20) | (m >> 3); lo = (m & 7u) << 29; }
  return __hiloint2double((int)hi, (int)lo);
}
__device__ __forceinline__ double to_double(double x) { return x; }
__device__ __forceinline__ double to_double(float x) { return f2d_bits(x); }

// error-free sum (Knuth): s + e = a + b exactly
__device__ __forceinline__ void two_sum(float a, float b, float &s, float &e) {
  s = a + b;
  float bb = s - a;
  e = (a - (s - bb)) + (b - bb);
}
// Face sums of the velocity reduction, (sum, error) pairs on the FP32 path:
// (h, l) += (h2, l2), and the finished value.
__device__ __forceinline__ void face_sum_add(float &h, float &l, float h2, float l2) {
  float s, e;
  two_sum(h, h2, s, e);
  h = s;
  l = (l + e) + l2;
}
__device__ __forceinline__ void face_sum_add(double &h, double &, double h2, double) { h += h2; }
__device__ __forceinline__ double face_sum_value(float h, float l) { return to_double(h) + to_double(l); }
__device__ __forceinline__ double face_sum_value(double h, double) { return h; }

// Component m of a cell's sum of S-weighted macro fluxes
__device__ __forceinline__ double cell_flux_sum(const Dev &d, int c, int m) {
  const int4 f = *reinterpret_cast<const int4 *>(d.cell_faces + 4 * c);
  const char4 g = *reinterpret_cast<const char4 *>(d.cell_sgn + 4 * c);
  double F = (double)g.x * d.fflux[4 * f.x + m];
  F += (double)g.y * d.fflux[4 * f.y + m];
  F += (double)g.z * d.fflux[4 * f.z + m];
  F += (double)g.w * d.fflux[4 * f.w + m];
  return F;
}

// Shakhov record in the arithmetic type from a cell record (double)
// and the finished 1 / (2 lam) and heat flux prefactor
template <typename T>
__device__ __forceinline__ void write_shrec(const Dev &d, const double *o, double il, double pref, double vol, T *r) {
  __align__(16) T v[NSH] = {};
  v[SH_HPRE] = (T)(o[CP_RHO] * o[CP_LAM] * M_1_PI);
  v[SH_UX] = (T)o[CP_UX];
  v[SH_UY] = (T)o[CP_UY];
  v[SH_LAM] = (T)o[CP_LAM];
  v[SH_QX] = (T)o[CP_QX];
  v[SH_QY] = (T)o[CP_QY];
  v[SH_PREF] = (T)pref;
  v[SH_IL] = (T)il;
  v[SH_ITAU] = (T)o[CP_ITAU];
  v[SH_VOL] = (T)vol;
  static_assert(NSH * sizeof(T) % 8 == 0, "record size");
#pragma unroll
  for (int m = 0; m < (int)(NSH * sizeof(T) / 8); ++m) reinterpret_cast<float2 *>(r)[m] = reinterpret_cast<float2 *>(v)[m];
}
template <typename T>
__device__ __forceinline__ void write_shrec(const Dev &d, const double *o, double vol, T *r) {
  write_shrec<T>(d, o, 1.0 / (2.0 * o[CP_LAM]), 4.0 * (1.0 - d.Pr) * o[CP_LAM] * o[CP_LAM] / (5.0 * o[CP_RHO]), vol, r);
}

template <typename T>
__device__ __forceinline__ typename Vec2<T>::type ldf(const void *base, size_t idx) {
  return reinterpret_cast<const typename Vec2<T>::type *>(base)[idx];
}
template <typename T>
__device__ __forceinline__ void stf(void *base, size_t idx, T h, T b) {
  typename Vec2<T>::type v;
  v.x = h;
  v.y = b;
  reinterpret_cast<typename Vec2<T>::type *>(base)[idx] = v;
}

// Pairs (h, b) of the arithmetic type.  FP32 pairs sit in one 64-bit register
// pair and take the packed FP32 instructions (add, multiply, fused
// multiply-add on both halves, each rounded as the scalar one): the velocity
// loops are bound by instruction issue, and h and b go through the same
// arithmetic almost everywhere.
struct alignas(8) PairF { unsigned long long v; };
struct alignas(16) PairD { double x, y; };
template <typename T> struct PairOf;
template <> struct PairOf<float> { typedef PairF type; };
template <> struct PairOf<double> { typedef PairD type; };
__device__ __forceinline__ PairF pr_make(float a, float b) {
  PairF r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ PairD pr_make(double a, double b) { return PairD{a, b}; }
__device__ __forceinline__ float2 pr_get(PairF a) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(a.v));
  return r;
}
__device__ __forceinline__ double2 pr_get(PairD a) { return double2{a.x, a.y}; }
__device__ __forceinline__ PairF pr_add(PairF a, PairF b) {
  PairF r;
  asm("add.rn.ftz.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ PairF pr_sub(PairF a, PairF b) {
  PairF r;
  asm("sub.rn.ftz.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ PairF pr_mul(PairF a, PairF b) {
  PairF r;
  asm("mul.rn.ftz.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ PairF pr_fma(PairF a, PairF b, PairF c) {
  PairF r;
  asm("fma.rn.ftz.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
  return r;
}
__device__ __forceinline__ PairD pr_add(PairD a, PairD b) { return PairD{a.x + b.x, a.y + b.y}; }
__device__ __forceinline__ PairD pr_sub(PairD a, PairD b) { return PairD{a.x - b.x, a.y - b.y}; }
__device__ __forceinline__ PairD pr_mul(PairD a, PairD b) { return PairD{a.x * b.x, a.y * b.y}; }
__device__ __forceinline__ PairD pr_fma(PairD a, PairD b, PairD c) {
  return PairD{fma(a.x, b.x, c.x), fma(a.y, b.y, c.y)};
}
template <typename T> __device__ __forceinline__ typename PairOf<T>::type pr_dup(T a) { return pr_make(a, a); }
template <typename P> struct alignas(16) Quad { P x, y; };       // two pairs: (x.h, x.b, y.h, y.b)

// the hardware's reciprocal (the factor of the fast approximate quotient)
__device__ __forceinline__ float rcp_approx(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

// The distribution f in its storage type: the arithmetic type's pair, or on
// the BF16-storage path (FP32 arithmetic) a bf16 pair rounded to nearest on
// store and widened exactly on load.  FB = 1 / 0 fixes the storage at
// compile time (the hot kernels are instantiated for both); FB = -1 reads
// d.fbf at run time.
template <typename T, int FB = -1>
__device__ __forceinline__ typename Vec2<T>::type ldF(const Dev &d, size_t idx) {
  if (sizeof(T) == 4 && (FB == 1 || (FB < 0 && d.fbf))) {
    float2 w = __bfloat1622float2(reinterpret_cast<const __nv_bfloat162 *>(d.f)[idx]);
    return typename Vec2<T>::type{(T)w.x, (T)w.y};
  }
  return ldf<T>(d.f, idx);
}
template <typename T, int FB = -1> __device__ __forceinline__ void stF(const Dev &d, size_t idx, T h, T b) {
  if (sizeof(T) == 4 && (FB == 1 || (FB < 0 && d.fbf)))
    reinterpret_cast<__nv_bfloat162 *>(d.f)[idx] = __floats2bfloat162_rn((float)h, (float)b);
  else
    stf<T>(d.f, idx, h, b);
}

// Asynchronous global -> shared copies (cp.async, sm_80+): a per-thread
// prefetch ring for the streaming inputs of the wavefront sweeps.
template <int BYTES> __device__ __forceinline__ void cp_async(void *smem, const void *gmem) {
  unsigned s = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2;\n" ::"r"(s), "l"(gmem), "n"(BYTES));
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::); }
template <int N> __device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;\n" ::"n"(N));
}

// shared::cta address
__device__ __forceinline__ unsigned smem_addr(const void *p) { return (unsigned)__cvta_generic_to_shared(p); }

template <typename T> __device__ __forceinline__ T dvx(const Dev &d, int k);
template <> __device__ __forceinline__ double dvx<double>(const Dev &d, int k) { return d.vx[k]; }
template <> __device__ __forceinline__ float dvx<float>(const Dev &d, int k) { return d.vxf[k]; }
template <typename T> __device__ __forceinline__ T dvy(const Dev &d, int k);
template <> __device__ __forceinline__ double dvy<double>(const Dev &d, int k) { return d.vy[k]; }
template <> __device__ __forceinline__ float dvy<float>(const Dev &d, int k) { return d.vyf[k]; }
template <typename T> __device__ __forceinline__ T dw(const Dev &d, int k);
template <> __device__ __forceinline__ double dw<double>(const Dev &d, int k) { return d.w[k]; }
template <> __device__ __forceinline__ float dw<float>(const Dev &d, int k) { return d.wf[k]; }
// the whole velocity grid (k < nv_all), also on a sharded context
template <typename T> __device__ __forceinline__ T dvxa(const Dev &d, int k);
template <> __device__ __forceinline__ double dvxa<double>(const Dev &d, int k) { return d.vxa[k]; }
template <> __device__ __forceinline__ float dvxa<float>(const Dev &d, int k) { return d.vxaf[k]; }
template <typename T> __device__ __forceinline__ T dvya(const Dev &d, int k);
template <> __device__ __forceinline__ double dvya<double>(const Dev &d, int k) { return d.vya[k]; }
template <> __device__ __forceinline__ float dvya<float>(const Dev &d, int k) { return d.vyaf[k]; }
template <typename T> __device__ __forceinline__ T dwa(const Dev &d, int k);
template <> __device__ __forceinline__ double dwa<double>(const Dev &d, int k) { return d.wa[k]; }
template <> __device__ __forceinline__ float dwa<float>(const Dev &d, int k) { return d.waf[k]; }

// Copy a record of N values (N * sizeof(T) a multiple of 16, 16-byte aligned)
// into registers with 128-bit loads.
template <typename T, int N> __device__ __forceinline__ void load_rec(const T *src, T *dst) {
  static_assert((N * sizeof(T)) % 16 == 0, "record size");
  const float4 *s = reinterpret_cast<const float4 *>(src);
  float4 *o = reinterpret_cast<float4 *>(dst);
#pragma unroll
  for (int q = 0; q < (int)(N * sizeof(T) / 16); ++q) o[q] = __ldg(s + q);
}

// Bivariate polynomials sum_{a+b<=D} c_ab cx^a cy^b, coefficients stored
// degree-major (index (a+b)(a+b+1)/2 + b), for the equilibrium parts of the
// interface flux: on the tensor velocity grid every such term is the face
// Maxwellian times a polynomial in c = v - U0.
template <int D, typename R = float> struct Poly2 {
  static constexpr int N = (D + 1) * (D + 2) / 2;
  R c[N];
  __host__ __device__ static constexpr int idx(int a, int b) { return (a + b) * (a + b + 1) / 2 + b; }
};
template <int D, typename R = float> __device__ __forceinline__ Poly2<D, R> p2_zero() {
  Poly2<D, R> r;
#pragma unroll
  for (int i = 0; i < Poly2<D, R>::N; ++i) r.c[i] = R(0);
  return r;
}
// a0 + ax cx + ay cy
template <typename R = float> __device__ __forceinline__ Poly2<1, R> p2_lin(R a0, R ax, R ay) {
  Poly2<1, R> r;
  r.c[0] = a0; r.c[Poly2<1, R>::idx(1, 0)] = ax; r.c[Poly2<1, R>::idx(0, 1)] = ay;
  return r;
}
template <int D1, int D2, typename R>
__device__ __forceinline__ Poly2<D1 + D2, R> p2_mul(const Poly2<D1, R> &x, const Poly2<D2, R> &y) {
  Poly2<D1 + D2, R> r = p2_zero<D1 + D2, R>();
#pragma unroll
  for (int s1 = 0; s1 <= D1; ++s1)
#pragma unroll
    for (int b1 = 0; b1 <= s1; ++b1)
#pragma unroll
      for (int s2 = 0; s2 <= D2; ++s2)
#pragma unroll
        for (int b2 = 0; b2 <= s2; ++b2)
          r.c[Poly2<D1 + D2, R>::idx(s1 - b1 + s2 - b2, b1 + b2)] +=
              x.c[Poly2<D1, R>::idx(s1 - b1, b1)] * y.c[Poly2<D2, R>::idx(s2 - b2, b2)];
  return r;
}
// alpha x + beta y (degrees D1 <= D2)
template <int D1, int D2, typename R>
__device__ __forceinline__ Poly2<D2, R> p2_axpby(R alpha, const Poly2<D1, R> &x, R beta, const Poly2<D2, R> &y) {
  Poly2<D2, R> r;
#pragma unroll
  for (int i = 0; i < Poly2<D2, R>::N; ++i) r.c[i] = beta * y.c[i] + (i < Poly2<D1, R>::N ? alpha * x.c[i] : R(0));
  return r;
}
// sum_ab c_ab Mx[a] My[b]
template <int D, typename R>
__device__ __forceinline__ R p2_sum(const Poly2<D, R> &x, const R *Mx, const R *My) {
  R s = R(0);
#pragma unroll
  for (int t = 0; t <= D; ++t)
#pragma unroll
    for (int b = 0; b <= t; ++b) s += x.c[Poly2<D, R>::idx(t - b, b)] * (Mx[t - b] * My[b]);
  return s;
}

// Equilibrium factors of the time-integrated interface distribution (Eq.
// fullSolution averaged over dt_s, Shakhov g0+ of Sec. 2.1) as cubics in
// c = v - U0 from a face record P: the interface distribution of one
// velocity is
//   h: q1 f + q2 w.grad f + H ih(c),   b: q1 f_b + q2 w.grad f_b + H ib(c),
// with H = rho0 lam0/pi exp(-lam0 c^2): ih = q3 (1 + g0+/g0) + q4 (w.(a.Psi))
// + q5 (A.Psi) in reduced form, ib the same for b (including its B/H =
// Keff/(2 lam0) factor).
template <typename R>
__device__ __forceinline__ void interface_polys(const R *P, R Keff, R Kint, Poly2<3, R> &ih, Poly2<3, R> &ib) {
  R ux = P[FP_UX], uy = P[FP_UY], lam = P[FP_LAM], il = P[FP_IL];
  const R *ax = P + FP_AX, *ay = P + FP_AY, *at = P + FP_AT;
  Poly2<1, R> vxp = p2_lin<R>(ux, R(1), R(0)), vyp = p2_lin<R>(uy, R(0), R(1));
  Poly2<2, R> v2 = p2_axpby(R(1), p2_mul(vxp, vxp), R(1), p2_mul(vyp, vyp));
  Poly2<2, R> c2 = p2_zero<2, R>();
  c2.c[Poly2<2, R>::idx(2, 0)] = R(1);
  c2.c[Poly2<2, R>::idx(0, 2)] = R(1);
  auto slope = [&](const R *s) {     // s0 + s1 vx + s2 vy + s3 v^2 / 2
    Poly2<2, R> r = p2_axpby(s[1], vxp, R(0.5) * s[3], v2);
    r = p2_axpby(s[2], vyp, R(1), r);
    r.c[0] += s[0];
    return r;
  };
  Poly2<2, R> bx = slope(ax), by = slope(ay), bt = slope(at);
  Poly2<1, R> wxp = p2_lin<R>(ux - P[FP_UFX], R(1), R(0)), wyp = p2_lin<R>(uy - P[FP_UFY], R(0), R(1));
  R eh = P[FP_EH], eb = P[FP_EB];
  Poly2<2, R> bxh = bx, byh = by, bxb = bx, byb = by;
  bxh.c[0] += ax[3] * eh; byh.c[0] += ay[3] * eh;
  bxb.c[0] += ax[3] * eb; byb.c[0] += ay[3] * eb;
  Poly2<3, R> sgh = p2_axpby(R(1), p2_mul(wxp, bxh), R(1), p2_mul(wyp, byh));
  Poly2<3, R> sgb = p2_axpby(R(1), p2_mul(wxp, bxb), R(1), p2_mul(wyp, byb));
  Poly2<2, R> sth = bt, stb = bt;
  sth.c[0] += at[3] * eh;
  stb.c[0] += at[3] * eb;
  Poly2<1, R> pc = p2_lin<R>(R(0), P[FP_PREF] * P[FP_QX], P[FP_PREF] * P[FP_QY]);
  Poly2<2, R> th = p2_axpby(R(0), c2, R(2) * lam, c2);
  th.c[0] -= R(4);                                        // 2 lam c^2 - 4
  Poly2<2, R> tb = p2_axpby(R(0), c2, R(2) * lam * Keff * il, c2);
  tb.c[0] += (-R(2) * Keff - R(2) * Kint) * il;           // ((2 lam c^2 - 2) Keff - 2 Kint) / (2 lam)
  R q3 = P[FP_Q3], q4 = P[FP_Q4], q5 = P[FP_Q5];
  ih = p2_axpby(q3, p2_mul(pc, th), q4, sgh);
  ih = p2_axpby(q5, sth, R(1), ih);
  ih.c[0] += q3;
  R kil = Keff * il;
  ib = p2_axpby(q3, p2_mul(pc, tb), q4 * kil, sgb);
  ib = p2_axpby(q5 * kil, stb, R(1), ib);
  ib.c[0] += q3 * kil;
}

// Store the two cubics into a face record (FP_IH, FP_IB).
template <typename R> __device__ __forceinline__ void store_polys(R *P, const Poly2<3, R> &ih, const Poly2<3, R> &ib) {
#pragma unroll
  for (int m = 0; m < 10; ++m) { P[FP_IH + m] = ih.c[m]; P[FP_IB + m] = ib.c[m]; }
}

}  // namespace ugks
