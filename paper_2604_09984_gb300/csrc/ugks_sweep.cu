// ugks_sweep.cu -- micro LU-SGS (arXiv 2604.09984 Sec. 2.2, Eq.
// dualTimeStepping_micro with the upwind flux variation): the forward sweep
// d* = (r - sum_lower c d*) / D and the backward sweep d = d* - sum_upper c d
// / D, f += d, over every block in lexicographic order (i fastest), for
// every discrete velocity independently.
//
// The sweep runs as a skewed wavefront.  A warp owns a band of rows of a block:
// 32 / QL groups of QL lanes, RG rows a group, VP velocities a lane.  At step s,
// group g takes column i = s - g of its RG rows one after the other: the lower
// neighbour along a row is the lane's own result of the step before, the one
// across rows the row just computed, and for the group's first row the last row
// of the group before, of its step before, one warp shuffle away: no barrier
// inside a band.  Bands of one block (warps of one CTA) pass the last row's
// values to the next band through a ring in shared memory with progress
// counters (bounded waits).  Cells of lower (upper) neighbours always come from
// earlier steps or rows, so the result is the lexicographic Gauss-Seidel exactly,
// and the same to the bit for every shape.
//
// What bounds it: while the arrays stay in the L2, the latency of a step (some
// hundred instructions of one warp, one to four warps a scheduler), beyond it
// the lines touched (shapes below).  So the only chain between steps is the
// shuffle and four operations a row; the rows of a lane share the step's
// overhead (copies, link, shuffle); (h, b) go through packed FP32 instructions,
// and so do the two faces of a direction in the coefficients; no copy is
// predicated, and the seam of a periodic row has a body of its own.  A lane's
// inputs (residual / forward result, f) and the cells' records come through the
// warp's ring of asynchronous copies.  FP64 is bound by its pipe (some 15 cycles
// a warp instruction and SM): one velocity a lane and few rows a group spread
// the work over the SMs, and a step reads and prepares the next one's
// coefficients behind its own results (FP32: in order, which holds fewer
// registers).
// Forward / backward, us, before (one row a group of 2 or 4 lanes, a warp
// shuffle and link a row, 64 bytes of a cell a warp) and after:
//   FP32  32x16 cells, 256 velocities            26.5 / 28.5   18.1 / 16.5
//   FP32  128x64 + 64x16 cells, 576 velocities    115 / 126      70 / 76
//   FP32  256x128 + 128x32 cells, 1024            284 / 400     190 / 236
//   FP32  512x256 + 2 x 192x48 cells, 4096       4602 / 5988   1713 / 2862
//   FP64  64x32 cells, 576                        445 / 405     135 / 141
//   FP64  96x48 + 64x16 cells, 1024               927 / 713     414 / 361
// (the largest one moves 9.8 / 14.7 GB: 5.7 / 5.1 TB/s)
#include <type_traits>
#include "ugks_internal.cuh"
#include "ugks_launch.h"

namespace ugks {

constexpr int WS_LR = 64;            // most ring entries between two bands (columns): the next band
                                     // trails by NGRP steps, the rest of the ring is slack; fewer
                                     // (a power of two >= 2) where shared memory is short

// Shared memory of a warp and ring step: per row and lane the lane's values
// (XB bytes; backward also f), per group its rows' records (16 bytes of padding:
// groups in distinct banks).
template <typename T, int PASS, int FB, int QL, int RG, int VP> struct WsCfg {
  typedef typename Vec2<T>::type T2;
  static constexpr int VPT = VP, NGRP = 32 / QL;                    // velocities a lane, groups a warp
  static constexpr bool BF = PASS == 1 && FB == 1;                  // bf16 f in the backward pass
  static constexpr int XB = VPT * (int)sizeof(T2);                  // bytes of a lane's values: 8 or 16
  static_assert(XB == 8 || XB == 16, "one access a lane and row");
  typedef typename std::conditional<XB == 16, float4, float2>::type XV;
  static constexpr int FB_ = PASS == 1 ? (BF ? VPT * 4 : XB) : 0;   // bytes of f of a lane and row
  static constexpr int RC = NSR * (int)sizeof(T) / 16, RGS = RG * RC + 1;   // chunks of a record, of a group's records
  static constexpr int OF = RG * XB * 32, OR = OF + RG * FB_ * 32, STEP = OR + NGRP * RGS * 16;   // bytes
};

// Shared memory of a sweep CTA with nw warps and ring depth ns.
template <typename T, int PASS, int FB, int QL, int RG, int VP>
__host__ __device__ constexpr size_t ws_smem(int nw, int ns, int lr = WS_LR) {
  typedef WsCfg<T, PASS, FB, QL, RG, VP> C;
  return (size_t)nw * ns * C::STEP + (size_t)nw * lr * QL * C::VPT * sizeof(typename Vec2<T>::type) +
         (size_t)nw * 2 * QL * sizeof(int);
}

__device__ __forceinline__ float pos(float x) { return fmaxf(x, 0.f); }
__device__ __forceinline__ float neg(float x) { return fminf(x, 0.f); }
// (FP64: by the sign bit, off the FP64 pipe)
__device__ __forceinline__ double pos(double x) { return __double2hiint(x) >= 0 ? x : 0.0; }
__device__ __forceinline__ double neg(double x) { return __double2hiint(x) < 0 ? x : 0.0; }
__device__ __forceinline__ float inv(float x) { return rcp_approx(x); }
__device__ __forceinline__ double inv(double x) { return 1.0 / x; }
// half w.S of a pair of faces: vx a + vy b - c
__device__ __forceinline__ PairF face_w(PairF vx, PairF vy, PairF a, PairF b, PairF c) {
  return pr_sub(pr_fma(vx, a, pr_mul(vy, b)), c);
}
__device__ __forceinline__ PairD face_w(PairD vx, PairD vy, PairD a, PairD b, PairD c) {
  return pr_fma(vx, a, pr_fma(vy, b, PairD{-c.x, -c.y}));
}
__device__ __forceinline__ PairF shfl_up_pair(PairF v, int n) {
  return PairF{__shfl_up_sync(0xffffffffu, v.v, n)};
}
__device__ __forceinline__ PairD shfl_up_pair(PairD v, int n) {
  return PairD{__shfl_up_sync(0xffffffffu, v.x, n), __shfl_up_sync(0xffffffffu, v.y, n)};
}
template <int BYTES> __device__ __forceinline__ void ws_copy(void *dst, const void *src) {
  if (BYTES == 16) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(smem_addr(dst)), "l"(src) : "memory");
  else cp_async<BYTES>(dst, src);
}

// work item: block, first velocity, velocity groups in this CTA
template <typename T, int PASS, int FB, int NS, int QL, int RG, int VP>
__global__ void __launch_bounds__(512) k_wsweep(Dev d, const int *work, int lr) {
  typedef typename Vec2<T>::type T2;
  typedef typename PairOf<T>::type P;
  typedef WsCfg<T, PASS, FB, QL, RG, VP> C;
  typedef typename C::XV XV;
  constexpr bool PIPE = sizeof(T) == 8;
  constexpr int NGRP = C::NGRP, WROWS = NGRP * RG, VPT = C::VPT, VW = QL * VPT;
  extern __shared__ __align__(16) unsigned char smraw[];
  const int nw = blockDim.x >> 5, w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int grp = lane / QL, q = lane - grp * QL;
  int b = work[3 * blockIdx.x], k0 = work[3 * blockIdx.x + 1], gpc = work[3 * blockIdx.x + 2];
  const int *bi = d.blk_info + 8 * b;
  const int ni = bi[0], nj = bi[1], off = d.cell_off[b];
  const bool per = bi[2] != 0;
  const int nb = (nj + WROWS - 1) / WROWS;        // bands of the block
  const int gw = w / nb, band = w - gw * nb;     // velocity group, band
  unsigned char *ring = smraw + (size_t)w * NS * C::STEP;
  P *links = reinterpret_cast<P *>(smraw + (size_t)nw * NS * C::STEP);
  volatile int *prog = reinterpret_cast<volatile int *>(links + (size_t)nw * lr * VW);
  volatile int *cons = prog + nw * QL;
  if (lane < QL) prog[w * QL + lane] = cons[w * QL + lane] = 0;
  __syncthreads();
  const int kw = k0 + gw * VW;                   // first velocity of the warp
  if (gw >= gpc || kw >= d.nvp) return;          // idle warp (no later CTA-wide barrier)
  const int kb = kw + q * VPT;                   // first velocity of the lane
  const int jb = WROWS * band + RG * grp;        // first row of the group (in sweep order)
  const int nr = min(max(nj - jb, 0), RG);       // rows of the group inside the block
  P vx[VPT], vy[VPT];
#pragma unroll
  for (int u = 0; u < VPT; ++u) {
    const bool kok = kb + u < d.nv;
    vx[u] = pr_dup(kok ? dvx<T>(d, kb + u) : T(0));
    vy[u] = pr_dup(kok ? dvy<T>(d, kb + u) : T(0));
  }
  const bool whole = kb + VPT <= d.nv, some = kb < d.nv;    // the lane's velocities inside the grid: all, the first
  // the lane's values and its groups' records at the column of the next copy,
  // row by row; rows and columns outside the block (and velocities past the
  // padding) take a copy of one inside, so that no copy is predicated
  const long cs = (PASS == 0 ? 1 : -1) * (long)d.nvp;       // to the next column (elements)
  const int rdir = PASS == 0 ? 1 : -1;
  const char *xp[RG], *fp[RG], *rp[RG];
  long xo[RG];                                   // stores: element offset of the current column
#pragma unroll
  for (int r = 0; r < RG; ++r) {
    const int jr = min(jb + r, nj - 1), row = PASS == 0 ? jr : nj - 1 - jr;
    const long c = (long)off + (long)row * ni + (PASS == 0 ? 0 : ni - 1);
    const long x = c * d.nvp + min(kb, d.nvp - VPT);
    xp[r] = reinterpret_cast<const char *>(reinterpret_cast<const T2 *>(d.dfs) + x);
    fp[r] = reinterpret_cast<const char *>(d.f) + x * (C::BF ? 4 : (long)sizeof(T2));
    rp[r] = reinterpret_cast<const char *>(reinterpret_cast<const T *>(d.srec) + c * NSR) + 16 * q;
    xo[r] = c * d.nvp + kb;
  }
  // copies of step st into ring slot sl
  auto issue = [&](int st, int sl) {
    unsigned char *dst = ring + sl * C::STEP;
#pragma unroll
    for (int r = 0; r < RG; ++r) {
      ws_copy<C::XB>(dst + (r * 32 + lane) * C::XB, xp[r]);
      if (PASS == 1) ws_copy<C::FB_>(dst + C::OF + (r * 32 + lane) * C::FB_, fp[r]);
#pragma unroll
      for (int m = 0; m < (C::RC + QL - 1) / QL; ++m)
        if (C::RC % QL == 0 || q + QL * m < C::RC) ws_copy<16>(dst + C::OR + (grp * C::RGS + r * C::RC + q + QL * m) * 16, rp[r] + 16 * QL * m);
    }
    const int il = st - grp;
    const bool on = il >= 0 && il < ni - 1;      // the next step's column is another one
    const long dx = on ? cs * (long)sizeof(T2) : 0, df = on ? cs * (C::BF ? 4 : (long)sizeof(T2)) : 0;
    const long dr = on ? rdir * NSR * (long)sizeof(T) : 0;
#pragma unroll
    for (int r = 0; r < RG; ++r) {
      xp[r] += dx;
      if (PASS == 1) fp[r] += df;
      rp[r] += dr;
    }
    cp_async_commit();
  };
  const int nsteps = ni + NGRP - 1;
  P val[RG][VPT];
  // the seam of a periodic row: increments of the first column and couplings of
  // the last one, written and read once a row, so they stay out of registers
  volatile T seam[RG][VPT][3];
#pragma unroll
  for (int r = 0; r < RG; ++r)
#pragma unroll
    for (int u = 0; u < VPT; ++u) val[r][u] = pr_dup(T(0));
  // inputs and coefficients of a step's cells: couplings along the row and
  // across rows, 1 / D, residual or forward result, f; a cell that is not solved
  // (or lies outside) keeps a zero increment
  struct Item { T cr, cc, idg; P in, f; };
  Item nx[RG][VPT];
  unsigned non = 0;                              // solved cells, bit r
  auto prepare = [&](int il, const unsigned char *st) {
    const bool act = il >= 0 && il < ni;
    non = 0;
#pragma unroll
    for (int r = 0; r < RG; ++r) {
      __align__(16) T rec[NSR];
#pragma unroll
      for (int m = 0; m < C::RC; ++m)
        reinterpret_cast<float4 *>(rec)[m] =
            reinterpret_cast<const float4 *>(st + C::OR)[grp * C::RGS + r * C::RC + m];
      __align__(16) P in[VPT], fv[VPT];
      *reinterpret_cast<XV *>(in) = reinterpret_cast<const XV *>(st)[r * 32 + lane];
      if (PASS == 1) {
        if (C::BF) {
          const __nv_bfloat162 *p = reinterpret_cast<const __nv_bfloat162 *>(st + C::OF) + (r * 32 + lane) * VPT;
#pragma unroll
          for (int u = 0; u < VPT; ++u) {
            const float2 x = __bfloat1622float2(p[u]);
            fv[u] = pr_make((T)x.x, (T)x.y);
          }
        } else {
          *reinterpret_cast<XV *>(fv) = reinterpret_cast<const XV *>(st + C::OF)[r * 32 + lane];
        }
      }
      const T dbase = rec[SR_DBASE];
      if (dbase != T(0) && r < nr && act) non |= 1u << r;
#pragma unroll
      for (int u = 0; u < VPT; ++u) {
        const auto wi = pr_get(face_w(vx[u], vy[u], pr_make(rec[0], rec[1]), pr_make(rec[2], rec[3]), pr_make(rec[4], rec[5])));
        const auto wj = pr_get(face_w(vx[u], vy[u], pr_make(rec[6], rec[7]), pr_make(rec[8], rec[9]), pr_make(rec[10], rec[11])));
        T dg = dbase;
        dg += pos(wi.x);
        dg += pos(wi.y);
        dg += pos(wj.x);
        dg += pos(wj.y);
        nx[r][u].idg = inv(dg);                  // FP32: the factor of the fast approximate quotient
        nx[r][u].cr = neg(PASS == 0 ? wi.x : wi.y);
        nx[r][u].cc = neg(PASS == 0 ? wj.x : wj.y);
        if (per && il == ni - 1) seam[r][u][2] = neg(PASS == 0 ? wi.y : wi.x);
        nx[r][u].in = in[u];
        if (PASS == 1) nx[r][u].f = fv[u];
      }
    }
  };
  // results of a step's rows; EDGE: a group may be at the first or last column
  // of a periodic row
  auto rows = [&](auto edge, int il, P *up) {
    constexpr bool EDGE = decltype(edge)::value;
    const bool wrap = EDGE && il == ni - 1;
#pragma unroll
    for (int r = 0; r < RG; ++r) {
      const bool on = (non >> r) & 1;
      __align__(16) P out[VPT];
#pragma unroll
      for (int u = 0; u < VPT; ++u) {
        const Item &x = nx[r][u];
        P a = pr_fma(pr_dup(x.cr), val[r][u], pr_mul(pr_dup(x.cc), up[u]));
        if (EDGE && wrap) a = pr_fma(pr_dup((T)seam[r][u][2]), pr_make((T)seam[r][u][0], (T)seam[r][u][1]), a);
        P v = PASS == 0 ? pr_mul(pr_sub(x.in, a), pr_dup(x.idg)) : pr_fma(a, pr_dup(-x.idg), x.in);
        if (!on) v = pr_dup(T(0));
        val[r][u] = v;
        up[u] = v;
        if (EDGE && il == 0) {
          const auto f0 = pr_get(v);
          seam[r][u][0] = f0.x;
          seam[r][u][1] = f0.y;
        }
        out[u] = PASS == 0 ? v : pr_add(x.f, v);
      }
      if (C::BF) {
#pragma unroll
        for (int u = 0; u < VPT; ++u) {
          const auto v = pr_get(out[u]);
          if (on && (u == 0 ? some : whole)) stF<T, FB>(d, (size_t)xo[r] + u, v.x, v.y);
        }
      } else {
        P *o = reinterpret_cast<P *>(PASS == 0 ? d.dfs : d.f) + xo[r];
        if (on && whole) *reinterpret_cast<XV *>(o) = *reinterpret_cast<const XV *>(out);
        if (VPT > 1 && on && some && !whole) o[0] = out[0];
      }
      xo[r] += il >= 0 ? cs : 0;
    }
  };
  // links to the bands before and after: values and progress, a lane of one
  // band with the lane of the other that has its velocities.  A wait that ran
  // out is recorded and the lane waits no more.
  const bool link_in = grp == 0 && band > 0, link_out = grp == NGRP - 1 && band + 1 < nb;
  const P *lin = links + (size_t)(w - 1) * lr * VW + q * VPT;
  P *lout = links + (size_t)w * lr * VW + q * VPT;
  volatile int *prog_in = prog + (w - 1) * QL + q, *cons_in = cons + (w - 1) * QL + q;
  volatile int *prog_out = prog + w * QL + q, *cons_out = cons + w * QL + q;
  // a consumer reports its progress every `report` columns (each one where the
  // ring is short)
  const int report = lr >= 32 ? 8 : 1;
  int polls = d.wait_polls, seen_p = 0, seen_c = 0;   // progress last seen of the band before / after
  int slot = 0;                                       // ring slot of step s
#pragma unroll
  for (int m = 0; m < NS; ++m) issue(m, m);
  if (PIPE) {
    cp_async_wait<NS - 1>();
    __syncwarp();
    prepare(-grp, ring);
  }
  for (int s = 0; s < nsteps; ++s) {
    const int il = s - grp;
    if (PIPE) {
      __syncwarp();                              // slot read by all lanes in the step before
      issue(s + NS, slot);
      slot = slot + 1 == NS ? 0 : slot + 1;
    } else {
      cp_async_wait<NS - 1>();
      __syncwarp();
      prepare(il, ring + slot * C::STEP);
      __syncwarp();
      issue(s + NS, slot);
      slot = slot + 1 == NS ? 0 : slot + 1;
    }
    // lower (upper) neighbour across rows of the group's first row: the last
    // row of the group before, of step s - 1, or for the band's first row the
    // previous band's last row through the link ring
    P up[VPT];
#pragma unroll
    for (int u = 0; u < VPT; ++u) {
      up[u] = shfl_up_pair(val[RG - 1][u], QL);
      if (grp == 0) up[u] = pr_dup(T(0));
    }
    if (link_in && il < ni) {                    // (group 0: il = s >= 0)
      if (seen_p <= il) {
        int n = 0;
        while ((seen_p = *prog_in) <= il && n < polls) {
          __nanosleep(32);               // leave the issue slots to the other warps
          ++n;
        }
        if (seen_p <= il) { polls = 0; atomicOr(d.err, EF_TIMEOUT); }
        __threadfence_block();
      }
      const P *src = lin + (size_t)(il & (lr - 1)) * VW;
#pragma unroll
      for (int u = 0; u < VPT; ++u) up[u] = src[u];
      if ((il + 1) % report == 0) {
        __threadfence_block();
        *cons_in = il + 1;
      }
    }
    __syncwarp();
    if (per && (s < NGRP || s >= ni - 1)) rows(std::true_type(), il, up);
    else rows(std::false_type(), il, up);
    // the next step's inputs: complete, and the group's records copied by its lanes
    if (PIPE) {
      cp_async_wait<NS - 1>();
      __syncwarp();
      prepare(il + 1, ring + slot * C::STEP);
    }
    // the band's last row feeds the next band
    if (link_out && il >= 0 && il < ni) {
      if (seen_c + lr <= il) {
        int n = 0;
        while ((seen_c = *cons_out) + lr <= il && n < polls) {
          __nanosleep(32);
          ++n;
        }
        if (seen_c + lr <= il) { polls = 0; atomicOr(d.err, EF_TIMEOUT); }
      }
      P *dst = lout + (size_t)(il & (lr - 1)) * VW;
#pragma unroll
      for (int u = 0; u < VPT; ++u) dst[u] = val[RG - 1][u];
      __threadfence_block();
      *prog_out = il + 1;
    }
    // (the vote also brings the lanes back together: without it they ran the
    // next step apart, at twice the time)
    if (__any_sync(0xffffffffu, polls == 0)) break;
  }
  cp_async_wait<0>();
}

// ring depths: one step only where 16 bands of four rows leave no room for two
template <int RG> constexpr int ws_depth(int n) { return n == 1 && RG < 4 ? 2 : n; }

template <typename T, int PASS, int FB, int QL, int RG, int VP>
static void ws_launch(const Dev &d, cudaStream_t s, const int *work, int nwork, int nw, int ns) {
  size_t lim = 227 * 1024;
  // deepest ring that fits (6, 4, 2 or 1 steps; 1 = no prefetch), no deeper
  // than asked; then the longest link ring that fits
  int n = ns >= 6 ? 6 : (ns >= 4 ? 4 : (ns >= 2 ? 2 : 1));
  while (n > ws_depth<RG>(1) && ws_smem<T, PASS, FB, QL, RG, VP>(nw, n) > lim) n = n == 2 ? 1 : n - 2;
  int lr = WS_LR;
  while (lr > 2 && ws_smem<T, PASS, FB, QL, RG, VP>(nw, n, lr) > lim) lr >>= 1;
  size_t sm = ws_smem<T, PASS, FB, QL, RG, VP>(nw, n, lr);
  int th = 32 * nw;
  if (n == 6) k_wsweep<T, PASS, FB, 6, QL, RG, VP><<<nwork, th, sm, s>>>(d, work, lr);
  else if (n == 4) k_wsweep<T, PASS, FB, 4, QL, RG, VP><<<nwork, th, sm, s>>>(d, work, lr);
  else if (n == 2) k_wsweep<T, PASS, FB, 2, QL, RG, VP><<<nwork, th, sm, s>>>(d, work, lr);
  else k_wsweep<T, PASS, FB, ws_depth<RG>(1), QL, RG, VP><<<nwork, th, sm, s>>>(d, work, lr);
}
template <typename T, int PASS, int FB, int QL, int RG, int VP> static void ws_attr_pass() {
  int lim = 227 * 1024;
  cudaFuncSetAttribute(k_wsweep<T, PASS, FB, ws_depth<RG>(1), QL, RG, VP>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
  cudaFuncSetAttribute(k_wsweep<T, PASS, FB, 2, QL, RG, VP>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
  cudaFuncSetAttribute(k_wsweep<T, PASS, FB, 4, QL, RG, VP>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
  cudaFuncSetAttribute(k_wsweep<T, PASS, FB, 6, QL, RG, VP>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
}

// what the host does with a shape: set up, shared memory of the backward sweep
// (the larger one) with ring depth ns and the longest link ring for ns > 1, the
// shortest for ns = 1, and launch
template <typename T, int QL, int RG, int VP> struct WsOps {
  static void attr() {
    ws_attr_pass<T, 0, 0, QL, RG, VP>();
    ws_attr_pass<T, 1, 0, QL, RG, VP>();
    if (sizeof(T) == 4) ws_attr_pass<T, 1, sizeof(T) == 4, QL, RG, VP>();
  }
  static size_t need(int fbf, int nw, int ns) {
    const int lr = ns > 1 ? WS_LR : 2, n = ns == 1 ? ws_depth<RG>(1) : ns;
    return fbf ? ws_smem<T, 1, sizeof(T) == 4, QL, RG, VP>(nw, n, lr) : ws_smem<T, 1, 0, QL, RG, VP>(nw, n, lr);
  }
  static void launch(const Dev &d, cudaStream_t s, int pass, const int *work, int nwork, int nw, int ns) {
    if (pass == 0) ws_launch<T, 0, 0, QL, RG, VP>(d, s, work, nwork, nw, ns);
    else if (sizeof(T) == 4 && d.fbf) ws_launch<T, 1, sizeof(T) == 4, QL, RG, VP>(d, s, work, nwork, nw, ns);
    else ws_launch<T, 1, 0, QL, RG, VP>(d, s, work, nwork, nw, ns);
  }
};
struct WsEntry {
  int ql, rg, vp;
  void (*attr)();
  size_t (*need)(int, int, int);
  void (*launch)(const Dev &, cudaStream_t, int, const int *, int, int, int);
};
template <typename T, int QL, int RG, int VP> constexpr WsEntry ws_entry() {
  typedef WsOps<T, QL, RG, VP> O;
  return {QL, RG, VP, O::attr, O::need, O::launch};
}
// Shapes: lanes a group, rows a group, velocities a lane; rows a band and the
// bytes of a cell that a warp touches.  FP32 forward / backward, us (bytes of one
// (cell, velocity) array; rows of the tallest block):
//                              4,2,1    4,2,2    8,2,1    8,2,2    8,4,2
//                              16 32 B  16 64 B  8 64 B   8 128 B  16 128 B
//   1 MB, 16 rows              18/17    22/20    20/21    27/23    31/35
//   14 MB, 32                  32/31    40/37    37/40    47/44    55/68
//   22 MB, 51 (21 x 21 vel.)   68/79    75/64    59/64    84/76    104/121
//   42 MB, 64                  70/72    84/76    76/82    98/93    113/137
//   75 MB, 64                  89/130   90/81    84/93    100/94   116/138
//   96 MB, 96                  124/131  136/123  125/138  164/156  187/239
//   170 MB, 96                 195/312  146/188  156/157  165/156  187/238
//   302 MB, 128                299/620  231/338  190/338  248/236  263/406
//   524 MB, 128                446/884  296/537  373/506  250/307  264/412
//   445 MB, 150                391/911  326/469  -        -        364/454
//   1188 MB, 200               1318/2231 903/1485 -       -        547/1020
//   4899 MB, 256               6700/10660 3488/5437 -     -        1713/2862
// While the arrays stay in the L2 a sweep is bound by the latency of its steps:
// few velocities a lane make them short.  Beyond it lines touched in parts are
// the bound, more so for the backward sweep (two arrays in, one out): a warp
// then takes whole lines, in bands of 8 rows where 16 bands reach (a step of
// two rows is the shorter one), else of 16.  The size is one context's: contexts
// stepped side by side share the L2, and the rule does not weigh that (12 of 2,448
// to 21,568 cells in one batch: 60.4 ms by the rule, 58.9 all in 4,2,2, 58.8 all in
// 8,2,2).
enum { WS32_4_2_1, WS32_4_2_2, WS32_8_2_1, WS32_8_2_2, WS32_8_4_2, WS32_4_4_2, WS64_4_1, WS64_4_2, WS64_4_4 };
static const WsEntry kWs[] = {
    ws_entry<float, 4, 2, 1>(), ws_entry<float, 4, 2, 2>(), ws_entry<float, 8, 2, 1>(), ws_entry<float, 8, 2, 2>(),
    ws_entry<float, 8, 4, 2>(), ws_entry<float, 4, 4, 2>(), ws_entry<double, 4, 1, 1>(), ws_entry<double, 4, 2, 1>(),
    ws_entry<double, 4, 4, 1>()};

void wsweep_setup() {
  for (const WsEntry &e : kWs) e.attr();
}
int wsweep_vw(int shape) { return kWs[shape].ql * kWs[shape].vp; }
int wsweep_rows(int shape) { return 32 / kWs[shape].ql * kWs[shape].rg; }
// By the table above.  FP64: as few rows as give at most 16 bands, more warps
// share its pipe (64x32 cells, 576 velocities: 1 row 134 / 140 us, 2 rows 191 /
// 195, 4 rows 311 / 334).  `forced` (>= 0): that FP32 shape where the block's
// bands fit.
int wsweep_shape(int fp32, int pass, int max_nj, double bytes, int forced) {
  if (!fp32) return max_nj <= 128 ? WS64_4_1 : max_nj <= 256 ? WS64_4_2 : WS64_4_4;
  if (forced >= WS32_4_2_1 && forced <= WS32_4_4_2 && max_nj <= 16 * wsweep_rows(forced)) return forced;
  if (max_nj > 256) return WS32_4_4_2;
  if (bytes <= (pass ? 16e6 : 60e6)) return WS32_4_2_1;
  if (max_nj > 128) return bytes > (pass ? 400e6 : 600e6) ? WS32_8_4_2 : WS32_4_2_2;
  if (pass == 0) return bytes <= 400e6 ? WS32_8_2_1 : WS32_8_2_2;
  return bytes <= 120e6 ? WS32_4_2_2 : WS32_8_2_2;
}
int wsweep_fits(int shape, int fbf, int nw, int ns) {
  return nw <= 16 && kWs[shape].need(fbf, nw, ns) <= 227 * 1024;
}
void launch_wsweep(const Dev &d, cudaStream_t s, int pass, const int *work, int nwork, int nw, int ns, int shape) {
  kWs[shape].launch(d, s, pass, work, nwork, nw, ns);
}

}  // namespace ugks
