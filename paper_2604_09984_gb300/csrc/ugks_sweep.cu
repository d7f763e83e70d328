// ugks_sweep.cu -- micro LU-SGS (arXiv 2604.09984 Sec. 2.2, Eq.
// dualTimeStepping_micro with the upwind flux variation): the forward sweep
// d* = (r - sum_lower c d*) / D and the backward sweep d = d* - sum_upper c d
// / D, f += d, over every block in lexicographic order (i fastest), for
// every discrete velocity independently.
//
// The sweep runs as a skewed wavefront.  A warp owns a band of 8 RG rows of a
// block: 8 groups of QL = 4 lanes, RG rows a group, two velocities a lane (one
// in FP64).  At step s, group g takes column i = s - g of its RG
// rows one after the other: the lower neighbour along a row is the lane's own
// result of the step before, the one across rows the row just computed, and
// for the group's first row the last row of the group before, of its step
// before, one warp shuffle away: no barrier inside a band.  Bands of one block
// (warps of one CTA) pass the last row's values to the next band through a
// ring in shared memory with progress counters (bounded waits).  Cells of
// lower (upper) neighbours always come from earlier steps or rows, so the
// result is the lexicographic Gauss-Seidel exactly.
//
// What bounds it: the latency of a step.  A step is some hundred instructions
// of one warp, and a mesh has only one to four warps for a scheduler (issue
// slots used: 31 %).  So the only chain between steps is the shuffle and four
// operations a row; the rows of a lane share the step's overhead (copies, link,
// shuffle); (h, b) go through packed FP32 instructions, and so do the two faces
// of a direction in the coefficients; no copy is predicated, and the seam of a
// periodic row has a body of its own.  A lane's inputs (residual / forward
// result, f) and the cells' records come through the warp's ring of
// asynchronous copies.  FP64 is bound by its pipe (some 15 cycles a warp
// instruction and SM): one velocity a lane and few rows a group spread the work
// over the SMs, and a step reads and prepares the next one's coefficients
// behind its own results (FP32: in order, which holds fewer registers).
// Forward / backward, us, before (one row a group of 2 or 4 lanes, one warp
// shuffle and link a row) and after:
//   FP32  32x16 cells, 256 velocities            26.5 / 28.5   22.5 / 19.0
//   FP32  128x64 + 64x16 cells, 576 velocities    115 / 126      86 / 74
//   FP32  256x128 + 128x32 cells, 1024            284 / 400     223 / 328
//   FP32  512x256 + 192x48 cells, 4096           4602 / 5988   3570 / 5534
//   FP64  64x32 cells, 576                        445 / 405     135 / 141
//   FP64  96x48 + 64x16 cells, 1024               927 / 713     414 / 361
// (the largest one moves 9 / 14 GB: 2.7 / 2.6 TB/s)
#include <type_traits>
#include "ugks_internal.cuh"
#include "ugks_launch.h"

namespace ugks {

constexpr int QL = 4, NGRP = 32 / QL;            // lanes a group, groups a warp
template <typename T> struct WsVpt { static constexpr int N = sizeof(T) == 4 ? 2 : 1; };   // velocities a lane
constexpr int WS_LR = 64;            // most ring entries between two bands (columns): the next band
                                     // trails by NGRP steps, the rest of the ring is slack; fewer
                                     // (a power of two >= 2) where shared memory is short

// Shared memory of a warp and ring step, in 16-byte chunks: per row and lane
// the lane's values (XC chunks; backward also f), per group its rows' records
// (one chunk of padding: groups in distinct banks).
template <typename T, int PASS, int RG, int FB> struct WsCfg {
  typedef typename Vec2<T>::type T2;
  static constexpr int VPT = WsVpt<T>::N;
  static constexpr bool BF = PASS == 1 && FB == 1;                  // bf16 f in the backward pass
  static constexpr int XC = VPT * (int)sizeof(T2) / 16;
  static constexpr int FBYTES = PASS == 1 ? (BF ? VPT * 4 : VPT * (int)sizeof(T2)) : 0;   // f of a lane and row
  static constexpr int FC = (FBYTES + 15) / 16;
  static constexpr int RC = NSR * (int)sizeof(T) / 16, RGS = RG * RC + 1;   // chunks of a record, of a group's records
  static constexpr int OF = RG * XC * 32, OR = OF + RG * FC * 32, STEP = OR + NGRP * RGS;
};

// Shared memory of a sweep CTA with nw warps and ring depth ns.
template <typename T, int PASS, int RG, int FB>
__host__ __device__ constexpr size_t ws_smem(int nw, int ns, int lr = WS_LR) {
  typedef WsCfg<T, PASS, RG, FB> C;
  return (size_t)nw * ns * C::STEP * 16 + (size_t)nw * lr * QL * C::VPT * sizeof(typename Vec2<T>::type) +
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
template <typename T, int PASS, int NS, int RG, int FB>
__global__ void __launch_bounds__(512) k_wsweep(Dev d, const int *work, int lr) {
  typedef typename Vec2<T>::type T2;
  typedef typename PairOf<T>::type P;
  typedef WsCfg<T, PASS, RG, FB> C;
  constexpr bool PIPE = sizeof(T) == 8;
  constexpr int WROWS = NGRP * RG, VPT = C::VPT, VW = QL * VPT;
  struct alignas(16) Chunk { unsigned char b[16]; };
  extern __shared__ __align__(16) unsigned char smraw[];
  const int nw = blockDim.x >> 5, w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int grp = lane / QL, q = lane - grp * QL;
  int b = work[3 * blockIdx.x], k0 = work[3 * blockIdx.x + 1], gpc = work[3 * blockIdx.x + 2];
  const int *bi = d.blk_info + 8 * b;
  const int ni = bi[0], nj = bi[1], off = d.cell_off[b];
  const bool per = bi[2] != 0;
  const int nb = (nj + WROWS - 1) / WROWS;        // bands of the block
  const int gw = w / nb, band = w - gw * nb;     // velocity group, band
  Chunk *ring = reinterpret_cast<Chunk *>(smraw) + (size_t)w * NS * C::STEP;
  P *links = reinterpret_cast<P *>(smraw + (size_t)nw * NS * C::STEP * 16);
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
    Chunk *dst = ring + sl * C::STEP;
#pragma unroll
    for (int r = 0; r < RG; ++r) {
#pragma unroll
      for (int m = 0; m < C::XC; ++m) ws_copy<16>(dst + (r * C::XC + m) * 32 + lane, xp[r] + 16 * m);
      if (PASS == 1) {
        if (C::BF) {
          ws_copy<VPT * 4>(dst + C::OF + r * 32 + lane, fp[r]);
        } else {
#pragma unroll
          for (int m = 0; m < C::FC; ++m) ws_copy<16>(dst + C::OF + (r * C::FC + m) * 32 + lane, fp[r] + 16 * m);
        }
      }
#pragma unroll
      for (int m = 0; m < C::RC / QL; ++m)
        ws_copy<16>(dst + C::OR + grp * C::RGS + r * C::RC + q + QL * m, rp[r] + 16 * QL * m);
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
  auto prepare = [&](int il, const Chunk *st) {
    const bool act = il >= 0 && il < ni;
    non = 0;
#pragma unroll
    for (int r = 0; r < RG; ++r) {
      __align__(16) T rec[NSR];
#pragma unroll
      for (int m = 0; m < C::RC; ++m)
        reinterpret_cast<float4 *>(rec)[m] = reinterpret_cast<const float4 *>(st + C::OR + grp * C::RGS + r * C::RC)[m];
      __align__(16) P in[VPT], fv[VPT];
#pragma unroll
      for (int m = 0; m < C::XC; ++m)
        reinterpret_cast<float4 *>(in)[m] = *reinterpret_cast<const float4 *>(st + (r * C::XC + m) * 32 + lane);
      if (PASS == 1) {
        if (C::BF) {
          const __nv_bfloat162 *p = reinterpret_cast<const __nv_bfloat162 *>(st + C::OF + r * 32 + lane);
#pragma unroll
          for (int u = 0; u < VPT; ++u) {
            const float2 x = __bfloat1622float2(p[u]);
            fv[u] = pr_make((T)x.x, (T)x.y);
          }
        } else {
#pragma unroll
          for (int m = 0; m < C::FC; ++m)
            reinterpret_cast<float4 *>(fv)[m] = *reinterpret_cast<const float4 *>(st + C::OF + (r * C::FC + m) * 32 + lane);
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
        if (on && whole) {
#pragma unroll
          for (int m = 0; m < C::XC; ++m) reinterpret_cast<float4 *>(o)[m] = reinterpret_cast<const float4 *>(out)[m];
        }
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

template <typename T, int PASS, int RG, int FB>
static void ws_launch(const Dev &d, cudaStream_t s, const int *work, int nwork, int nw, int ns) {
  size_t lim = 227 * 1024;
  // deepest ring that fits (6, 4, 2 or 1 steps; 1 = no prefetch), no deeper
  // than asked; then the longest link ring that fits
  int n = ns >= 6 ? 6 : (ns >= 4 ? 4 : (ns >= 2 ? 2 : 1));
  while (n > ws_depth<RG>(1) && ws_smem<T, PASS, RG, FB>(nw, n) > lim) n = n == 2 ? 1 : n - 2;
  int lr = WS_LR;
  while (lr > 2 && ws_smem<T, PASS, RG, FB>(nw, n, lr) > lim) lr >>= 1;
  size_t sm = ws_smem<T, PASS, RG, FB>(nw, n, lr);
  int th = 32 * nw;
  if (n == 6) k_wsweep<T, PASS, 6, RG, FB><<<nwork, th, sm, s>>>(d, work, lr);
  else if (n == 4) k_wsweep<T, PASS, 4, RG, FB><<<nwork, th, sm, s>>>(d, work, lr);
  else if (n == 2) k_wsweep<T, PASS, 2, RG, FB><<<nwork, th, sm, s>>>(d, work, lr);
  else k_wsweep<T, PASS, ws_depth<RG>(1), RG, FB><<<nwork, th, sm, s>>>(d, work, lr);
}

template <typename T, int PASS, int RG, int FB> static void ws_attr() {
  int lim = 227 * 1024;
  cudaFuncSetAttribute(k_wsweep<T, PASS, ws_depth<RG>(1), RG, FB>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
  cudaFuncSetAttribute(k_wsweep<T, PASS, 2, RG, FB>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
  cudaFuncSetAttribute(k_wsweep<T, PASS, 4, RG, FB>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
  cudaFuncSetAttribute(k_wsweep<T, PASS, 6, RG, FB>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
}
template <int RG> static void ws_attr_all() {
  if (RG > 1) { ws_attr<float, 0, RG, 0>(); ws_attr<float, 1, RG, 0>(); ws_attr<float, 1, RG, 1>(); }
  ws_attr<double, 0, RG, 0>(); ws_attr<double, 1, RG, 0>();
}
void wsweep_setup() {
  ws_attr_all<1>();
  ws_attr_all<2>();
  ws_attr_all<4>();
}

int wsweep_vw(int fp32) { return QL * (fp32 ? WsVpt<float>::N : WsVpt<double>::N); }
int wsweep_rows(int rg) { return NGRP * rg; }
// Rows a group: as few as give at most 16 bands (warps of a CTA).  FP64: more
// warps share its pipe (64x32 cells, 576 velocities: 1 row 134 / 140 us, 2
// rows 191 / 195, 4 rows 311 / 334).  FP32: not below 2, where the lag of the
// bands outgrows the shorter step (256x128 + 128x32 cells, 1024 velocities: 1 row
// 246 / 392 us, 2 rows 223 / 329, 4 rows 238 / 352).
int wsweep_rg(int max_nj, int fp32) { return max_nj <= 128 && !fp32 ? 1 : max_nj <= 256 ? 2 : 4; }

// shared memory of the backward sweep (the larger one) with ring depth ns
// and the longest link ring for ns > 1, the shortest for ns = 1
template <int RG> static size_t ws_need(int fp32, int fbf, int nw, int ns) {
  int lr = ns > 1 ? WS_LR : 2;
  ns = ns == 1 ? ws_depth<RG>(1) : ns;
  if (!fp32) return ws_smem<double, 1, RG, 0>(nw, ns, lr);
  return fbf ? ws_smem<float, 1, RG, 1>(nw, ns, lr) : ws_smem<float, 1, RG, 0>(nw, ns, lr);
}
int wsweep_fits(int fp32, int fbf, int rg, int nw, int ns) {
  size_t need = rg == 4 ? ws_need<4>(fp32, fbf, nw, ns) : rg == 2 ? ws_need<2>(fp32, fbf, nw, ns) : ws_need<1>(fp32, fbf, nw, ns);
  return nw <= 16 && need <= 227 * 1024;
}

template <int RG>
static void ws_dispatch(const Dev &d, cudaStream_t s, int pass, const int *work, int nwork, int nw, int ns, int fp32) {
  if (!fp32) {
    if (pass == 0) ws_launch<double, 0, RG, 0>(d, s, work, nwork, nw, ns);
    else ws_launch<double, 1, RG, 0>(d, s, work, nwork, nw, ns);
    return;
  }
  constexpr int RF = RG > 1 ? RG : 2;
  if (pass == 0) ws_launch<float, 0, RF, 0>(d, s, work, nwork, nw, ns);
  else if (d.fbf) ws_launch<float, 1, RF, 1>(d, s, work, nwork, nw, ns);
  else ws_launch<float, 1, RF, 0>(d, s, work, nwork, nw, ns);
}
void launch_wsweep(const Dev &d, cudaStream_t s, int pass, const int *work, int nwork, int nw, int ns, int rg, int fp32) {
  if (rg == 4) ws_dispatch<4>(d, s, pass, work, nwork, nw, ns, fp32);
  else if (rg == 2) ws_dispatch<2>(d, s, pass, work, nwork, nw, ns, fp32);
  else ws_dispatch<1>(d, s, pass, work, nwork, nw, ns, fp32);
}

}  // namespace ugks
