// ugks_macro.cu -- macro LU-SGS of an inner iteration (arXiv 2604.09984 Sec.
// 2.2 Step 4, Eq. dualTimeStepping_macro with the Euler-flux variation
// (1/4) S (dF_E,j - Gamma dW_j)): the records of the sweep, the forward and
// backward sweep over every block in lexicographic order (i fastest), and the
// predictor W' with its cell records.
//
// A block is swept by one CTA as a skewed wavefront without barriers inside a
// warp.  LPR lanes hold a row; row j takes cell i = t - j at diagonal t, so
// its lower neighbour along the row is its own result of diagonal t - 1 and
// its lower neighbour across rows is row j - 1's, one warp shuffle away.  A
// cell evaluates the variation of both Cartesian fluxes for its own increment
// once and sends the finished couplings (4 values) to its two next
// neighbours, so the chain from one diagonal to the next is one reciprocal, a
// dozen fused multiply-adds and a shuffle.  Bands of 32 / LPR rows (one warp
// each) hand their last row's couplings on through a ring in shared memory;
// a band trails the one before it by K - 1 further diagonals, so that one CTA
// barrier per K diagonals orders the ring (no polling).
//
// What bounds it: the latency of that chain (one SM per block).  The four
// vectors a cell needs per pass arrive D - 1 diagonals ahead in a ring in
// shared memory (asynchronous 16-byte copies, coalesced over the rows of a
// diagonal), and the next diagonal's are moved into registers while the
// current one is evaluated; padding around the diagonals and rows holds
// records of a cell at rest that couples to nothing, so the loop has no
// bounds checks.  FP64: the pipe retires a warp instruction in tens of cycles,
// so four lanes share a row (one component each) while all bands fit in one
// CTA.  Measured (sweep alone, 256 x 128 + 128 x 32 cells, FP32): 115 us for
// both passes, 0.15 us a diagonal, against 608 us for the form with one CTA
// barrier and one 32 KB record copy per diagonal; the same loop with the
// records prefetched straight into registers took 200 us (eight loads in
// flight wait on each other's scoreboards).  FP64, 64 x 32 cells: 1.53 ms to
// 0.37 ms with its record gather and predictor.
#include "ugks_internal.cuh"
#include "ugks_launch.h"

namespace ugks {

// planes of the sweep records, one vector of 4 per cell each:
//   VAL  R of Step 4, then the increment (forward, then final)
//   ST   rho, V_x, V_y, p of W
//   F1   1/diag, couplings sent across the i-high face   F2 the j-high face
//   B1   1/diag, couplings sent across the i-low face    B2 the j-low face
// A coupling (a, b, g) gives the neighbour a dF_x + b dF_y - g dW.
enum { MP_VAL = 0, MP_ST, MP_F1, MP_F2, MP_B1, MP_B2, NMP };

template <typename T> struct alignas(16) MV4 { T v[4]; };

// rows of a block in the record array
__host__ __device__ __forceinline__ int macro_rows(int nj) { return (nj + 31) / 32 * 32; }

// Launch shape by the rows of the tallest block: lanes a row, diagonals per
// barrier and ring depth.  Eight diagonals a barrier cost 7 more per band and
// hide the barrier; D - 1 diagonals of copies in flight cover the L2 latency
// (about 1 us at 0.12 us a diagonal), fewer where 16 bands share the memory.
struct MacroShape { int lpr, k, d; };
constexpr MacroShape kShape32{1, 8, 8}, kShape32Tall{1, 8, 6}, kShape64{4, 2, 4}, kShape64Tall{1, 2, 3};
static MacroShape macro_shape(int rows, int fp32) {
  if (fp32) return rows <= 256 ? kShape32 : kShape32Tall;
  return rows <= 128 ? kShape64 : kShape64Tall;
}
static int macro_bands(int rows, const MacroShape &m) { int rpb = 32 / m.lpr; return (rows + rpb - 1) / rpb; }

// diagonals of padding before the first and after the last one: the trailing
// bands' offsets, the rounding to whole barriers and the copies ahead
int macro_pad(int rows, int fp32) {
  MacroShape m = macro_shape(rows, fp32);
  return (macro_bands(rows, m) - 1) * (m.k - 1) + m.k + m.d;
}
// records (cells with padding) of one block
size_t macro_cells(int ni, int nj, int pad) { return (size_t)(ni + nj - 1 + 2 * pad) * macro_rows(nj); }
size_t macro_record_bytes(int fp32) { return NMP * (fp32 ? sizeof(MV4<float>) : sizeof(MV4<double>)); }

// vector index of plane 0 of row `row` on diagonal t of block b
__device__ __forceinline__ long macro_at(const Dev &d, int b, int t, int row) {
  int njp = macro_rows(d.blk_info[8 * b + 1]);
  return (long)NMP * ((long)d.mrec_off[b] + (long)(t + d.mpad) * njp) + row;
}
__device__ __forceinline__ long macro_at_cell(const Dev &d, int c, int &njp) {
  int b = d.cell_block[c];
  int ni = d.blk_info[8 * b], loc = c - d.cell_off[b];
  int j = loc / ni, i = loc - j * ni;
  njp = macro_rows(d.blk_info[8 * b + 1]);
  return macro_at(d, b, i + j, j);
}

// every record a cell at rest without couplings (once per mesh: the padding
// keeps it)
template <typename T> __global__ void k_macro_pad(Dev d, int b) {
  int njp = macro_rows(d.blk_info[8 * b + 1]), nd = d.blk_info[8 * b] + d.blk_info[8 * b + 1] - 1 + 2 * d.mpad;
  MV4<T> *rec = reinterpret_cast<MV4<T> *>(d.mrec) + (long)NMP * d.mrec_off[b];
  for (long q = (long)blockIdx.x * blockDim.x + threadIdx.x; q < (long)nd * NMP * njp; q += (long)gridDim.x * blockDim.x) {
    int plane = (int)(q / njp % NMP);
    T one = plane == MP_ST ? T(1) : T(0);
    rec[q] = MV4<T>{{one, T(0), T(0), one}};
  }
}

// Gather the records of every cell (parallel): R, 1/diag, the state and the
// couplings to the solved neighbours.
template <typename T> __global__ void k_macro_prep(Dev d) {
  int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= d.nc) return;
  int njp;
  MV4<T> *o = reinterpret_cast<MV4<T> *>(d.mrec) + macro_at_cell(d, c, njp);
  int mask = d.cmask[c];
  const bool on = mask & 1;
  double r[4] = {0, 0, 0, 0}, st[4] = {1, 0, 0, 1}, idg = 0.0;
  double cp[4][3] = {{0, 0, 0}, {0, 0, 0}, {0, 0, 0}, {0, 0, 0}};
  if (on) {
    double vol = d.vol_new[c], idt = 1.0 / d.stepc[0], W[4];
    for (int m = 0; m < 4; ++m) {
      W[m] = d.W[4 * c + m];
      r[m] = d.TW[4 * c + m] - vol * idt * W[m] - 0.5 * d.Fc[4 * c + m];
    }
    double ir = 1.0 / W[0];
    st[0] = W[0];
    st[1] = W[1] * ir;
    st[2] = W[2] * ir;
    st[3] = 2.0 / (2.0 + d.Keff) * (W[3] - 0.5 * (W[1] * st[1] + W[2] * st[2]));
    double diag = vol * (d.cfl_s / (d.cfl_pseudo * d.dts[c]) + idt);
    for (int s = 0; s < 4; ++s) {
      int f = d.cell_faces[4 * c + s];
      double sq = 0.25 * d.S[f] * d.gam[f];
      diag += sq;
      if (mask & (2 << s)) {      // the receiver's outward normal is the opposite of this cell's
        double sg = -0.25 * (double)d.cell_sgn[4 * c + s];
        cp[s][0] = sg * d.Sn[2 * f];
        cp[s][1] = sg * d.Sn[2 * f + 1];
        cp[s][2] = sg * d.SUn[f] + sq;
      }
    }
    idg = 1.0 / diag;
  }
  auto put = [&](int plane, double a, double b, double e, double g) {
    o[(long)plane * njp] = MV4<T>{{(T)a, (T)b, (T)e, (T)g}};
  };
  put(MP_VAL, r[0], r[1], r[2], r[3]);
  put(MP_ST, st[0], st[1], st[2], st[3]);
  put(MP_F1, idg, cp[1][0], cp[1][1], cp[1][2]);
  put(MP_F2, cp[3][0], cp[3][1], cp[3][2], 0.0);
  put(MP_B1, idg, cp[0][0], cp[0][1], cp[0][2]);
  put(MP_B2, cp[2][0], cp[2][1], cp[2][2], 0.0);
}

__device__ __forceinline__ double m_rcp(double x) { return 1.0 / x; }
__device__ __forceinline__ float m_rcp(float x) { return __fdividef(1.0f, x); }   // 2 ulp

// One pass (0 forward, 1 backward) over block b for this warp's band.
template <typename T, int LPR, int K, int D, int PASS>
__device__ __forceinline__ void macro_pass(const Dev &d, int b, int ni, int nj, bool per, int nb, MV4<T> *ring, T *links) {
  constexpr int RPB = 32 / LPR, NC = 4 / LPR;          // rows a band, components a lane
  constexpr unsigned FULL = 0xffffffffu;
  static_assert(K % 2 == 0 && D >= 3, "register pair by step parity; a copy, a read and a free slot");
  typedef MV4<T> V;
  struct Rec { T v[NC]; V st, c1, c2; };
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int sub = lane % LPR, lr = lane / LPR, row = w * RPB + lr;
  const int njp = macro_rows(nj), nd = ni + nj - 1;
  const int lead = PASS == 0 ? w : nb - 1 - w;         // position of the band in the sweep order
  const int total = (nd + (nb - 1) * (K - 1) + K - 1) / K * K;
  const int t0 = PASS == 0 ? -lead * (K - 1) : nd - 1 + lead * (K - 1);
  const long stride = (PASS == 0 ? 1 : -1) * (long)NMP * njp;      // to the next diagonal (vectors)
  V *ps = reinterpret_cast<V *>(d.mrec) + macro_at(d, b, t0, row); // this step's cell, plane 0
  // the band's copies of a diagonal: planes VAL, ST and this pass's two, RPB
  // vectors each, as 16-byte chunks over the lanes
  constexpr int P1 = PASS == 0 ? MP_F1 : MP_B1, P2 = PASS == 0 ? MP_F2 : MP_B2;
  constexpr int CPV = (int)sizeof(V) / 16, CPP = RPB * CPV, NCH = 4 * CPP / 32;
  static_assert(CPP * 4 % 32 == 0, "whole copies per lane");
  const char *src[NCH];
#pragma unroll
  for (int m = 0; m < NCH; ++m) {
    const int q = lane + 32 * m, pl = q / CPP, plane = pl == 0 ? MP_VAL : pl == 1 ? MP_ST : pl == 2 ? P1 : P2;
    src[m] = reinterpret_cast<const char *>(reinterpret_cast<const V *>(d.mrec) + macro_at(d, b, t0, w * RPB) +
                                            (long)plane * njp) + 16 * (q - pl * CPP);
  }
  V *rg = ring + (size_t)w * D * 4 * RPB;
  auto copy = [&](int slot) {
    char *dst = reinterpret_cast<char *>(rg + slot * 4 * RPB) + 16 * lane;
#pragma unroll
    for (int m = 0; m < NCH; ++m) {
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(smem_addr(dst + 512 * m)), "l"(src[m]) : "memory");
      src[m] += stride * (long)sizeof(V);
    }
    cp_async_commit();
  };
  auto read = [&](int slot, Rec &r) {
    const V *s = rg + slot * 4 * RPB + lr;
#pragma unroll
    for (int m = 0; m < NC; ++m) r.v[m] = s[0].v[LPR == 1 ? m : sub];
    r.st = s[RPB];
    r.c1 = s[2 * RPB];
    r.c2 = s[3 * RPB];
  };
#pragma unroll
  for (int u = 0; u < D - 1; ++u) copy(u);
  // couplings that wrap around a periodic row: from its first cell of the
  // pass to its last, with the coefficients of the other pass's record
  T wrap[NC], wc[3] = {T(0), T(0), T(0)};
  const int ifirst = PASS == 0 ? 0 : ni - 1, ilast = PASS == 0 ? ni - 1 : 0;
  if (per && row < nj) {
    const V x = (reinterpret_cast<const V *>(d.mrec) + macro_at(d, b, ifirst + row, row))[(long)(PASS == 0 ? MP_B1 : MP_F1) * njp];
    for (int m = 0; m < 3; ++m) wc[m] = x.v[1 + m];
  }
  T *rin = links + (size_t)lead * 2 * K * 4, *rout = rin + 2 * K * 4;     // link 0 stays zero
  for (int q = lane; q < 2 * K * 4; q += 32) {
    rout[q] = T(0);
    if (lead == 0) rin[q] = T(0);
  }
  T carry[NC], outj[NC];
#pragma unroll
  for (int m = 0; m < NC; ++m) { carry[m] = T(0); outj[m] = T(0); wrap[m] = T(0); }
  const bool efirst = PASS == 0 ? lr == 0 : lr == RPB - 1;      // the band's first / last row of the pass
  const bool elast = PASS == 0 ? lr == RPB - 1 : lr == 0;
  int i = t0 - row;
  const T g1 = T(2) / (T(2) + (T)d.Keff);              // gamma - 1
  const T ig1 = T(1) + (T(2) + (T)d.Keff) * T(0.5);    // 1 + 1 / (gamma - 1)
  int sc = D - 1, sr = 1;                              // ring slots: next copy, next read
  Rec rec[2];
  cp_async_wait<D - 2>();
  __syncwarp();
  read(0, rec[0]);
  for (int c = 0; c < total; c += K) {
    // the link half written before this barrier is read after it, and the
    // half read before it is written after it
    asm volatile("bar.sync 1, %0;" ::"r"(32 * nb) : "memory");
    const int hw = (c / K & 1) * K, hr = K - hw;
#pragma unroll
    for (int u = 0; u < K; ++u) {
      const Rec &r = rec[u & 1];
      copy(sc);                                        // into the slot read the step before last
      sc = sc + 1 == D ? 0 : sc + 1;
      cp_async_wait<D - 2>();
      if (CPV * LPR > 1) __syncwarp();                 // (else a lane reads what it copied itself)
      read(sr, rec[(u & 1) ^ 1]);
      sr = sr + 1 == D ? 0 : sr + 1;
      T in[NC], val[NC], dw[4];
#pragma unroll
      for (int m = 0; m < NC; ++m) {
        T up = PASS == 0 ? __shfl_up_sync(FULL, outj[m], LPR) : __shfl_down_sync(FULL, outj[m], LPR);
        T lk = rin[(hr + u) * 4 + (LPR == 1 ? m : sub)];
        in[m] = carry[m] + (efirst ? lk : up);
      }
      if (per && i == ilast) {
#pragma unroll
        for (int m = 0; m < NC; ++m) in[m] += wrap[m];
      }
      const T idg = r.c1.v[0];
      const bool on = idg != T(0);                     // a solved cell; the others keep a zero increment
#pragma unroll
      for (int m = 0; m < NC; ++m) {
        T x = PASS == 0 ? (r.v[m] - in[m]) * idg : r.v[m] - in[m] * idg;
        val[m] = on ? x : T(0);
      }
      if (on) {
        if (LPR == 1) {
          V x;
#pragma unroll
          for (int m = 0; m < 4; ++m) x.v[m] = val[m % NC];
          ps[0] = x;
        } else {
          ps[0].v[sub] = val[0];
        }
      }
#pragma unroll
      for (int m = 0; m < 4; ++m) dw[m] = LPR == 1 ? val[m % NC] : __shfl_sync(FULL, val[0], (lane & ~(LPR - 1)) + m);
      // variation of the Cartesian Euler fluxes between W and W + dW, written
      // in the increments (no difference of two fluxes)
      const T rho = r.st.v[0], vx = r.st.v[1], vy = r.st.v[2], p = r.st.v[3];
      const T hh = ig1 * p + T(0.5) * rho * (vx * vx + vy * vy);      // rho E + p
      const T ri = m_rcp(rho + dw[0]);
      const T du = (dw[1] - vx * dw[0]) * ri, dv = (dw[2] - vy * dw[0]) * ri;
      const T m1 = rho * vx + dw[1], m2 = rho * vy + dw[2];
      const T dk = dw[1] * vx + dw[2] * vy + m1 * du + m2 * dv;       // variation of rho |V|^2
      const T dp = g1 * (dw[3] - T(0.5) * dk);
      const T dh = dw[3] + dp, h1 = hh + dh;
#pragma unroll
      for (int m = 0; m < NC; ++m) {
        const int q = LPR == 1 ? m : sub;
        const T al = q == 1 ? dw[1] : q == 2 ? dw[2] : dh;
        const T be = q == 1 ? m1 : q == 2 ? m2 : h1;
        T fx = al * vx + be * du, fy = al * vy + be * dv;
        if (q == 1) fx += dp;
        if (q == 2) fy += dp;
        if (q == 0) { fx = dw[1]; fy = dw[2]; }
        const T dq = LPR == 1 ? dw[m] : val[0];
        carry[m] = r.c1.v[1] * fx + r.c1.v[2] * fy - r.c1.v[3] * dq;
        outj[m] = r.c2.v[0] * fx + r.c2.v[1] * fy - r.c2.v[2] * dq;
        if (per && i == ifirst) wrap[m] = wc[0] * fx + wc[1] * fy - wc[2] * dq;
      }
      if (elast) {
#pragma unroll
        for (int m = 0; m < NC; ++m) rout[(hw + u) * 4 + (LPR == 1 ? m : sub)] = outj[m];
      }
      ps += stride;
      i += PASS == 0 ? 1 : -1;
    }
  }
  cp_async_wait<0>();
}

template <typename T, int LPR, int K, int D> __host__ __device__ constexpr size_t macro_ring(int nb) {
  return (size_t)nb * D * 4 * (32 / LPR) * sizeof(MV4<T>);
}

template <typename T, int LPR, int K, int D> __global__ void __launch_bounds__(512) k_macro_sweep(Dev d) {
  extern __shared__ __align__(16) unsigned char smraw[];
  const int b = blockIdx.x;
  const int *bi = d.blk_info + 8 * b;
  const int ni = bi[0], nj = bi[1], nb = (nj + 32 / LPR - 1) / (32 / LPR);
  const bool per = bi[2] != 0;
  MV4<T> *ring = reinterpret_cast<MV4<T> *>(smraw);                              // [nb][D][4][RPB]
  T *links = reinterpret_cast<T *>(smraw + macro_ring<T, LPR, K, D>(nb));        // [nb + 1][2 K][4]
  if ((int)(threadIdx.x >> 5) >= nb) return;           // the named barrier counts the block's bands
  macro_pass<T, LPR, K, D, 0>(d, b, ni, nj, per, nb, ring, links);
  // the increments stored above are copied by the same band's lanes in the
  // next pass; the links are free
  __threadfence();
  asm volatile("bar.sync 1, %0;" ::"r"(32 * nb) : "memory");
  macro_pass<T, LPR, K, D, 1>(d, b, ni, nj, per, nb, ring, links);
}

// W' = W + dW and the predictor cell record (Step 4 result) for Step 5.
template <typename T> __global__ void k_macro_post(Dev d) {
  int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= d.nc) return;
  T *sr = reinterpret_cast<T *>(d.srec) + (size_t)NSR * c;
  int mask = d.cmask[c];
  *reinterpret_cast<int *>(sr + SR_MASK) = mask;
  if (!(mask & 1)) {
    for (int m = 0; m < 4; ++m) d.Wp[4 * c + m] = d.W[4 * c + m];
    return;
  }
  int njp;
  const MV4<T> inc = reinterpret_cast<const MV4<T> *>(d.mrec)[macro_at_cell(d, c, njp)];
  for (int m = 0; m < 4; ++m) d.Wp[4 * c + m] = d.W[4 * c + m] + (double)inc.v[m];
  Prim p = primitive(d.Wp + 4 * c, d.Keff);
  double *o = d.cpar + NCP * c;
  o[CP_RHO] = p.rho; o[CP_UX] = p.ux; o[CP_UY] = p.uy; o[CP_LAM] = p.lam;
  o[CP_QX] = d.q[2 * c]; o[CP_QY] = d.q[2 * c + 1];
  o[CP_ITAU] = 1.0 / collision_time(p.rho, p.lam, d.mu_ref, d.omega);
  o[CP_DBASE] = d.vol_new[c] * (d.cfl_s / (d.cfl_pseudo * d.dts[c]) + 1.0 / d.stepc[0] + 0.5 * o[CP_ITAU]);
  sr[SR_DBASE] = (T)o[CP_DBASE];
  write_shrec<T>(d, o, d.vol_new[c], reinterpret_cast<T *>(d.shp) + (size_t)NSH * c);
}

// ------------------------------------------------------- launch wrappers
static inline int nblk(size_t n, int b) { return (int)((n + b - 1) / b); }

void launch_macro_pad(const Dev &d, cudaStream_t s, int fp32) {
  for (int b = 0; b < d.nblocks; ++b) {
    if (fp32) k_macro_pad<float><<<256, 256, 0, s>>>(d, b);
    else k_macro_pad<double><<<256, 256, 0, s>>>(d, b);
  }
}

// The sweep records are gathered on the caller's stream before the fork, so
// the sweep kernel is the first work of the side stream: it then takes its
// empty SMs before the flux kernel launched beside it fills the GPU.
void launch_macro_prep(const Dev &d, cudaStream_t s, int fp32) {
  if (fp32) k_macro_prep<float><<<nblk(d.nc, 128), 128, 0, s>>>(d);
  else k_macro_prep<double><<<nblk(d.nc, 128), 128, 0, s>>>(d);
}

// the whole shared memory of an SM: the sweep's SMs take no CTA of the
// kernels running beside it on the main stream
constexpr int kMacroSmem = 227 * 1024;

template <typename T, int LPR, int K, int D> static void macro_launch(const Dev &d, cudaStream_t s, int nb) {
  k_macro_sweep<T, LPR, K, D><<<d.nblocks, 32 * nb, kMacroSmem, s>>>(d);
}
#define UGKS_MACRO(T, S) T, S.lpr, S.k, S.d
void launch_macro_sweep(const Dev &d, cudaStream_t s, int rows, int fp32) {
  int nb = macro_bands(rows, macro_shape(rows, fp32));
  if (fp32) {
    if (rows <= 256) macro_launch<UGKS_MACRO(float, kShape32)>(d, s, nb);
    else macro_launch<UGKS_MACRO(float, kShape32Tall)>(d, s, nb);
    k_macro_post<float><<<nblk(d.nc, 128), 128, 0, s>>>(d);
  } else {
    if (rows <= 128) macro_launch<UGKS_MACRO(double, kShape64)>(d, s, nb);
    else macro_launch<UGKS_MACRO(double, kShape64Tall)>(d, s, nb);
    k_macro_post<double><<<nblk(d.nc, 128), 128, 0, s>>>(d);
  }
}

template <typename T, int LPR, int K, int D, int NB> static void macro_attr() {
  static_assert(macro_ring<T, LPR, K, D>(NB) + (NB + 1) * 2 * K * 4 * sizeof(T) <= kMacroSmem, "ring and links fit");
  cudaFuncSetAttribute(k_macro_sweep<T, LPR, K, D>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMacroSmem);
}
void macro_setup() {
  macro_attr<UGKS_MACRO(float, kShape32), 8>();
  macro_attr<UGKS_MACRO(float, kShape32Tall), 16>();
  macro_attr<UGKS_MACRO(double, kShape64), 16>();
  macro_attr<UGKS_MACRO(double, kShape64Tall), 16>();
}
#undef UGKS_MACRO

}  // namespace ugks
