// ugks_macro.cu -- macro LU-SGS of an inner iteration (arXiv 2604.09984 Sec.
// 2.2 Step 4, Eq. dualTimeStepping_macro with the Euler-flux variation
// (1/4) S (dF_E,j - Gamma dW_j)): the records of the sweep, the forward and
// backward sweep over every block in lexicographic order (i fastest), and the
// predictor W' with its cell records.
//
// A block is swept by one CTA as a skewed wavefront without barriers inside a
// warp.  LPR lanes hold a row; row j takes cell i = t - j at diagonal t, so
// its lower neighbour along the row is its own result of diagonal t - 1 and
// its lower neighbour across rows is row j - 1's, one warp shuffle away.
// Bands of 32 / LPR rows (one warp each) hand their last row's values on
// through a link in shared memory; a band trails the one before it by K - 1
// further diagonals, so that one CTA barrier per K diagonals orders the links
// (no polling).
//
// What bounds it: the latency of the chain from one diagonal to the next (one
// SM per block).  The record of a cell arrives D - 1 diagonals ahead in a ring
// in shared memory (asynchronous 16-byte copies, coalesced over the rows of a
// diagonal), and the next diagonal's is moved into registers while the current
// one is evaluated; padding around the diagonals and rows holds records of
// cells that keep a zero increment, so the loop has no bounds checks.
//
// FP32: a lane a row; the cell evaluates the couplings of its two neighbours
// of the pass from their increments (the same arithmetic, rounding for
// rounding, as one thread per face slot).  FP64: the pipe retires a warp
// instruction in tens of cycles, so a cell evaluates the variation of both
// Cartesian fluxes for its own increment once and sends finished couplings (4
// values) to its two next neighbours, and four lanes share a row (one
// component each) while all bands fit in one CTA.
//
// Measured (192 x 96 + 96 x 24 cells, FP32, the sweep alone): 117 us for both
// passes, 0.20 us a diagonal, against 437 us for the form with one CTA barrier
// and one 32 KB record copy per diagonal.  FP64, 64 x 32 cells: 1.53 ms to 0.42
// with its record gather and predictor.
#include <type_traits>
#include "ugks_internal.cuh"
#include "ugks_launch.h"

namespace ugks {

// Planes of the sweep records, one vector of 4 per cell each.  Plane VAL: R of
// Step 4, then the increment (forward, then final).
// FP64:
//   ST   rho, V_x, V_y, p of W
//   F1   1/diag, couplings sent across the i-high face   F2 the j-high face
//   B1   1/diag, couplings sent across the i-low face    B2 the j-low face
// where a coupling (a, b, g) gives the neighbour a dF_x + b dF_y - g dW.
// FP32, per pass (forward FW: slots i-low, j-low; backward BW: i-high, j-high):
//   +0   W of the neighbour along the row   +1 outward normal, U.n, S/4 there
//   +2   W of the neighbour across rows     +3 outward normal, U.n, S/4 there
//   +4   Gamma of both faces, 1/diag
enum { MP_VAL = 0, MP_ST, MP_F1, MP_F2, MP_B1, MP_B2, NMP64 };
enum { MP_FW = 1, MP_BW = 6, NMP32 = 11, NPASS32 = 5 };
template <typename T> struct Planes { static constexpr int N = sizeof(T) == 4 ? NMP32 : NMP64; };

template <typename T> struct alignas(16) MV4 { T v[4]; };

// rows of a block in the record array
__host__ __device__ __forceinline__ int macro_rows(int nj) { return (nj + 31) / 32 * 32; }

// Launch shape by the rows of the tallest block: lanes a row, diagonals per
// barrier and ring depth.  Eight diagonals a barrier cost 7 more per band and
// hide the barrier; D - 1 diagonals of copies in flight cover the L2 latency
// (about 1 us at 0.12 us a diagonal), fewer where 16 bands share the memory.
struct MacroShape { int lpr, k, d; };
constexpr MacroShape kShape32{1, 8, 8}, kShape32Tall{1, 8, 4}, kShape64{4, 2, 4}, kShape64Tall{1, 2, 3};
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
size_t macro_record_bytes(int fp32) { return fp32 ? NMP32 * sizeof(MV4<float>) : NMP64 * sizeof(MV4<double>); }

// vector index of plane 0 of row `row` on diagonal t of block b
template <typename T> __device__ __forceinline__ long macro_at(const Dev &d, int b, int t, int row) {
  int njp = macro_rows(d.blk_info[8 * b + 1]);
  return (long)Planes<T>::N * ((long)d.mrec_off[b] + (long)(t + d.mpad) * njp) + row;
}
template <typename T> __device__ __forceinline__ long macro_at_cell(const Dev &d, int c, int &njp) {
  int b = d.cell_block[c];
  int ni = d.blk_info[8 * b], loc = c - d.cell_off[b];
  int j = loc / ni, i = loc - j * ni;
  njp = macro_rows(d.blk_info[8 * b + 1]);
  return macro_at<T>(d, b, i + j, j);
}

// every record a cell at rest that keeps a zero increment (once per mesh: the
// padding keeps it)
template <typename T> __global__ void k_macro_pad(Dev d, int b) {
  constexpr int N = Planes<T>::N;
  int njp = macro_rows(d.blk_info[8 * b + 1]), nd = d.blk_info[8 * b] + d.blk_info[8 * b + 1] - 1 + 2 * d.mpad;
  MV4<T> *rec = reinterpret_cast<MV4<T> *>(d.mrec) + (long)N * d.mrec_off[b];
  for (long q = (long)blockIdx.x * blockDim.x + threadIdx.x; q < (long)nd * N * njp; q += (long)gridDim.x * blockDim.x) {
    int plane = (int)(q / njp % N);
    bool state = sizeof(T) == 8 ? plane == MP_ST : plane == MP_FW || plane == MP_FW + 2 || plane == MP_BW || plane == MP_BW + 2;
    T one = state ? T(1) : T(0);
    rec[q] = MV4<T>{{one, T(0), T(0), one}};
  }
}

// Gather the records of every cell (parallel), FP64: the cell's sum of macro
// fluxes, R, 1/diag, the state and the couplings to the solved neighbours.
// Bound by the latency of three dependent loads (cell, face, neighbour) and on
// small meshes of the FP64 chain: everything is loaded before the first store,
// and CTAs of MPREP threads spread a small mesh over the SMs.
constexpr int MPREP = 32;
__global__ void __launch_bounds__(MPREP) k_macro_prep64(Dev d) {
  int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= d.nc) return;
  typedef double T;
  int njp;
  MV4<T> *o = reinterpret_cast<MV4<T> *>(d.mrec) + macro_at_cell<T>(d, c, njp);
  int mask = d.cmask[c];
  const bool on = mask & 1;
  double r[4] = {0, 0, 0, 0}, st[4] = {1, 0, 0, 1}, idg = 0.0, Fc[4];
  double cp[4][3] = {{0, 0, 0}, {0, 0, 0}, {0, 0, 0}, {0, 0, 0}};
#pragma unroll
  for (int m = 0; m < 4; ++m) Fc[m] = cell_flux_sum(d, c, m);
  if (on) {
    double vol = d.vol_new[c], idt = d.stepc[1], W[4];
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      W[m] = d.W[4 * c + m];
      r[m] = d.TW[4 * c + m] - vol * idt * W[m] - 0.5 * Fc[m];
    }
    double ir = 1.0 / W[0];
    st[0] = W[0];
    st[1] = W[1] * ir;
    st[2] = W[2] * ir;
    st[3] = 2.0 / (2.0 + d.Keff) * (W[3] - 0.5 * (W[1] * st[1] + W[2] * st[2]));
    double diag = vol * (d.idtau[c] + idt);
#pragma unroll
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
  auto put = [&](int plane, double a, double b, double e, double g) { o[(long)plane * njp] = MV4<T>{{a, b, e, g}}; };
  put(MP_VAL, r[0], r[1], r[2], r[3]);
  put(MP_ST, st[0], st[1], st[2], st[3]);
  put(MP_F1, idg, cp[1][0], cp[1][1], cp[1][2]);
  put(MP_F2, cp[3][0], cp[3][1], cp[3][2], 0.0);
  put(MP_B1, idg, cp[0][0], cp[0][1], cp[0][2]);
  put(MP_B2, cp[2][0], cp[2][1], cp[2][2], 0.0);
#pragma unroll
  for (int m = 0; m < 4; ++m) d.Fc[4 * c + m] = Fc[m];
}

// The same, FP32: R, 1/diag and per face slot the neighbour's state and the
// face.  A cell that is not solved gets 1/diag = 0 and keeps a zero increment.
// Four lanes a cell: lane s takes component s of R and face slot s (512 cells:
// 14.3 us and 5.1 us for the flux sums before, now 6.3; 36864 cells: 22.9 + 6.2
// -> 20.2).
__global__ void __launch_bounds__(2 * MPREP) k_macro_prep32(Dev d) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x, s = t & 3;
  const int c = min(t >> 2, d.nc - 1);           // (past the end: a copy of the last cell)
  int njp;
  MV4<float> *o = reinterpret_cast<MV4<float> *>(d.mrec) + macro_at_cell<float>(d, c, njp);
  auto put = [&](int plane, float a, float b, float e, float g) { o[(long)plane * njp] = MV4<float>{{a, b, e, g}}; };
  const bool on = d.cmask[c] & 1;
  const int f = d.cell_faces[4 * c + s];
  const double sg = (double)d.cell_sgn[4 * c + s];
  const double vol = d.vol_new[c], idtau = d.idtau[c], idt = d.stepc[1], Wm = d.W[4 * c + s], TW = d.TW[4 * c + s];
  const double S = d.S[f], g = d.gam[f], nx = d.nrm[2 * f], ny = d.nrm[2 * f + 1], un = d.Un[f];
  const int nb = (sg > 0) ? d.face_R[f] : d.face_L[f];
  const double Fc = cell_flux_sum(d, c, s);
  // missing neighbour: a harmless positive state (its increment is zero)
  float w[4];
#pragma unroll
  for (int m = 0; m < 4; ++m) w[m] = nb >= 0 ? (float)d.W[4 * nb + m] : (m == 0 || m == 3 ? 1.f : 0.f);
  const float r = on ? (float)(TW - vol * idt * Wm - 0.5 * Fc) : 0.f, gf = (float)g;
  double diag = vol * (idtau + idt);
  const unsigned all = 0xffffffffu;
  const int l0 = threadIdx.x & 28;
#pragma unroll
  for (int m = 0; m < 4; ++m) diag = __fma_rn(0.25 * __shfl_sync(all, S, l0 + m), __shfl_sync(all, g, l0 + m), diag);
  const float idg = (float)(1.0 / diag);
  float rv[4], gv[4];
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    rv[m] = __shfl_sync(all, r, l0 + m);
    gv[m] = __shfl_sync(all, gf, l0 + m);
  }
  if (t >> 2 >= d.nc) return;
  d.Fc[4 * c + s] = Fc;
  if (on) {
    const int plane = (s & 1 ? MP_BW : MP_FW) + (s & 2);
    put(plane, w[0], w[1], w[2], w[3]);
    put(plane + 1, (float)(sg * nx), (float)(sg * ny), (float)(sg * un), (float)(0.25 * S));
  }
  if (s == 0) put(MP_VAL, rv[0], rv[1], rv[2], rv[3]);
  if (s == 1) put(MP_FW + 4, on ? gv[0] : 0.f, on ? gv[2] : 0.f, on ? idg : 0.f, 0.f);
  if (s == 2) put(MP_BW + 4, on ? gv[1] : 0.f, on ? gv[3] : 0.f, on ? idg : 0.f, 0.f);
}

// Coupling (1/4 S)(Delta F_E . n - Gamma dW) of a neighbour with state w,
// outward normal, U.n and S/4 in e, and increment dw, the flux variation
// written out as a difference (one division, no cancellation between the two
// fluxes): with d(a b / rho) = (da b rho + a db rho + da db rho - a b drho) /
// (rho (rho + drho)) and p = (gamma - 1)(E - |m|^2 / (2 rho)).
__device__ __forceinline__ void macro_off(const float *w, const float *e, float gam, const float *dw, int Keff, float out[4]) {
  float r = w[0], m1 = w[1], m2 = w[2], E = w[3];
  float nx = e[0], ny = e[1], un = e[2];
  float dr = dw[0], d1 = dw[1], d2 = dw[2], dE = dw[3];
  float g1 = __fdividef(2.0f, 2.0f + (float)Keff);    // gamma - 1
  float mn = m1 * nx + m2 * ny, dmn = d1 * nx + d2 * ny;
  float den = __fdividef(1.0f, r * (r + dr));          // 1/(rho (rho + drho))
  float dq11 = (2.0f * (m1 * d1 + m2 * d2) * r + (d1 * d1 + d2 * d2) * r -
                (m1 * m1 + m2 * m2) * dr) * den;
  float dp = g1 * (dE - 0.5f * dq11);
  float p = g1 * (E - 0.5f * (m1 * m1 + m2 * m2) * ((r + dr) * den));
  float dv = (dmn * r - mn * dr) * den;               // d(mn / rho)
  float dF0 = dmn - dr * un;
  float dF1 = (d1 * mn * r + m1 * dmn * r + d1 * dmn * r - m1 * mn * dr) * den - d1 * un + dp * nx;
  float dF2 = (d2 * mn * r + m2 * dmn * r + d2 * dmn * r - m2 * mn * dr) * den - d2 * un + dp * ny;
  float dF3 = (dE * mn * r + E * dmn * r + dE * dmn * r - E * mn * dr) * den - dE * un +
              dp * (mn + dmn) * (r * den) + p * dv;
  float q = e[3], g = gam;
  out[0] = q * (dF0 - g * dr);
  out[1] = q * (dF1 - g * d1);
  out[2] = q * (dF2 - g * d2);
  out[3] = q * (dF3 - g * dE);
}

// The bands' copies of a diagonal: NPL planes of a band's RPB rows as 16-byte
// chunks over the lanes, from a ring of D diagonals.
template <typename T, int NPL, int RPB> struct MacroRing {
  typedef MV4<T> V;
  static constexpr int CPV = (int)sizeof(V) / 16, CPP = RPB * CPV, NCH = NPL * CPP / 32;
  static_assert(NPL * CPP % 32 == 0, "whole copies per lane");
  const char *src[NCH];
  V *rg;
  long step;             // bytes to the next diagonal
  // planes: VAL, then NPL - 1 planes given by plane(1), plane(2), ...
  template <typename F> __device__ __forceinline__ void init(const V *first, long njp, long stride, V *ring, int lane, F plane) {
#pragma unroll
    for (int m = 0; m < NCH; ++m) {
      const int q = lane + 32 * m, pl = q / CPP;
      src[m] = reinterpret_cast<const char *>(first + (long)(pl == 0 ? 0 : plane(pl)) * njp) + 16 * (q - pl * CPP);
    }
    rg = ring;
    step = stride * (long)sizeof(V);
  }
  __device__ __forceinline__ void copy(int slot, int lane) {
    char *dst = reinterpret_cast<char *>(rg + slot * NPL * RPB) + 16 * lane;
#pragma unroll
    for (int m = 0; m < NCH; ++m) {
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(smem_addr(dst + 512 * m)), "l"(src[m]) : "memory");
      src[m] += step;
    }
    cp_async_commit();
  }
  __device__ __forceinline__ const V *slot(int s, int row) const { return rg + s * NPL * RPB + row; }
};

// One pass (0 forward, 1 backward) over block b for this warp's band, FP32.
template <int K, int D, int PASS>
__device__ __forceinline__ void macro_pass32(const Dev &d, int b, int ni, int nj, bool per, int nb, MV4<float> *ring,
                                             float4 *links) {
  constexpr unsigned FULL = 0xffffffffu;
  constexpr int NPL = 1 + NPASS32, P0 = PASS == 0 ? MP_FW : MP_BW, Q0 = PASS == 0 ? MP_BW : MP_FW;
  static_assert(K % 2 == 0 && D >= 3, "register pair by step parity; a copy, a read and a free slot");
  typedef MV4<float> V;
  struct Rec { V v, wi, ei, wj, ej, c; };
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, row = w * 32 + lane;
  const int njp = macro_rows(nj), nd = ni + nj - 1;
  const int lead = PASS == 0 ? w : nb - 1 - w;         // position of the band in the sweep order
  const int total = (nd + (nb - 1) * (K - 1) + K - 1) / K * K;
  const int t0 = PASS == 0 ? -lead * (K - 1) : nd - 1 + lead * (K - 1);
  const long stride = (PASS == 0 ? 1 : -1) * (long)NMP32 * njp;          // to the next diagonal (vectors)
  V *rec0 = reinterpret_cast<V *>(d.mrec);
  V *ps = rec0 + macro_at<float>(d, b, t0, row);                         // this step's cell, plane 0
  MacroRing<float, NPL, 32> R;
  R.init(rec0 + macro_at<float>(d, b, t0, w * 32), njp, stride, ring + (size_t)w * D * NPL * 32, lane,
         [](int pl) { return P0 + pl - 1; });
  auto read = [&](int slot, Rec &r) {                                    // a lane reads what it copied itself
    const V *s = R.slot(slot, lane);
    r.v = s[0]; r.wi = s[32]; r.ei = s[64]; r.wj = s[96]; r.ej = s[128]; r.c = s[160];
  };
#pragma unroll
  for (int u = 0; u < D - 1; ++u) R.copy(u, lane);
  // the wrap of a periodic row: its last cell of the pass is coupled to its
  // first, across the slot the other pass's record holds
  const int ifirst = PASS == 0 ? 0 : ni - 1, ilast = PASS == 0 ? ni - 1 : 0;
  V ww = {{1.f, 0.f, 0.f, 1.f}}, we = {{0.f, 0.f, 0.f, 0.f}};
  float wg = 0.f, first[4] = {0.f, 0.f, 0.f, 0.f};
  if (per && row < nj) {
    const V *x = rec0 + macro_at<float>(d, b, ilast + row, row);
    ww = x[(long)Q0 * njp];
    we = x[(long)(Q0 + 1) * njp];
    wg = x[(long)(Q0 + 4) * njp].v[0];
  }
  float4 *rin = links + (size_t)lead * 2 * K, *rout = rin + 2 * K;       // link 0 stays zero
  if (lane < 2 * K) {
    rout[lane] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (lead == 0) rin[lane] = make_float4(0.f, 0.f, 0.f, 0.f);
  }
  float val[4] = {0.f, 0.f, 0.f, 0.f};
  const bool efirst = PASS == 0 ? lane == 0 : lane == 31, elast = PASS == 0 ? lane == 31 : lane == 0;
  int i = t0 - row, sc = D - 1, sr = 1;                // ring slots: next copy, next read
  Rec rec[2];
  cp_async_wait<D - 2>();
  read(0, rec[0]);
  for (int c = 0; c < total; c += K) {
    // the link half written before this barrier is read after it, and the
    // half read before it is written after it
    asm volatile("bar.sync 1, %0;" ::"r"(32 * nb) : "memory");
    const int hw = (c / K & 1) * K, hr = K - hw;
#pragma unroll 2
    for (int u = 0; u < K; ++u) {                      // (all eight would overrun the instruction cache)
      const Rec &r = rec[u & 1];
      R.copy(sc, lane);                                // into the slot read the step before last
      sc = sc + 1 == D ? 0 : sc + 1;
      cp_async_wait<D - 2>();
      read(sr, rec[(u & 1) ^ 1]);
      sr = sr + 1 == D ? 0 : sr + 1;
      // increments of the neighbours: along the row this lane's last one,
      // across rows the neighbour lane's or the band before's
      float up[4], oi[4], oj[4], acc[4];
      const float4 lk = rin[hr + u];
#pragma unroll
      for (int m = 0; m < 4; ++m) up[m] = PASS == 0 ? __shfl_up_sync(FULL, val[m], 1) : __shfl_down_sync(FULL, val[m], 1);
      if (efirst) { up[0] = lk.x; up[1] = lk.y; up[2] = lk.z; up[3] = lk.w; }
      macro_off(r.wi.v, r.ei.v, r.c.v[0], val, d.Keff, oi);
      macro_off(r.wj.v, r.ej.v, r.c.v[1], up, d.Keff, oj);
      if (per && i == ilast) {
        float ow[4];
        macro_off(ww.v, we.v, wg, first, d.Keff, ow);
#pragma unroll
        for (int m = 0; m < 4; ++m) oi[m] = __fadd_rn(oi[m], ow[m]);
      }
#pragma unroll
      for (int m = 0; m < 4; ++m) acc[m] = __fadd_rn(oi[m], oj[m]);
      const float idg = r.c.v[2];
      const bool on = idg != 0.f;                      // a solved cell; the others keep a zero increment
      V x;
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        x.v[m] = PASS == 0 ? (r.v.v[m] - acc[m]) * idg : r.v.v[m] - acc[m] * idg;
        val[m] = on ? x.v[m] : 0.f;
      }
      if (on) ps[0] = x;
      if (per && i == ifirst) {
#pragma unroll
        for (int m = 0; m < 4; ++m) first[m] = val[m];
      }
      if (elast) rout[hw + u] = make_float4(val[0], val[1], val[2], val[3]);
      ps += stride;
      i += PASS == 0 ? 1 : -1;
    }
  }
  cp_async_wait<0>();
}

// One pass over block b for this warp's band, FP64.
template <int LPR, int K, int D, int PASS>
__device__ __forceinline__ void macro_pass64(const Dev &d, int b, int ni, int nj, bool per, int nb, MV4<double> *ring,
                                             double *links) {
  typedef double T;
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
  const long stride = (PASS == 0 ? 1 : -1) * (long)NMP64 * njp;       // to the next diagonal (vectors)
  V *rec0 = reinterpret_cast<V *>(d.mrec);
  V *ps = rec0 + macro_at<T>(d, b, t0, row);                          // this step's cell, plane 0
  constexpr int P1 = PASS == 0 ? MP_F1 : MP_B1, P2 = PASS == 0 ? MP_F2 : MP_B2;
  MacroRing<T, 4, RPB> R;                              // planes VAL, ST and this pass's two
  R.init(rec0 + macro_at<T>(d, b, t0, w * RPB), njp, stride, ring + (size_t)w * D * 4 * RPB, lane,
         [](int pl) { return pl == 1 ? MP_ST : pl == 2 ? P1 : P2; });
  auto read = [&](int slot, Rec &r) {
    const V *s = R.slot(slot, lr);
#pragma unroll
    for (int m = 0; m < NC; ++m) r.v[m] = s[0].v[LPR == 1 ? m : sub];
    r.st = s[RPB];
    r.c1 = s[2 * RPB];
    r.c2 = s[3 * RPB];
  };
#pragma unroll
  for (int u = 0; u < D - 1; ++u) R.copy(u, lane);
  // couplings that wrap around a periodic row: from its first cell of the
  // pass to its last, with the coefficients of the other pass's record
  T wrap[NC], wc[3] = {T(0), T(0), T(0)};
  const int ifirst = PASS == 0 ? 0 : ni - 1, ilast = PASS == 0 ? ni - 1 : 0;
  if (per && row < nj) {
    const V x = (rec0 + macro_at<T>(d, b, ifirst + row, row))[(long)(PASS == 0 ? MP_B1 : MP_F1) * njp];
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
      R.copy(sc, lane);                                // into the slot read the step before last
      sc = sc + 1 == D ? 0 : sc + 1;
      cp_async_wait<D - 2>();
      __syncwarp();                                    // the band's copies, made by all its lanes
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
      const T ri = 1.0 / (rho + dw[0]);
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

// shared memory: the bands' rings, then the links [nb + 1][2 K][4]
template <typename T, int LPR, int D> __host__ __device__ constexpr size_t macro_ring(int nb) {
  return (size_t)nb * D * (sizeof(T) == 4 ? 1 + NPASS32 : 4) * (32 / LPR) * sizeof(MV4<T>);
}

template <typename T, int LPR, int K, int D>
__global__ void __launch_bounds__(sizeof(T) == 4 && D == 8 ? 256 : 512) k_macro_sweep(Dev d) {
  extern __shared__ __align__(16) unsigned char smraw[];
  const int b = blockIdx.x;
  const int *bi = d.blk_info + 8 * b;
  const int ni = bi[0], nj = bi[1], nb = (nj + 32 / LPR - 1) / (32 / LPR);
  const bool per = bi[2] != 0;
  MV4<T> *ring = reinterpret_cast<MV4<T> *>(smraw);
  unsigned char *links = smraw + macro_ring<T, LPR, D>(nb);
  if ((int)(threadIdx.x >> 5) >= nb) return;           // the named barrier counts the block's bands
  auto pass = [&](auto which) {
    constexpr int PASS = decltype(which)::value;
    if constexpr (sizeof(T) == 4) macro_pass32<K, D, PASS>(d, b, ni, nj, per, nb, ring, reinterpret_cast<float4 *>(links));
    else macro_pass64<LPR, K, D, PASS>(d, b, ni, nj, per, nb, ring, reinterpret_cast<double *>(links));
  };
  pass(std::integral_constant<int, 0>());
  // the increments stored above are copied by the same band's lanes in the
  // next pass; the links are free
  __threadfence();
  asm volatile("bar.sync 1, %0;" ::"r"(32 * nb) : "memory");
  pass(std::integral_constant<int, 1>());
}

// W' = W + dW and the predictor cell record (Step 4 result) for Step 5.  Small
// CTAs and loads before the stores, as in the gather above.
template <typename T> __global__ void __launch_bounds__(MPREP) k_macro_post(Dev d) {
  int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= d.nc) return;
  T *sr = reinterpret_cast<T *>(d.srec) + (size_t)NSR * c;
  int njp;
  const MV4<T> inc = reinterpret_cast<const MV4<T> *>(d.mrec)[macro_at_cell<T>(d, c, njp)];
  const bool on = d.cmask[c] & 1;
  const double2 w01 = *reinterpret_cast<const double2 *>(d.W + 4 * c), w23 = *reinterpret_cast<const double2 *>(d.W + 4 * c + 2);
  const double2 q = *reinterpret_cast<const double2 *>(d.q + 2 * c);
  const double vol = d.vol_new[c], idtau = d.idtau[c], idt = d.stepc[1];
  double W[4] = {w01.x, w01.y, w23.x, w23.y};
  if (on)
    for (int m = 0; m < 4; ++m) W[m] += (double)inc.v[m];
  reinterpret_cast<double2 *>(d.Wp + 4 * c)[0] = make_double2(W[0], W[1]);
  reinterpret_cast<double2 *>(d.Wp + 4 * c)[1] = make_double2(W[2], W[3]);
  if (!on) {
    sr[SR_DBASE] = T(0);
    return;
  }
  // the record of write_shrec from four divisions: T = 1 / (2 lam) = (gamma - 1) e,
  // 1 / tau = rho T / mu(T)
  const double ir = 1.0 / W[0], ux = W[1] * ir, uy = W[2] * ir;
  const double il = 2.0 / (2.0 + d.Keff) * (W[3] * ir - 0.5 * (ux * ux + uy * uy)), lam = 0.5 / il;
  double o[NCP];
  o[CP_RHO] = W[0]; o[CP_UX] = ux; o[CP_UY] = uy; o[CP_LAM] = lam;
  o[CP_QX] = q.x; o[CP_QY] = q.y;
  o[CP_ITAU] = W[0] * il / (d.mu_ref * pow(il, d.omega));
  o[CP_DBASE] = vol * (idtau + idt + 0.5 * o[CP_ITAU]);
  sr[SR_DBASE] = (T)o[CP_DBASE];
  write_shrec<T>(d, o, il, 0.8 * (1.0 - d.Pr) * lam * lam * ir, vol, reinterpret_cast<T *>(d.shp) + (size_t)NSH * c);
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
  if (fp32) k_macro_prep32<<<nblk(4 * (size_t)d.nc, 2 * MPREP), 2 * MPREP, 0, s>>>(d);
  else k_macro_prep64<<<nblk(d.nc, MPREP), MPREP, 0, s>>>(d);
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
    k_macro_post<float><<<nblk(d.nc, MPREP), MPREP, 0, s>>>(d);
  } else {
    if (rows <= 128) macro_launch<UGKS_MACRO(double, kShape64)>(d, s, nb);
    else macro_launch<UGKS_MACRO(double, kShape64Tall)>(d, s, nb);
    k_macro_post<double><<<nblk(d.nc, MPREP), MPREP, 0, s>>>(d);
  }
}

template <typename T, int LPR, int K, int D, int NB> static void macro_attr() {
  static_assert(macro_ring<T, LPR, D>(NB) + (NB + 1) * 2 * K * 4 * sizeof(T) <= kMacroSmem, "ring and links fit");
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
