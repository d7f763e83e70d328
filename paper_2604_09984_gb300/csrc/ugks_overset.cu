// ugks_overset.cu -- overset assembly (arXiv 2604.09984 Sec. 3.1) and
// inverse-distance interpolation (Sec. 3.2) on the device.
//
// Every geometric predicate uses explicit round-to-nearest FP64 operations
// (__dadd_rn, __dmul_rn, ...) so no multiply-add is contracted: the result is
// bit-identical to a plain FP64 evaluation of the same expressions in the
// same order.  Readings of the garbled classification sentence of Sec. 3.1:
//   * wall distance of a node to a zone: min squared distance to the zone's
//     wall segments (+inf without walls);
//   * a node of zone Z is inactive if it lies inside another zone's body
//     polygon, or inside a core cell (not within n_fringe + n_gap layers of an
//     overset edge) of a zone D with a smaller wall distance (ties: higher
//     priority wins);
//   * cells: all nodes inactive -> hole, mixed -> boundary, fringe layers ->
//     receptor; active face neighbours of boundary or hole cells form the
//     buffer layer (receptors); the rest are field cells;
//   * donor: the containing cell of another zone, field cells before
//     receptor cells, then (priority desc, block, cell index); stencil =
//     donor + its non-hole face neighbours (order i-1, i+1, j-1, j+1),
//     weights d^-2 normalised in that order (Sec. 3.2).
//
// The FP64 predicates decide everything; float filters in front of them only
// skip work whose outcome they already know exactly: with rn() the
// round-to-nearest map to float (monotone), rn(a) > rn(b) implies a > b.
#include <algorithm>

#include "ugks_internal.cuh"
#include "ugks_launch.h"

namespace ugks {

enum { CL_ACTIVE = 0, CL_MIXED = 1, CL_HOLE = 2, CL_FRINGE = 3 };

__device__ __forceinline__ double ad(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ double sb(double a, double b) { return __dsub_rn(a, b); }
__device__ __forceinline__ double ml(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ double dv(double a, double b) { return __ddiv_rn(a, b); }

// squared distance of (x, y) to wall segment s (exact FP64 expression)
__device__ __forceinline__ double seg_dist2(const Dev &d, int s, double x, double y) {
  int a = d.wall_seg[2 * s], b = d.wall_seg[2 * s + 1];
  double ax = d.X_new[2 * a], ay = d.X_new[2 * a + 1];
  double ex = sb(d.X_new[2 * b], ax), ey = sb(d.X_new[2 * b + 1], ay);
  double px = sb(x, ax), py = sb(y, ay);
  double t = dv(ad(ml(px, ex), ml(py, ey)), ad(ml(ex, ex), ml(ey, ey)));
  t = fmin(fmax(t, 0.0), 1.0);
  double dx = sb(px, ml(t, ex)), dy = sb(py, ml(t, ey));
  return ad(ml(dx, dx), ml(dy, dy));
}

// Wall distances and the body test of a node run over a group of NLANES lanes
// (each takes every NLANES-th segment; all of them get the result).
constexpr int NLANES = 8;
struct Group {
  unsigned mask;
  int lane;
  __device__ Group() : mask(0xffu << (threadIdx.x & 24)), lane(threadIdx.x & (NLANES - 1)) {}
  template <typename V> __device__ V down(V v, int o) const { return __shfl_xor_sync(mask, v, o); }
};
static_assert(NLANES == 8, "the group's lane mask");

// Segment nearest to (x, y) in float, and a bracket [lo, hi] of the squared
// distance to the nearest one in floats that allow for all roundings: lo from
// the distances to the segments' bounding boxes, shrunk, hi from the point
// found on the near segment (any point on it bounds), widened by 1e-6 of the
// coordinates (some 16 float roundings of 6e-8).
// `seg` holds the float endpoints (A.x, A.y, B.x, B.y) of every segment
// (shared memory, or the global copy when they do not fit there).
__device__ __forceinline__ float seg_size(float4 AB, float xf, float yf) {
  return fabsf(xf) + fabsf(yf) + fabsf(AB.x) + fabsf(AB.y) + fabsf(AB.z) + fabsf(AB.w);
}
__device__ __forceinline__ float seg_bound(float4 AB, float xf, float yf) {
  float lx = fminf(AB.x, AB.z), hx = fmaxf(AB.x, AB.z), ly = fminf(AB.y, AB.w), hy = fmaxf(AB.y, AB.w);
  float tol = 2.4e-7f * seg_size(AB, xf, yf);
  float gx = fmaxf(fmaxf(lx - xf, xf - hx) - tol, 0.f);
  float gy = fmaxf(fmaxf(ly - yf, yf - hy) - tol, 0.f);
  return (gx * gx + gy * gy) * 0.99999f;
}
__device__ int near_segment(const Group &g, const float4 *seg, int s0, int s1, float xf, float yf, float &lo, float &hi) {
  int sg = s0;
  float gbest = __int_as_float(0x7f800000);
  lo = hi = gbest;
  for (int s = s0 + g.lane; s < s1; s += NLANES) {
    float4 AB = seg[s];
    float ex = AB.z - AB.x, ey = AB.w - AB.y, px = xf - AB.x, py = yf - AB.y;
    float ee = ex * ex + ey * ey;
    float t = ee > 0.f ? fminf(fmaxf(__fdividef(px * ex + py * ey, ee), 0.f), 1.f) : 0.f;
    float dx = fabsf(px - t * ex), dy = fabsf(py - t * ey), d2 = dx * dx + dy * dy;
    if (d2 < gbest) {
      gbest = d2;
      sg = s;
      const float tol = 1e-6f * seg_size(AB, xf, yf);
      hi = ((dx + tol) * (dx + tol) + (dy + tol) * (dy + tol)) * 1.00001f;
    }
    lo = fminf(lo, seg_bound(AB, xf, yf));
  }
#pragma unroll
  for (int o = NLANES / 2; o > 0; o >>= 1) {
    const float ob = g.down(gbest, o), oh = g.down(hi, o), ol = g.down(lo, o);
    const int os = g.down(sg, o);
    if (ob < gbest || (ob == gbest && os < sg)) { gbest = ob; sg = os; }
    hi = fminf(hi, oh);
    lo = fminf(lo, ol);
  }
  return sg;
}

// Minimum squared distance to the zone's wall segments exactly (+inf without):
// the near segment's exact distance bounds it; then only segments whose float
// lower bound does not exceed that bound are evaluated exactly.  The skipped
// ones are farther than the minimum.
__device__ double wall_dist2(const Group &g, const Dev &d, const float4 *seg, int blk, double x, double y) {
  double best = __longlong_as_double(0x7ff0000000000000LL);   // +inf
  int s0 = d.wall_seg_off[blk], s1 = d.wall_seg_off[blk + 1];
  if (s1 <= s0) return best;
  float xf = __double2float_rn(x), yf = __double2float_rn(y), lo, hi;
  int sg = near_segment(g, seg, s0, s1, xf, yf, lo, hi);
  best = seg_dist2(d, sg, x, y);
  float bestf = __double2float_ru(best);
  for (int s = s0 + g.lane; s < s1; s += NLANES) {
    if (s == sg || seg_bound(seg[s], xf, yf) > bestf) continue;
    double d2 = seg_dist2(d, s, x, y);
    if (d2 < best) { best = d2; bestf = __double2float_ru(best); }
  }
#pragma unroll
  for (int o = NLANES / 2; o > 0; o >>= 1) best = fmin(best, g.down(best, o));
  return best;
}

__device__ bool inside_quad(const Dev &d, int c, double x, double y) {
  const int *nd = d.cell_nodes + 4 * c;
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    int a = nd[e], b = nd[(e + 1) & 3];
    double ax = d.X_new[2 * a], ay = d.X_new[2 * a + 1];
    double bx = d.X_new[2 * b], by = d.X_new[2 * b + 1];
    double cr = sb(ml(sb(bx, ax), sb(y, ay)), ml(sb(by, ay), sb(x, ax)));
    if (!(cr >= 0.0)) return false;
  }
  return true;
}

// Float boxes of each block's body polygon and of its bins, rounded outward (one
// warp per block): a point outside the first is outside the polygon, outside
// the second in no bin.  (A coordinate rounded to float keeps its side of a
// float bound, so the tests against them need no FP64.)
__global__ void k_body_box(Dev d) {
  int b = blockIdx.x, lane = threadIdx.x;
  int r0 = d.body_ring_off[b], r1 = d.body_ring_off[b + 1];
  double xl = 1e300, xh = -1e300, yl = 1e300, yh = -1e300;
  for (int i = r0 + lane; i < r1; i += 32) {
    int a = d.body_ring[i];
    double x = d.X_new[2 * a], y = d.X_new[2 * a + 1];
    xl = fmin(xl, x); xh = fmax(xh, x); yl = fmin(yl, y); yh = fmax(yh, y);
  }
  for (int o = 16; o > 0; o >>= 1) {
    xl = fmin(xl, __shfl_xor_sync(0xffffffffu, xl, o));
    xh = fmax(xh, __shfl_xor_sync(0xffffffffu, xh, o));
    yl = fmin(yl, __shfl_xor_sync(0xffffffffu, yl, o));
    yh = fmax(yh, __shfl_xor_sync(0xffffffffu, yh, o));
  }
  if (lane == 0)
    d.body_bb[b] = make_float4(__double2float_rd(xl), __double2float_rd(yl), __double2float_ru(xh),
                               __double2float_ru(yh));
  if (lane == 0) {      // the bins' box, widened past the roundings of bin_of
    const double *g = d.bin_geo + 4 * b;
    const double w = d.bin_dim[3 * b] / g[2], h = d.bin_dim[3 * b + 1] / g[3];
    const double px = 1e-12 * (fabs(g[0]) + w), py = 1e-12 * (fabs(g[1]) + h);
    d.bin_bb[b] = make_float4(__double2float_rd(g[0] - px), __double2float_rd(g[1] - py),
                              __double2float_ru(g[0] + w + px), __double2float_ru(g[1] + h + py));
  }
}

__device__ __forceinline__ bool in_box(float4 bb, float x, float y) {
  return !(x < bb.x || x > bb.z || y < bb.y || y > bb.w);
}
__device__ __forceinline__ bool in_body_box(const Dev &d, int blk, float x, float y) {
  return d.body_ring_off[blk + 1] > d.body_ring_off[blk] && in_box(d.body_bb[blk], x, y);
}

__device__ bool inside_body(const Group &g, const Dev &d, int blk, double x, double y) {
  float yf = __double2float_rn(y);
  if (!in_body_box(d, blk, __double2float_rn(x), yf)) return false;
  int r0 = d.body_ring_off[blk], r1 = d.body_ring_off[blk + 1];
  int M = r1 - r0, in = 0;
  for (int i = g.lane; i < M; i += NLANES) {
    int a = d.body_ring[r0 + i], b = d.body_ring[r0 + (i + 1 < M ? i + 1 : 0)];
    // side of y for each end from the floats where they differ, else exactly
    float af = d.Xf[a].y, bf = d.Xf[b].y;
    int sa = af > yf ? 1 : (af < yf ? -1 : 0), sbv = bf > yf ? 1 : (bf < yf ? -1 : 0);
    if (sa != 0 && sa == sbv) continue;                   // both above or both below
    double ax = d.X_new[2 * a], ay = d.X_new[2 * a + 1];
    double bx = d.X_new[2 * b], by = d.X_new[2 * b + 1];
    bool crosses = (ay > y) != (by > y);
    if (crosses) {
      double xint = ad(ax, dv(ml(sb(y, ay), sb(bx, ax)), sb(by, ay)));
      if (x < xint) in ^= 1;
    }
  }
#pragma unroll
  for (int o = NLANES / 2; o > 0; o >>= 1) in ^= g.down(in, o);
  return in != 0;
}

__device__ __forceinline__ bool in_layer(const int *bi, int i, int j, int L) {
  int ni = bi[0], nj = bi[1], mask = bi[6];
  if ((mask & 1) && i < L) return true;
  if ((mask & 2) && i >= ni - L) return true;
  if ((mask & 4) && j < L) return true;
  if ((mask & 8) && j >= nj - L) return true;
  return false;
}

// ---------------------------------------------------------------- bins
// Per block a uniform grid of bins over a box containing the block at
// t^{n+1}; every cell is registered in the bins its bounding box overlaps.
// A point lies in the bin (floor((x-x0)/hx), floor((y-y0)/hy)); a cell that
// contains the point overlaps that bin (floor is monotone), so the minimum
// index among the bin's candidates that contain the point equals the minimum
// over all cells: same result as a scan of the whole block.
__device__ __forceinline__ void bin_range(const Dev &d, int b, double lo, double hi, int axis,
                                          int &i0, int &i1) {
  const double *g = d.bin_geo + 4 * b;
  int n = d.bin_dim[3 * b + axis];
  double x0 = g[axis], ih = g[2 + axis];
  double a = floor((lo - x0) * ih), c = floor((hi - x0) * ih);
  i0 = a < 0.0 ? 0 : (a > n - 1 ? n - 1 : (int)a);
  i1 = c < 0.0 ? 0 : (c > n - 1 ? n - 1 : (int)c);
}

__device__ __forceinline__ int bin_of(const Dev &d, int b, double x, double y) {
  const double *g = d.bin_geo + 4 * b;
  int nx = d.bin_dim[3 * b], ny = d.bin_dim[3 * b + 1];
  double a = floor((x - g[0]) * g[2]), c = floor((y - g[1]) * g[3]);
  if (a < 0.0 || c < 0.0 || a > nx - 1 || c > ny - 1) return -1;
  return d.bin_dim[3 * b + 2] + (int)c * nx + (int)a;
}

__global__ void k_node_f(Dev d) {
  int n = blockIdx.x * blockDim.x + threadIdx.x;
  if (n == 0) *d.node_todo_n = 0;
  if (n < d.nn)
    d.Xf[n] = make_float2(__double2float_rn(d.X_new[2 * n]), __double2float_rn(d.X_new[2 * n + 1]));
  if (n < d.nseg) {      // float endpoints of wall segment n, one record each
    int a = d.wall_seg[2 * n], b = d.wall_seg[2 * n + 1];
    d.segf[n] = make_float4(__double2float_rn(d.X_new[2 * a]), __double2float_rn(d.X_new[2 * a + 1]),
                            __double2float_rn(d.X_new[2 * b]), __double2float_rn(d.X_new[2 * b + 1]));
  }
}

// bounding box and bin range of every cell (at most 2048 bins an axis)
__global__ void k_bin_count(Dev d) {
  int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= d.nc) return;
  int b = d.cell_block[c];
  const int4 n4 = *reinterpret_cast<const int4 *>(d.cell_nodes + 4 * c);
  const double2 *X = reinterpret_cast<const double2 *>(d.X_new);
  const double2 p0 = X[n4.x], p1 = X[n4.y], p2 = X[n4.z], p3 = X[n4.w];
  const double xl = fmin(fmin(fmin(p0.x, p1.x), p2.x), p3.x), xh = fmax(fmax(fmax(p0.x, p1.x), p2.x), p3.x);
  const double yl = fmin(fmin(fmin(p0.y, p1.y), p2.y), p3.y), yh = fmax(fmax(fmax(p0.y, p1.y), p2.y), p3.y);
  d.cbb[c] = make_float4(__double2float_rd(xl), __double2float_rd(yl), __double2float_ru(xh),
                         __double2float_ru(yh));
  int ix0, ix1, iy0, iy1;
  bin_range(d, b, xl, xh, 0, ix0, ix1);
  bin_range(d, b, yl, yh, 1, iy0, iy1);
  d.bin_rng[c] = make_int2(ix0 | iy0 << 16, ix1 | iy1 << 16);
  int nx = d.bin_dim[3 * b], base = d.bin_dim[3 * b + 2];
  for (int iy = iy0; iy <= iy1; ++iy)
    for (int ix = ix0; ix <= ix1; ++ix) atomicAdd(&d.bin_cnt[base + iy * nx + ix], 1);
}

// Exclusive scan of the bin counts.  Each CTA adds the counts before its
// chunk itself (75,000 bins: at most 73 loads of 16 bytes a thread, from L2),
// so the CTAs need no order among them: 110 us with one CTA, 11 so.
constexpr int SCAN_THREADS = 256, SCAN_CHUNK = 4 * SCAN_THREADS;
__global__ void __launch_bounds__(SCAN_THREADS) k_bin_scan(Dev d) {
  __shared__ int wsum[2][SCAN_THREADS / 32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, n = d.nbins;
  const int4 *cnt = reinterpret_cast<const int4 *>(d.bin_cnt);
  int before = 0;
#pragma unroll 8
  for (int q = threadIdx.x; q < (int)blockIdx.x * SCAN_THREADS; q += SCAN_THREADS) {
    const int4 v = cnt[q];
    before += v.x + v.y + v.z + v.w;
  }
  const int i0 = blockIdx.x * SCAN_CHUNK + 4 * threadIdx.x;
  int v[4];
#pragma unroll
  for (int m = 0; m < 4; ++m) v[m] = i0 + m < n ? d.bin_cnt[i0 + m] : 0;
  const int mine = v[0] + v[1] + v[2] + v[3];
  int incl = mine;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int t = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += t;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) before += __shfl_xor_sync(0xffffffffu, before, o);
  if (lane == 31) { wsum[0][w] = before; wsum[1][w] = incl; }
  __syncthreads();
  int run = incl - mine;
#pragma unroll
  for (int q = 0; q < SCAN_THREADS / 32; ++q) {
    run += wsum[0][q];
    if (q < w) run += wsum[1][q];
  }
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    if (i0 + m < n) d.bin_start[i0 + m] = run;
    run += v[m];
    if (i0 + m == n - 1) {
      d.bin_start[n] = run;
      if (run > d.bin_cap) atomicOr(d.err, EF_BINS);
    }
  }
}

// (the counts run down as the bins fill)
__global__ void k_bin_fill(Dev d) {
  int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= d.nc) return;
  const int2 rng = d.bin_rng[c];
  const int b = d.cell_block[c], nx = d.bin_dim[3 * b], base = d.bin_dim[3 * b + 2];
  for (int iy = rng.x >> 16; iy <= rng.y >> 16; ++iy)
    for (int ix = rng.x & 0xffff; ix <= (rng.y & 0xffff); ++ix) {
      const int bin = base + iy * nx + ix;
      const int pos = d.bin_start[bin] + atomicSub(&d.bin_cnt[bin], 1) - 1;
      if (pos < d.bin_cap) d.bin_items[pos] = c;
    }
}

// lowest-index cell of block b containing (x, y) among the cells accepted by
// `ok` (bins guarantee the same answer as a scan of the block); the group's
// lanes share the bin's candidates (a bin at a stretched wall holds a hundred)
template <typename Pred>
__device__ int first_containing(const Group &g, const Dev &d, int b, double x, double y, Pred ok) {
  const float xf = __double2float_rn(x), yf = __double2float_rn(y);
  if (!in_box(d.bin_bb[b], xf, yf)) return -1;
  int bin = bin_of(d, b, x, y);
  if (bin < 0) return -1;
  int best = 0x7fffffff;
  int q1 = min(d.bin_start[bin + 1], d.bin_cap);
  for (int q = d.bin_start[bin] + g.lane; q < q1; q += NLANES) {
    int c = d.bin_items[q];
    if (c >= best) continue;
    if (!in_box(d.cbb[c], xf, yf)) continue;     // the cell lies inside its box
    if (ok(c) && inside_quad(d, c, x, y)) best = c;
  }
#pragma unroll
  for (int o = NLANES / 2; o > 0; o >>= 1) best = min(best, g.down(best, o));
  return best == 0x7fffffff ? -1 : best;
}

// Whether a cell of block b outside its outer layers contains (x, y)
__device__ bool in_core(const Group &g, const Dev &d, int b, double x, double y) {
  const int *bi = d.blk_info + 8 * b;
  const int ni = bi[0], L = bi[4] + bi[5], c0 = d.cell_off[b];
  return first_containing(g, d, b, x, y, [&](int c) {
    int loc = c - c0;
    return !in_layer(bi, loc % ni, loc / ni, L);
  }) >= 0;
}

// Node classification.  Most nodes lie in no other zone's bins and no body's
// box: one thread a node finds them active from float boxes.  The others go to
// a list, whose nodes take a group of lanes each in a second launch: their
// loops over a bin's candidates, wall segments and body edges (some 20,000
// instructions a node for three blocks with 192 segments) belong to
// neighbouring nodes, so that one thread a node left them to few warps (150784
// nodes: 128 us, 6 + 64 in two launches).
__global__ void __launch_bounds__(128) k_node_classify(Dev d) {
  const int n = blockIdx.x * blockDim.x + threadIdx.x;
  bool todo = false;
  if (n < d.nn) {
    const int z = d.node_block[n];
    const float2 X = d.Xf[n];
    for (int b = 0; b < d.nblocks && !todo; ++b)
      todo = b != z && (in_box(d.bin_bb[b], X.x, X.y) || in_body_box(d, b, X.x, X.y));
    d.node_active[n] = 1;
  }
  const unsigned all = __ballot_sync(0xffffffffu, todo);
  if (!all) return;
  const int lane = threadIdx.x & 31;
  int at = 0;
  if (lane == 0) at = atomicAdd(d.node_todo_n, __popc(all));
  at = __shfl_sync(0xffffffffu, at, 0);
  if (todo) d.node_todo[at + __popc(all & ((1u << lane) - 1u))] = n;
}

// the wall segments' float records are staged in shared memory when they fit
// (STAGE)
template <bool STAGE> __global__ void __launch_bounds__(256) k_node_todo(Dev d) {
  extern __shared__ float4 seg_s[];
  const int count = *d.node_todo_n;
  if ((int)(blockIdx.x * blockDim.x / NLANES) >= count) return;
  if (STAGE) {
    for (int q = threadIdx.x; q < d.nseg; q += blockDim.x) seg_s[q] = d.segf[q];
    __syncthreads();
  }
  const float4 *seg = STAGE ? seg_s : d.segf;
  const Group g;
  const float inf = __int_as_float(0x7f800000);
  for (int t = (blockIdx.x * blockDim.x + threadIdx.x) / NLANES; t < count; t += gridDim.x * blockDim.x / NLANES) {
    const int n = d.node_todo[t], z = d.node_block[n];
    const double x = d.X_new[2 * n], y = d.X_new[2 * n + 1];
    const float xf = __double2float_rn(x), yf = __double2float_rn(y);
    auto bracket = [&](int b, float &lo, float &hi) {        // of the distance to b's walls; both +inf without
      lo = hi = inf;
      const int s0 = d.wall_seg_off[b], s1 = d.wall_seg_off[b + 1];
      if (s1 > s0) near_segment(g, seg, s0, s1, xf, yf, lo, hi);
    };
    // the exact distances are needed only where their brackets overlap:
    // elsewhere the brackets decide db < dz (or db > dz) as they would
    double dz = 0.0;
    float zlo = 0.f, zhi = 0.f;
    bool have_z = false, have_dz = false, inact = false;
    for (int b = 0; b < d.nblocks && !inact; ++b) {
      if (b == z) continue;
      if (inside_body(g, d, b, x, y)) {
        inact = true;
        break;
      }
      if (!in_core(g, d, b, x, y)) continue;
      if (!have_z) {
        bracket(z, zlo, zhi);
        have_z = true;
      }
      float blo, bhi;
      bracket(b, blo, bhi);
      if (bhi < zlo) {                  // db <= bhi < zlo <= dz
        inact = true;
      } else if (!(blo > zhi)) {        // brackets overlap: exact values
        if (!have_dz) {
          dz = wall_dist2(g, d, seg, z, x, y);
          have_dz = true;
        }
        double db = wall_dist2(g, d, seg, b, x, y);
        if (db < dz || (db == dz && d.blk_info[8 * b + 3] > d.blk_info[8 * z + 3])) inact = true;
      }                                 // else db >= blo > zhi >= dz: stays active
    }
    if (inact && g.lane == 0) d.node_active[n] = 0;
  }
}

__global__ void k_cell_classify(Dev d) {
  int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= d.nc) return;
  const int *nd = d.cell_nodes + 4 * c;
  int na = d.node_active[nd[0]] + d.node_active[nd[1]] + d.node_active[nd[2]] + d.node_active[nd[3]];
  int b = d.cell_block[c];
  const int *bi = d.blk_info + 8 * b;
  int loc = c - d.cell_off[b];
  int i = loc % bi[0], j = loc / bi[0];
  int cl;
  if (na == 0) cl = CL_HOLE;
  else if (na < 4) cl = CL_MIXED;
  else if (in_layer(bi, i, j, bi[4])) cl = CL_FRINGE;
  else cl = CL_ACTIVE;
  d.cls[c] = cl;
}

// status from the classes; buffer layer; fresh cells (hole -> field) flagged
// with bit 8 of prev_status scratch
__global__ void k_cell_buffer(Dev d, int *prev_status) {
  int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= d.nc) return;
  int cl = d.cls[c];
  int st;
  if (cl == CL_HOLE) st = ST_HOLE;
  else if (cl == CL_MIXED || cl == CL_FRINGE) st = ST_RECEPTOR;
  else {
    st = ST_FIELD;
    for (int s = 0; s < 4; ++s) {
      if (d.nb_kind[4 * c + s] != NB_CELL) continue;
      int nc2 = d.cls[d.nb_id[4 * c + s]];
      if (nc2 == CL_MIXED || nc2 == CL_HOLE) st = ST_RECEPTOR;
    }
  }
  int prev = prev_status[c];
  prev_status[c] = (prev == ST_HOLE && st == ST_FIELD) ? 1 : 0;   // fresh flag
  d.status[c] = st;
}

// Donor search and IDW weights of receptor and fresh cells; all other rows are
// cleared.  A CTA lists the searching ones of its 32 cells and gives each a group of lanes
// (bins' candidates, then a lane per donor); one thread a cell left the search,
// a chain of dependent loads, to a few lanes of a warp (149504 cells: 43 us,
// 22 so).
constexpr int DONOR_CELLS = 32, DONOR_THREADS = DONOR_CELLS * NLANES;
__global__ void __launch_bounds__(DONOR_THREADS) k_donor(Dev d, const int *fresh_flag, const int *blk_order,
                                                         int *n_orphan) {
  __shared__ int list[DONOR_CELLS], count;
  if (threadIdx.x == 0) count = 0;
  __syncthreads();
  const int c0 = blockIdx.x * DONOR_CELLS, cells = min(DONOR_CELLS, d.nc - c0), here = c0 + threadIdx.x;
  if ((int)threadIdx.x < cells && (d.status[here] == ST_RECEPTOR || fresh_flag[here])) list[atomicAdd(&count, 1)] = here;
  for (int t = threadIdx.x; t < 5 * cells; t += DONOR_THREADS) {
    d.donors[5 * (size_t)c0 + t] = -1;
    d.dwgt[5 * (size_t)c0 + t] = 0.0;
  }
  __syncthreads();
  const Group g;
  const int t = threadIdx.x / NLANES;
  if (t < count) {
    const int c = list[t], own = d.cell_block[c];
    const double x = d.xc_new[2 * c], y = d.xc_new[2 * c + 1];
    int found = -1;
    for (int cls = ST_FIELD; cls <= ST_RECEPTOR && found < 0; ++cls)
      for (int o = 0; o < d.nblocks && found < 0; ++o) {
        int b = blk_order[o];
        if (b != own) found = first_containing(g, d, b, x, y, [&](int q) { return d.status[q] == cls; });
      }
    if (found < 0) {
      if (g.lane == 0) atomicAdd(n_orphan, 1);
      return;
    }
    // lane 0: the found cell, lanes 1 to 4 its neighbours that are no holes
    int e = g.lane == 0 ? found : -1;
    if (g.lane >= 1 && g.lane < 5 && d.nb_kind[4 * found + g.lane - 1] == NB_CELL) {
      e = d.nb_id[4 * found + g.lane - 1];
      if (d.status[e] == ST_HOLE) e = -1;
    }
    double d2 = 1.0;
    if (e >= 0) {
      const double ex = sb(x, d.xc_new[2 * e]), ey = sb(y, d.xc_new[2 * e + 1]);
      d2 = ad(ml(ex, ex), ml(ey, ey));
    }
    const int shift = threadIdx.x & 24;
    const unsigned valid = __ballot_sync(g.mask, e >= 0) >> shift & 0xffu;
    const unsigned zero = __ballot_sync(g.mask, e >= 0 && d2 == 0.0) >> shift & 0xffu;
    const int m = __popc(valid & ((1u << g.lane) - 1u));          // the lane's place in the row
    const double inv = dv(1.0, d2);
    double tot = 0.0;
#pragma unroll
    for (int l = 0; l < 5; ++l) {                                 // in the row's order
      const double v = __shfl_sync(g.mask, inv, l, NLANES);
      if (valid >> l & 1u) tot = ad(tot, v);
    }
    if (e >= 0) {
      d.donors[5 * (size_t)c + m] = e;
      d.dwgt[5 * (size_t)c + m] = zero ? (g.lane == __ffs(zero) - 1 ? 1.0 : 0.0) : dv(inv, tot);
    }
  }
}

// Receptor and fresh-cell lists, compacted on the device in ascending cell
// order (two passes over 1024-cell chunks: count, then scan and write), so
// that no host round trip sits between the assembly and the step.
constexpr int LCHUNK = 1024;

__global__ void __launch_bounds__(LCHUNK) k_list_count(Dev d, const int *fresh_flag) {
  int c = blockIdx.x * LCHUNK + threadIdx.x;
  bool in = c < d.nc;
  int st = in ? d.status[c] : -1;
  int nr = __syncthreads_count(in && st == ST_RECEPTOR);
  int nfr = __syncthreads_count(in && fresh_flag[c] != 0);
  int nfd = __syncthreads_count(in && st == ST_FIELD);
  int no = __syncthreads_count(in && st != ST_FIELD && st != ST_RECEPTOR);
  if (threadIdx.x == 0) d.conn_chunk[blockIdx.x] = make_int4(nr, nfr, nfd, no);
}

__global__ void __launch_bounds__(LCHUNK) k_list_write(Dev d, const int *fresh_flag, const int *n_orphan) {
  __shared__ int base[2];
  __shared__ int wcnt[2][LCHUNK / 32];
  int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  if (w == 0) {   // offsets of this chunk: totals of the earlier chunks
    int a = 0, b = 0;
    for (int q = lane; q < (int)blockIdx.x; q += 32) {
      int4 v = d.conn_chunk[q];
      a += v.x;
      b += v.y;
    }
    for (int o = 16; o >= 1; o >>= 1) {
      a += __shfl_xor_sync(0xffffffffu, a, o);
      b += __shfl_xor_sync(0xffffffffu, b, o);
    }
    if (lane == 0) { base[0] = a; base[1] = b; }
  }
  int c = blockIdx.x * LCHUNK + threadIdx.x;
  bool in = c < d.nc;
  bool isr = in && d.status[c] == ST_RECEPTOR;
  bool isf = in && fresh_flag[c] != 0;
  unsigned mr = __ballot_sync(0xffffffffu, isr), mf = __ballot_sync(0xffffffffu, isf);
  if (lane == 0) { wcnt[0][w] = __popc(mr); wcnt[1][w] = __popc(mf); }
  __syncthreads();
  int orr = base[0], off = base[1];
  for (int q = 0; q < w; ++q) { orr += wcnt[0][q]; off += wcnt[1][q]; }
  unsigned below = (1u << lane) - 1u;
  int ir = orr + __popc(mr & below), jf = off + __popc(mf & below);
  if (isr && ir < d.cap_interp) d.rec_list[ir] = c;
  if (isf && jf < d.cap_interp) d.fresh_list[jf] = c;
  if (blockIdx.x == gridDim.x - 1 && w == 0) {   // totals and their checks
    int t[4] = {0, 0, 0, 0};
    for (int q = lane; q < (int)gridDim.x; q += 32) {
      int4 v = d.conn_chunk[q];
      t[0] += v.x; t[1] += v.y; t[2] += v.z; t[3] += v.w;
    }
#pragma unroll
    for (int m = 0; m < 4; ++m)
      for (int o = 16; o >= 1; o >>= 1) t[m] += __shfl_xor_sync(0xffffffffu, t[m], o);
    if (lane == 0) {
      int no = *n_orphan;
      d.conn_cnt[0] = t[0]; d.conn_cnt[1] = t[1]; d.conn_cnt[2] = t[2]; d.conn_cnt[3] = t[3];
      d.conn_cnt[4] = no;
      if (t[0] > d.cap_interp || t[1] > d.cap_interp) atomicOr(d.err, EF_CAPACITY);
      if (no > 0) atomicOr(d.err, EF_ORPHAN);
    }
  }
}

// Jacobi interpolation: gather into staging, then scatter.  The list length
// is read on the device (*cnt, clamped to the staging capacity); a fixed grid
// strides over it.
// parts: bit 0 the distributions, bit 1 W and q (the two may run apart: the
// distributions right after the micro sweep, W and q after Step 7)
//
// A CTA takes one receptor and up to INTERP_CHUNK velocities at a time, so that
// list, donors and weights are read (and the weights converted, which passes
// the FP64 pipe) once a warp and not once a velocity; the first warp's lanes
// take the components of W and q.  Both parts, gather and scatter: 256x128 +
// 128x32 cells, 1024 velocities 33 us -> 21; 512x256 + 2 x 192x48, 4096: 305 ->
// 121.
constexpr int INTERP_THREADS = 256, INTERP_CHUNK = 2 * INTERP_THREADS;
template <typename T> __global__ void __launch_bounds__(INTERP_THREADS) k_interp_gather(Dev d, const int *list,
                                                                                       const int *cnt, int parts) {
  const int n = min(*cnt, d.cap_interp), lane = threadIdx.x & 31;
  const int nch = (parts & 1) ? (d.nvp + INTERP_CHUNK - 1) / INTERP_CHUNK : 1;
  for (int u = blockIdx.x; u < n * nch; u += gridDim.x) {
    const int r = u / nch, ch = u - r * nch, c = list[r];
    const int e0 = lane < 5 ? d.donors[5 * c + lane] : -1;
    const double w0 = lane < 5 ? d.dwgt[5 * c + lane] : 0.0;
    const T t0 = (T)w0;
    int e[5];
#pragma unroll
    for (int m = 0; m < 5; ++m) e[m] = __shfl_sync(0xffffffffu, e0, m);
    if (parts & 1) {
      // f in the arithmetic type (its storage type): FP32 weights and sums on
      // the mixed path keep the FP64 pipe out of the per-velocity loop
      T w[5];
#pragma unroll
      for (int m = 0; m < 5; ++m) w[m] = __shfl_sync(0xffffffffu, t0, m);
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const int k = ch * INTERP_CHUNK + j * INTERP_THREADS + threadIdx.x;
        if (k >= d.nvp) continue;
        T ah = T(0), ab = T(0);
#pragma unroll
        for (int m = 0; m < 5; ++m) {
          if (e[m] < 0) continue;
          auto v = ldF<T>(d, (size_t)e[m] * d.nvp + k);
          ah = ah + w[m] * v.x;
          ab = ab + w[m] * v.y;
        }
        stf<T>(d.itmp, (size_t)r * d.nvp + k, ah, ab);
      }
    }
    if ((parts & 2) && ch == 0 && threadIdx.x < 32) {
      double acc = 0.0;
#pragma unroll
      for (int m = 0; m < 5; ++m) {
        const double w = __shfl_sync(0xffffffffu, w0, m);
        if (e[m] < 0 || lane >= 6) continue;
        acc = acc + w * (lane < 4 ? d.W[4 * e[m] + lane] : d.q[2 * e[m] + lane - 4]);
      }
      if (lane < 6) d.itmpW[6 * r + lane] = acc;
    }
  }
}

template <typename T> __global__ void __launch_bounds__(INTERP_THREADS) k_interp_scatter(Dev d, const int *list,
                                                                                        const int *cnt, int parts) {
  const int n = min(*cnt, d.cap_interp);
  const int nch = (parts & 1) ? (d.nvp + INTERP_CHUNK - 1) / INTERP_CHUNK : 1;
  for (int u = blockIdx.x; u < n * nch; u += gridDim.x) {
    const int r = u / nch, ch = u - r * nch, c = list[r];
    if (d.donors[5 * c] < 0) continue;          // orphan: keep its values
    if (parts & 1) {
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const int k = ch * INTERP_CHUNK + j * INTERP_THREADS + threadIdx.x;
        if (k >= d.nvp) continue;
        auto v = ldf<T>(d.itmp, (size_t)r * d.nvp + k);
        stF<T>(d, (size_t)c * d.nvp + k, v.x, v.y);
      }
    }
    if ((parts & 2) && ch == 0 && threadIdx.x < 6) {
      const int m = threadIdx.x;
      const double v = d.itmpW[6 * r + m];
      if (m < 4) d.W[4 * c + m] = v;
      else d.q[2 * c + m - 4] = v;
    }
  }
}

static inline int nblk(size_t n, int b) { return (int)((n + b - 1) / b); }

void launch_connect(const Dev &d, cudaStream_t s, int *prev_status, const int *blk_order,
                    int *n_orphan) {
  cudaMemsetAsync(d.bin_cnt, 0, sizeof(int) * d.nbins, s);
  k_node_f<<<nblk(d.nn > d.nseg ? d.nn : d.nseg, 256), 256, 0, s>>>(d);
  k_body_box<<<d.nblocks, 32, 0, s>>>(d);
  k_bin_count<<<nblk(d.nc, 256), 256, 0, s>>>(d);
  k_bin_scan<<<nblk(d.nbins, SCAN_CHUNK), SCAN_THREADS, 0, s>>>(d);
  k_bin_fill<<<nblk(d.nc, 256), 256, 0, s>>>(d);
  k_node_classify<<<nblk(d.nn, 128), 128, 0, s>>>(d);
  const int todo = std::min(nblk((size_t)d.nn * NLANES, 256), 152 * 8);      // CTAs, strided over the list
  size_t segb = sizeof(float4) * (size_t)d.nseg;
  if (segb <= 48 * 1024) k_node_todo<true><<<todo, 256, segb, s>>>(d);
  else k_node_todo<false><<<todo, 256, 0, s>>>(d);
  k_cell_classify<<<nblk(d.nc, 256), 256, 0, s>>>(d);
  k_cell_buffer<<<nblk(d.nc, 256), 256, 0, s>>>(d, prev_status);
  k_donor<<<nblk(d.nc, DONOR_CELLS), DONOR_THREADS, 0, s>>>(d, prev_status, blk_order, n_orphan);
}

void launch_lists(const Dev &d, cudaStream_t s, const int *fresh_flag, const int *n_orphan) {
  int nch = nblk(d.nc, LCHUNK);
  k_list_count<<<nch, LCHUNK, 0, s>>>(d, fresh_flag);
  k_list_write<<<nch, LCHUNK, 0, s>>>(d, fresh_flag, n_orphan);
}

void launch_interp(const Dev &d, cudaStream_t s, const int *list, const int *cnt, int nsm, int fp32, int parts) {
  // W and q alone take one warp a receptor
  const int th = (parts & 1) ? INTERP_THREADS : 32;
  const size_t units = (size_t)d.cap_interp * ((parts & 1) ? nblk(d.nvp, INTERP_CHUNK) : 1);
  const int grid = (int)std::max<size_t>(1, std::min<size_t>(units, (size_t)(2048 / th) * std::max(nsm, 1)));
  if (fp32) {
    k_interp_gather<float><<<grid, th, 0, s>>>(d, list, cnt, parts);
    k_interp_scatter<float><<<grid, th, 0, s>>>(d, list, cnt, parts);
  } else {
    k_interp_gather<double><<<grid, th, 0, s>>>(d, list, cnt, parts);
    k_interp_scatter<double><<<grid, th, 0, s>>>(d, list, cnt, parts);
  }
}

}  // namespace ugks
