// ugks_tile.cu -- the two velocity-resolved passes over f of every inner
// iteration (arXiv 2604.09984 Sec. 2.2, Steps 3 and 5) and the micro residual:
//   k_face_reduce  per face, the velocity sums of W0 (the interface
//                  equilibrium's moments) and of the f-dependent parts of the
//                  macro flux (Eq. macroscopicFlux);
//   k_flux         flux divergence D = sum_faces S F_hat per (cell, velocity)
//                  (Eqs. microscopicFlux, fullSolution, wall condition) from
//                  the face reconstruction the reduction stored; it does not
//                  depend on the macro predictor, so it runs while the macro
//                  LU-SGS sweep runs on another stream;
//   k_residual     the micro residual r from D (reading R4).
//
// A CTA takes an 8x8 cell tile of a block and a share of the velocity chunks.
// In the reduction, per chunk, f of the tile plus a two-cell halo (ghost cells
// hold the Maxwellian of their ghost state) is staged in shared memory with
// asynchronous copies, double-buffered so the next chunk arrives while the
// current one is reconstructed.  A thread owns one face slot of the tile and
// one half of every chunk's velocities: everything that does not depend on the
// velocity -- the face geometry, which region cells are its two sides, and for
// the flux the interface record of Eq. fullSolution -- is loaded once and kept
// in registers for the whole velocity loop.  The reduction accumulates its 12
// face sums in registers across all chunks (partial sums added with an
// error-free transformation on the FP32 path) and writes them once, with no
// atomics: the result does not depend on scheduling.  It also stores the
// reconstruction of every (face, velocity), so the flux pass reads one
// 4-vector per (face, velocity) instead of re-staging f and recomputing the
// limited gradients.
#include "ugks_internal.cuh"
#include "ugks_launch.h"

namespace ugks {

constexpr int TX = 8, TY = 8, RW = TX + 4, RH = TY + 4, NR = RW * RH;
constexpr int NSI = (TX + 1) * TY;          // i-face slots: tile row w, column x = 0..TX
constexpr int NSLOT = NSI + TX * (TY + 1);  // + j-face slots: row y = 0..TY, tile column w
// Two threads a face slot, adjacent lanes, take interleaved velocities of a
// chunk (kk = half + 2 q), so they store whole 32-byte sectors of
// reconstructions.
constexpr int NT = 2 * NSLOT;
static_assert(NR == NSLOT, "two threads a region cell as well");

// region cell (i, j) of block b -> cell id (>= 0), ghost (-2 - face id) or
// none (-1).  Periodic blocks wrap in i.
__device__ __forceinline__ int region_gid(const Dev &d, const int *bi, int off, int i, int j) {
  int ni = bi[0], nj = bi[1], per = bi[2];
  if (per) i = ((i % ni) + ni) % ni;
  bool iin = i >= 0 && i < ni, jin = j >= 0 && j < nj;
  if (iin && jin) return off + j * ni + i;
  int c = -1, s = -1;
  if (jin && !iin) {
    if (i == -1) { c = off + j * ni; s = 0; }
    else if (i == ni) { c = off + j * ni + ni - 1; s = 1; }
  } else if (iin && !jin) {
    if (j == -1) { c = off + i; s = 2; }
    else if (j == nj) { c = off + (nj - 1) * ni + i; s = 3; }
  }
  if (c < 0) return -1;
  if (d.nb_kind[4 * c + s] == NB_GHOST) return -2 - d.nb_id[4 * c + s];
  return -1;
}

// Face id of slot (dir, w, x): dir 0 the i-face left of tile column x of tile
// row w (x = TX: right of the last column), dir 1 the j-face below tile row
// x of tile column w; -1 where the face lies outside the block.
__device__ __forceinline__ int tile_face_id(const Dev &d, int dir, int off, int ni, int nj, int i0, int j0,
                                            int w, int x) {
  if (dir == 0) {
    int i = i0 + x, j = j0 + w;
    if (j >= nj || i > ni) return -1;
    return (i < ni) ? d.cell_faces[4 * (off + j * ni + i) + 0] : d.cell_faces[4 * (off + j * ni + ni - 1) + 1];
  }
  int i = i0 + w, j = j0 + x;
  if (i >= ni || j > nj) return -1;
  return (j < nj) ? d.cell_faces[4 * (off + j * ni + i) + 2] : d.cell_faces[4 * (off + (nj - 1) * ni + i) + 3];
}

// Gradient cells: the 10x10 block of region cells (rows and columns 1..10)
// that can be the upwind side of a tile face; g = (ry - 1) * GW + rx - 1.
constexpr int GW = TX + 2, NG = GW * (TY + 2);
__device__ __forceinline__ int region_of_g(int g) {
  int gy = g / GW;
  return (gy + 1) * RW + (g - gy * GW) + 1;
}
__device__ __forceinline__ int g_of_region(int r) {
  int ry = r / RW;
  return (ry - 1) * GW + (r - ry * RW) - 1;
}

// a b + c d with one product rounded by itself (written out where results must
// not depend on the compiler's choice)
__device__ __forceinline__ float mul_add2(float a, float b, float c, float d) { return __fmaf_rn(a, b, __fmul_rn(c, d)); }
// S w.n of a face at one velocity.  At a wall its sign splits the velocities into
// incident and reflected ones, and the reduction and the flux pass have to split
// alike (along a wall that slides in its own plane w.n is zero up to its rounding):
// both take these forms, every rounding written out.  FP64: from the row's part,
// vy S n_y - S U.n.
__device__ __forceinline__ float face_ws(float vx, float vy, float snx, float sny, float sun) {
  return __fsub_rn(mul_add2(vx, snx, vy, sny), sun);
}
__device__ __forceinline__ double face_ws_row(double vy, double sny, double sun) { return __fma_rn(vy, sny, -sun); }
__device__ __forceinline__ double face_ws(double vx, double snx, double row) { return __fma_rn(vx, snx, row); }
// Half of the van Leer slopes 2 a b / (a + b) (0 where a b <= 0) of a pair of
// differences, FP32 (the factor 2 goes into the inverse Jacobian: exact).
__device__ __forceinline__ float2 pr_vanleer_half(PairF a, PairF b) {
  const PairF p = pr_mul(a, b), s = pr_add(a, b);
  const float2 pv = pr_get(p), sv = pr_get(s);
  const float2 q = pr_get(pr_mul(p, pr_make(rcp_approx(sv.x), rcp_approx(sv.y))));
  return make_float2(pv.x > 0.f ? q.x : 0.f, pv.y > 0.f ? q.y : 0.f);
}
// FP64: both quotients from one reciprocal, 1/s_x = s_y / (s_x s_y), the
// hardware estimate refined by Newton's iteration r <- r + r (1 - x r)
// (quadratic: 2^-20 -> 2^-40 -> 2^-80, i.e. to rounding); a double-precision
// division costs a dozen instructions of a pipe that retires one in tens of
// cycles.  A product below 2^-960 counts as no common sign (slopes below 1e-144).
__device__ __forceinline__ PairD pr_vanleer(PairD a, PairD b) {
  const double px = a.x * b.x, py = a.y * b.y;
  const bool ox = __double2hiint(px) >= 0x03f00000, oy = __double2hiint(py) >= 0x03f00000;
  const double sx = ox ? a.x + b.x : 1.0, sy = oy ? a.y + b.y : 1.0;
  const double x = sx * sy;
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
  r = fma(r, fma(-x, r, 1.0), r);
  r = fma(r, fma(-x, r, 1.0), r);
  return PairD{ox ? 2.0 * px * (r * sy) : 0.0, oy ? 2.0 * py * (r * sx) : 0.0};
}

// Chunks of the velocity loop: every row of the velocity grid (fixed v_y) is
// cut into `per_row` chunks of `len` <= VK velocities (the last may be
// shorter), so that within a chunk every velocity sum is a sum of moments in
// v_x; rows of even length get even chunks (16-byte copies of FP32 pairs).
struct Chunks { int per_row, len, total; };
template <int VK> __host__ __device__ __forceinline__ Chunks face_chunks(int nvx, int nv) {
  Chunks c;
  c.per_row = (nvx + VK - 1) / VK;
  c.len = (nvx + c.per_row - 1) / c.per_row;
  if (nvx % 2 == 0) c.len = (c.len + 1) / 2 * 2;
  c.per_row = (nvx + c.len - 1) / c.len;
  c.total = nv / nvx * c.per_row;
  return c;
}

// Shared memory of the FP64 reduction: the double-buffered region of f, the
// limited Cartesian gradients of the chunk, the v_x table of both buffered
// chunks (weights times powers of v_x), and per region cell its slope cases
// and inverse Jacobian.
constexpr int VK64 = 8, VKP64 = VK64, VKG64 = VK64 + 2;
struct Smem64 {
  struct alignas(16) Tab { double w[4], vx, pad; };
  PairD F[2][NR][VKP64];
  Quad<PairD> G[NG][VKG64];      // (d_x h, d_x b), (d_y h, d_y b)
  Tab tab[2][VK64];
  double4 J[NR];
  int fl[NR];
};

template <typename T> __device__ __forceinline__ T grid_vx(const Dev &d, int ix);
template <> __device__ __forceinline__ double grid_vx<double>(const Dev &d, int ix) { return d.vx1[ix]; }
template <> __device__ __forceinline__ float grid_vx<float>(const Dev &d, int ix) { return d.vxf[ix]; }
template <typename T> __device__ __forceinline__ T grid_vy(const Dev &d, int iy);      // iy of the whole grid
template <> __device__ __forceinline__ double grid_vy<double>(const Dev &d, int iy) { return d.vy1[iy]; }
template <> __device__ __forceinline__ float grid_vy<float>(const Dev &d, int iy) { return d.vy1f[iy]; }

// Slot -> (direction, tile row / column w, position x) and the region cells
// A (lower logical side) and B of the face.
__device__ __forceinline__ void slot_geom(int slot, int &dir, int &w, int &x, int &A, int &B) {
  if (slot < NSI) {
    dir = 0;
    w = slot / (TX + 1);
    x = slot - w * (TX + 1);
    A = (x + 1) + (w + 2) * RW;
    B = A + 1;
  } else {
    int s = slot - NSI;
    dir = 1;
    x = s / TX;
    w = s - x * TX;
    A = (w + 2) + (x + 1) * RW;
    B = A + RW;
  }
}

// The stored reconstruction of (face, velocity k), a 4-vector: (f_face h,
// f_face b, w.grad f h, w.grad f b).  Tile-major, [tile][k / 2][slot][k % 2]
// with the face's slot in the tile that owns it, so that the threads of a CTA,
// two a slot on interleaved velocities, store and load consecutive vectors
// (row by row of a face, a warp's 16 faces touch 16 cache lines an access:
// those cost the reduction a third of its shared/global data cycles).
// fval_at: offset of (slot 0, k = 0) plus the slot's two vectors.
__host__ __device__ constexpr size_t fval_tile(int nvp) { return (size_t)(nvp / 2) * 2 * NSLOT; }
__device__ __forceinline__ size_t fval_at(int k, int slot) { return (size_t)(k >> 1) * (2 * NSLOT) + 2 * slot + (k & 1); }

// Owner (tile, slot) of the face of slot `slot` of tile `tile` at (i0, j0) of
// a block: the tile of the cell on its high side; a closing face belongs to
// the block's last tile, the seam of a periodic row to its first.
__device__ __forceinline__ void fval_owner(const int *bi, int i0, int j0, int tile, int slot, int &otile, int &oslot) {
  const int ni = bi[0], nj = bi[1], per = bi[2], ntx = (ni + TX - 1) / TX;
  int dir, w, x, A, B;
  slot_geom(slot, dir, w, x, A, B);
  int i = dir == 0 ? i0 + x : i0 + w, j = dir == 0 ? j0 + w : j0 + x;
  if (dir == 0 && per && i == ni) i = 0;
  int ti = i / TX, tj = j / TY;
  if (dir == 0 && i == ni) ti = (ni - 1) / TX;
  if (dir == 1 && j == nj) tj = (nj - 1) / TY;
  otile = tile + (tj - j0 / TY) * ntx + (ti - i0 / TX);
  oslot = dir == 0 ? (j - TY * tj) * (TX + 1) + (i - TX * ti) : NSI + (j - TY * tj) * TX + (i - TX * ti);
}
size_t face_values(int ntiles, int nvp) { return (size_t)ntiles * fval_tile(nvp); }

// ------------------------------------------------------------ face reduction
// Per owned face (the i- and j-faces on the low side of the tile's cells, and
// the closing faces at a non-periodic block end) the 12 sums over all
// velocities: W0 = sum V Psi f_face (interior faces), and the incident-part
// sums sum V Psi w.S f_face and sum V Psi w.S (w.grad f) (Eq. macroscopicFlux
// with the time integrals q1, q2 applied afterwards).  The reconstruction of
// every (face, velocity) -- the upwind face value and w.grad f of Eq.
// fullSolution -- is stored for the flux pass, which then needs neither f nor
// its gradients.
//
// gridDim.y CTAs share a tile's chunks where the tiles alone leave SMs idle
// (face_splits): each then leaves its (sum, error) pairs for the interface
// state kernel, which adds them in order.

// This thread's face of the reduction.
struct RedFace {
  int fid, A, B, Lr, Rr;         // region cells A (lower logical side), B; L and R
  bool act, wall;
};
template <typename T> __device__ __forceinline__ RedFace red_face(const Dev &d, const int *bi, int off, int i0, int j0, int slot) {
  RedFace f;
  const int ni = bi[0], nj = bi[1], per = bi[2];
  int dir, w, x;
  slot_geom(slot, dir, w, x, f.A, f.B);
  f.fid = tile_face_id(d, dir, off, ni, nj, i0, j0, w, x);
  f.act = f.wall = false;
  f.Lr = f.Rr = f.A;
  if (f.fid >= 0) {
    const int i = dir == 0 ? i0 + x : i0 + w, j = dir == 0 ? j0 + w : j0 + x;
    const bool own = dir == 0 ? ((i < ni && x < TX) || (!per && i == ni)) : ((j < nj && x < TY) || j == nj);
    f.act = own && d.face_kind[f.fid] != BC_OVERSET;
    if (f.act) {
      const int Lg = d.face_L[f.fid], Rg = d.face_R[f.fid];
      f.act = d.status[Lg] == ST_FIELD || (Rg >= 0 && d.status[Rg] == ST_FIELD);
    }
  }
  if (f.act) {
    f.wall = d.face_kind[f.fid] == BC_WALL;
    const int gA = region_gid(d, bi, off, i0 - 2 + f.A % RW, j0 - 2 + f.A / RW);
    f.Lr = (gA == d.face_L[f.fid]) ? f.A : f.B;
    f.Rr = (f.Lr == f.A) ? f.B : f.A;
  }
  return f;
}

// The two parts of a face meet in shared memory (xs: 2 NFS NSLOT values, free
// once every thread has passed the barrier), summed in part order.
template <typename T>
__device__ __forceinline__ void red_finish(const Dev &d, T *xs, const RedFace &f, int slot, int half, const T *hi, const T *lo) {
  __syncthreads();
  if (half > 0 && slot < NSLOT) {
#pragma unroll
    for (int m = 0; m < NFS; ++m) { xs[(2 * m) * NSLOT + slot] = hi[m]; xs[(2 * m + 1) * NSLOT + slot] = lo[m]; }
  }
  __syncthreads();
  if (half == 0 && f.act) {
#pragma unroll
    for (int m = 0; m < NFS; ++m) {
      T h = hi[m], l = lo[m];
      face_sum_add(h, l, xs[(2 * m) * NSLOT + slot], xs[(2 * m + 1) * NSLOT + slot]);
      if (f.wall && m < FS_FF) h = l = T(0);       // walls take W0 from the interior cell
      if (gridDim.y == 1) {
        d.fsum[(size_t)NFS * f.fid + m] = face_sum_value(h, l);
      } else {
        T *o = reinterpret_cast<T *>(d.fpart) + 2 * (((size_t)blockIdx.y * NFS + m) * d.nf + f.fid);
        o[0] = h;
        o[1] = l;
      }
    }
  }
}

// FP32.  Per chunk of VK32 consecutive velocities: staging of the next chunk;
// phase A, the limited gradients of the tile's 100 gradient cells, a thread
// walking down five cells of a column at one velocity (the column's values
// stay in registers: three shared loads a cell instead of five); phase B, the
// face values and the sums.  Bound by the shared-memory data path and by
// instruction issue together: the limiter runs on (h, b) pairs in packed FP32
// instructions, the sums on (f_face, w.grad f) pairs, and every shared and
// global access of a warp covers whole lines (staging 128 bytes of a cell,
// stores 512 consecutive bytes).  Two chunks are summed plainly, then folded
// into (sum, error) pairs by an error-free sum.
constexpr int VK32 = 16, VKP32 = VK32 + 2, VKG32 = VK32 + 2;   // rows in distinct banks
constexpr int NT32 = 2 * GW * VK32;                            // two threads a gradient column and velocity
static_assert(NT32 >= NT && NT32 % 32 == 0 && TY + 2 == 10, "phase A: five of a column's ten cells a thread");
struct Smem32 {
  PairF F[2][NR][VKP32];
  float4 G[NG][VKG32];     // gradients: d_x h, d_x b, d_y h, d_y b
  float4 tab[2][VK32];     // vx, vy, weight, |v|^2 / 2
  float4 J[NR];            // twice the inverse Jacobian (real cells), ghost state rho lam / pi, Vx, Vy, lam (ghosts)
  int gid[NR];
};

template <int FB> __global__ void __launch_bounds__(NT32, 2) k_face_reduce32(Dev d) {
  extern __shared__ __align__(16) unsigned char smraw[];
  Smem32 &S = *reinterpret_cast<Smem32 *>(smraw);
  const int tile = blockIdx.x, tid = threadIdx.x;
  const int b = d.tiles[3 * tile], i0 = d.tiles[3 * tile + 1], j0 = d.tiles[3 * tile + 2];
  const int *bi = d.blk_info + 8 * b;
  const int off = d.cell_off[b];
  for (int r = tid; r < NR; r += NT32) {
    const int g = region_gid(d, bi, off, i0 - 2 + r % RW, j0 - 2 + r / RW);
    float4 J = make_float4(0.f, 0.f, 0.f, 0.f);
    if (g >= 0) {
      J = d.jinvf[g];
      J = make_float4(2.f * J.x, 2.f * J.y, 2.f * J.z, 2.f * J.w);
    } else if (g <= -2) {
      Prim p = primitive(d.ghostW + 4 * (-2 - g), d.Keff);
      J = make_float4((float)(p.rho * p.lam * M_1_PI), (float)p.ux, (float)p.uy, (float)p.lam);
    }
    S.J[r] = J;
    S.gid[r] = g;
  }
  __syncthreads();
  const int nch = (d.nv + VK32 - 1) / VK32, npair = (nch + 1) / 2;
  const int ch0 = 2 * (int)((long)npair * blockIdx.y / gridDim.y);
  const int ch1 = min(nch, 2 * (int)((long)npair * (blockIdx.y + 1) / gridDim.y));
  // copies of chunk ch into buffer buf: real cells by asynchronous 16-byte
  // copies (bf16 storage: load and widen), ghost cells the Maxwellian of their
  // ghost state, no cell / padding velocities zero; and the velocity table
  auto stage = [&](int ch, int buf) {
    const int kb = ch * VK32;
#pragma unroll
    for (int m = 0; m < (NR * VK32 / 2 + NT32 - 1) / NT32; ++m) {
      const int it = tid + m * NT32, r = it / (VK32 / 2), e = 2 * (it % (VK32 / 2)), k = kb + e;
      if (it >= NR * VK32 / 2) break;
      const int g = S.gid[r];
      PairF *dst = &S.F[buf][r][e];
      if (g >= 0 && k < d.nv) {
        if (FB) {
          for (int q = 0; q < 2; ++q) {
            auto v = ldF<float, 1>(d, (size_t)g * d.nvp + k + q);
            dst[q] = pr_make(v.x, v.y);
          }
        } else {
          // k < nv <= nvp, nvp a multiple of 16 and k even: the pair stays in
          // the cell's row (padding velocities hold zero)
          cp_async<16>(dst, reinterpret_cast<const PairF *>(d.f) + (size_t)g * d.nvp + k);
        }
      } else {
        for (int q = 0; q < 2; ++q) {
          V2<float> v = {0.f, 0.f};
          if (g <= -2 && k + q < d.nv) {
            const float4 p = S.J[r];
            v = maxwellian_pre<float>(p.x, p.y, p.z, p.w, (float)d.Keff / (2.f * p.w), d.vxf[k + q], d.vyf[k + q]);
          }
          dst[q] = pr_make(v.h, v.b);
        }
      }
    }
    if (tid < VK32) {
      const int k = kb + tid;
      const float vx = k < d.nv ? d.vxf[k] : 0.f, vy = k < d.nv ? d.vyf[k] : 0.f, w = k < d.nv ? d.wf[k] : 0.f;
      S.tab[buf][tid] = make_float4(vx, vy, w, 0.5f * (vx * vx + vy * vy));
    }
    cp_async_commit();
  };
  if (ch0 < ch1) stage(ch0, 0);
  // phase A task: column and five rows of the gradient cells, one velocity
  const int akk = tid % VK32, acol = (tid / VK32) % GW, arow = 5 * (tid / (VK32 * GW));
  int afl = 0;                             // slope cases of the five cells, 4 bits each
#pragma unroll
  for (int m = 0; m < 5; ++m) {
    const int g = S.gid[(arow + m + 1) * RW + acol + 1];
    if (g >= 0) afl |= d.slope_flags[g] << (4 * m);
  }
  auto gradients = [&](int buf) {
    const PairF *c = &S.F[buf][(arow + 1) * RW + acol + 1][akk];
    const float4 *J = &S.J[(arow + 1) * RW + acol + 1];
    float4 *o = &S.G[arow * GW + acol][akk];
    PairF jm = c[-RW * VKP32], fc = c[0];
#pragma unroll
    for (int m = 0; m < 5; ++m) {
      const PairF jp = c[RW * VKP32], ia = pr_sub(fc, c[-VKP32]), ib = pr_sub(c[VKP32], fc);
      const PairF ja = pr_sub(fc, jm), jb = pr_sub(jp, fc);
      const float4 J2 = *J;
      float2 si = pr_vanleer_half(ia, ib), sj = pr_vanleer_half(ja, jb);
      if (afl != 0xfffff) {
        // one-sided where one neighbour is missing, none without both (twice
        // the inverse Jacobian: one-sided slopes enter by half)
        const int fl = afl >> (4 * m);
        const PairF h = pr_make(0.5f, 0.5f);
        const float2 z = make_float2(0.f, 0.f);
        if ((fl & 3) != 3) si = (fl & 1) ? pr_get(pr_mul(h, ia)) : (fl & 2) ? pr_get(pr_mul(h, ib)) : z;
        if ((fl & 12) != 12) sj = (fl & 4) ? pr_get(pr_mul(h, ja)) : (fl & 8) ? pr_get(pr_mul(h, jb)) : z;
      }
      float4 G = make_float4(mul_add2(J2.x, si.x, J2.y, sj.x), mul_add2(J2.x, si.y, J2.y, sj.y),
                             mul_add2(J2.z, si.x, J2.w, sj.x), mul_add2(J2.z, si.y, J2.w, sj.y));
      if (afl != 0xfffff && !((afl >> (4 * m)) & 15)) G = make_float4(0.f, 0.f, 0.f, 0.f);   // (ghost: J holds its state)
      *o = G;
      jm = fc;
      fc = jp;
      c += RW * VKP32;
      J += RW;
      o += GW * VKG32;
    }
  };
  const int slot = tid >> 1, half = tid & 1;
  RedFace f;
  f.act = false;
  if (tid < NT) f = red_face<float>(d, bi, off, i0, j0, slot);
  float snx = 0.f, sny = 0.f, sun = 0.f, ufx = 0.f, ufy = 0.f, dxl = 0.f, dyl = 0.f, dxr = 0.f, dyr = 0.f;
  int oL = 0, oR = 0, gL = 0, gR = 0;      // region and gradient rows of the two sides
  if (f.act) {
    __align__(16) float Gr[NFG];
    load_rec<float, NFG>(reinterpret_cast<const float *>(d.fgeo) + (size_t)f.fid * NFG, Gr);
    snx = Gr[FG_SNX]; sny = Gr[FG_SNY]; sun = Gr[FG_SUN]; ufx = Gr[FG_UFX]; ufy = Gr[FG_UFY];
    dxl = Gr[FG_DXLX]; dyl = Gr[FG_DXLY]; dxr = Gr[FG_DXRX]; dyr = Gr[FG_DXRY];
    oL = f.Lr * VKP32; oR = f.Rr * VKP32;
    gL = g_of_region(f.Lr) * VKG32; gR = g_of_region(f.Rr) * VKG32;
  }
  float hi[NFS], lo[NFS], w0[4];
  PairF fg[4];                             // (FF, WG) sums of the fold
#pragma unroll
  for (int m = 0; m < NFS; ++m) { hi[m] = 0.f; lo[m] = 0.f; }
#pragma unroll
  for (int m = 0; m < 4; ++m) { w0[m] = 0.f; fg[m] = pr_make(0.f, 0.f); }
  float4 *fv = reinterpret_cast<float4 *>(d.fval) + (size_t)tile * fval_tile(d.nvp) + tid;
  for (int ch = ch0; ch < ch1; ++ch) {
    const int buf = (ch - ch0) & 1, kb = ch * VK32;
    cp_async_wait<0>();
    __syncthreads();                       // chunk ch visible; phase B of ch - 1 done everywhere
    if (ch + 1 < ch1) stage(ch + 1, buf ^ 1);
    gradients(buf);
    __syncthreads();
    if (f.act) {
      const PairF *F = S.F[buf][0];
      const float4 *G = S.G[0];
#pragma unroll 4
      for (int q = 0; q < VK32 / 2; ++q) {
        const int kk = half + 2 * q;
        const float4 t = S.tab[buf][kk];
        const float vx = t.x, vy = t.y;
        const float wS = face_ws(vx, vy, snx, sny, sun);
        const bool r = !f.wall && wS < 0.f;
        const float wx = vx - ufx, wy = vy - ufy;
        V2<float> ff, wg;
        auto side = [&](const PairF *c, const float4 *gp, float dx, float dy, V2<float> &a, V2<float> &e) {
          const float2 fc = pr_get(*c);
          const float4 g = *gp;
          a.h = __fmaf_rn(dy, g.z, __fmaf_rn(dx, g.x, fc.x));
          a.b = __fmaf_rn(dy, g.w, __fmaf_rn(dx, g.y, fc.y));
          e.h = mul_add2(wx, g.x, wy, g.z);
          e.b = mul_add2(wx, g.y, wy, g.w);
        };
        side(F + (r ? oR : oL) + kk, G + (r ? gR : gL) + kk, r ? dxr : dxl, r ? dyr : dyl, ff, wg);
        if (wS == 0.f && !f.wall) {        // exactly along the face: the mean of both sides
          V2<float> f2, g2;
          side(F + oR + kk, G + gR + kk, dxr, dyr, f2, g2);
          ff = {0.5f * (ff.h + f2.h), 0.5f * (ff.b + f2.b)};
          wg = {0.5f * (wg.h + g2.h), 0.5f * (wg.b + g2.b)};
        }
        // the flux pass reads the reconstruction from here
        if (kb + kk < d.nv) fv[(size_t)(kb / 2 + q) * NT] = make_float4(ff.h, ff.b, wg.h, wg.b);
        // reflected velocities of a wall carry no f; p = w Psi f_face, g = w Psi (w.grad f) in pairs
        const float w = f.wall && !(wS > 0.f) ? 0.f : t.z, hw = 0.5f * w;
        const PairF a = pr_mul(pr_make(w, w), pr_make(ff.h, wg.h));
        const PairF p1 = pr_mul(pr_make(vx, vx), a), p2 = pr_mul(pr_make(vy, vy), a);
        const PairF p3 = pr_fma(pr_make(hw, hw), pr_make(ff.b, wg.b), pr_mul(pr_make(t.w, t.w), a)), ws = pr_make(wS, wS);
        w0[0] += pr_get(a).x; w0[1] += pr_get(p1).x; w0[2] += pr_get(p2).x; w0[3] += pr_get(p3).x;
        fg[0] = pr_fma(ws, a, fg[0]); fg[1] = pr_fma(ws, p1, fg[1]);
        fg[2] = pr_fma(ws, p2, fg[2]); fg[3] = pr_fma(ws, p3, fg[3]);
      }
      if ((ch & 1) || ch + 1 == ch1) {
#pragma unroll
        for (int m = 0; m < NFS; ++m) {
          const float2 p = pr_get(fg[m & 3]);
          const float x = m < FS_FF ? w0[m & 3] : m < FS_WG ? p.x : p.y;
          float t, e;
          two_sum(hi[m], x, t, e);
          hi[m] = t;
          lo[m] += e;
        }
#pragma unroll
        for (int m = 0; m < 4; ++m) { w0[m] = 0.f; fg[m] = pr_make(0.f, 0.f); }
      }
    }
  }
  static_assert(sizeof(S.F) >= sizeof(float) * 2 * NFS * NSLOT, "the parts' sums fit in the region buffers");
  red_finish<float>(d, reinterpret_cast<float *>(S.F), f, slot, half, hi, lo);
}

// FP64.  Bound by the FP64 pipe, so the operation count decides: the limited
// gradients of a chunk are formed once per cell (phase A) and pass through
// shared memory, the limiter shares one reciprocal between h and b, and a
// chunk lies in one velocity row, so phase B only adds up the moments sum w
// v_x^n (h, b) of the face value and of w.grad f (n <= 3); the 12 sums follow
// from them once per fold (two chunks or a row's end) with the row's v_y.
// Which side of a face is upwind changes at most once along a row, so chunks
// with one sign of w.n at both ends take their side once; only the chunk that
// holds the change selects per velocity.
__global__ void __launch_bounds__(NT, 1) k_face_reduce64(Dev d) {
  typedef double T;
  typedef PairD P;
  constexpr int VK = VK64, VKP = VKP64, VKG = VKG64;
  extern __shared__ __align__(16) unsigned char smraw[];
  Smem64 &S = *reinterpret_cast<Smem64 *>(smraw);
  const int tile = blockIdx.x, tid = threadIdx.x;
  const int b = d.tiles[3 * tile], i0 = d.tiles[3 * tile + 1], j0 = d.tiles[3 * tile + 2];
  const int *bi = d.blk_info + 8 * b;
  const int off = d.cell_off[b];
  // this thread's region cell and its half of the staged copies
  const int rc = tid >> 1, half = tid & 1;
  const int gid = region_gid(d, bi, off, i0 - 2 + rc % RW, j0 - 2 + rc / RW);
  double4 gst = {0.0, 0.0, 0.0, 0.0};              // ghost state
  {
    double4 J = {0.0, 0.0, 0.0, 0.0};
    int fl = 0;
    if (gid >= 0) {
      fl = d.slope_flags[gid];
      J.x = d.jinv[4 * gid]; J.y = d.jinv[4 * gid + 1]; J.z = d.jinv[4 * gid + 2]; J.w = d.jinv[4 * gid + 3];
    } else if (gid <= -2) {
      Prim p = primitive(d.ghostW + 4 * (-2 - gid), d.Keff);
      gst.x = p.rho * p.lam * M_1_PI; gst.y = p.ux; gst.z = p.uy; gst.w = p.lam;
    } else {                                       // no cell: zero in both buffers, once
      for (int q = half; q < VKP; q += 2) S.F[0][rc][q] = S.F[1][rc][q] = pr_dup(0.0);
    }
    if (half == 0) { S.J[rc] = J; S.fl[rc] = fl; }
  }
  const Chunks ck = face_chunks<VK>(d.nvx, d.nv);
  const int ch0 = (int)((long)ck.total * blockIdx.y / gridDim.y), ch1 = (int)((long)ck.total * (blockIdx.y + 1) / gridDim.y);
  // position of a chunk: its row (of this context) and first column
  struct Pos { int iy, x0; };
  auto advance = [&](Pos &p) {
    p.x0 += ck.len;
    if (p.x0 >= d.nvx) { p.x0 = 0; ++p.iy; }
  };
  auto count = [&](const Pos &p) { return min(ck.len, d.nvx - p.x0); };
  auto stage = [&](const Pos &p, int buf) {
    const int n = count(p), k0 = p.iy * d.nvx + p.x0;
    P *dst = S.F[buf][rc];
    if (gid >= 0) {
      const P *src = reinterpret_cast<const P *>(d.f) + (size_t)gid * d.nvp + k0;
      for (int e = half; e < n; e += 2) cp_async<16>(dst + e, src + e);
    } else if (gid <= -2) {
      for (int e = half; e < n; e += 2) {
        V2<T> m = maxwellian_pre<T>(gst.x, gst.y, gst.z, gst.w, (T)d.Keff / (T(2) * gst.w), d.vx1[p.x0 + e],
                                    d.vy1[d.iy0 + p.iy]);
        dst[e] = pr_make(m.h, m.b);
      }
    }
    for (int e = tid; e < n; e += NT) {
      const T vx = d.vx1[p.x0 + e], w = d.wx1[p.x0 + e];
      S.tab[buf][e] = Smem64::Tab{{w, w * vx, w * (vx * vx), w * (vx * vx) * vx}, vx, 0.0};
    }
    cp_async_commit();
  };
  // phase A: the limited Cartesian gradient of (h, b) of gradient cell g and
  // chunk velocity kk (ghost and missing cells carry none)
  auto gradient = [&](int g, int kk, int buf) {
    const int r = region_of_g(g);
    const int fl = S.fl[r];
    Quad<P> out = {pr_dup(0.0), pr_dup(0.0)};
    if (fl) {
      const double4 J = S.J[r];
      const P *c = &S.F[buf][r][kk];
      const P fc = c[0];
      const P ia = pr_sub(fc, c[-VKP]), ib = pr_sub(c[VKP], fc);
      const P ja = pr_sub(fc, c[-RW * VKP]), jb = pr_sub(c[RW * VKP], fc);
      P si = pr_vanleer(ia, ib), sj = pr_vanleer(ja, jb);
      if (fl != 15) {      // one-sided where one neighbour is missing, none without both
        const P z = pr_dup(0.0);
        if ((fl & 3) != 3) si = (fl & 1) ? ia : (fl & 2) ? ib : z;
        if ((fl & 12) != 12) sj = (fl & 4) ? ja : (fl & 8) ? jb : z;
      }
      out.x = pr_fma(pr_dup(J.x), si, pr_mul(pr_dup(J.y), sj));
      out.y = pr_fma(pr_dup(J.z), si, pr_mul(pr_dup(J.w), sj));
    }
    S.G[g][kk] = out;
  };
  const int slot = tid >> 1;
  const RedFace f = red_face<T>(d, bi, off, i0, j0, slot);
  T snx = 0.0, sny = 0.0, sun = 0.0, ufx = 0.0, ufy = 0.0, dxl = 0.0, dyl = 0.0, dxr = 0.0, dyr = 0.0;
  if (f.act) {
    __align__(16) T Gr[NFG];
    load_rec<T, NFG>(reinterpret_cast<const T *>(d.fgeo) + (size_t)f.fid * NFG, Gr);
    snx = Gr[FG_SNX]; sny = Gr[FG_SNY]; sun = Gr[FG_SUN]; ufx = Gr[FG_UFX]; ufy = Gr[FG_UFY];
    dxl = Gr[FG_DXLX]; dyl = Gr[FG_DXLY]; dxr = Gr[FG_DXRX]; dyr = Gr[FG_DXRY];
  }
  const int Lg = g_of_region(f.Lr), Rg = g_of_region(f.Rr);
  T hi[NFS], lo[NFS];
#pragma unroll
  for (int m = 0; m < NFS; ++m) { hi[m] = 0.0; lo[m] = 0.0; }
  P M[4], Q[4];                                    // moments of the face value and of w.grad f
#pragma unroll
  for (int n = 0; n < 4; ++n) { M[n] = pr_dup(0.0); Q[n] = pr_dup(0.0); }
  Pos cur = {ch0 / ck.per_row, (ch0 % ck.per_row) * ck.len}, nxt = cur;
  if (ch0 < ch1) stage(cur, 0);
  advance(nxt);
  const unsigned magic = ((1u << 20) + ck.len - 1) / ck.len;
  for (int ch = ch0; ch < ch1; ++ch) {
    const int buf = (ch - ch0) & 1, n = count(cur);
    cp_async_wait<0>();
    __syncthreads();                       // chunk ch visible; phase B of ch-1 done everywhere
    if (ch + 1 < ch1) stage(nxt, buf ^ 1);
    // it / len by its reciprocal (it < 2^10, len <= 8: exact)
    for (int it = tid; it < NG * ck.len; it += NT) {
      const int g = (int)(((unsigned)it * magic) >> 20), kk = it - g * ck.len;
      if (kk < n) gradient(g, kk, buf);
    }
    __syncthreads();
    if (f.act) {
      const Smem64::Tab *tab = S.tab[buf];
      const T vy = d.vy1[d.iy0 + cur.iy], cy = face_ws_row(vy, sny, sun), wy = vy - ufy;
      Quad<P> *fv = reinterpret_cast<Quad<P> *>(d.fval) + (size_t)tile * fval_tile(d.nvp);
      const int k0 = cur.iy * d.nvx + cur.x0;
      const P wyp = pr_dup(wy);
      auto reconstruct = [&](const P *F, const Quad<P> *G, P dx, P dy, int kk, P &ff, P &wg) {
        const Quad<P> g = G[kk];
        ff = pr_fma(dx, g.x, pr_fma(dy, g.y, F[kk]));
        wg = pr_fma(pr_dup(tab[kk].vx - ufx), g.x, pr_mul(wyp, g.y));
      };
      auto accumulate = [&](const Smem64::Tab &t, P ff, P wg) {
#pragma unroll
        for (int m = 0; m < 4; ++m) {
          M[m] = pr_fma(pr_dup(t.w[m]), ff, M[m]);
          Q[m] = pr_fma(pr_dup(t.w[m]), wg, Q[m]);
        }
      };
      // w.S at the chunk's ends, rounded as for each velocity: monotone in v_x
      const T wa = face_ws(tab[0].vx, snx, cy), wb = face_ws(tab[n - 1].vx, snx, cy);
      const bool allL = wa > 0.0 && wb > 0.0, allR = wa < 0.0 && wb < 0.0;
      if (allL || (allR && !f.wall)) {
        const P *F = S.F[buf][allL ? f.Lr : f.Rr];
        const Quad<P> *G = S.G[allL ? Lg : Rg];
        const P dx = pr_dup(allL ? dxl : dxr), dy = pr_dup(allL ? dyl : dyr);
        for (int kk = half; kk < n; kk += 2) {
          P ff, wg;
          reconstruct(F, G, dx, dy, kk, ff, wg);
          fv[fval_at(k0 + kk, slot)] = Quad<P>{ff, wg};                // the flux pass reads the reconstruction from here
          accumulate(tab[kk], ff, wg);
        }
      } else {
        // the upwind side changes inside the chunk (w.S = 0 exactly: the mean
        // of both sides); a wall takes its interior side, summed over the
        // incident part
        for (int kk = half; kk < n; kk += 2) {
          const T wS = face_ws(tab[kk].vx, snx, cy);
          const bool r = !f.wall && wS < 0.0;
          P ff, wg;
          reconstruct(S.F[buf][r ? f.Rr : f.Lr], S.G[r ? Rg : Lg], pr_dup(r ? dxr : dxl), pr_dup(r ? dyr : dyl), kk, ff, wg);
          if (wS == 0.0 && !f.wall) {
            P f2, g2;
            reconstruct(S.F[buf][f.Rr], S.G[Rg], pr_dup(dxr), pr_dup(dyr), kk, f2, g2);
            ff = pr_mul(pr_dup(0.5), pr_add(ff, f2));
            wg = pr_mul(pr_dup(0.5), pr_add(wg, g2));
          }
          fv[fval_at(k0 + kk, slot)] = Quad<P>{ff, wg};
          if (!f.wall || wS > 0.0) accumulate(tab[kk], ff, wg);
        }
      }
      // fold after two chunks, at the end of the row and at the last chunk
      if (((cur.x0 / ck.len) & 1) || cur.x0 + n >= d.nvx || ch + 1 == ch1) {
        const T ww = d.wy1[d.iy0 + cur.iy], hv = 0.5 * ww, vy2 = vy * vy;
        auto sums = [&](const P *m, T *o, bool flux) {
          const T e0 = m[2].x + vy2 * m[0].x + m[0].y;       // sum w (|v|^2 h + b)
          if (!flux) {
            o[0] += ww * m[0].x; o[1] += ww * m[1].x; o[2] += ww * (vy * m[0].x); o[3] += hv * e0;
          } else {
            const T e1 = m[3].x + vy2 * m[1].x + m[1].y;
            const T f0 = snx * m[1].x + cy * m[0].x;
            o[0] += ww * f0; o[1] += ww * (snx * m[2].x + cy * m[1].x); o[2] += ww * (vy * f0);
            o[3] += hv * (snx * e1 + cy * e0);
          }
        };
        sums(M, hi + FS_W0, false);
        sums(M, hi + FS_FF, true);
        sums(Q, hi + FS_WG, true);
#pragma unroll
        for (int m = 0; m < 4; ++m) { M[m] = pr_dup(0.0); Q[m] = pr_dup(0.0); }
      }
    }
    cur = nxt;
    advance(nxt);
  }
  static_assert(sizeof(S.F) >= sizeof(T) * 2 * NFS * NSLOT, "the parts' sums fit in the region buffers");
  red_finish<T>(d, &S.F[0][0][0].x, f, slot, half, hi, lo);
}

// -------------------------------------------------------- flux divergence
// Every face slot of the tile (faces shared with a neighbouring tile are
// evaluated by both) computes S F_hat per velocity into shared memory from
// the reconstruction the reduction pass stored; then each (tile cell,
// velocity) sums its four faces with the cell's orientation signs and stores
// D.  A chunk is at most VK velocities of one velocity row, and the rows are
// walked for a fixed range of columns; the interface cubics become cubics in
// c_x whose coefficients a row shares.  SEP: the Maxwellian as the product of
// a v_x factor, one exponential per column and range, and a v_y factor, one
// per row; FP64 always (an exponential costs some thirty instructions of its
// pipe), FP32 where N_v_x is a multiple of 16, else one exponential an item
// (the hardware's takes two instructions; each form keeps its own rounding).
//
// A thread's own (face, velocity) items come through a ring of FS stages with
// per-thread asynchronous copies: nobody else reads them, so a chunk needs one
// barrier (the face fluxes, double-buffered) and FS - 1 chunks are in flight.
// (One bulk copy per face row instead, completing on an mbarrier: its operands
// are uniform, so lanes with different addresses issue one by one, some 1,400
// warp instructions a chunk against 36.)  gridDim.y CTAs share a tile's rows.
// Streaming: 16 bytes in per (face, velocity), 8 out per (cell, velocity) in
// FP32; FP64 is bound by its pipe.
template <typename T> struct FluxCfg;
template <> struct FluxCfg<float> { static constexpr int VK = 8, FS = 4, CTAS = 2; };
template <> struct FluxCfg<double> { static constexpr int VK = 8, FS = 3, CTAS = 1; };
template <typename T> static constexpr size_t flux_smem() {
  typedef typename PairOf<T>::type P;
  typedef FluxCfg<T> C;
  return sizeof(Quad<P>) * C::FS * C::VK / 2 * NT + sizeof(P) * 2 * NSLOT * (C::VK + 2);
}

// EVAL: the sums go to the caller's array (ncells x nv x 2, FP64; zero outside
// the field) instead of the residual's buffer.  (One thread a cell and velocity
// that gathered the gradients and fluxes of its four faces from the cells:
// 5.1 ms for 192 x 96 + 96 x 24 cells and 1024 velocities, 6.03 ms the call;
// from the face values that the reduction leaves, 0.83 ms the call.)
// PAIR (FP32 joint form, by flux_pairs): two ranges of columns in turn, row by row,
// so that a cell's sums of both are stored close together (300x150 + 2 x 120x30
// cells, 33x33 velocities: 731 -> 649 us; in the separable form the longer
// registers cost more: 256x128 + 128x32, 32x32: 313 -> 431).
template <typename T, bool SEP, bool PAIR, bool EVAL>
__global__ void __launch_bounds__(NT, FluxCfg<T>::CTAS) k_flux(Dev d, double *eval) {
  typedef typename PairOf<T>::type P;
  constexpr int VK = FluxCfg<T>::VK, FS = FluxCfg<T>::FS, VH = VK / 2, VKG = VK + 2;
  extern __shared__ __align__(16) unsigned char smraw[];
  Quad<P> *FV = reinterpret_cast<Quad<P> *>(smraw);                         // [FS][VH][NT]
  P *Fs = reinterpret_cast<P *>(smraw + sizeof(Quad<P>) * FS * VH * NT);    // [2][NSLOT][VKG]
  const int tile = blockIdx.x, tid = threadIdx.x;
  const int b = d.tiles[3 * tile], i0 = d.tiles[3 * tile + 1], j0 = d.tiles[3 * tile + 2];
  const int *bi = d.blk_info + 8 * b;
  const int ni = bi[0], nj = bi[1], off = d.cell_off[b];
  // this thread's cell of the sums (four threads a cell)
  int g = -1;
  bool field = false;
  P sg[4];
  const P *fa = Fs, *fc = Fs;
  const bool wide = !EVAL || (reinterpret_cast<uintptr_t>(eval) & 15) == 0;    // the caller's array: 8-byte aligned at least
  {
    const int c = tid >> 2, tx = c % TX, ty = c / TX, i = i0 + tx, j = j0 + ty;
    if (tid < 4 * TX * TY && i < ni && j < nj) {
      g = off + j * ni + i;
      field = d.status[g] == ST_FIELD;
      if (!EVAL && !field) g = -1;
    }
    const char4 sc = g >= 0 ? reinterpret_cast<const char4 *>(d.cell_sgn)[g] : make_char4(0, 0, 0, 0);
    sg[0] = pr_dup((T)sc.x); sg[1] = pr_dup((T)sc.y); sg[2] = pr_dup((T)sc.z); sg[3] = pr_dup((T)sc.w);
    fa += (ty * (TX + 1) + tx) * VKG;
    fc += (NSI + ty * TX + tx) * VKG;
  }
  // this thread's face
  const int slot = tid >> 1, half = tid & 1;
  bool act = false;
  int fid;
  {
    int dir, w, x, A, B;
    slot_geom(slot, dir, w, x, A, B);
    fid = tile_face_id(d, dir, off, ni, nj, i0, j0, w, x);
    if (fid >= 0 && d.face_kind[fid] != BC_OVERSET) {
      int Lg = d.face_L[fid], Rg = d.face_R[fid];
      act = d.status[Lg] == ST_FIELD || (Rg >= 0 && d.status[Rg] == ST_FIELD);
    }
  }
  if (!act)
    for (int e = half; e < 2 * VKG; e += 2) Fs[((e >= VKG) * NSLOT + slot) * VKG + e % VKG] = pr_dup(T(0));
  const bool wall = act && d.face_kind[fid] == BC_WALL;
  __align__(16) T P_[NFP];
  if (act) {
    load_rec<T, NFP>(reinterpret_cast<const T *>(d.fparT) + (size_t)fid * NFP, P_);
  } else {
#pragma unroll
    for (int m = 0; m < NFP; ++m) P_[m] = T(0);
  }
  const Chunks ck = face_chunks<VK>(d.nvx, d.nv);
  const int rows = d.nv / d.nvx;
  const int r0 = (int)((long)rows * blockIdx.y / gridDim.y), r1 = (int)((long)rows * (blockIdx.y + 1) / gridDim.y);
  const int nch = ck.per_row * (r1 - r0);
  struct Pos { int x0, iy, odd; };
  auto advance = [&](Pos &p) {
    if (PAIR && !p.odd && p.x0 + ck.len < d.nvx) {
      p.odd = 1;
      p.x0 += ck.len;
      return;
    }
    if (PAIR && p.odd) {
      p.odd = 0;
      p.x0 -= ck.len;
    }
    if (++p.iy == r1) { p.iy = r0; p.x0 += (PAIR ? 2 : 1) * ck.len; }
  };
  int otile = tile, oslot = slot;
  if (act) fval_owner(bi, i0, j0, tile, slot, otile, oslot);
  const Quad<P> *fown = reinterpret_cast<const Quad<P> *>(d.fval) + (size_t)otile * fval_tile(d.nvp);
  Quad<P> *ring = FV + tid;
  auto stage = [&](const Pos &p, int st) {
    if (act && p.x0 < d.nvx) {
      const int n = min(ck.len, d.nvx - p.x0) - half;
      const int k0 = p.iy * d.nvx + p.x0 + half;
      const Quad<P> *src = fown + fval_at(k0, oslot);      // k0 + 2 q: NT vectors further each
#pragma unroll
      for (int q = 0; q < VH; ++q)
        if (2 * q < n) {
          char *dst = reinterpret_cast<char *>(ring + (st * VH + q) * NT);
#pragma unroll
          for (int e = 0; e < (int)sizeof(Quad<P>) / 16; ++e)
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(smem_addr(dst + 16 * e)),
                         "l"(reinterpret_cast<const char *>(src + q * NT) + 16 * e) : "memory");
        }
    }
    cp_async_commit();
  };
  Pos cur = {0, r0, 0}, nxt = cur;
  if (r0 == r1) nxt.x0 = d.nvx;
#pragma unroll
  for (int s = 0; s < FS - 1; ++s) { stage(nxt, s); advance(nxt); }
  const T Keff = (T)d.Keff;
  const P snx2 = pr_dup(P_[FP_SNX]), nux2 = pr_dup(-P_[FP_UX]), q12 = pr_dup(P_[FP_Q1]), q22 = pr_dup(P_[FP_Q2]);
  P cub[10];
#pragma unroll
  for (int m = 0; m < 10; ++m) cub[m] = pr_make(P_[FP_IH + m], P_[FP_IB + m]);
  P vx2[VH];
  T ex[VH];                                            // SEP: the columns' factors of the Maxwellian
  T vxr[PAIR ? 2 : 1][VH];                             // PAIR: the columns of both ranges
  int xcur = -1, st = 0, sn = FS - 1;                  // ring stages: this chunk's, the next copy's
  for (int ch = 0; ch < nch; ++ch) {
    const int n = min(ck.len, d.nvx - cur.x0);
    if (PAIR) {
      if (!cur.odd && cur.x0 != xcur) {                // another pair of ranges
        xcur = cur.x0;
#pragma unroll
        for (int h = 0; h < (PAIR ? 2 : 1); ++h)
#pragma unroll
          for (int q = 0; q < VH; ++q) {
            const int x = xcur + h * ck.len + half + 2 * q;
            vxr[h][q] = x < d.nvx ? grid_vx<T>(d, x) : T(0);
          }
      }
#pragma unroll
      for (int q = 0; q < VH; ++q) {
        vx2[q] = pr_dup(cur.odd ? vxr[PAIR ? 1 : 0][q] : vxr[0][q]);
        ex[q] = T(0);
      }
    } else if (cur.x0 != xcur) {                       // another range of columns
      xcur = cur.x0;
#pragma unroll
      for (int q = 0; q < VH; ++q) {
        const int kk = half + 2 * q;
        const T vx = kk < n ? grid_vx<T>(d, xcur + kk) : T(0), cx = vx - P_[FP_UX];
        vx2[q] = pr_dup(vx);
        ex[q] = SEP ? r_exp<T>(-P_[FP_LAM] * (cx * cx)) : T(0);
      }
    }
    const T vy = grid_vy<T>(d, d.iy0 + cur.iy);
    cp_async_wait<FS - 2>();
    P *fso = Fs + ((ch & 1) * NSLOT + slot) * VKG + half;
    const Quad<P> *fvb = ring + st * VH * NT;
    if (act) {
      // per-row factors: the c_y parts of the cubics and of the Maxwellian
      const T cy = vy - P_[FP_UY];
      const P cy2 = pr_dup(cy);
      const P a0 = pr_fma(cy2, pr_fma(cy2, pr_fma(cy2, cub[9], cub[5]), cub[2]), cub[0]);
      const P a1 = pr_fma(cy2, pr_fma(cy2, cub[8], cub[4]), cub[1]);
      const P a2 = pr_fma(cy2, cub[7], cub[3]), a3 = cub[6];
      const T ey = SEP ? P_[FP_HPRE] * r_exp<T>(-P_[FP_LAM] * (cy * cy)) : T(0);
      P wsy2;
      if constexpr (sizeof(T) == 8) wsy2 = pr_dup(face_ws_row(vy, P_[FP_SNY], P_[FP_SUN]));
      else wsy2 = pr_dup(vy * P_[FP_SNY] - P_[FP_SUN]);
#pragma unroll
      for (int q = 0; q < VH; ++q) {
        if (half + 2 * q < n) {
          // Eq. fullSolution averaged over dt_s: q1 f + q2 w.grad f + H ih(c)
          // (and b), the equilibrium factors as per-face cubics in c = v - U0
          const Quad<P> fv = fvb[q * NT];
          const P cx = pr_add(vx2[q], nux2);
          const P ph = pr_fma(cx, pr_fma(cx, pr_fma(cx, a3, a2), a1), a0);
          P I = pr_fma(q12, fv.x, pr_mul(q22, fv.y)), wS;
          T H;
          // (pr_fma and the sum of the joint form round as face_ws)
          if (SEP && (!wall || sizeof(T) == 8)) wS = pr_fma(vx2[q], snx2, wsy2);
          else wS = pr_add(pr_fma(vx2[q], snx2, pr_dup(vy * P_[FP_SNY])), pr_dup(-P_[FP_SUN]));
          if (SEP && !wall) {
            H = ey * ex[q];
          } else {
            H = P_[FP_HPRE] * r_exp<T>(-P_[FP_LAM] * (pr_get(cx).x * pr_get(cx).x + cy * cy));
          }
          I = pr_fma(pr_dup(H), ph, I);
          P out = pr_mul(wS, I);
          if (wall && !(pr_get(wS).x > T(0))) {
            // reflected part: wall Maxwellian at the face velocity (Eq. maxWalldes)
            const T w = pr_get(wS).x, wx = pr_get(vx2[q]).x - P_[FP_UFX], wy = vy - P_[FP_UFY], lw = P_[FP_LAMW];
            const T Hw = P_[FP_RHOW] * (lw * T(M_1_PI)) * r_exp<T>(-lw * (wx * wx + wy * wy));
            out = pr_make(w * Hw, w * Keff / (T(2) * lw) * Hw);
          }
          fso[2 * q] = out;
        }
      }
    }
    stage(nxt, sn);                                    // into the stage read one chunk ago
    advance(nxt);
    __syncthreads();                                   // face fluxes complete
    if (g >= 0) {
      const int o = (ch & 1) * NSLOT * VKG;
      const int k0 = cur.iy * d.nvx + cur.x0;
      P *out = reinterpret_cast<P *>(d.Dbuf) + (size_t)g * d.nvp + k0;
#pragma unroll
      for (int m = 0; m < VK / 4; ++m) {
        const int kk = (tid & 3) + 4 * m;
        if (kk < n) {
          P D = pr_mul(sg[0], fa[o + kk]);
          D = pr_fma(sg[1], fa[o + VKG + kk], D);
          D = pr_fma(sg[2], fc[o + kk], D);
          D = pr_fma(sg[3], fc[o + TX * VKG + kk], D);
          if (EVAL) {
            const auto v = pr_get(D);
            double *o2 = eval + 2 * ((size_t)g * d.nv + k0 + kk);
            const double2 w = field ? make_double2((double)v.x, (double)v.y) : make_double2(0.0, 0.0);
            if (wide) {
              *reinterpret_cast<double2 *>(o2) = w;
            } else {
              o2[0] = w.x;
              o2[1] = w.y;
            }
          } else {
            out[kk] = D;
          }
        }
      }
    }
    advance(cur);
    st = st + 1 == FS ? 0 : st + 1;
    sn = sn + 1 == FS ? 0 : sn + 1;
  }
  cp_async_wait<0>();
}

// Micro residual (Steps 3, 5; reading R4), elementwise over (cell, velocity):
//   r = T - Omega^{n+1} f / dt + (Omega^{n+1} (f+(W') - f)/tau' - D) / 2,
// with the level-n term T = Omega^n f^n / dt + (Omega^n (f+(W^n) - f^n)/tau^n
// - D^n) / 2 formed on the first inner iteration.  r goes to the sweep buffer.
//
// FP32: streaming (f, D, T in, r out; 6.4 TB/s).  Where the macro sweep, whose
// W' it needs, outlasts the flux pass that runs beside it (small velocity grids
// against the sweep's length: residual_split), a first pass (PART 1) forms the
// part without W', P = T_n - Omega^{n+1} f / dt - D / 2, within the sweep, and a
// second one (PART 2) adds the collision term; else one pass (PART 0), with the
// same roundings (256x128 + 128x32 cells, 1024 velocities: two passes 190 + 158
// us, one 203).  FP64: its pipe; the exponential of f+ (some
// thirty of its instructions) splits into a factor per column and one per row of
// the CTA's velocities, tabulated first, and f+ is written with the fewest
// operations (96x48 + 64x16 cells, 1024 velocities: 524 -> 334 us).
constexpr int RES_NT = 256;                      // most threads of a CTA
// pairs of adjacent velocities a thread takes (FP64: the tables and the
// constants of a cell serve two)
template <typename T> struct ResPairs { static constexpr int N = sizeof(T) == 8 ? 2 : 1; };
template <typename T> struct ResTable {          // exponentials per column and row of a CTA's velocities
  T ex[2 * RES_NT * ResPairs<T>::N], ey[2 * RES_NT * ResPairs<T>::N];
};
template <typename T>
__device__ __forceinline__ void res_table(const Dev &d, const T *rec, int k0, int n, ResTable<T> &tb) {
  // n consecutive velocities from k0: at most min(n, nvx) columns (from k0's
  // on) and the rows iy0 .. iy1
  const int iy0 = k0 / d.nvx, iy1 = (k0 + n - 1) / d.nvx;
  for (int i = threadIdx.x; i < min(n, d.nvx); i += blockDim.x) {
    const int k = k0 + i;                        // (columns of the first n velocities: all of them)
    const T cx = dvx<T>(d, k) - rec[SH_UX];
    tb.ex[i] = r_exp<T>(-rec[SH_LAM] * cx * cx);
  }
  for (int i = threadIdx.x; i <= iy1 - iy0; i += blockDim.x) {
    const T cy = dvy<T>(d, (iy0 + i) * d.nvx) - rec[SH_UY];
    tb.ey[i] = rec[SH_HPRE] * r_exp<T>(-rec[SH_LAM] * cy * cy);
  }
}
template <typename T, int FB, int PART> __global__ void __launch_bounds__(RES_NT) k_residual(Dev d, int first_iter) {
  typedef typename Vec2<T>::type T2;
  constexpr bool SEP = sizeof(T) == 8;
  __shared__ ResTable<T> tp, tn0;
  // grid: cells x velocity chunks; a thread takes pairs of adjacent velocities
  // (nvp is a multiple of 16, so a pair stays inside the cell's row)
  constexpr int NP = ResPairs<T>::N;
  const int c = blockIdx.x, kc = 2 * NP * blockIdx.y * blockDim.x;
  if (!(d.cmask[c] & 1)) return;
  const T *cp = reinterpret_cast<const T *>(d.shp) + (size_t)NSH * c;
  const T *cn = reinterpret_cast<const T *>(d.shn) + (size_t)NSH * c;
  if (SEP) {
    const int n = min(2 * NP * (int)blockDim.x, d.nv - kc);
    res_table<T>(d, cp, kc, n, tp);
    if (first_iter) res_table<T>(d, cn, kc, n, tn0);
    __syncthreads();
  }
  // (PART 1 runs before the cell record of W' is there; the record holds this volume)
  const T itau = PART == 1 ? T(0) : cp[SH_ITAU], vol1 = PART == 1 ? (T)d.vol_new[c] : cp[SH_VOL];
  const T hv = T(0.5) * vol1, hi = hv * itau;
  const T idt = sizeof(T) == 4 ? (T)reinterpret_cast<const float *>(d.stepc)[4] : (T)d.stepc[1];
#pragma unroll
  for (int m = 0; m < NP; ++m) {
    const int k0 = kc + 2 * (threadIdx.x + m * blockDim.x);
    if (k0 >= d.nv) return;
    T2 fv[2], D[2], tn[2];
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      size_t t = (size_t)c * d.nvp + k0 + u;
      fv[u] = ldF<T, FB>(d, t);
      if (PART == 2) {
        tn[u] = ldf<T>(d.dfs, t);                // P
      } else {
        D[u] = ldf<T>(d.Dbuf, t);
        if (!first_iter) tn[u] = ldf<T>(d.Tn, t);
      }
    }
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      int k = k0 + u;
      if (k >= d.nv) break;
      size_t t = (size_t)c * d.nvp + k;
      T vx = dvx<T>(d, k), vy = dvy<T>(d, k);
      auto equilibrium = [&](const T *rec, const ResTable<T> &tb) {
        if (!SEP) return shakhov_rec<T>(rec, vx, vy, (T)d.Keff, (T)d.Kint);
        const int i = k - kc, row = k / d.nvx - kc / d.nvx;
        return shakhov_short<T>(rec, vx, vy, tb.ex[i % d.nvx] * tb.ey[row], (T)d.Keff, (T)d.Kint);
      };
      V2<T> fp = {T(0), T(0)};
      if (PART != 1) fp = equilibrium(cp, tp);
      if (PART != 2 && first_iter) {
        T itn = cn[SH_ITAU];
        V2<T> fn = equilibrium(cn, tn0);
        T vol0 = cn[SH_VOL];
        tn[u].x = vol0 * idt * fv[u].x + T(0.5) * (vol0 * (fn.h - fv[u].x) * itn - D[u].x);
        tn[u].y = vol0 * idt * fv[u].y + T(0.5) * (vol0 * (fn.b - fv[u].y) * itn - D[u].y);
        stf<T>(d.Tn, t, tn[u].x, tn[u].y);
      }
      const T ph = PART == 2 ? tn[u].x : tn[u].x - vol1 * idt * fv[u].x - T(0.5) * D[u].x;
      const T pb = PART == 2 ? tn[u].y : tn[u].y - vol1 * idt * fv[u].y - T(0.5) * D[u].y;
      if (PART == 1) stf<T>(d.dfs, t, ph, pb);
      else if (SEP) stf<T>(d.dfs, t, ph + hi * (fp.h - fv[u].x), pb + hi * (fp.b - fv[u].y));
      else stf<T>(d.dfs, t, ph + hv * (fp.h - fv[u].x) * itau, pb + hv * (fp.b - fv[u].y) * itau);
    }
  }
}

// CTAs that share a tile's velocity chunks (by the sizes alone: the workspace is
// laid out by them, without a device): the share that ends a pass soonest
// on 152 SMs with two resident CTAs each (FP64: one), with ~4 us of set-up and
// finish a CTA against ~7 us a pair of chunks (FP32, the fold's unit) or ~22 us
// a chunk (FP64).  8 tiles at 16 x 16 velocities (32 x 16 cells): 8 CTAs a tile,
// reduction 62 -> 14 us; 88 tiles in FP64 (96 x 48 + 64 x 16 cells, 32 x 32
// velocities): 4.2 -> 1.7 ms; from about 600 tiles on a tile keeps its CTA.
int face_splits(int ntiles, int nvx, int nv, int fp32) {
  const int chunks = fp32 ? (nv + 2 * VK32 - 1) / (2 * VK32) : face_chunks<VK64>(nvx, nv).total;
  const int slots = fp32 ? 304 : 152;
  const double setup = 4.0, per = fp32 ? 7.0 : 22.0;
  int best = 1;
  double tb = 1e300;
  for (int n = 1; n <= chunks && n <= 32; ++n) {
    const double t = ((long)ntiles * n + slots - 1) / slots * (setup + per * ((chunks + n - 1) / n));
    if (t < 0.97 * tb) { tb = t; best = n; }
  }
  return best;
}

void face_tile_shape(int fp32, int *vk, int *nh) {
  *vk = fp32 ? VK32 : VK64;
  *nh = 2;
}

template <typename T, bool SEP> static void flux_attr() {
  cudaFuncSetAttribute(k_flux<T, SEP, false, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)flux_smem<T>());
  cudaFuncSetAttribute(k_flux<T, SEP, false, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)flux_smem<T>());
  if (!SEP) cudaFuncSetAttribute(k_flux<T, SEP, !SEP, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)flux_smem<T>());
}
void tile_setup() {
  cudaFuncSetAttribute(k_face_reduce32<0>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(Smem32));
  cudaFuncSetAttribute(k_face_reduce32<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(Smem32));
  cudaFuncSetAttribute(k_face_reduce64, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(Smem64));
  flux_attr<float, true>(); flux_attr<float, false>(); flux_attr<double, true>();
}

int tile_count(int ni, int nj) { return ((ni + TX - 1) / TX) * ((nj + TY - 1) / TY); }
void tile_origins(int ni, int nj, int *out) {   // (i0, j0) pairs
  int q = 0;
  for (int tj = 0; tj < (nj + TY - 1) / TY; ++tj)
    for (int ti = 0; ti < (ni + TX - 1) / TX; ++ti) { out[q++] = ti * TX; out[q++] = tj * TY; }
}

void launch_face_reduce(const Dev &d, cudaStream_t s, int fp32) {
  const dim3 grid(d.ntiles, d.nsplit);
  if (!fp32) k_face_reduce64<<<grid, NT, sizeof(Smem64), s>>>(d);
  else if (d.fbf) k_face_reduce32<1><<<grid, NT32, sizeof(Smem32), s>>>(d);
  else k_face_reduce32<0><<<grid, NT32, sizeof(Smem32), s>>>(d);
}
// Pairs of ranges where neighbouring ranges share the 32-byte sectors of D (rows of
// a multiple of four columns do not) and a sector written in part leaves the L2
// before its other part comes: D exceeds it, and one CTA walks all rows of its
// tile for a range, some 2.8 KB an item and 304 CTAs (126 MB and more from 21 rows
// on; a few rows less each where CTAs share a tile).  Flux pass, us, single ranges
// and pairs (MB of D): 256x128 + 128x32 cells, 17 columns 132 / 133 (90), 21: 194 /
// 189 (132), 22: 177 / 180, 25: 294 / 265, 31: 445 / 361, 33: 565 / 457, 49: 1321 /
// 995 (713); 300x150 + 2 x 120x30, 33: 731 / 649; multiples of four there, 24: 245
// / 272, 40: 659 / 714; CTAs that share tiles, 192x96 + 96x24, 31: 205 / 220,
// 300x150 + 120x30, 33: 579 / 596.
bool flux_pairs(size_t items, int nvx, int nsplit) {
  return nvx % 4 != 0 && nsplit == 1 && 8.0 * (double)items > 120e6;
}
template <bool EVAL> static void flux(const Dev &d, cudaStream_t s, int fp32, double *eval) {
  const dim3 grid(d.ntiles, d.nsplit);
  if (!fp32) k_flux<double, true, false, EVAL><<<grid, NT, flux_smem<double>(), s>>>(d, eval);
  else if (d.nvx % 16 == 0) k_flux<float, true, false, EVAL><<<grid, NT, flux_smem<float>(), s>>>(d, eval);
  else if (!EVAL && d.flux_pair) k_flux<float, false, true, false><<<grid, NT, flux_smem<float>(), s>>>(d, nullptr);
  else k_flux<float, false, false, EVAL><<<grid, NT, flux_smem<float>(), s>>>(d, eval);
}
void launch_flux(const Dev &d, cudaStream_t s, int fp32) { flux<false>(d, s, fp32, nullptr); }
void launch_flux_eval(const Dev &d, cudaStream_t s, double *D, int fp32) { flux<true>(d, s, fp32, D); }
// Whether the macro sweep (steps: diagonals of its two passes, some 0.25 us each)
// outlasts the flux pass and the residual's first pass (8.4 + 5.0 ps an item, a
// cell and velocity).  A step of 10 iterations in two passes and in one, ms, by
// the items a diagonal: 1.28e4 (128x64 + 64x16 cells, 23x23 velocities) 4.48 /
// 4.54, 1.39e4 (24x24) 4.42 / 4.49, 1.51e4 (25x25) 4.79 / 4.79, 1.76e4 (27x27)
// 5.16 / 5.05; 1.45e4 (192x96 + 96x24, 20x20) 7.51 / 7.35, 1.75e4 (22x22) 8.04 /
// 7.79; 1.40e4 (64x32, 36x36) 2.57 / 2.59, 1.56e4 (38x38) 2.82 / 2.74; 1.46e4
// (160x80 + 2 x 96x24, 20x20) 6.00 / 6.10; 2.8e4 (256x128 + 128x32, 24x24) 13.57 /
// 12.96, 4.9e4 (32x32) 18.08 / 16.85: they meet near 1.5e4.
bool residual_split(long items, long steps, int fp32) { return fp32 && (double)items < 1.5e4 * (double)steps; }

template <typename T, int FB, int PART> static void residual(const Dev &d, cudaStream_t s, int first_iter) {
  const int n = (d.nv + 2 * ResPairs<T>::N - 1) / (2 * ResPairs<T>::N);      // threads a cell
  const int bt = n >= RES_NT ? RES_NT : ((n + 31) / 32) * 32;
  k_residual<T, FB, PART><<<dim3(d.nc, (n + bt - 1) / bt), bt, 0, s>>>(d, first_iter);
}
template <int FB> static void residual32(const Dev &d, cudaStream_t s, int first_iter, int part) {
  if (part == 1) residual<float, FB, 1>(d, s, first_iter);
  else if (part == 2) residual<float, FB, 2>(d, s, first_iter);
  else residual<float, FB, 0>(d, s, first_iter);
}
void launch_residual(const Dev &d, cudaStream_t s, int first_iter, int fp32, int part) {
  if (!fp32) residual<double, 0, 0>(d, s, first_iter);
  else if (d.fbf) residual32<1>(d, s, first_iter, part);
  else residual32<0>(d, s, first_iter, part);
}

}  // namespace ugks
