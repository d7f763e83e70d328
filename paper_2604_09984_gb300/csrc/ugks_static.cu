// ugks_static.cu -- allocation-free receptor interpolation.
//
// Some callers cannot allocate device memory at all: code running inside a
// host framework that owns every device allocation and hands out only the
// buffers it manages, or code that must not call cudaMalloc while another
// component is capturing or replaying work.  ugks_idw_interpolate_static
// serves them: it takes the fields, receptor list and donor stencils as
// caller buffers and stages the interpolated values in a fixed-size scratch
// array that lives in this file as a static __device__ variable (every GPU
// that loads the library holds it until the process exits).
//
// Host code must not use the array's name as a device address: on the host
// that symbol is only a stand-in.  The device address is obtained with
// cudaGetSymbolAddress (with the device current) on the first call in each
// CUDA context and passed to the kernels; a new context on a device (after
// cudaDeviceReset, for instance) reloads the module and triggers a new
// lookup on its first call.
#include <cuda.h>
#include <cuda_runtime.h>
#include <cstdint>
#include <mutex>

#include "ugks.h"

namespace {

__device__ __align__(256) double g_idw_scratch[UGKS_STATIC_SCRATCH_DOUBLES];

constexpr int kMaxDevices = 64;
double *g_scratch_addr[kMaxDevices];
CUcontext g_scratch_ctx[kMaxDevices];     // context the address belongs to
std::mutex g_scratch_mutex;

typedef CUresult (*CtxGetCurrentFn)(CUcontext *);

// The calling thread's current CUDA context (driver entry point reached
// through the runtime, so the library needs no link against libcuda).
CUcontext current_context() {
  static CtxGetCurrentFn fn = nullptr;
  static bool tried = false;
  if (!tried) {
    void *p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuCtxGetCurrent", &p, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<CtxGetCurrentFn>(p);
    cudaGetLastError();
    tried = true;
  }
  CUcontext c = nullptr;
  if (fn && fn(&c) != CUDA_SUCCESS) c = nullptr;
  return c;
}

// The scratch array's device address in the current context (looked up on
// the first call in that context).
int scratch_for_current_device(double **out) {
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) {
    cudaGetLastError();
    return UGKS_ERR_CUDA;
  }
  std::lock_guard<std::mutex> lock(g_scratch_mutex);
  // (no context yet: null, which never matches, so the lookup below runs
  // and the next call records the context it created)
  CUcontext ctx = current_context();
  if (!g_scratch_addr[dev] || ctx == nullptr || ctx != g_scratch_ctx[dev]) {
    void *p = nullptr;
    if (cudaGetSymbolAddress(&p, g_idw_scratch) != cudaSuccess || p == nullptr) {
      cudaGetLastError();
      return UGKS_ERR_CUDA;
    }
    g_scratch_addr[dev] = static_cast<double *>(p);
    g_scratch_ctx[dev] = ctx;
  }
  *out = g_scratch_addr[dev];
  return UGKS_OK;
}

// Pass 1: every receptor row from its donors' values before the call
// (Jacobi), into the scratch.  Donor ids outside [0, ncells) are skipped and
// the remaining weights of the row renormalised to their sum (a row with no
// donor left keeps its values, flagged by a zero weight sum).  Grid:
// (receptor, velocity chunk).
__global__ void k_idw_gather_static(double *scratch, const double *f, const double *W,
                                    const double *q, int ncells, int nv, int nrec,
                                    const int32_t *donors, const double *weights) {
  int r = blockIdx.x;
  int k = blockIdx.y * blockDim.x + threadIdx.x;
  const int32_t *dn = donors + 5 * (size_t)r;
  const double *wt = weights + 5 * (size_t)r;
  double wv[5], wsum = 0.0;
  bool skipped = false;
  for (int m = 0; m < 5; ++m) {
    int e = dn[m];
    bool ok = e >= 0 && e < ncells;
    skipped = skipped || (e != -1 && !ok);
    wv[m] = ok ? wt[m] : 0.0;
    wsum = wsum + wv[m];
  }
  if (skipped && wsum != 0.0)
    for (int m = 0; m < 5; ++m) wv[m] = wv[m] / wsum;
  double *sw = scratch + 2 * (size_t)nrec * nv + 7 * (size_t)r;
  if (k < nv) {
    double ah = 0.0, ab = 0.0;
    for (int m = 0; m < 5; ++m) {
      int e = dn[m];
      if (e < 0 || e >= ncells) continue;
      const double *fe = f + 2 * ((size_t)e * nv + k);
      ah = ah + wv[m] * fe[0];
      ab = ab + wv[m] * fe[1];
    }
    scratch[2 * ((size_t)r * nv + k)] = ah;
    scratch[2 * ((size_t)r * nv + k) + 1] = ab;
  }
  if (blockIdx.y == 0 && threadIdx.x == 0) {
    double acc[6] = {0, 0, 0, 0, 0, 0};
    for (int m = 0; m < 5; ++m) {
      int e = dn[m];
      if (e < 0 || e >= ncells) continue;
      if (W)
        for (int c = 0; c < 4; ++c) acc[c] = acc[c] + wv[m] * W[4 * (size_t)e + c];
      if (q) {
        acc[4] = acc[4] + wv[m] * q[2 * (size_t)e];
        acc[5] = acc[5] + wv[m] * q[2 * (size_t)e + 1];
      }
    }
    for (int c = 0; c < 6; ++c) sw[c] = acc[c];
    sw[6] = wsum;
  }
}

// Pass 2: scatter the staged rows; rows without a donor stay unchanged.
__global__ void k_idw_scatter_static(const double *scratch, double *f, double *W, double *q,
                                     int ncells, int nv, int nrec, const int32_t *receptors,
                                     const int32_t *donors) {
  int r = blockIdx.x;
  int k = blockIdx.y * blockDim.x + threadIdx.x;
  const double *sw = scratch + 2 * (size_t)nrec * nv + 7 * (size_t)r;
  if (donors[5 * (size_t)r] < 0 || sw[6] == 0.0) return;
  int c = receptors[r];
  if (c < 0 || c >= ncells) return;
  if (k < nv) {
    double *fc = f + 2 * ((size_t)c * nv + k);
    fc[0] = scratch[2 * ((size_t)r * nv + k)];
    fc[1] = scratch[2 * ((size_t)r * nv + k) + 1];
  }
  if (blockIdx.y == 0 && threadIdx.x == 0) {
    if (W)
      for (int m = 0; m < 4; ++m) W[4 * (size_t)c + m] = sw[m];
    if (q) {
      q[2 * (size_t)c] = sw[4];
      q[2 * (size_t)c + 1] = sw[5];
    }
  }
}

// One pass: a value depends on its donors' values at the same velocity only, so
// a CTA that takes CH (h, b) pairs of every receptor (the pairs of W and q
// follow those of f) reads them all before it writes the first, and no scratch
// and no second launch are needed.  A call is bound by its launches, by two
// dependent loads and by the instructions themselves: they are fetched anew on
// every call, so loops are not unrolled (unrolled fourfold with the values in
// registers: 16.4 us), and weights, their sum and a division of the FP64 pipe
// are formed once a receptor in shared memory (280 receptors, 576 velocities:
// 14.4 us a call in two passes, 8.5 in one; with 256 threads 10.2).
constexpr int ITHREADS = 512, ONE_PASS_NV = 8192;
struct IdwRow { double w[5]; int e[5], target; };      // e: valid donors, else -1
template <int CH, typename V>
__global__ void __launch_bounds__(ITHREADS) k_idw_one_pass(double *f, double *W, double *q, int ncells, int nv, int nrec,
                                                           const int32_t *receptors, const int32_t *donors,
                                                           const double *weights) {
  extern __shared__ __align__(16) unsigned char smraw[];
  IdwRow *row = reinterpret_cast<IdwRow *>(smraw);
  double2 *val = reinterpret_cast<double2 *>(row + nrec);
#pragma unroll 1
  for (int r = threadIdx.x; r < nrec; r += ITHREADS) {
    const int c = receptors[r];
    double wsum = 0.0;
    bool skipped = false;
#pragma unroll
    for (int m = 0; m < 5; ++m) {
      const int e = donors[5 * (size_t)r + m];
      const bool ok = e >= 0 && e < ncells;
      const double w = ok ? weights[5 * (size_t)r + m] : 0.0;
      skipped = skipped || (e != -1 && !ok);
      row[r].e[m] = ok ? e : -1;
      row[r].w[m] = w;
      wsum = wsum + w;
    }
    row[r].target = donors[5 * (size_t)r] < 0 || wsum == 0.0 || c < 0 || c >= ncells ? -1 : c;
    if (skipped && wsum != 0.0)
#pragma unroll 1
      for (int m = 0; m < 5; ++m) row[r].w[m] = row[r].w[m] / wsum;
  }
  __syncthreads();
  const int p = blockIdx.x * CH + threadIdx.x % CH;
  // pair p of a cell: f, then W, then q (none where the array is not given)
  V *base = reinterpret_cast<V *>(p < nv ? f + 2 * p : p < nv + 2 ? W : q);
  if (p >= nv && p < nv + 2 && W) base += 2 * sizeof(double) / sizeof(V) * (p - nv);
  const long stride = (p < nv ? 2L * nv : p < nv + 2 ? 4 : 2) * sizeof(double) / sizeof(V);
  const bool live = p < nv || (p < nv + 2 ? W != nullptr : p == nv + 2 && q);
  constexpr int NX = 2 * sizeof(double) / sizeof(V);
#pragma unroll 1
  for (int r = threadIdx.x / CH; r < nrec; r += ITHREADS / CH) {
    if (!live || row[r].target < 0) continue;
    double ah = 0.0, ab = 0.0;
#pragma unroll
    for (int m = 0; m < 5; ++m) {
      const int e = row[r].e[m];
      if (e < 0) continue;
      double x[2];
#pragma unroll
      for (int i = 0; i < NX; ++i) reinterpret_cast<V *>(x)[i] = base[stride * e + i];
      ah = ah + row[r].w[m] * x[0];
      ab = ab + row[r].w[m] * x[1];
    }
    val[CH * r + threadIdx.x % CH] = make_double2(ah, ab);
  }
  __syncthreads();
#pragma unroll 1
  for (int r = threadIdx.x / CH; r < nrec; r += ITHREADS / CH) {
    if (!live || row[r].target < 0) continue;
    const double2 v = val[CH * r + threadIdx.x % CH];
    const double x[2] = {v.x, v.y};
#pragma unroll
    for (int i = 0; i < NX; ++i) base[stride * row[r].target + i] = reinterpret_cast<const V *>(x)[i];
  }
}
template <int CH> size_t one_pass_smem(int nrec) { return (size_t)nrec * (sizeof(IdwRow) + CH * sizeof(double2)); }
template <int CH>
void one_pass(double *f, double *W, double *q, int ncells, int nv, int nrec, const int32_t *receptors,
              const int32_t *donors, const double *weights, cudaStream_t s) {
  const int grid = (nv + 3 + CH - 1) / CH;
  const size_t sm = one_pass_smem<CH>(nrec);
  const bool aligned = ((reinterpret_cast<uintptr_t>(f) | reinterpret_cast<uintptr_t>(W) | reinterpret_cast<uintptr_t>(q)) & 15) == 0;
  if (aligned) k_idw_one_pass<CH, double2><<<grid, ITHREADS, sm, s>>>(f, W, q, ncells, nv, nrec, receptors, donors, weights);
  else k_idw_one_pass<CH, double><<<grid, ITHREADS, sm, s>>>(f, W, q, ncells, nv, nrec, receptors, donors, weights);
}

}  // namespace

extern "C" int ugks_idw_interpolate_static(double *f, double *W, double *q, int ncells, int nv,
                                           const int32_t *receptors, int nrec,
                                           const int32_t *donors, const double *weights,
                                           void *stream) {
  if (!f || ncells <= 0 || nv <= 0 || nrec < 0 || (nrec > 0 && (!receptors || !donors || !weights)))
    return UGKS_ERR_ARG;
  if (nrec == 0) return UGKS_OK;
  // staged values: 2 per (receptor, velocity) plus 7 per receptor
  unsigned long long need = 2ull * nrec * nv + 7ull * nrec;
  if (need > UGKS_STATIC_SCRATCH_DOUBLES) return UGKS_ERR_ARG;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  // One pass where a CTA's shared memory (48 KB) holds every receptor: four pairs
  // (a line of 64 bytes) a CTA, two where four would leave SMs idle.  Else two
  // passes through the scratch; so too beyond ONE_PASS_NV velocities, which leave
  // few receptors (the scratch bounds their product) and a CTA with four pairs of
  // each mostly idle threads, CTA after CTA (one pass / two, us a call back to
  // back: 4096 velocities, 1 and 63 receptors 6.3 / 10.4 and 10.4 / 18.5; 8192, 1
  // and 31 receptors 10.3 / 10.3 and 12.4 / 18.4; 16000, 1 and 16 receptors
  // 14.5 / 10.3 and 16.5 / 18.5, with cold caches 21.1 / 15.0 and 25.2 / 21.2;
  // 262000, 1 receptor 172 / 18).
  const bool four = nv >= 4 * 128 && one_pass_smem<4>(nrec) <= 48 * 1024;
  if (nv <= ONE_PASS_NV && (four || one_pass_smem<2>(nrec) <= 48 * 1024)) {
    if (four) one_pass<4>(f, W, q, ncells, nv, nrec, receptors, donors, weights, s);
    else one_pass<2>(f, W, q, ncells, nv, nrec, receptors, donors, weights, s);
    if (cudaPeekAtLastError() != cudaSuccess) {
      cudaGetLastError();
      return UGKS_ERR_CUDA;
    }
    return UGKS_OK;
  }
  double *scratch = nullptr;
  int r = scratch_for_current_device(&scratch);
  if (r != UGKS_OK) return r;
  int bt = nv >= 256 ? 256 : ((nv + 31) / 32) * 32;
  dim3 grid(nrec, (nv + bt - 1) / bt);
  k_idw_gather_static<<<grid, bt, 0, s>>>(scratch, f, W, q, ncells, nv, nrec, donors, weights);
  k_idw_scatter_static<<<grid, bt, 0, s>>>(scratch, f, W, q, ncells, nv, nrec, receptors, donors);
  if (cudaPeekAtLastError() != cudaSuccess) {
    cudaGetLastError();
    return UGKS_ERR_CUDA;
  }
  return UGKS_OK;
}
