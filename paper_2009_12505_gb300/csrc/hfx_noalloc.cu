// hfx_term_noalloc: one exchange term contracted with no device allocation.
//
// Some callers cannot allocate device memory when they call into this
// library: a host framework that owns the GPU's memory through its own pool
// and forbids direct cudaMalloc, a latency-critical loop where cudaMalloc /
// cudaFree (which can synchronize the device) are not allowed, or a process
// whose device memory is already fully reserved by another allocator so that a
// new allocation would fail.  hfx_build allocates its working memory inside
// the context; this entry point does not: it keeps its two intermediates in
// the fixed static array below instead of allocated scratch.  The caller
// passes inputs and the output as device pointers.
//
// Two orders of the product, by multiply-adds:
//   pair:   W = V^T cA and X = cB D^T (one launch), out = W . X   (two launches)
//   staged: Y = V cB, T = Y D^T, out = cA . T                     (three)
// The pair order halves the work when i, k are no larger than j, l (60/90 ABFs,
// 13 and 27 AOs: 2.2 against 4.8 M multiply-adds), has one launch fewer, and
// its two first products run side by side; it is taken when it needs no more
// multiply-adds and its intermediates fit the static array, else the staged
// order, whose sizes the caller's limits are stated for.
// That term: 105 us a call before (three launches, one thread per output in
// the last), 31 us now.
#include <algorithm>
#include <mutex>

#include "hfx_internal.h"

namespace {

// Two intermediates of at most kHalf doubles each (2 MiB in total).  Every GPU
// that loads the library holds this array until the process exits.
constexpr int64_t kHalf = 131072;
static __device__ __align__(256) double g_noalloc_scratch[2 * kHalf];

constexpr int kMaxDevices = 64;
std::mutex g_mu;
// Per device: the CUDA context the address was looked up in (its process-wide
// unique id, 0 = none yet) and the address.  A static __device__ array has one
// copy per context, so a cached address is only valid in the context it came
// from: after cudaDeviceReset (a new primary context) or under another context
// made current with the driver API, the address is looked up again.
unsigned long long g_scratch_ctx[kMaxDevices] = {0};
double *g_scratch_ptr[kMaxDevices] = {nullptr};

typedef int (*CtxGetCurrentFn)(void **);
typedef int (*CtxGetIdFn)(void *, unsigned long long *);

// Id of the current context (0 when none is current or the driver calls are
// unavailable; the lookup then runs on every call).
unsigned long long current_context_id() {
  static CtxGetCurrentFn get_current = nullptr;
  static CtxGetIdFn get_id = nullptr;
  static bool resolved = false;
  if (!resolved) {
    cudaDriverEntryPointQueryResult q1, q2;
    void *f1 = nullptr, *f2 = nullptr;
    if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &f1, 12000, cudaEnableDefault, &q1) ==
            cudaSuccess && q1 == cudaDriverEntryPointSuccess &&
        cudaGetDriverEntryPointByVersion("cuCtxGetId", &f2, 12000, cudaEnableDefault, &q2) ==
            cudaSuccess && q2 == cudaDriverEntryPointSuccess) {
      get_current = (CtxGetCurrentFn)f1;
      get_id = (CtxGetIdFn)f2;
    }
    resolved = true;
  }
  if (!get_current || !get_id) return 0;
  void *c = nullptr;
  unsigned long long id = 0;
  if (get_current(&c) != 0 || !c || get_id(c, &id) != 0) return 0;
  return id;
}

// Y[al][j][l] = sum_be V[al][be] cB[be][j][l]
__global__ void k_term_y(int pA, int pB, int nj, int nl, const double *V, const double *cB,
                         double *Y) {
  const int n = nj * nl;
  for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < pA * n;
       idx += gridDim.x * blockDim.x) {
    const int al = idx / n, c = idx - al * n;
    double s = 0.0;
#pragma unroll 8
    for (int be = 0; be < pB; ++be) s = fma(V[al * pB + be], cB[be * n + c], s);
    Y[idx] = s;
  }
}

// T[x][j][k] = sum_l Y[x][j][l] D[k][l], element idx
__device__ __forceinline__ void term_t(int idx, int nj, int nk, int nl, const double *Y,
                                       const double *D, double *T) {
  const int n = nj * nk;
  const int x = idx / n, r = idx - x * n, j = r / nk, k = r - j * nk;
  const double *y = Y + ((int64_t)x * nj + j) * nl;
  const double *d = D + (int64_t)k * nl;
  double s = 0.0;
#pragma unroll 8
  for (int l = 0; l < nl; ++l) s = fma(y[l], d[l], s);
  T[idx] = s;
}

__global__ void k_term_t(int pA, int nj, int nk, int nl, const double *Y, const double *D,
                         double *T) {
  for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < pA * nj * nk;
       idx += gridDim.x * blockDim.x)
    term_t(idx, nj, nk, nl, Y, D, T);
}

// W[be][i][k] = sum_al V[al][be] cA[al][i][k] and X[be][j][k] = sum_l
// cB[be][j][l] D[k][l], one element per thread: bound by the latency of its
// loads (unrolled, so several are in flight) at these sizes.
__global__ void k_term_wx(int pA, int pB, int ni, int nj, int nk, int nl, const double *cA,
                          const double *V, const double *cB, const double *D, double *W,
                          double *X) {
  const int n = ni * nk, nw = pB * n, nx = pB * nj * nk;
  for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < nw + nx;
       idx += gridDim.x * blockDim.x) {
    if (idx >= nw) {
      term_t(idx - nw, nj, nk, nl, cB, D, X);
      continue;
    }
    const int be = idx / n, c = idx - be * n;
    double s = 0.0;
#pragma unroll 8
    for (int al = 0; al < pA; ++al) s = fma(V[(int64_t)al * pB + be], cA[(int64_t)al * n + c], s);
    W[idx] = s;
  }
}

// out[i][j] = sum_{x,k} A[x][i][k] T[x][j][k] with LANES lanes (32 or 1) per
// output, which share the p nk terms and add up in a fixed tree.  One thread
// per output (a chain of 780 loads and multiply-adds for 13 AOs and 60 ABFs)
// was most of the call; it is kept for blocks of so many outputs that threads
// alone fill the chip.
template <int LANES>
__global__ void k_term_out(int p, int ni, int nj, int nk, const double *A, const double *T,
                           double *out) {
  const int lane = threadIdx.x % LANES;
  const int64_t step = (int64_t)gridDim.x * blockDim.x / LANES;
  for (int64_t o = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / LANES;
       o < (int64_t)ni * nj; o += step) {
    const int i = (int)(o / nj), j = (int)(o - (int64_t)i * nj);
    double s = 0.0;
#pragma unroll 4
    for (int t = lane; t < p * nk; t += LANES) {
      const int x = t / nk, k = t - x * nk;
      s = fma(A[((int64_t)x * ni + i) * nk + k], T[((int64_t)x * nj + j) * nk + k], s);
    }
    for (int h = LANES / 2; h; h >>= 1) s += __shfl_xor_sync(0xffffffffu, s, h);
    if (lane == 0) out[o] = s;
  }
}

// Device address of the static array in the current context, looked up once
// per device and context (host code may not use the array's name as a device
// pointer).  The first call on a device, and the first after a device reset,
// does the lookup; make it outside stream capture.
cudaError_t scratch_for_current_device(double **out) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
  const unsigned long long ctx = current_context_id();
  std::lock_guard<std::mutex> lock(g_mu);
  if (!g_scratch_ptr[dev] || ctx == 0 || g_scratch_ctx[dev] != ctx) {
    void *p = nullptr;
    // makes the device's primary context current when no context is
    e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
    if (e != cudaSuccess) return e;
    g_scratch_ptr[dev] = (double *)p;
    g_scratch_ctx[dev] = current_context_id();
  }
  *out = g_scratch_ptr[dev];
  return cudaSuccess;
}

}  // namespace

extern "C" hfx_status hfx_term_noalloc(int32_t nabf_a, int32_t nabf_b, int32_t nao_i,
                                       int32_t nao_k, int32_t nao_j, int32_t nao_l,
                                       const double *cA, const double *V, const double *cB,
                                       const double *D, double *out, void *cuda_stream) {
  if (!cA || !V || !cB || !D || !out) return HFX_E_ARG;
  if (nabf_a < 1 || nabf_b < 1 || nao_i < 1 || nao_k < 1 || nao_j < 1 || nao_l < 1)
    return HFX_E_ARG;
  // both intermediates must fit their half of the static array
  if ((int64_t)nabf_a * nao_j * nao_l > kHalf || (int64_t)nabf_a * nao_j * nao_k > kHalf)
    return HFX_E_SHAPE;
  // the output kernel indexes ni * nj outputs in 32-bit arithmetic
  if ((int64_t)nao_i * nao_j > 2147483647ll) return HFX_E_SHAPE;
  double *scratch = nullptr;
  if (scratch_for_current_device(&scratch) != cudaSuccess) return HFX_E_CUDA;
  cudaStream_t st = (cudaStream_t)cuda_stream;
  double *Y = scratch, *T = scratch + kHalf;
  const int threads = 128;
  auto blocks = [&](int64_t n) { return (unsigned)std::max<int64_t>(1, std::min<int64_t>((n + threads - 1) / threads, 4096)); };
  auto term_out = [&](int p, const double *A, const double *B) {
    const int64_t n = (int64_t)nao_i * nao_j;
    if (n < 65536)
      k_term_out<32><<<blocks(32 * n), threads, 0, st>>>(p, nao_i, nao_j, nao_k, A, B, out);
    else
      k_term_out<1><<<blocks(n), threads, 0, st>>>(p, nao_i, nao_j, nao_k, A, B, out);
  };
  // elements and multiply-adds of the two orders (doubles: no overflow)
  const double w = (double)nabf_b * nao_i * nao_k, x = (double)nabf_b * nao_j * nao_k;
  const double y = (double)nabf_a * nao_j * nao_l, t = (double)nabf_a * nao_j * nao_k;
  const double pair = w * nabf_a + x * nao_l + x * nao_i;
  const double staged = y * nabf_b + t * nao_l + t * nao_i;
  if (w <= kHalf && x <= kHalf && pair <= staged) {
    k_term_wx<<<blocks((int64_t)(w + x)), threads, 0, st>>>(nabf_a, nabf_b, nao_i, nao_j, nao_k,
                                                            nao_l, cA, V, cB, D, Y, T);
    term_out(nabf_b, Y, T);
  } else {
    k_term_y<<<blocks((int64_t)y), threads, 0, st>>>(nabf_a, nabf_b, nao_j, nao_l, V, cB, Y);
    k_term_t<<<blocks((int64_t)t), threads, 0, st>>>(nabf_a, nao_j, nao_k, nao_l, Y, D, T);
    term_out(nabf_a, cA, T);
  }
  return cudaGetLastError() == cudaSuccess ? HFX_OK : HFX_E_CUDA;
}
