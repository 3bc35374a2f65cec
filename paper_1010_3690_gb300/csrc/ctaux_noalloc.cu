// ctaux_invert_noalloc: the blocked Gauss-Jordan inversion of the from-scratch
// recomputation (ctaux_inverse.cu), for callers that cannot allocate device
// memory.  Its scratch (the matrix, the slices, pivots and flags) lives in one
// file-scope static device array; nothing here calls cudaMalloc, cudaFree or an
// allocating library routine.  Declared in include/ctaux.h.
#include <cuda_runtime.h>

#include <mutex>

#include "../../include/ctaux.h"
#include "ctaux_dev.cuh"
#include "ctaux_inverse.cuh"

namespace {

using namespace ctaux;

constexpr int kM = CTAUX_NOALLOC_MAX_M;

// Scratch layout, bytes: the work area of one matrix, then the pivot arrays,
// the order and the view.
constexpr size_t kWork = ((size_t)kM * kM + (size_t)kM * 114 + 1024) * sizeof(double);   // ld^2 + inv_extra_doubles(kM, 1)
constexpr size_t kPerm = kWork, kPcol = kPerm + kM * sizeof(int), kUsed = kPcol + kM * sizeof(int),
                 kStatus = kUsed + kM, kOrder = kStatus + 16, kBalance = kOrder + 16, kView = kBalance + 32 * sizeof(int),
                 kColExp = kView + (sizeof(InvView) + 15) / 16 * 16, kRowExp = kColExp + kM * sizeof(int),
                 kEnd = kRowExp + kM * sizeof(int);
static_assert(kEnd <= CTAUX_NOALLOC_SCRATCH_BYTES, "scratch size in the header");
static_assert(kM < kInvTwoLevel, "one level: one image per row block, and the balance");

// Shared by every call on a device; held by each device that loads the library.
static __device__ __align__(1024) unsigned char g_noalloc_scratch[CTAUX_NOALLOC_SCRATCH_BYTES];

// Columns and rows of extreme magnitude are brought near 1 by powers of two (A' =
// 2^-r A 2^-c, so A^-1 = 2^-c A'^-1 2^-r): the products of the elimination have no
// subnormal numbers, which would cost a matrix near the smallest or largest
// normal number its digits (entries of 2^-1010: error 8e-3 without).  Magnitudes from
// 2^-kPlain to 2^kPlain stay as they are.  Order 310: 795 -> 799 us.
constexpr int kPlain = 256;
__device__ __forceinline__ int exponent_field(double x) { return (__double2hiint(x) >> 20) & 0x7ff; }
__device__ __forceinline__ int scale_exponent(int largest_field) {
  if (largest_field == 0) return -1050;   // zero, or subnormal: 2^-1074 to 2^-1022
  if (largest_field == 0x7ff) return 0;
  const int e = largest_field - 1023;
  return abs(e) <= kPlain ? 0 : e;
}

// The matrix into the scratch, a CTA per column, with the state the inversion starts
// from (the previous call's must not leak in).
__global__ void __launch_bounds__(256) k_noalloc_load(const double* __restrict__ A, int lda, int m, InvView v,
                                                      unsigned char* scratch) {
  __shared__ int part[8];
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    *reinterpret_cast<InvView*>(scratch + kView) = v;
    *reinterpret_cast<int*>(scratch + kOrder) = m;
    *v.status = 0;
  }
  const int j = blockIdx.x;
  int most = 0;
  for (int i = threadIdx.x; i < m; i += blockDim.x) most = max(most, exponent_field(A[(size_t)j * lda + i]));
  most = __reduce_max_sync(0xffffffffu, most);
  if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = most;
  __syncthreads();
  for (int w = 0; w < 8; ++w) most = max(most, part[w]);
  const int e = scale_exponent(most);
  if (threadIdx.x == 0) {
    v.used[j] = 0;
    v.pcol[j] = -1;
    reinterpret_cast<int*>(scratch + kColExp)[j] = e;
  }
  for (int i = threadIdx.x; i < m; i += blockDim.x) {
    const double x = A[(size_t)j * lda + i];
    v.X[(size_t)j * v.ld + i] = e ? scalbn(x, -e) : x;
  }
}

// The rows of extreme magnitude, 32 rows per CTA, a lane per row.
__global__ void __launch_bounds__(256) k_noalloc_rows(int m, InvView v, int* row_exp) {
  __shared__ int part[8][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, i = blockIdx.x * 32 + lane;
  int most = 0;
  if (i < m) {
#pragma unroll 16
    for (int j = warp; j < m; j += 8) most = max(most, exponent_field(v.X[(size_t)j * v.ld + i]));
  }
  part[warp][lane] = most;
  __syncthreads();
  for (int w = 0; w < 8; ++w) most = max(most, part[w][lane]);
  const int e = scale_exponent(most);
  if (i >= m) return;
  if (warp == 0) row_exp[i] = e;
  if (e == 0) return;
  for (int j = warp; j < m; j += 8) v.X[(size_t)j * v.ld + i] = scalbn(v.X[(size_t)j * v.ld + i], -e);
}

// The inverse in the caller's order, and log|det| (the pivots' logarithms, in a
// fixed order).  All NaN where a bounded wait of the inversion gave up.
__global__ void __launch_bounds__(256) k_noalloc_store(double* __restrict__ Ainv, int ldi, int m, InvView v,
                                                       const int* __restrict__ col_exp,
                                                       const int* __restrict__ row_exp, double* logdet) {
  const int status = *v.status;
  const double poison = (status & ~DS_SINGULAR) ? nan("") : 0.0;
  for (int j = blockIdx.x; j < m; j += gridDim.x) {
    const int pj = inv_column(status, DS_SINGULAR, v.perm, j), re = row_exp[pj];
    for (int c = threadIdx.x; c < m; c += blockDim.x) {
      const double x = v.X[(size_t)j * v.ld + v.perm[c]] + poison;   // inv[c][perm[j]]
      const int e = re + col_exp[c];
      Ainv[(size_t)pj * ldi + c] = e ? scalbn(x, -e) : x;
    }
  }
  if (blockIdx.x == 0 && logdet) {
    __shared__ double part[8];
    __shared__ int exps;
    double s = 0.0;
    int e = 0;
    for (int k = threadIdx.x; k < m; k += blockDim.x) {
      s += log(fabs(v.piv[k]));
      e += col_exp[k] + row_exp[k];
    }
    s = warp_sum(s);
    e = __reduce_add_sync(0xffffffffu, e);
    if (threadIdx.x == 0) exps = 0;
    __syncthreads();
    if ((threadIdx.x & 31) == 0) {
      part[threadIdx.x >> 5] = s;
      atomicAdd(&exps, e);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      double t = 0.0;
      for (int w = 0; w < 8; ++w) t += part[w];
      *logdet = fma((double)exps, 0.69314718055994530942, t) + poison;   // ln 2
    }
  }
}

struct DeviceSetup {
  std::once_flag once;
  cudaError_t err = cudaSuccess;
  unsigned char* scratch = nullptr;  // device address of g_noalloc_scratch
  InvShape shape;
};
constexpr int kMaxDevices = 64;
DeviceSetup g_setup[kMaxDevices];

}  // namespace

extern "C" ctaux_status ctaux_invert_noalloc(const double* d_a, int lda, double* d_inv, int ld_inv,
                                             int m, double* d_logdet, void* cuda_stream) {
  if (!d_a || !d_inv || m < 1 || lda < m || ld_inv < m) return CTAUX_EINVAL;
  if (m > CTAUX_NOALLOC_MAX_M) return CTAUX_ECAPACITY;
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess) return CTAUX_ECUDA;
  if (dev < 0 || dev >= kMaxDevices) return CTAUX_EINVAL;
  DeviceSetup& s = g_setup[dev];
  // once per device, with that device current: the host-side name of the
  // array is only a stand-in, so resolve its device address here
  std::call_once(s.once, [&s, dev]() {
    s.err = cudaGetSymbolAddress(reinterpret_cast<void**>(&s.scratch), g_noalloc_scratch);
    int sms = 0;
    InvDevice d{};
    if (s.err == cudaSuccess) s.err = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (s.err == cudaSuccess) s.err = inv_device(sms, true, &d);
    if (s.err == cudaSuccess) s.shape = inv_shapes({kM}, d)[0];
  });
  if (s.err != cudaSuccess || !s.scratch) return CTAUX_ECUDA;
  InvView v{};
  inv_layout(reinterpret_cast<double*>(s.scratch), kM, 1, v);
  v.width = inv_width(kM, s.shape.dev);
  v.perm = reinterpret_cast<int*>(s.scratch + kPerm);
  v.pcol = reinterpret_cast<int*>(s.scratch + kPcol);
  v.used = reinterpret_cast<int8_t*>(s.scratch + kUsed);
  v.status = reinterpret_cast<int*>(s.scratch + kStatus);
  v.balance = reinterpret_cast<int*>(s.scratch + kBalance);   // a caller's rows may differ in scale
  cudaStream_t st = reinterpret_cast<cudaStream_t>(cuda_stream);
  int* const col_exp = reinterpret_cast<int*>(s.scratch + kColExp);
  int* const row_exp = reinterpret_cast<int*>(s.scratch + kRowExp);
  k_noalloc_load<<<m, 256, 0, st>>>(d_a, lda, m, v, s.scratch);
  k_noalloc_rows<<<(m + 31) / 32, 256, 0, st>>>(m, v, row_exp);
  cudaError_t e = cudaSuccess;
  launch_inverse(reinterpret_cast<const InvView*>(s.scratch + kView), reinterpret_cast<const int*>(s.scratch + kOrder),
                 1, m, s.shape, st, &e);
  if (e == cudaSuccess) {
    k_noalloc_store<<<m, 256, 0, st>>>(d_inv, ld_inv, m, v, col_exp, row_exp, d_logdet);
    e = cudaGetLastError();
  }
  return e == cudaSuccess ? CTAUX_OK : CTAUX_ECUDA;
}
