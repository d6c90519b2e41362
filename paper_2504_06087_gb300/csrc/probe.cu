// Diagnostics of the SIMT pipes (float32 and float64): the matrix product on
// its own, and the FMA-rate probe.
//
// The roofline fractions of the kernels that run on the FP32 or FP64 pipe
// (the restricted log-det contraction, the Gauss-Jordan inverse, the float64
// LU) are quoted against the rate this kernel measures on the device at hand,
// instead of a rate derived from unit counts and clocks.
//
// Each thread runs eight independent multiply-add chains x <- x * a + b for
// `iters` rounds (eight dependent chains hide the pipe latency at full
// occupancy); the chains are written out at the end so no round can be
// dropped.  FLOPs = 2 * 8 * iters * blocks * threads.
#include <cuda_runtime.h>

#include "../../include/fire.h"
#include "gemm.cuh"

namespace {

template <typename T>
__device__ __forceinline__ T fma_rn(T x, T a, T b);

template <>
__device__ __forceinline__ float fma_rn<float>(float x, float a, float b) {
  float y;
  asm volatile("fma.rn.f32 %0, %1, %2, %3;" : "=f"(y) : "f"(x), "f"(a), "f"(b));
  return y;
}

template <>
__device__ __forceinline__ double fma_rn<double>(double x, double a, double b) {
  double y;
  asm volatile("fma.rn.f64 %0, %1, %2, %3;" : "=d"(y) : "d"(x), "d"(a), "d"(b));
  return y;
}

template <typename T>
__global__ void __launch_bounds__(256) fma_probe_kernel(T* __restrict__ out, long long iters, T a, T b) {
  const long long tid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  T x0 = (T)(threadIdx.x & 7), x1 = x0 + (T)1, x2 = x0 + (T)2, x3 = x0 + (T)3;
  T x4 = x0 + (T)4, x5 = x0 + (T)5, x6 = x0 + (T)6, x7 = x0 + (T)7;
  for (long long k = 0; k < iters; ++k) {
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      x0 = fma_rn<T>(x0, a, b);
      x1 = fma_rn<T>(x1, a, b);
      x2 = fma_rn<T>(x2, a, b);
      x3 = fma_rn<T>(x3, a, b);
      x4 = fma_rn<T>(x4, a, b);
      x5 = fma_rn<T>(x5, a, b);
      x6 = fma_rn<T>(x6, a, b);
      x7 = fma_rn<T>(x7, a, b);
    }
  }
  out[tid] = ((x0 + x1) + (x2 + x3)) + ((x4 + x5) + (x6 + x7));
}

}  // namespace

extern "C" int fire_selftest_fma_rate(int32_t dtype, int64_t iters, int32_t blocks, void* out, void* stream) {
  if ((dtype != 0 && dtype != 1) || iters < 1 || blocks < 1 || !out) return FIRE_ERR_INVALID_ARG;
  cudaStream_t s = (cudaStream_t)stream;
  // each loop round does four multiply-adds per chain
  const long long rounds = (iters + 3) / 4;
  if (dtype == 0)
    fma_probe_kernel<double><<<blocks, 256, 0, s>>>((double*)out, rounds, 0.9999999, 1e-7);
  else
    fma_probe_kernel<float><<<blocks, 256, 0, s>>>((float*)out, rounds, 0.9999f, 1e-4f);
  return cudaGetLastError() == cudaSuccess ? FIRE_OK : FIRE_ERR_CUDA;
}

extern "C" int fire_selftest_simt_gemm(int32_t dtype, int64_t M, int32_t N, int32_t K, int32_t batch, int32_t transB,
                                       int32_t accumulate, const void* A, int64_t lda, const void* B, int64_t ldb,
                                       int64_t sB, void* C, int64_t ldc, int64_t sC, void* stream) {
  if ((dtype != 0 && dtype != 1) || M < 1 || N < 1 || K < 1 || batch < 1 || lda < K || ldb < (transB ? K : N) ||
      ldc < N || sB < 0 || sC < 0 || !A || !B || !C)
    return FIRE_ERR_INVALID_ARG;
  cudaStream_t s = (cudaStream_t)stream;
  if (dtype == 0)
    fire::gemm<double>(s, (const double*)A, lda, (const double*)B, ldb, transB != 0, (double*)C, ldc, 0, M, nullptr,
                       M, N, K, batch, 0, sB, sC, accumulate != 0);
  else
    fire::gemm<float>(s, (const float*)A, lda, (const float*)B, ldb, transB != 0, (float*)C, ldc, 0, M, nullptr, M, N,
                      K, batch, 0, sB, sC, accumulate != 0);
  return cudaGetLastError() == cudaSuccess ? FIRE_OK : FIRE_ERR_CUDA;
}

extern "C" int fire_selftest_simt_layer(int32_t dtype, int64_t M, int32_t N, int32_t K, int32_t one, const void* A,
                                        int64_t lda, const void* B, const void* bias, const void* R, int64_t ldr,
                                        void* C, int64_t ldc, void* stream) {
  if ((dtype != 0 && dtype != 1) || M < 1 || N < 1 || K < 1 || lda < K || ldc < N || !A || !B || !bias || !C ||
      (R && ldr < N))
    return FIRE_ERR_INVALID_ARG;
  cudaStream_t s = (cudaStream_t)stream;
  if (dtype == 0)
    fire::gemm<double>(s, (const double*)A, lda, (const double*)B, N, false, (double*)C, ldc, 0, M, nullptr, M, N, K, 1,
                       0, 0, 0, false, (const double*)bias, (const double*)R, ldr, one != 0);
  else
    fire::gemm<float>(s, (const float*)A, lda, (const float*)B, N, false, (float*)C, ldc, 0, M, nullptr, M, N, K, 1, 0,
                      0, 0, false, (const float*)bias, (const float*)R, ldr, one != 0);
  return cudaGetLastError() == cudaSuccess ? FIRE_OK : FIRE_ERR_CUDA;
}
