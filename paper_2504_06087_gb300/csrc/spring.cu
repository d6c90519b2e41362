// SPRING parameter update (Methods, "Variational Monte Carlo", eq. spring):
//
//   Obar_i = O_i - mean_j O_j,   eps_i = E_L,i - mean_j E_L,j,
//   delta  = Obar^T (Obar Obar^T + lambda I)^-1 (eps - eta Obar delta_prev) + eta delta_prev,
//
// with the N x P matrix O of per-walker rows d ln|Psi| / d theta (the output
// of fire_grad_logpsi).  The N x N Gram matrix is the only dense contraction
// (2 N^2 P flops): it runs on the tensor cores as a split-bf16 product (three
// bf16 components per operand, six component products, FP32 accumulation in
// tensor memory) over chunks of the parameter axis, each chunk's rows
// converted once and its partial Gram matrix summed in float64.  The product
// takes the uncentred rows (G = O O^T) and the centring is applied exactly in
// float64 to the N x N matrix, Obar Obar^T = P G P with P = I - 1 1^T / N:
// centring the rows first would leave every row carrying the mean of the
// largest ones, whose float32 rounding then swamps the small eigenvalues, and
// the exact projection keeps 1 an exact null vector.  The damped N x N
// system is solved by a float64 blocked Cholesky factorisation of
// P G P + lambda I + mu 1 1^T / N (mu = the mean of diag P G P): the right-hand
// side is orthogonal to 1, so the added term changes no solution but keeps
// the null direction away from zero;
// the column means, the projection Obar delta_prev and the final
// Obar^T x are single streaming passes over O (HBM-bound).
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/fire.h"
#include "plan.h"
#include "tc_api.h"

namespace fire {
namespace spring {

// Parameters per Gram chunk (multiple of 64).  The tensor cores accumulate a
// chunk in float32 with an error that grows with the number of K steps
// (about 2^-22 of the running sum per 16-deep step, measured); chunks of 4096
// keep it near 6e-5 of sqrt(G_ii G_jj), and the chunks are summed in float64.
constexpr int kChunk = 1 << 12;
constexpr int kNC = 3;            // bf16 components per operand
constexpr int kB = 64;            // Cholesky block

inline size_t align_up(size_t x) { return (x + 255) & ~(size_t)255; }

struct Layout {
  int64_t Np;       // N rounded up to the Cholesky block
  int64_t pc;       // chunk width used (<= kChunk, multiple of 64)
  int groups;       // chunks whose products run together
  size_t mean, pack, cch, kacc, rowdot, b, a, rinv, scal, err, total;
};

// Chunks per product launch: the fewest that keep nine tenths of the SMs (a
// CTA of 128 x 128 outputs each) busy to the last round, within 512 MB of
// packed rows.  N = 1024 (64 tiles of a chunk): 7.
inline int chunk_groups(int64_t N, int64_t pc, int64_t nchunk) {
  const int64_t tiles = ((N + 127) / 128) * ((N + 127) / 128);
  int best = 1;
  double eff = 0.0;
  for (int64_t g = 1; g <= kSMs && g <= nchunk && (g == 1 || g * kNC * N * pc * 2 <= (512ll << 20)); ++g) {
    const int64_t t = tiles * g;
    const double e = (double)t / (double)((t + kSMs - 1) / kSMs * kSMs);
    if (e > eff) { eff = e; best = (int)g; }
    if (e >= 0.9) break;
  }
  return best;
}

inline Layout layout(int64_t N, int64_t P) {
  Layout L{};
  L.Np = (N + kB - 1) / kB * kB;
  int64_t pc = (P + 63) / 64 * 64;
  L.pc = pc < kChunk ? pc : kChunk;
  L.groups = chunk_groups(N, L.pc, (P + L.pc - 1) / L.pc);
  size_t o = 0;
  L.mean = o;   o = align_up(o + (size_t)P * 8);
  L.pack = o;   o = align_up(o + (size_t)kNC * N * L.pc * L.groups * 2);
  L.cch = o;    o = align_up(o + (size_t)N * N * L.groups * 4);
  L.kacc = o;   o = align_up(o + (size_t)L.Np * L.Np * 8);
  L.rowdot = o; o = align_up(o + (size_t)N * 8);
  L.b = o;      o = align_up(o + (size_t)L.Np * 8);
  L.a = o;      o = align_up(o + (size_t)N * 8);
  L.rinv = o;   o = align_up(o + (size_t)L.Np * 8);
  L.scal = o;   o = align_up(o + 32);
  L.err = o;    o = align_up(o + 16);
  L.total = o;
  return L;
}

// A float32 as float64 by integer operations: on GB300 a widening conversion
// takes the float64 pipe like an addition (even one that is predicated off),
// and the streaming passes over O below are bound by that pipe: 10^9 elements
// with a conversion and an addition each took 3.8 ms, without the conversion
// 2.1 ms, against 0.6 ms of HBM reads.  Subnormals are scaled into the normal
// range first; the exponent of infinities and NaNs is filled.
__device__ __forceinline__ double widen(float v) {
  const uint32_t e = __float_as_uint(v) & 0x7f800000u;
  const bool tiny = e == 0u;
  const uint32_t u = __float_as_uint(tiny ? v * 16777216.f : v), m = u & 0x7fffffffu;
  uint32_t hi = (m >> 3) + (tiny ? 0x38000000u - (24u << 20) : (e == 0x7f800000u ? 0x70000000u : 0x38000000u));
  hi = m == 0u ? 0u : hi;
  return __hiloint2double((int)((u & 0x80000000u) | hi), (int)(u << 29));
}

// mean[p] = (1/N) sum_i O[i][p]; one thread per column, rows streamed (each
// warp reads 128 contiguous bytes of a row per step), eight loads ahead.
// 1024 x 10^6: 3.8 -> 2.0 ms.
__global__ void __launch_bounds__(256) colmean_kernel(int64_t N, int64_t P, const float* __restrict__ O, int64_t ldo,
                                                      double* __restrict__ mean) {
  const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= P) return;
  double s[4] = {0.0, 0.0, 0.0, 0.0};
  int64_t i = 0;
  for (; i + 8 <= N; i += 8) {
    float v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) v[u] = O[(i + u) * ldo + p];
#pragma unroll
    for (int u = 0; u < 8; ++u) s[u & 3] += widen(v[u]);
  }
  for (; i + 4 <= N; i += 4)
#pragma unroll
    for (int u = 0; u < 4; ++u) s[u] += widen(O[(i + u) * ldo + p]);
  for (; i < N; ++i) s[0] += widen(O[i * ldo + p]);
  mean[p] = ((s[0] + s[1]) + (s[2] + s[3])) / (double)N;
}

// Rows of the columns [p0, p0 + width) as kNC bf16 components dst[c][i][q]
// (q < width; zero beyond P), and rowdot[i] += sum_q O_iq dprev[p0 + q] (the
// mean's share of the projection Obar delta_prev is one number for every row:
// meandot_kernel).  Block (x, y): kPackRows rows, 4096 columns, 16 per thread;
// dprev is widened once for all rows and the rows' sums are reduced together
// (transpose-halving), so an element costs one float64 multiply-add.
// 1024 x 10^6: 11.5 -> 2.4 ms.
constexpr int kPackRows = 16;
__global__ void __launch_bounds__(256) pack_kernel(int64_t N, int64_t P, const float* __restrict__ O, int64_t ldo,
                                                   int64_t p0, int64_t width, __nv_bfloat16* __restrict__ dst,
                                                   const float* __restrict__ dprev, double* __restrict__ rowdot,
                                                   int vec) {
  __shared__ double red[8][kPackRows];
  const int64_t i0 = (int64_t)blockIdx.y * kPackRows;
  const int nr = (int)(N - i0 < kPackRows ? N - i0 : kPackRows);
  double acc[kPackRows];
#pragma unroll
  for (int r = 0; r < kPackRows; ++r) acc[r] = 0.0;
  for (int u = 0; u < 4; ++u) {
    const int64_t q = (int64_t)blockIdx.x * 4096 + u * 1024 + threadIdx.x * 4;
    if (q >= width) break;
    const int64_t p = p0 + q;
    const int left = (int)(P - p < 4 ? (P > p ? P - p : 0) : 4);
    double d[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) d[k] = dprev && k < left ? widen(dprev[p + k]) : 0.0;
#pragma unroll
    for (int r = 0; r < kPackRows; ++r) {
      if (r >= nr) break;
      const float* src = O + (i0 + r) * ldo + p;
      float v[4];
      if (vec && left == 4) {
        const float4 x = *reinterpret_cast<const float4*>(src);
        v[0] = x.x; v[1] = x.y; v[2] = x.z; v[3] = x.w;
      } else {
#pragma unroll
        for (int k = 0; k < 4; ++k) v[k] = k < left ? src[k] : 0.f;
      }
      if (dprev) {
#pragma unroll
        for (int k = 0; k < 4; ++k)
          if (k < left) acc[r] = fma(widen(v[k]), d[k], acc[r]);
      }
      __nv_bfloat16* out = dst + (i0 + r) * width + q;
#pragma unroll
      for (int c = 0; c < kNC; ++c) {
        struct alignas(8) { __nv_bfloat16 x[4]; } h;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          h.x[k] = __float2bfloat16_rn(v[k]);
          v[k] -= __bfloat162float(h.x[k]);
        }
        *reinterpret_cast<uint2*>(out + (int64_t)c * N * width) = *reinterpret_cast<const uint2*>(&h);
      }
    }
  }
  if (!dprev) return;
  // lane L ends with the warp sum of row L & 15
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int s = 8; s >= 1; s >>= 1) {
    const bool up = (lane & s) != 0;
#pragma unroll
    for (int k = 0; k < s; ++k) {
      const double send = up ? acc[k] : acc[k + s], keep = up ? acc[k + s] : acc[k];
      acc[k] = keep + __shfl_xor_sync(0xffffffffu, send, s);
    }
  }
  acc[0] += __shfl_xor_sync(0xffffffffu, acc[0], 16);
  if (lane < kPackRows) red[threadIdx.x >> 5][lane] = acc[0];
  __syncthreads();
  if (threadIdx.x < nr) {
    double s = 0.0;
    for (int w = 0; w < 8; ++w) s += red[w][threadIdx.x];
    atomicAdd(&rowdot[i0 + threadIdx.x], s);
  }
}

// *out += sum_p mean[p] dprev[p].
__global__ void __launch_bounds__(256) meandot_kernel(int64_t P, const double* __restrict__ mean,
                                                      const float* __restrict__ dprev, double* __restrict__ out) {
  __shared__ double red[8];
  double s = 0.0;
  for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < P; p += (int64_t)gridDim.x * blockDim.x)
    s = fma(mean[p], widen(dprev[p]), s);
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < 8; ++w) t += red[w];
    atomicAdd(out, t);
  }
}

// K[i][j] (+)= sum_g C[g][i][j] in float64, the groups in order, over the N x N
// block of the padded Np x Np matrix; the padding gets the identity when
// first == 1.
__global__ void accum_kernel(int64_t N, int64_t Np, const float* __restrict__ C, int groups, double* __restrict__ K,
                             int first) {
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= Np * Np) return;
  const int64_t i = e / Np, j = e % Np;
  if (i < N && j < N) {
    double k = (double)C[i * N + j];
    if (!first) k = K[e] + k;
    for (int g = 1; g < groups; ++g) k += (double)C[((int64_t)g * N + i) * N + j];
    K[e] = k;
  } else if (first) {
    K[e] = (i == j) ? 1.0 : 0.0;
  }
}

// a[i] = (1/N) sum_j G[i][j] (row means of the uncentred Gram matrix), one
// warp per row.
__global__ void rowmean_kernel(int64_t N, int64_t Np, const double* __restrict__ K, double* __restrict__ a) {
  const int64_t i = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (i >= N) return;
  double s = 0.0;
  for (int64_t j = lane; j < N; j += 32) s += K[i * Np + j];
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (lane == 0) a[i] = s / (double)N;
}

// K <- P G P = G - a 1^T - 1 a^T + abar 1 1^T (abar = mean of a), in place
// over the N x N block; one CTA of 1024 threads forms abar first.
__global__ void center_kernel(int64_t N, int64_t Np, double* __restrict__ K, const double* __restrict__ a,
                              double* __restrict__ abar_out) {
  __shared__ double red[32];
  __shared__ double s_abar;
  double s = 0.0;
  for (int64_t i = threadIdx.x; i < N; i += blockDim.x) s += a[i];
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += red[w];
    s_abar = t / (double)N;
    if (blockIdx.x == 0 && abar_out) *abar_out = s_abar;
  }
  __syncthreads();
  const double abar = s_abar;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < N * N; e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = e / N, j = e % N;
    K[i * Np + j] = ((K[i * Np + j] - a[i]) - a[j]) + abar;
  }
}

// b[i] = (E_i - mean E) - eta (rowdot[i] - *meandot) (zero in the padding); *mu = the
// mean of diag K (before the damping); then K[i][i] += lambda.
__global__ void rhs_kernel(int64_t N, int64_t Np, const double* __restrict__ e_loc, const double* __restrict__ rowdot,
                           const double* __restrict__ meandot, double eta, double lambda, double* __restrict__ b,
                           double* __restrict__ K, double* __restrict__ mu) {
  __shared__ double red[2][32];
  __shared__ double s_mean;
  double s = 0.0, dsum = 0.0;
  for (int64_t i = threadIdx.x; i < N; i += blockDim.x) {
    s += e_loc[i];
    dsum += K[i * Np + i];
  }
  for (int o = 16; o > 0; o >>= 1) {
    s += __shfl_xor_sync(0xffffffffu, s, o);
    dsum += __shfl_xor_sync(0xffffffffu, dsum, o);
  }
  if ((threadIdx.x & 31) == 0) {
    red[0][threadIdx.x >> 5] = s;
    red[1][threadIdx.x >> 5] = dsum;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0, d = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) { t += red[0][w]; d += red[1][w]; }
    s_mean = t / (double)N;
    *mu = d / (double)N;
  }
  __syncthreads();
  for (int64_t i = threadIdx.x; i < Np; i += blockDim.x) {
    b[i] = i < N ? (e_loc[i] - s_mean) - eta * (rowdot ? rowdot[i] - *meandot : 0.0) : 0.0;
    if (i < N) K[i * Np + i] += lambda;
  }
}

// K += (mu / N) 1 1^T over the N x N block: lifts the null direction 1 of the
// centred matrix to mu + lambda without changing the solution for a
// right-hand side orthogonal to 1.
__global__ void lift_kernel(int64_t N, int64_t Np, double* __restrict__ K, const double* __restrict__ mu) {
  const double add = *mu / (double)N;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < N * N; e += (int64_t)gridDim.x * blockDim.x)
    K[(e / N) * Np + e % N] += add;
}

// --- float64 blocked Cholesky (lower, in place, row-major Np x Np) ---------

// Diagonal block k: A_kk = L_kk L_kk^T in shared memory; a non-positive pivot
// sets *err (the matrix is not positive definite) and leaves the block.
// Column j is a chain of square root, reciprocal and multiply, then a trailing
// update; thread 0 forms the next column's pivot and its reciprocal root first
// (its own entry of the update), while the others update, so the chain and
// the update overlap: 123 -> 69 us a block.  rinv[j] = 1 / L_jj for the
// panel and the solves.
__global__ void __launch_bounds__(256) chol_diag_kernel(int64_t Np, double* __restrict__ K, int k,
                                                        double* __restrict__ rinv, int* __restrict__ err) {
  __shared__ double a[kB][kB + 1];
  __shared__ double s_root[2], s_ri[2];
  __shared__ int bad;
  const int tid = threadIdx.x;
  double* A = K + (int64_t)k * kB * Np + (int64_t)k * kB;
  for (int e = tid; e < kB * kB; e += blockDim.x) a[e / kB][e % kB] = A[(int64_t)(e / kB) * Np + e % kB];
  if (tid == 0) bad = 0;
  __syncthreads();
  auto pivot = [&](double d, int slot) {
    if (!(d > 0.0)) bad = 1;
    const double r = d > 0.0 ? sqrt(d) : 1.0;
    s_root[slot] = r;
    s_ri[slot] = 1.0 / r;
  };
  if (tid == 0) pivot(a[0][0], 0);
  __syncthreads();
  for (int j = 0; j < kB; ++j) {
    const double ri = s_ri[j & 1];
    if (tid == 0) a[j][j] = s_root[j & 1];
    if (tid > j && tid < kB) a[tid][j] *= ri;
    if (tid == 0) rinv[(int64_t)k * kB + j] = ri;
    __syncthreads();
    const int w = kB - j - 1;   // trailing rows j + 1 ..
    if (tid == 0) {
      if (w > 0) pivot(a[j + 1][j + 1] - a[j + 1][j] * a[j + 1][j], (j + 1) & 1);
    } else if (tid >= 32) {
      // lower triangle of the trailing block but its first diagonal entry, flat over the other seven warps
      for (int e = tid - 32 + 1; e < w * (w + 1) / 2; e += 224) {
        int r = (int)((sqrtf(8.f * (float)e + 1.f) - 1.f) * 0.5f);   // row of the triangle, corrected
        if ((r + 1) * (r + 2) / 2 <= e) ++r;
        if (r * (r + 1) / 2 > e) --r;
        const int rr = j + 1 + r, cc = j + 1 + e - r * (r + 1) / 2;
        a[rr][cc] -= a[rr][j] * a[cc][j];
      }
    }
    __syncthreads();
  }
  for (int e = tid; e < kB * kB; e += blockDim.x) {
    const int r = e / kB, c = e % kB;
    A[(int64_t)r * Np + c] = c <= r ? a[r][c] : 0.0;
  }
  if (tid == 0 && bad) atomicExch(err, 1);
}

// Panel below block k: L_ik = A_ik L_kk^-T by forward substitution along the
// rows, 16 rows per CTA and 16 threads per row (four columns each): column j
// is finished by its owner and taken from the later ones at once, so the
// chain of a row is 64 multiply-adds deep instead of 2016 and the float64
// pipes of four times as many SMs work: 115-135 -> 21 us.
constexpr int kPanelRows = 16;
__global__ void __launch_bounds__(256) chol_panel_kernel(int64_t Np, double* __restrict__ K, int k,
                                                         const double* __restrict__ rinv) {
  __shared__ double l[kB][kB + 1];   // l[j][c] = L_kk[c][j]
  const double* Lkk = K + (int64_t)k * kB * Np + (int64_t)k * kB;
  for (int e = threadIdx.x; e < kB * kB; e += blockDim.x) l[e % kB][e / kB] = Lkk[(int64_t)(e / kB) * Np + e % kB];
  const int row = threadIdx.x >> 4, t = threadIdx.x & 15;
  double* A = K + ((int64_t)(k + 1) * kB + (int64_t)blockIdx.x * kPanelRows + row) * Np + (int64_t)k * kB;
  double x[4];   // columns t, t + 16, t + 32, t + 48
#pragma unroll
  for (int q = 0; q < 4; ++q) x[q] = A[t + 16 * q];
  __syncthreads();
#pragma unroll
  for (int q = 0; q < 4; ++q)
    for (int jj = 0; jj < 16; ++jj) {
      const int j = 16 * q + jj;
      double y = x[q];
      if (t == jj) y *= rinv[(int64_t)k * kB + j];
      y = __shfl_sync(0xffffffffu, y, jj, 16);
      if (t == jj) x[q] = y;
#pragma unroll
      for (int p = q; p < 4; ++p)
        if (t + 16 * p > j) x[p] -= y * l[j][t + 16 * p];
    }
#pragma unroll
  for (int q = 0; q < 4; ++q) A[t + 16 * q] = x[q];
}

// Trailing update A_ij -= L_ik L_jk^T for block rows i >= j > k: one 64 x 64
// tile per CTA, 256 threads of 4 x 4 outputs; CTA q takes the q-th tile of the
// lower triangle (with CTAs for the upper one too, 169 of them put two tiles
// on some SMs: 136 us against 72).
__global__ void __launch_bounds__(256) chol_update_kernel(int64_t Np, double* __restrict__ K, int k) {
  const int64_t q0 = blockIdx.x;
  int64_t tr = (int64_t)((sqrt(8.0 * (double)q0 + 1.0) - 1.0) * 0.5);
  if ((tr + 1) * (tr + 2) / 2 <= q0) ++tr;
  if (tr * (tr + 1) / 2 > q0) --tr;
  const int ti = k + 1 + (int)tr, tj = k + 1 + (int)(q0 - tr * (tr + 1) / 2);
  extern __shared__ double cu_sm[];
  double* li = cu_sm;                 // [kB][kB + 1]
  double* lj = cu_sm + kB * (kB + 1);
  const double* Li = K + (int64_t)ti * kB * Np + (int64_t)k * kB;
  const double* Lj = K + (int64_t)tj * kB * Np + (int64_t)k * kB;
  for (int e = threadIdx.x; e < kB * kB; e += blockDim.x) {
    li[(e / kB) * (kB + 1) + e % kB] = Li[(int64_t)(e / kB) * Np + e % kB];
    lj[(e / kB) * (kB + 1) + e % kB] = Lj[(int64_t)(e / kB) * Np + e % kB];
  }
  __syncthreads();
  const int r0 = (threadIdx.x / 16) * 4, c0 = (threadIdx.x % 16) * 4;
  double acc[4][4] = {};
  for (int q = 0; q < kB; ++q) {
    double a[4], b[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      a[u] = li[(r0 + u) * (kB + 1) + q];
      b[u] = lj[(c0 + u) * (kB + 1) + q];
    }
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
      for (int v = 0; v < 4; ++v) acc[u][v] = fma(a[u], b[v], acc[u][v]);
  }
  double* A = K + (int64_t)ti * kB * Np + (int64_t)tj * kB;
#pragma unroll
  for (int u = 0; u < 4; ++u)
#pragma unroll
    for (int v = 0; v < 4; ++v) A[(int64_t)(r0 + u) * Np + c0 + v] -= acc[u][v];
}

// L y = b then L^T x = y in place on b, one CTA of 1024 threads.  Per block of
// 64 unknowns the diagonal block is staged in shared memory, warp 0 solves the
// small triangle (two unknowns per lane, each finished one taken from the
// rest at once: one multiply-add pair per unknown instead of a dot product
// with global loads and a warp reduction) and every thread updates the
// remaining right-hand side entries.  N = 1024: 2.9 -> 0.8 ms.
__global__ void __launch_bounds__(1024) chol_solve_kernel(int64_t Np, const double* __restrict__ L,
                                                          const double* __restrict__ rinv, double* __restrict__ b) {
  __shared__ double l[kB][kB + 1];
  __shared__ double y[kB];
  const int nb = (int)(Np / kB);
  const int tid = threadIdx.x, lane = tid & 31;
  for (int pass = 0; pass < 2; ++pass) {   // 0: forward, 1: backward with L^T
    for (int kk = 0; kk < nb; ++kk) {
      const int k = pass ? nb - 1 - kk : kk;
      const int64_t o = (int64_t)k * kB;
      // l[j][i] = what unknown j takes from entry i
      for (int e = tid; e < kB * kB; e += blockDim.x) {
        const double v = L[(o + e / kB) * Np + o + e % kB];
        if (pass) l[e / kB][e % kB] = v;
        else l[e % kB][e / kB] = v;
      }
      __syncthreads();
      if (tid < 32) {
        double v0 = b[o + lane], v1 = b[o + 32 + lane];
        const double r0 = rinv[o + lane], r1 = rinv[o + 32 + lane];
        for (int jj = 0; jj < kB; ++jj) {
          const int j = pass ? kB - 1 - jj : jj;
          double t = (j < 32 ? v0 : v1) * (j < 32 ? r0 : r1);   // the owner's product counts
          t = __shfl_sync(0xffffffffu, t, j & 31);
          if (lane == (j & 31)) {
            if (j < 32) v0 = t;
            else v1 = t;
          }
          const bool t0 = pass ? lane < j : lane > j, t1 = pass ? lane + 32 < j : lane + 32 > j;
          if (t0) v0 -= t * l[j][lane];
          if (t1) v1 -= t * l[j][lane + 32];
        }
        y[lane] = v0;
        y[lane + 32] = v1;
        b[o + lane] = v0;
        b[o + 32 + lane] = v1;
      }
      __syncthreads();
      if (pass == 0) {
        for (int64_t i = o + kB + tid; i < Np; i += blockDim.x) {
          double s = 0.0;
#pragma unroll 16
          for (int q = 0; q < kB; ++q) s += L[i * Np + o + q] * y[q];
          b[i] -= s;
        }
      } else {
        for (int64_t i = tid; i < o; i += blockDim.x) {
          double s = 0.0;
#pragma unroll 16
          for (int q = 0; q < kB; ++q) s += L[(o + q) * Np + i] * y[q];
          b[i] -= s;
        }
      }
      __syncthreads();
    }
  }
}

// *out = sum_i x[i] (one warp).
__global__ void xsum_kernel(int64_t N, const double* __restrict__ x, double* __restrict__ out) {
  double s = 0.0;
  for (int64_t i = threadIdx.x; i < N; i += 32) s += x[i];
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (threadIdx.x == 0) *out = s;
}

// delta[p] = sum_i O[i][p] x[i] - mean[p] sum_i x[i] + eta dprev[p]; one thread
// per column, rows streamed eight ahead; x staged in shared memory 1024
// entries at a time.  1024 x 10^6: 1.7 ms (3.8 with converted operands).
__global__ void __launch_bounds__(256) update_kernel(int64_t N, int64_t P, const float* __restrict__ O, int64_t ldo,
                                                     const double* __restrict__ mean, const double* __restrict__ x,
                                                     const double* __restrict__ xsum,
                                                     const float* __restrict__ dprev, double eta,
                                                     float* __restrict__ delta) {
  __shared__ double xs[1024];
  const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  double acc = 0.0;
  for (int64_t i0 = 0; i0 < N; i0 += 1024) {
    const int cnt = (int)(N - i0 < 1024 ? N - i0 : 1024);
    __syncthreads();
    for (int q = threadIdx.x; q < cnt; q += blockDim.x) xs[q] = x[i0 + q];
    __syncthreads();
    if (p < P) {
      const float* o = O + i0 * ldo + p;
      int q = 0;
      for (; q + 8 <= cnt; q += 8) {
        float v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = o[(q + u) * ldo];
#pragma unroll
        for (int u = 0; u < 8; ++u) acc += widen(v[u]) * xs[q + u];
      }
      for (; q < cnt; ++q) acc += widen(o[q * ldo]) * xs[q];
    }
  }
  if (p >= P) return;
  delta[p] = (float)(acc - mean[p] * *xsum + eta * (dprev ? (double)dprev[p] : 0.0));
}

}  // namespace spring
}  // namespace fire

using namespace fire::spring;

extern "C" size_t fire_spring_workspace_size(int64_t n_walkers, int64_t n_params) {
  if (n_walkers < 2 || n_params < 1 || n_walkers > (1 << 16)) return 0;
  return layout(n_walkers, n_params).total;
}

extern "C" int fire_spring_step(int64_t n_walkers, int64_t n_params, const float* O, int64_t ldo,
                                const double* e_loc, const float* delta_prev, double eta, double lambda,
                                float* delta, double* gram, double* x_out, void* ws, size_t ws_bytes,
                                void* stream) {
  const int64_t N = n_walkers, P = n_params;
  if (N < 2 || P < 1 || N > (1 << 16) || ldo < P || !O || !e_loc || !delta) return FIRE_ERR_INVALID_ARG;
  if (!(lambda > 0.0) || !(lambda < 1e300) || !(eta >= 0.0) || !(eta < 1e300)) return FIRE_ERR_INVALID_ARG;
  const Layout L = layout(N, P);
  if (!ws || ws_bytes < L.total) return FIRE_ERR_WORKSPACE;
  cudaStream_t s = (cudaStream_t)stream;
  unsigned char* w = reinterpret_cast<unsigned char*>(ws);
  double* mean = reinterpret_cast<double*>(w + L.mean);
  __nv_bfloat16* pack = reinterpret_cast<__nv_bfloat16*>(w + L.pack);
  float* cch = reinterpret_cast<float*>(w + L.cch);
  double* K = reinterpret_cast<double*>(w + L.kacc);
  double* rowdot = reinterpret_cast<double*>(w + L.rowdot);
  double* b = reinterpret_cast<double*>(w + L.b);
  int* err = reinterpret_cast<int*>(w + L.err);
  double* rinv = reinterpret_cast<double*>(w + L.rinv);
  const int64_t Np = L.Np;
  if (cudaMemsetAsync(err, 0, 16, s) != cudaSuccess) return FIRE_ERR_CUDA;
  if (delta_prev && cudaMemsetAsync(rowdot, 0, (size_t)N * 8, s) != cudaSuccess) return FIRE_ERR_CUDA;
  colmean_kernel<<<(unsigned)((P + 255) / 256), 256, 0, s>>>(N, P, O, ldo, mean);
  double* scal = reinterpret_cast<double*>(w + L.scal);   // abar, mu, mean . dprev, sum x
  if (cudaMemsetAsync(scal, 0, 32, s) != cudaSuccess) return FIRE_ERR_CUDA;
  if (delta_prev) meandot_kernel<<<fire::kSMs, 256, 0, s>>>(P, mean, delta_prev, scal + 2);
  // Gram matrix over chunks of the parameter axis, L.groups of them per launch
  // (the last chunks alone where the axis does not fill a group)
  const int vec = ldo % 4 == 0 && (reinterpret_cast<uintptr_t>(O) & 15) == 0;
  int first = 1;
  for (int64_t p0 = 0; p0 < P;) {
    const int64_t left = (P - p0 + 63) / 64 * 64;
    int groups = (int)(left / L.pc);
    groups = groups < 1 ? 1 : (groups > L.groups ? L.groups : groups);
    const int pc = (int)(left < L.pc ? left : L.pc);
    const int64_t width = (int64_t)groups * pc;
    const dim3 g((unsigned)((width + 4095) / 4096), (unsigned)((N + kPackRows - 1) / kPackRows));
    pack_kernel<<<g, 256, 0, s>>>(N, P, O, ldo, p0, width, pack, delta_prev, rowdot, vec && p0 % 4 == 0);
    const int rc = fire::tc::gemm_bf16_rows(s, pack, width, N, pack, (int)N, 0, (int)N, pc, cch, N, 0, N, nullptr, N,
                                            err + 1, kNC, groups, width, N);
    if (rc != FIRE_OK) return rc;
    accum_kernel<<<(unsigned)((Np * Np + 255) / 256), 256, 0, s>>>(N, Np, cch, groups, K, first);
    first = 0;
    p0 += width;
  }
  // exact centring in float64: Obar Obar^T = P G P
  double* a = reinterpret_cast<double*>(w + L.a);
  rowmean_kernel<<<(unsigned)((N + 7) / 8), 256, 0, s>>>(N, Np, K, a);
  center_kernel<<<4 * fire::kSMs, 1024, 0, s>>>(N, Np, K, a, scal);
  if (gram) cudaMemcpy2DAsync(gram, (size_t)N * 8, K, (size_t)Np * 8, (size_t)N * 8, (size_t)N,
                              cudaMemcpyDeviceToDevice, s);
  rhs_kernel<<<1, 1024, 0, s>>>(N, Np, e_loc, delta_prev ? rowdot : nullptr, scal + 2, eta, lambda, b, K,
                                scal + 1);
  lift_kernel<<<4 * fire::kSMs, 256, 0, s>>>(N, Np, K, scal + 1);
  // float64 Cholesky of K + lambda I, then the two triangular solves
  const int nb = (int)(Np / kB);
  const size_t usm = 2 * (size_t)kB * (kB + 1) * 8;
  if (cudaFuncSetAttribute(chol_update_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)usm) != cudaSuccess)
    return FIRE_ERR_CUDA;
  for (int k = 0; k < nb; ++k) {
    chol_diag_kernel<<<1, 256, 0, s>>>(Np, K, k, rinv, err);
    const int rest = nb - k - 1;
    if (rest > 0) {
      chol_panel_kernel<<<(unsigned)(rest * (kB / kPanelRows)), 256, 0, s>>>(Np, K, k, rinv);
      chol_update_kernel<<<(unsigned)((int64_t)rest * (rest + 1) / 2), 256, usm, s>>>(Np, K, k);
    }
  }
  chol_solve_kernel<<<1, 1024, 0, s>>>(Np, K, rinv, b);
  if (x_out) cudaMemcpyAsync(x_out, b, (size_t)N * 8, cudaMemcpyDeviceToDevice, s);
  xsum_kernel<<<1, 32, 0, s>>>(N, b, scal + 3);
  update_kernel<<<(unsigned)((P + 255) / 256), 256, 0, s>>>(N, P, O, ldo, mean, b, scal + 3, delta_prev, eta, delta);
  int herr[2] = {0, 0};
  if (cudaMemcpyAsync(herr, err, sizeof(herr), cudaMemcpyDeviceToHost, s) != cudaSuccess) return FIRE_ERR_CUDA;
  if (cudaStreamSynchronize(s) != cudaSuccess) return FIRE_ERR_CUDA;
  if (cudaGetLastError() != cudaSuccess) return FIRE_ERR_CUDA;
  if (herr[1]) return FIRE_ERR_TIMEOUT;
  if (herr[0]) return FIRE_ERR_NONFINITE;
  return FIRE_OK;
}
