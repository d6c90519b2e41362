// Building blocks of the per-walker parameter gradient (adjoint).
#pragma once

#include "common.cuh"
#include "gemm.cuh"

namespace fire {

// The electrons of a walker in block order are two runs of rows, spin-up then
// spin-down; a per-walker sum walks both.  Row k of walker w of a matrix with
// row stride ld: base + w wld[0] + k ld for k < n0, base + off1 + w wld[1] +
// (k - n0) ld beyond.
struct SpinRows {
  int n0, n1;
  int64_t w0, w1, off1;   // rows per walker of each run, rows before run 1
  __device__ __forceinline__ int64_t row(int w, int k) const {
    return k < n0 ? w * w0 + k : off1 + w * w1 + (k - n0);
  }
};
inline SpinRows spin_rows(int wc, int n_up, int n_dn) { return {n_up, n_dn, n_up, n_dn, (int64_t)wc * n_up}; }
inline SpinRows one_spin(int ns) { return {ns, 0, ns, 0, 0}; }      // one run alone (base pointer at its first row)
inline SpinRows walker_rows() { return {1, 0, 1, 0, 0}; }           // one row per walker

// Per-walker transposed products, the outer-product sums over a walker's
// electrons that give weight gradients: for every walker w and batch q
//   C[w sc + q cb + (b / nbk) scb + a ldc + b % nbk] = sum_k X[row(w, k) ldx + q xb + a] Y[row(w, k) ldy + q yb + b],
// a < Na, b < Nb.  The rows of X and Y are the slabs of a product with the sum
// over rows, so nothing is transposed: 64 x 64 tiles, 16 rows of each operand
// ahead in registers, 8 x 8 outputs per thread in float32 (packed
// multiply-adds), 4 x 4 in float64.  Each C entry is written once.
// C26H24, 128 walkers, all weights: 10.9 -> 5.1 ms (32 x 32 tiles, one launch per
// determinant and spin and a read of C for the second spin before).
template <typename T>
struct TnArgs {
  const T *X, *Y;
  T* C;
  int64_t ldx, ldy, ldc, sc, xb, yb, cb, scb;
  SpinRows rows;
  int Na, Nb, nbk, nbatch;
  int va, vb;   // 16-byte loads of X and of Y
};

template <typename T, int TM, int TN>
__global__ void __launch_bounds__((64 / TM) * (64 / TN)) tn_kernel(TnArgs<T> g) {
  constexpr int BT = 64, BK = 16, NT = (BT / TM) * (BT / TN), VE = 16 / (int)sizeof(T);
  constexpr int PER = BK * BT / VE / NT, NCH = BT / VE;   // chunks of a slab per thread, per row
  constexpr int RM = TM / 4, RN = TN / 4;
  static_assert(PER >= 1 && NT % NCH == 0, "slab");
  __shared__ __align__(16) T xs[2][BK][BT];
  __shared__ __align__(16) T ys[2][BK][BT];
  const int w = blockIdx.z / g.nbatch, q = blockIdx.z % g.nbatch;
  const int a0 = blockIdx.x * BT, b0 = blockIdx.y * BT;
  const T* X = g.X + q * g.xb;
  const T* Y = g.Y + q * g.yb;
  const int tid = threadIdx.x;
  const int tx = tid % (BT / TN), ty = tid / (BT / TN);
  const int kr = tid / NCH, kc = (tid % NCH) * VE;   // first slab row and column of this thread's chunks
  const int K = g.rows.n0 + g.rows.n1;
  T rx[PER][VE], ry[PER][VE];
  T acc[TM][TN];
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j) acc[i][j] = T(0);
  auto chunk = [&](T (&v)[VE], const T* p, int left, int vec) {
    if (vec) {
      if (left > 0) ld_vec<T, VE>(v, p);
      else
#pragma unroll
        for (int i = 0; i < VE; ++i) v[i] = T(0);
    } else {
#pragma unroll
      for (int i = 0; i < VE; ++i) v[i] = i < left ? p[i] : T(0);
    }
  };
  auto load = [&](int k0) {
#pragma unroll
    for (int u = 0; u < PER; ++u) {
      const int k = k0 + kr + u * (NT / NCH);
      const int64_t row = g.rows.row(w, k < K ? k : 0);
      chunk(rx[u], X + row * g.ldx + a0 + kc, k < K ? g.Na - a0 - kc : 0, g.va);
      chunk(ry[u], Y + row * g.ldy + b0 + kc, k < K ? g.Nb - b0 - kc : 0, g.vb);
    }
  };
  auto store = [&](int buf) {
    struct alignas(16) Vec { T x[VE]; };
#pragma unroll
    for (int u = 0; u < PER; ++u) {
      *reinterpret_cast<Vec*>(&xs[buf][kr + u * (NT / NCH)][kc]) = *reinterpret_cast<const Vec*>(rx[u]);
      *reinterpret_cast<Vec*>(&ys[buf][kr + u * (NT / NCH)][kc]) = *reinterpret_cast<const Vec*>(ry[u]);
    }
  };
  load(0);
  store(0);
  __syncthreads();
  int buf = 0;
  for (int k0 = 0; k0 < K; k0 += BK) {
    const bool more = k0 + BK < K;
    if (more) load(k0 + BK);
#pragma unroll
    for (int kk = 0; kk < BK; ++kk) {
      T a[RM][4], b[RN][4];
#pragma unroll
      for (int p = 0; p < RM; ++p) ld_vec<T, 4>(a[p], &xs[buf][kk][p * (BT / RM) + ty * 4]);
#pragma unroll
      for (int p = 0; p < RN; ++p) ld_vec<T, 4>(b[p], &ys[buf][kk][p * (BT / RN) + tx * 4]);
#pragma unroll
      for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN; j += 2)
          fma_pair(acc[i][j], acc[i][j + 1], a[i / 4][i % 4], b[j / 4][j % 4], b[j / 4][j % 4 + 1]);
    }
    if (more) {
      store(buf ^ 1);
      __syncthreads();
      buf ^= 1;
    }
  }
  T* C = g.C + (int64_t)w * g.sc + q * g.cb;
#pragma unroll
  for (int i = 0; i < TM; ++i) {
    const int a = a0 + (i / 4) * (BT / RM) + ty * 4 + i % 4;
    if (a >= g.Na) continue;
#pragma unroll
    for (int j = 0; j < TN; ++j) {
      const int b = b0 + (j / 4) * (BT / RN) + tx * 4 + j % 4;
      if (b < g.Nb) C[(int64_t)(b / g.nbk) * g.scb + (int64_t)a * g.ldc + b % g.nbk] = acc[i][j];
    }
  }
}

template <typename T>
inline void tn_batched(cudaStream_t s, int W, int Na, int Nb, const SpinRows& rows, const T* X, int64_t ldx,
                       const T* Y, int64_t ldy, T* C, int64_t ldc, int64_t sc, int nbatch = 1, int64_t xb = 0,
                       int64_t yb = 0, int64_t cb = 0, int nbk = 0, int64_t scb = 0) {
  if (W <= 0 || Na <= 0 || Nb <= 0 || rows.n0 + rows.n1 <= 0) return;
  constexpr int VE = 16 / (int)sizeof(T);
  auto al = [](const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; };
  TnArgs<T> g{X, Y, C, ldx, ldy, ldc, sc, xb, yb, cb, scb, rows, Na, Nb, nbk > 0 ? nbk : Nb, nbatch, 0, 0};
  g.va = al(X) && ldx % VE == 0 && xb % VE == 0 && Na % VE == 0;
  g.vb = al(Y) && ldy % VE == 0 && yb % VE == 0 && Nb % VE == 0;
  // grid.z is limited to 65535
  const int wz = 65535 / nbatch;
  for (int w0 = 0; w0 < W; w0 += wz) {
    const int nw = W - w0 < wz ? W - w0 : wz;
    TnArgs<T> h = g;
    h.X += (int64_t)w0 * rows.w0 * ldx;
    h.Y += (int64_t)w0 * rows.w0 * ldy;
    h.rows.off1 += (int64_t)w0 * (rows.w1 - rows.w0);
    h.C += (int64_t)w0 * sc;
    const dim3 grid((unsigned)((Na + 63) / 64), (unsigned)((Nb + 63) / 64), (unsigned)(nw * nbatch));
    if constexpr (sizeof(T) == 4) tn_kernel<T, 8, 8><<<grid, 64, 0, s>>>(h);
    else tn_kernel<T, 4, 4><<<grid, 256, 0, s>>>(h);
  }
}

// C[w sc + b] = sum_k Y[row(w, k) ldy + b]  (bias gradients).
template <typename T>
__global__ void colsum_batched_kernel(int Nb, SpinRows rows, const T* __restrict__ Y, int64_t ldy, T* __restrict__ C,
                                      int64_t sc, int w0) {
  const int w = w0 + blockIdx.y;
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= Nb) return;
  T acc = T(0);
  const int K = rows.n0 + rows.n1;
#pragma unroll 8
  for (int k = 0; k < K; ++k) acc += Y[rows.row(w, k) * ldy + b];
  C[(int64_t)w * sc + b] = acc;
}

template <typename T>
inline void colsum_batched(cudaStream_t s, int W, int Nb, const SpinRows& rows, const T* Y, int64_t ldy, T* C,
                           int64_t sc) {
  if (W <= 0 || Nb <= 0 || rows.n0 + rows.n1 <= 0) return;
  for (int w0 = 0; w0 < W; w0 += 65535) {
    const int nw = W - w0 < 65535 ? W - w0 : 65535;
    const dim3 grid((unsigned)((Nb + 127) / 128), (unsigned)nw);
    colsum_batched_kernel<T><<<grid, 128, 0, s>>>(Nb, rows, Y, ldy, C, sc, w0);
  }
}

// Elementwise helpers over dense [rows][ncol] matrices.
// mode 0: out = d * SiLU'(z + b)           (back through y = SiLU(z + b))
// mode 1: out = d * SiLU(z + b)            (used by products)
template <typename T, typename W>
__global__ void silu_bwd_kernel(int64_t rows, int ncol, const T* __restrict__ D, int64_t ldd,
                                const T* __restrict__ Z, int64_t ldz, const W* bias, T* __restrict__ O,
                                int64_t ldo) {
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= rows * ncol) return;
  const int64_t r = e / ncol;
  const int c = (int)(e % ncol);
  T f, f1, f2;
  silu3<T>(Z[r * ldz + c] + (bias ? T(bias[c]) : T(0)), f, f1, f2);
  O[r * ldo + c] = D[r * ldd + c] * f1;
}

}  // namespace fire
