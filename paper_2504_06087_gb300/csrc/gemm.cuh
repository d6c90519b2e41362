// SIMT matrix product C = A * op(B) over row ranges of the forward-Laplacian
// tensors, for the float32 and float64 forms.
//
// A is row-major [M][K] (lda), B row-major [K][N] (ldb) or, with TB,
// [N][K]; C row-major [M][N] (ldc).  The row range may live on the device
// (m_range = {begin, end}), so a launch can be enqueued before the ragged row
// counts are known; tiles past the end exit at once.  grid.z batches
// independent products with element strides sA, sB, sC.  Products of one A
// with several B whose results lie side by side are one product whose
// columns come from B in blocks of nb (element stride sB between blocks).
//
// Every output is one chain of fused multiply-adds over k in ascending order,
// whatever the tile, so the result does not depend on the tile chosen.
#pragma once

#include "common.cuh"
#include "plan.h"

namespace fire {

template <typename T>
struct GemmArgs {
  const T* A;
  const T* B;
  T* C;
  int64_t lda, ldb, ldc;
  int64_t sA, sB, sC;
  int64_t m_begin, m_end;        // used when m_range == nullptr
  const int64_t* m_range;        // device {begin, end} or nullptr
  int N, K;
  int nb;                        // columns per block of B
  int accumulate;
  int va, vb, vc;                // 16-byte loads of A and of B, 16-byte stores of C
  const T* bias;                 // ACT: C = (R ? R : 0) + SiLU(product + bias), R with row stride ldr
  const T* R;
  int64_t ldr;
  int one;                       // ACT: R is added to x * logistic(x) in one rounding or in two
};

// One BM x BN tile per CTA; a thread owns TM x TN outputs as groups of at most
// four consecutive rows and columns, so a warp's shared loads are 128-bit
// broadcasts without bank conflicts.  The next BK-deep slab is in registers
// while the current one is multiplied.
template <typename T, int BM, int BN, int BK, int TM, int TN, bool TB, bool ACT = false>
__global__ void __launch_bounds__((BM / TM) * (BN / TN))
gemm_kernel(GemmArgs<T> g) {
  constexpr int NT = (BM / TM) * (BN / TN);
  constexpr int VE = 16 / (int)sizeof(T);          // elements of a 16-byte load
  constexpr int GM = TM < 4 ? TM : 4, GN = TN < 4 ? TN : 4;
  constexpr int RM = TM / GM, RN = TN / GN;        // row and column groups of a thread
  constexpr int NX = BN / TN;                      // threads along the columns
  constexpr int LX = NX < 8 ? NX : 8, LY = 32 / LX;   // warp: LY x LX threads
  static_assert(NT % 32 == 0 && (BM / TM) % LY == 0 && NX % LX == 0, "warp layout");
  constexpr int AC = BM * BK / VE / NT, KC = BK / VE;
  static_assert(AC >= 1 && NT % KC == 0, "A slab");
  constexpr int BC = BK * BN / VE / NT, NC = BN / VE;
  static_assert(BC >= 1 && (TB ? NT % KC == 0 : NT % NC == 0 || NC % NT == 0), "B slab");
  constexpr int PAD = 4;
  __shared__ __align__(16) T As[2][BK][BM + PAD];
  __shared__ __align__(16) T Bs[2][BK][BN + PAD];
  int64_t mb = g.m_begin, me = g.m_end;
  if (g.m_range) { mb = g.m_range[0]; me = g.m_range[1]; }
  const int64_t m0 = mb + (int64_t)blockIdx.x * BM;
  if (m0 >= me) return;
  const int n0 = blockIdx.y * BN;
  const T* A = g.A + g.sA * blockIdx.z;
  const T* B = g.B + g.sB * blockIdx.z;
  T* C = g.C + g.sC * blockIdx.z;
  const int tid = threadIdx.x;
  const int wid = tid >> 5, lane = tid & 31;
  const int tx = (wid % (NX / LX)) * LX + lane % LX, ty = (wid / (NX / LX)) * LY + lane / LX;
  // A slab: thread loads VE elements of row ar + q (NT / KC) at column ak
  const int ar = tid / KC, ak = (tid % KC) * VE;
  const T* Ap = A + (m0 + ar) * g.lda + ak;
  const int64_t mleft = me - m0 - ar;
  // B slab: as rows k (VE columns) or, with TB, as rows n (VE k's)
  const T* Bp[BC];
  int bk[BC], bn[BC];
  int bl[BC];   // columns left from this one on
#pragma unroll
  for (int q = 0; q < BC; ++q) {
    const int e = tid + q * NT;
    bk[q] = TB ? (e % KC) * VE : e / NC;
    bn[q] = TB ? e / KC : (e % NC) * VE;
    const int gn = n0 + bn[q];
    bl[q] = g.N - gn;
    const int z = gn / g.nb, c = gn - z * g.nb;
    Bp[q] = B + (int64_t)z * g.sB + (TB ? (int64_t)c * g.ldb + bk[q] : (int64_t)bk[q] * g.ldb + c);
  }
  T ra[AC][VE], rb[BC][VE];
  T acc[TM][TN];
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j) acc[i][j] = T(0);

  auto load = [&](int k0) {
#pragma unroll
    for (int q = 0; q < AC; ++q) {
      const T* p = Ap + (int64_t)q * (NT / KC) * g.lda + k0;
      const bool row = q * (NT / KC) < mleft;
      if (g.va) {
        if (row && k0 + ak < g.K) ld_vec<T, VE>(ra[q], p);
        else
#pragma unroll
          for (int i = 0; i < VE; ++i) ra[q][i] = T(0);
      } else {
#pragma unroll
        for (int i = 0; i < VE; ++i) ra[q][i] = (row && k0 + ak + i < g.K) ? p[i] : T(0);
      }
    }
#pragma unroll
    for (int q = 0; q < BC; ++q) {
      const T* p = Bp[q] + (TB ? (int64_t)k0 : (int64_t)k0 * g.ldb);
      const bool in = TB ? bl[q] > 0 : k0 + bk[q] < g.K;
      const int left = TB ? g.K - k0 - bk[q] : bl[q];   // elements along the load
      if (g.vb) {
        if (in && left > 0) ld_vec<T, VE>(rb[q], p);
        else
#pragma unroll
          for (int i = 0; i < VE; ++i) rb[q][i] = T(0);
      } else if (TB) {
#pragma unroll
        for (int i = 0; i < VE; ++i) rb[q][i] = (in && i < left) ? p[i] : T(0);
      } else {
        // columns may cross into the next block of B
        int c = (n0 + bn[q]) % g.nb;
#pragma unroll
        for (int i = 0; i < VE; ++i) {
          rb[q][i] = (in && i < left) ? *p : T(0);
          ++p;
          if (++c == g.nb) { c = 0; p += g.sB - g.nb; }
        }
      }
    }
  };
  auto store = [&](int buf) {
#pragma unroll
    for (int q = 0; q < AC; ++q)
#pragma unroll
      for (int i = 0; i < VE; ++i) As[buf][ak + i][ar + q * (NT / KC)] = ra[q][i];
#pragma unroll
    for (int q = 0; q < BC; ++q) {
      if (TB) {
#pragma unroll
        for (int i = 0; i < VE; ++i) Bs[buf][bk[q] + i][bn[q]] = rb[q][i];
      } else {
        struct alignas(16) Vec { T x[VE]; } u;
#pragma unroll
        for (int i = 0; i < VE; ++i) u.x[i] = rb[q][i];
        *reinterpret_cast<Vec*>(&Bs[buf][bk[q]][bn[q]]) = u;
      }
    }
  };

  load(0);
  store(0);
  __syncthreads();
  int buf = 0;
  for (int k0 = 0; k0 < g.K; k0 += BK) {
    const bool more = (k0 + BK) < g.K;
    if (more) load(k0 + BK);
#pragma unroll
    for (int kk = 0; kk < BK; ++kk) {
      T a[RM][GM], b[RN][GN];
#pragma unroll
      for (int p = 0; p < RM; ++p) ld_vec<T, GM>(a[p], &As[buf][kk][p * (BM / RM) + ty * GM]);
#pragma unroll
      for (int p = 0; p < RN; ++p) ld_vec<T, GN>(b[p], &Bs[buf][kk][p * (BN / RN) + tx * GN]);
#pragma unroll
      for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN; j += 2)
          fma_pair(acc[i][j], acc[i][j + 1], a[i / GM][i % GM], b[j / GN][j % GN], b[j / GN][j % GN + 1]);
    }
    if (more) {
      store(buf ^ 1);
      __syncthreads();
      buf ^= 1;
    }
  }
#pragma unroll
  for (int i = 0; i < TM; ++i) {
    const int64_t gm = m0 + (i / GM) * (BM / RM) + ty * GM + i % GM;
    if (gm >= me) continue;
    if constexpr (ACT) {
#pragma unroll
      for (int p = 0; p < RN; ++p) {
        const int gn = n0 + p * (BN / RN) + tx * GN;
        T* o = C + gm * g.ldc + gn;
        const T* rr = g.R ? g.R + gm * g.ldr + gn : nullptr;
        const bool whole = g.vc && gn + GN <= g.N;   // (R is as aligned as C then)
        T y[GN];
        if (whole && rr) ld_vec<T, GN>(y, rr);
        else
#pragma unroll
          for (int j = 0; j < GN; ++j) y[j] = rr && gn + j < g.N ? rr[j] : T(0);
#pragma unroll
        for (int j = 0; j < GN; ++j) {
          const T x = acc[i][p * GN + j] + (gn + j < g.N ? g.bias[gn + j] : T(0));
          const T sg = T(1) / (T(1) + dexp<T>(-x));
          const T f = mul_rn(x, sg);
          y[j] = !rr ? f : g.one ? fma(x, sg, y[j]) : add_rn(y[j], f);
        }
        if (whole) {
          constexpr int W = VE < GN ? VE : GN;
          struct alignas(W * sizeof(T)) Vec { T x[W]; };
#pragma unroll
          for (int q = 0; q < GN; q += W) {
            Vec u;
#pragma unroll
            for (int j = 0; j < W; ++j) u.x[j] = y[q + j];
            *reinterpret_cast<Vec*>(o + q) = u;
          }
        } else {
#pragma unroll
          for (int j = 0; j < GN; ++j)
            if (gn + j < g.N) o[j] = y[j];
        }
      }
      continue;
    }
#pragma unroll
    for (int p = 0; p < RN; ++p) {
      const int gn = n0 + p * (BN / RN) + tx * GN;
      T* o = C + gm * g.ldc + gn;
      if (g.vc && gn + GN <= g.N) {
        constexpr int W = VE < GN ? VE : GN;
        struct alignas(W * sizeof(T)) Vec { T x[W]; };
#pragma unroll
        for (int q = 0; q < GN; q += W) {
          Vec u;
          if (g.accumulate) {
            u = *reinterpret_cast<const Vec*>(o + q);
#pragma unroll
            for (int j = 0; j < W; ++j) u.x[j] = u.x[j] + acc[i][p * GN + q + j];
          } else {
#pragma unroll
            for (int j = 0; j < W; ++j) u.x[j] = acc[i][p * GN + q + j];
          }
          *reinterpret_cast<Vec*>(o + q) = u;
        }
      } else {
#pragma unroll
        for (int j = 0; j < GN; ++j)
          if (gn + j < g.N) o[j] = g.accumulate ? (o[j] + acc[i][p * GN + j]) : acc[i][p * GN + j];
      }
    }
  }
}

template <typename T, int BM, int BN, int BK, int TM, int TN>
inline void gemm_launch(cudaStream_t s, const GemmArgs<T>& g, bool tb, int64_t m_cap, int batch) {
  const dim3 grid((unsigned)((m_cap + BM - 1) / BM), (unsigned)((g.N + BN - 1) / BN), batch);
  constexpr int NT = (BM / TM) * (BN / TN);
  if (g.bias) gemm_kernel<T, BM, BN, BK, TM, TN, false, true><<<grid, NT, 0, s>>>(g);
  else if (tb) gemm_kernel<T, BM, BN, BK, TM, TN, true><<<grid, NT, 0, s>>>(g);
  else gemm_kernel<T, BM, BN, BK, TM, TN, false><<<grid, NT, 0, s>>>(g);
}

// Host launcher.  m_cap bounds end - begin (grid sizing).  With bias (plain
// products only) the epilogue is a SiLU layer, C = (R ? R : 0) + SiLU(A B + bias):
// a move's products are so short that the layer's own launch took a third of
// their time.  C must not be A or R's rows of another tile (R may be A).  With
// `one` the residual sum is a single multiply-add, as in mcmc_act_kernel;
// without it product and sum are rounded one by one, as in fl_act4_kernel: a
// row comes out the same whichever kernel took its layer.
//
// float32: tiles of 64 x 64 (64 threads, 8 x 8 outputs each, 168 registers)
// reach 55-59 of the 77 TFLOP/s of plain multiply-adds once a few tiles per SM
// exist: 400 k rows, K = N = 256 in 885 us, and N = 180 in 672 us (2200 and
// 2064 us with one 128 x 128 tile of scalar loads and unpacked multiply-adds).
// Larger tiles measured no faster (128 x 64: 905 us, 128 x 128 with 16 x 8
// outputs: 1000 us).  32 x 32 tiles keep more SMs busy where there are few
// outputs and a product is one chain of K dependent steps (128 x 256, K = 256:
// 47 -> 9 us); 128 x 16 tiles avoid computing padding columns
// (400 k rows, N = 16: 695 -> 138 us).
// float64: every tile shape runs at the float64 pipe's rate (1.2 TFLOP/s), so
// the smallest one, which pads least and spreads furthest, is the only one
// (81920 rows, K = 64, N = 10: 578 -> 142 us; 256 rows: 70 -> 9 us).
template <typename T>
inline void gemm(cudaStream_t s, const T* A, int64_t lda, const T* B, int64_t ldb, bool transB,
                 T* C, int64_t ldc, int64_t m_begin, int64_t m_end, const int64_t* m_range,
                 int64_t m_cap, int N, int K, int batch = 1, int64_t sA = 0, int64_t sB = 0,
                 int64_t sC = 0, bool accumulate = false, const T* bias = nullptr, const T* R = nullptr,
                 int64_t ldr = 0, int one = 0) {
  if (m_cap <= 0 || N <= 0 || K <= 0 || batch <= 0) return;
  GemmArgs<T> g{A, B, C, lda, ldb, ldc, sA, sB, sC, m_begin, m_end, m_range, N, K, N, accumulate ? 1 : 0, 0, 0, 0,
                bias, R, ldr, one};
  if (bias && (transB || batch != 1 || accumulate)) return;   // the fused layer is a plain product
  if (batch > 1 && sA == 0 && sC == N) {   // side by side: one product of batch * N columns
    g.N = N * batch;
    batch = 1;
  }
  constexpr int VE = 16 / (int)sizeof(T);
  auto al = [](const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; };
  g.va = al(A) && lda % VE == 0 && K % VE == 0 && sA % VE == 0;
  g.vb = al(B) && ldb % VE == 0 && sB % VE == 0 && (transB ? K : N) % VE == 0;
  g.vc = al(C) && ldc % VE == 0 && sC % VE == 0 && (!R || (al(R) && ldr % VE == 0));
  if constexpr (sizeof(T) == 8) {
    gemm_launch<T, 16, 16, 32, 1, 2>(s, g, transB, m_cap, batch);
  } else {
    // the tile of least estimated time, in outputs of the 64 x 64 tile's rate:
    // all tiles over the SMs, but no less than one tile alone takes (a lone
    // 64-thread tile is a chain of loads and barriers: 3700 rows, N = K = 128,
    // 11 us against 8 with 32 x 32 tiles)
    struct Tile { int bm, bn; float eff, lone; };
    constexpr Tile t[] = {{64, 64, 1.f, 18500.f}, {32, 32, 0.38f, 11700.f}, {128, 16, 0.42f, 16000.f}};
    int best = 0;
    float cost = 3.4e38f;
    for (int q = 0; q < 3; ++q) {
      const int64_t tiles = ((m_cap + t[q].bm - 1) / t[q].bm) * ((g.N + t[q].bn - 1) / t[q].bn) * batch;
      float c = (float)tiles * t[q].bm * t[q].bn / ((float)kSMs * t[q].eff);
      if (c < t[q].lone) c = t[q].lone + 1e-3f * c;
      if (c < cost) { cost = c; best = q; }
    }
    if (best == 0) gemm_launch<T, 64, 64, 16, 8, 8>(s, g, transB, m_cap, batch);
    else if (best == 1) gemm_launch<T, 32, 32, 32, 2, 4>(s, g, transB, m_cap, batch);
    else gemm_launch<T, 128, 16, 32, 4, 4>(s, g, transB, m_cap, batch);
  }
}

}  // namespace fire
