// Two-electron swap ratios for the S+ operator (Supplementary "Low-rank
// updates in S+ operator": R_beta = 1 - sum_alpha Psi(pi_{alpha beta} r)/Psi(r),
// pi swapping the positions of the spin-up electron alpha and the spin-down
// electron beta; Methods "Low-rank wave function updates": only the
// embeddings within c of either electron change).
//
// A swap moves alpha to r_beta and beta to r_alpha, each keeping its spin.
// h^0 and its message projections depend on the position alone, so the new
// h^0 of alpha is the cached h^0 of beta and vice versa; the envelope rows
// of both are recomputed with their own spin's weights.  The update set is
// {alpha, beta} and every electron within c of r_alpha or r_beta; the
// orbital rows of the update set, the MLP-Jastrow rows and the attention
// registers are recomputed as for a single-electron move, and the
// determinant ratios come from the same |U| x |U| determinant lemma.
// (Included by pipeline.cuh after mcmc.cuh.)
#pragma once

#include <stdint.h>

#include "../../include/fire.h"

namespace fire {

// rk = r_beta (alpha's new position), rk2 = r_alpha (beta's), and the update
// set.  One warp per walker.
static __global__ void swap_propose_kernel(int n, int n_up, int a, int b, const double* __restrict__ r, double c2,
                                           int Umax, double* __restrict__ rk, double* __restrict__ rk2,
                                           int32_t* __restrict__ Ul, int32_t* __restrict__ Uc,
                                           int32_t* __restrict__ Ucu, DevStatus* st) {
  const int w = blockIdx.x;
  const int lane = threadIdx.x;
  const double* rw = r + (int64_t)w * n * 3;
  if (lane < 3) {
    rk[(int64_t)w * 3 + lane] = rw[3 * b + lane];
    rk2[(int64_t)w * 3 + lane] = rw[3 * a + lane];
  }
  // members: a, and every j within c of r_a or of r_b (b among them)
  update_set(w, lane, n, n_up, a, rw, rw + 3 * b, c2, Umax, Ul, Uc, Ucu, st, true);
}

// h^1 of every member i of U after the swap (value only).  For i = a or b
// every term changes: the neighbour list at the new position is rebuilt with
// the swapped positions and h^0 / projections (position-only) taken from the
// other electron's block.  For any other i the terms of the pairs (i, a) and
// (i, b) change: h^1_i - old (i, a) - old (i, b) + new (i, a) + new (i, b),
// the new terms at the swapped positions with the swapped projections and
// the spin channel of the pair unchanged.  CTAs 0 and 1 of a walker take a and
// b, the others 8 members each (four terms); blockDim == d; dynamic shared
// memory n ints.  256 walkers of C8H10: 500 -> 78 us a swap.
template <typename T, typename W>
__global__ void __launch_bounds__(kFilterThreads<T>) swap_msg_kernel(
    int Wn, int n, int n_up, int d, int a, int b, int Umax, const double* __restrict__ r, double cut, Params<W> p,
    const int32_t* __restrict__ Ul, const int32_t* __restrict__ Uc, const int32_t* __restrict__ Urow,
    const T* __restrict__ H0, const T* __restrict__ PQ, const T* __restrict__ H1, T* __restrict__ X,
    T* __restrict__ H1n) {
  constexpr int GM = kMsgPairs / 4;   // members of a CTA: four terms each
  __shared__ MsgBatch<T> B;
  extern __shared__ int sw_nbr[];
  __shared__ int s_cnt[2], s_u;
  const int groups = 2 + (Umax + GM - 1) / GM;
  const int w = blockIdx.x / groups, g = blockIdx.x % groups;
  const int uc = Uc[w], u0 = (g - 2) * GM;
  if (g > 1 && u0 >= uc) return;
  const int c = threadIdx.x;
  const int64_t ld4 = 4 * (int64_t)d;
  const double* rw = r + (int64_t)w * n * 3;
  const int32_t* U = Ul + (int64_t)w * Umax;
  const int32_t* rows = Urow + (int64_t)w * Umax;
  const MsgWeights<T, W> mw(p, d, c);
  // positions and position-dependent blocks after the swap
  auto src = [&](int j) { return j == a ? b : (j == b ? a : j); };
  auto qrow = [&](int j) { return PQ + (int64_t)block_index(w, src(j), Wn, n, n_up) * ld4; };
  if (g < 2) {
    const int i = g == 0 ? a : b;
    auto pos = [&](int j, int t) -> double { return rw[3 * src(j) + t]; };
    if (c == 0) s_u = -1;
    __syncthreads();
    if (c < 32) warp_neighbours(n, n_up, i, cut, pos, sw_nbr, s_cnt);
    for (int u = c; u < uc; u += blockDim.x)
      if (U[u] == i) s_u = u;
    __syncthreads();
    if (s_u < 0) return;   // the update set was cut short (reported as an overflow)
    const int64_t bi = block_index(w, src(i), Wn, n, n_up);
    const T acc = msg_of_moved<T, W>(mw, B, p, i, d, cut, pos, qrow, PQ + bi * ld4, sw_nbr, s_cnt, H0[bi * d + c]);
    const int64_t row = rows[s_u];
    X[row * d + c] = acc;
    H1n[row * d + c] = acc;
    return;
  }
  const int nm = min(GM, uc - u0);
  if (c < 4 * nm) {   // pairs 4 m ..: (i, a) old, new, (i, b) old, new
    const int i = U[u0 + c / 4], kk = (c & 2) ? b : a;
    const int sk = (c & 1) ? src(kk) : kk;   // the position and blocks the pair uses
    const double dd[3] = {rw[3 * i] - rw[3 * sk], rw[3 * i + 1] - rw[3 * sk + 1], rw[3 * i + 2] - rw[3 * sk + 2]};
    const bool in = i != a && i != b && dd[0] * dd[0] + dd[1] * dd[1] + dd[2] * dd[2] <= cut * cut;
    B.put(c, dd, in ? PQ + (int64_t)block_index(w, sk, Wn, n, n_up) * ld4 : nullptr,
          ((i < n_up) == (kk < n_up)) ? 0 : 1);
  }
  __syncthreads();
  B.features(4 * nm, p, cut);
  __syncthreads();
  for (int m = 0; m < nm; ++m) {
    const int i = U[u0 + m];
    if (i == a || i == b) continue;
    const int64_t bi = block_index(w, i, Wn, n, n_up);
    const T* Pi = PQ + bi * ld4;
    T acc = H1[bi * d + c];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int s = 4 * m + q;
      if (!B.Q[s]) continue;
      T gam, f;
      mw.term(B.feat[s], Pi, B.Q[s], B.ch[s], d, c, gam, f);
      acc += (q & 1) == 0 ? -(gam * f) : gam * f;
    }
    const int64_t row = rows[u0 + m];
    X[row * d + c] = acc;
    H1n[row * d + c] = acc;
  }
}
inline int swap_msg_groups(int Umax) { return 2 + (Umax + kMsgPairs / 4 - 1) / (kMsgPairs / 4); }

// ratios[w][a] = Psi(swapped) / Psi for the walkers (signed).
template <typename T>
__global__ void swap_accum_kernel(int Wn, int n, int n_up, int D, int a, int b, int Umax, uint32_t flags,
                                  const double* __restrict__ r, const double* __restrict__ rk,
                                  const double* __restrict__ rk2, const int32_t* __restrict__ Ul,
                                  const int32_t* __restrict__ Uc, const int32_t* __restrict__ Urow, McmcJastrow jp,
                                  const T* __restrict__ F1, const T* __restrict__ F2, const T* __restrict__ F1n,
                                  const T* __restrict__ F2n, const T* __restrict__ G1, const T* __restrict__ G2,
                                  const T* __restrict__ G1n, const T* __restrict__ G2n,
                                  const double* __restrict__ ldabs, const double* __restrict__ lsign,
                                  const double* __restrict__ lrat, const double* __restrict__ srat,
                                  double* __restrict__ ratios) {
  const int w = blockIdx.x;
  const WalkerRatio wr = walker_ratio<T>(w, Wn, n, n_up, D, a, Umax, flags, r + (int64_t)w * n * 3,
                                         rk + (int64_t)w * 3, b, rk2 + (int64_t)w * 3, Ul, Uc, Urow, jp, F1, F2, F1n,
                                         F2n, G1, G2, G1n, G2n, ldabs, lsign, lrat, srat);
  if (threadIdx.x == 0) ratios[(int64_t)w * n_up + a] = wr.sign * exp(wr.logr);
}

// r_beta[w] = 1 - sum_a ratios[w][a] (in index order).
static __global__ void swap_sum_kernel(int Wn, int n_up, const double* __restrict__ ratios,
                                       double* __restrict__ rb) {
  const int w = blockIdx.x * blockDim.x + threadIdx.x;
  if (w >= Wn) return;
  double sm = 0.0;
  for (int a = 0; a < n_up; ++a) sm += ratios[(int64_t)w * n_up + a];
  rb[w] = 1.0 - sm;
}

}  // namespace fire
