// Backward (adjoint) kernels of d log|Psi| / d theta per walker (Methods,
// eq. spring: the gradient rows O_i of SPRING).  The forward value path
// (embeddings recomputed in the same call) leaves its intermediates in the
// workspace; these kernels walk it in reverse.  Per-walker weight gradients
// that are sums over a walker's electrons are written by tn_batched /
// colsum_batched; per-edge and per-nucleus sums accumulate with atomics.
#pragma once

#include "common.cuh"
#include "embed.cuh"

namespace fire {

// d log|sum_d det Phi_d| / d Phi_d[i][l] = w_d A_d[l][i] with w_d the signed
// weight of determinant d; back through Phi = o * phi:
//   dO[i][d*n + l] = G phi,  dF[i][d*n + l] = G o.   One CTA per (walker, d).
template <typename T>
__global__ void det_bwd_kernel(int Wc, int n, int n_up, int D, const double* __restrict__ ldabs,
                               const double* __restrict__ lsign, const T* __restrict__ AT,
                               const T* __restrict__ Ov, const T* __restrict__ Fenv, T* __restrict__ dO,
                               T* __restrict__ dF) {
  const int w = blockIdx.x / D, dd = blockIdx.x % D;
  __shared__ double s_w;
  if (threadIdx.x == 0) {
    double lmax = -INFINITY;
    for (int q = 0; q < D; ++q)
      if (lsign[(int64_t)w * D + q] != 0.0 && ldabs[(int64_t)w * D + q] > lmax) lmax = ldabs[(int64_t)w * D + q];
    double S = 0.0, mine = 0.0;
    for (int q = 0; q < D; ++q) {
      const double sg = lsign[(int64_t)w * D + q];
      const double t = sg != 0.0 ? sg * exp(ldabs[(int64_t)w * D + q] - lmax) : 0.0;
      S += t;
      if (q == dd) mine = t;
    }
    s_w = mine / S;
  }
  __syncthreads();
  const T om = T(s_w);
  const int64_t Dn = (int64_t)D * n;
  const T* A = AT + ((int64_t)w * D + dd) * n * n;
  for (int e = threadIdx.x; e < n * n; e += blockDim.x) {
    const int i = e / n, l = e % n;
    const int64_t b = block_index(w, i, Wc, n, n_up);
    const T g = om * A[(int64_t)i * n + l];
    const int64_t col = b * Dn + (int64_t)dd * n + l;
    dO[col] = g * Fenv[col];
    dF[col] = g * Ov[col];
  }
}

// d sigma_me += sum_i dQ[i][me] * (-|r_i - R_m|) * q_ime.  One CTA per walker.
template <typename T>
__global__ void env_sigma_bwd_kernel(int Wc, int n, int n_up, int N, int E, const double* __restrict__ r,
                                     const double* __restrict__ R, const T* __restrict__ Q,
                                     const T* __restrict__ dQ, T* __restrict__ g, int64_t P, int64_t off) {
  const int w = blockIdx.x;
  const int NE = N * E;
  for (int q = threadIdx.x; q < NE; q += blockDim.x) {
    const int m = q / E;
    T acc = T(0);
    for (int i = 0; i < n; ++i) {
      const double* ri = r + ((int64_t)w * n + i) * 3;
      const double dx = ri[0] - R[3 * m], dy = ri[1] - R[3 * m + 1], dz = ri[2] - R[3 * m + 2];
      const T dist = T(sqrt(dx * dx + dy * dy + dz * dz));
      const int64_t b = block_index(w, i, Wc, n, n_up);
      acc += dQ[b * NE + q] * (-dist) * Q[b * NE + q];
    }
    g[(int64_t)w * P + off + q] += acc;
  }
}

// Seeds of the Jastrow-MLP backward: per electron row the adjoint of the
// readout f (1 for MLP1, 1/sum_i MLP2 for MLP2), then dY2 = df * w3.
template <typename T>
__global__ void jseed_kernel(int Wc, int n, int n_up, int J, const T* __restrict__ F2, const T* b32,
                             const T* __restrict__ w3, int second, T* __restrict__ df, T* __restrict__ dY) {
  const int w = blockIdx.x;
  __shared__ T s_inv;
  if (second) {
    if (threadIdx.x == 0) {
      T S = T(0);
      for (int i = 0; i < n; ++i) S += F2[block_index(w, i, Wc, n, n_up)] + b32[0];
      s_inv = T(1) / S;
    }
    __syncthreads();
  }
  const T f = second ? s_inv : T(1);
  for (int i = 0; i < n; ++i) {
    const int64_t b = block_index(w, i, Wc, n, n_up);
    if (threadIdx.x == 0) df[b] = f;
    for (int c = threadIdx.x; c < J; c += blockDim.x) dY[b * J + c] = f * w3[c];
  }
}

// Same seeds for the register readouts (one row per walker): dg1 = 1,
// dg2 = 1 / g2.
template <typename T>
__global__ void vseed_kernel(int J, const T* __restrict__ G2, const T* b32, const T* __restrict__ w3, int second,
                             T* __restrict__ df, T* __restrict__ dY) {
  const int w = blockIdx.x;
  const T f = second ? T(1) / (G2[w] + b32[0]) : T(1);
  if (threadIdx.x == 0) df[w] = f;
  for (int c = threadIdx.x; c < J; c += blockDim.x) dY[(int64_t)w * J + c] = f * w3[c];
}

// Back through the registers V_r = sum_i a_ir u_ir, a_ir = softmax_i(s_ir):
//   du_ir = a_ir dV_r,  da_ir = dV_r . u_ir,  ds_ir = a_ir (da_ir - sum_k a_kr da_kr).
// One CTA per walker, one thread per column of V.  dSU has the layout of SU.
template <typename T>
__global__ void att_bwd_kernel(int Wc, int n, int n_up, int R, int dr, const T* __restrict__ SU, int64_t ld,
                               const T* __restrict__ dV, T* __restrict__ dSU) {
  extern __shared__ unsigned char ab_smem[];
  T* a = reinterpret_cast<T*>(ab_smem);      // [n][R] softmax weights
  T* da = a + (int64_t)n * R;                // [n][R]
  T* smax = da + (int64_t)n * R;             // [R]
  T* zs = smax + R;                          // [R]
  T* dd = zs + R;                            // [R]  sum_k a_kr da_kr
  const int w = blockIdx.x;
  const int RD = R * dr;
  const int col = threadIdx.x;
  const int rg = col / dr;
  for (int q = threadIdx.x; q < R; q += blockDim.x) {
    T m = -INFINITY;
    for (int i = 0; i < n; ++i) m = fmax(m, SU[(int64_t)block_index(w, i, Wc, n, n_up) * ld + q]);
    T z = T(0);
    for (int i = 0; i < n; ++i) z += dexp<T>(SU[(int64_t)block_index(w, i, Wc, n, n_up) * ld + q] - m);
    smax[q] = m;
    zs[q] = z;
  }
  __syncthreads();
  for (int e = threadIdx.x; e < n * R; e += blockDim.x) {
    const int i = e / R, q = e % R;
    a[e] = dexp<T>(SU[(int64_t)block_index(w, i, Wc, n, n_up) * ld + q] - smax[q]) / zs[q];
    da[e] = T(0);
  }
  __syncthreads();
  // da_ir = sum_c dV_rc u_irc : per (i, r) a reduction over the dr columns
  for (int e = threadIdx.x; e < n * R; e += blockDim.x) {
    const int i = e / R, q = e % R;
    const int64_t row = (int64_t)block_index(w, i, Wc, n, n_up) * ld;
    T s = T(0);
    for (int c = 0; c < dr; ++c) s += dV[(int64_t)w * RD + q * dr + c] * SU[row + R + q * dr + c];
    da[e] = s;
  }
  __syncthreads();
  for (int q = threadIdx.x; q < R; q += blockDim.x) {
    T s = T(0);
    for (int i = 0; i < n; ++i) s += a[i * R + q] * da[i * R + q];
    dd[q] = s;
  }
  __syncthreads();
  for (int i = 0; i < n; ++i) {
    const int64_t row = (int64_t)block_index(w, i, Wc, n, n_up) * ld;
    if (col < RD) dSU[row + R + col] = a[i * R + rg] * dV[(int64_t)w * RD + col];
    for (int q = threadIdx.x; q < R; q += blockDim.x) dSU[row + q] = a[i * R + q] * (da[i * R + q] - dd[q]);
  }
}

// ---------------------------------------------------------------------------
// Backward of the filters Gamma = (a W_2) * (chi W_env), a = SiLU(x W_1 + b_1),
// shared by the message and the electron-nucleus passes.  blockDim == d, one
// column each; pairs go in batches of kGradPairs:
//   forward  the caller forms Gamma's factors of every pair from the features
//            in shared memory and leaves s_e = dGamma chi-factor and s_g =
//            dGamma a-factor of its column in shared memory;
//   columns  d W_2[h][c] += a_h s_e[c], d W_env[g][c] += chi_g s_g[c], the
//            running sums in shared memory between batches (in registers beside
//            the 48 weights of the forward they left one CTA per SM);
//   rows     sum_c s_e[c] W_2[h][c] and sum_c s_g[c] W_env[g][c], a product of
//            [pairs x d] with [d x 48]: a warp takes four pairs and 24 of the
//            48 outputs, so a weight is loaded once for four pairs, and reduces
//            its 96 sums by transpose-halving; then d W_1, d b_1 and d sigma of
//            each pair into the CTA's sums.
// One pair at a time, with derivative features and a 48-value CTA reduction per
// pair, the electron-nucleus pass of C26H24 (128 walkers) took 27.3 ms and the
// message pass 18.0 ms; now 3.8 and 4.3 ms.
// ---------------------------------------------------------------------------
constexpr int kGradPairs = 16;
// Widest CTA of the two kernels (two of them per SM in float32).
constexpr int kGradThreads = 256;

template <typename T>
struct FilterGrad {
  PairFeat<T, 1> feat[kGradPairs];
  T dv[kGradPairs][3], r[kGradPairs];
  T acc[5 * kEdgeHidden + kGauss];   // d W_1 (4 x H), d b_1, d sigma
};
// Dynamic shared memory: FilterGrad, s_e and s_g [kGradPairs][d], column sums [48][d].
template <typename T>
inline size_t filter_grad_smem(int d) {
  return ((sizeof(FilterGrad<T>) + 15) & ~(size_t)15) + (size_t)(2 * kGradPairs + kEdgeHidden + kGauss) * d * sizeof(T);
}
template <typename T>
struct FilterGradMem {
  FilterGrad<T>* f;
  T *se, *sg, *col;
  __device__ __forceinline__ FilterGradMem(unsigned char* sm, int d) {
    f = reinterpret_cast<FilterGrad<T>*>(sm);
    se = reinterpret_cast<T*>(sm + ((sizeof(FilterGrad<T>) + 15) & ~(size_t)15));
    sg = se + kGradPairs * d;
    col = sg + kGradPairs * d;
    const int c = threadIdx.x;
    for (int t = 0; t < kEdgeHidden + kGauss; ++t) col[t * d + c] = T(0);
    for (int t = c; t < 5 * kEdgeHidden + kGauss; t += blockDim.x) f->acc[t] = T(0);
  }
};

// The column and row sums of a batch of nb pairs (barriers inside: the
// features, s_e and s_g must be in place before; both are free after).
template <typename T, typename W>
__device__ __forceinline__ void filter_grad_batch(const FilterGradMem<T>& m, int nb, int d, const W* w1, const W* b1,
                                                  const W* w2, const W* wenv, const W* sigma) {
  constexpr int H = kEdgeHidden, G = kGauss;
  const int c = threadIdx.x;
  {
    T a[H + G];
#pragma unroll
    for (int t = 0; t < H + G; ++t) a[t] = m.col[t * d + c];
    for (int q = 0; q < nb; ++q) {
      const T e = m.se[q * d + c], g = m.sg[q * d + c];
#pragma unroll
      for (int t = 0; t < H + G; t += 4) {
        T f[4];
        ld_vec<T, 4>(f, &m.f->feat[q].f[t][0]);
#pragma unroll
        for (int i = 0; i < 4; ++i) a[t + i] += f[i] * (t < H ? e : g);
      }
    }
#pragma unroll
    for (int t = 0; t < H + G; ++t) m.col[t * d + c] = a[t];
  }
  __syncthreads();   // s_e and s_g of every column
  constexpr int NO = (H + G) / 2, NQ = 4;   // outputs and pairs of a warp's task
  const int lane = c & 31, nw = blockDim.x >> 5;
  for (int task = c >> 5; task < 2 * (kGradPairs / NQ); task += nw) {
    const int q0 = (task >> 1) * NQ, t0 = (task & 1) * NO;
    if (q0 >= nb) continue;
    T v[NQ * NO];
#pragma unroll
    for (int k = 0; k < NQ * NO; ++k) v[k] = T(0);
    for (int k = lane; k < d; k += 32) {
      T e[NQ], g[NQ];
#pragma unroll
      for (int q = 0; q < NQ; ++q) {   // rows past nb hold an earlier batch: their sums are dropped
        e[q] = m.se[(q0 + q) * d + k];
        g[q] = m.sg[(q0 + q) * d + k];
      }
#pragma unroll
      for (int o = 0; o < NO; ++o) {
        const int t = t0 + o;
        const T w = T(t < H ? w2[t * d + k] : wenv[(t - H) * d + k]);
#pragma unroll
        for (int q = 0; q < NQ; ++q) v[q * NO + o] += w * (t < H ? e[q] : g[q]);
      }
    }
    // lane L ends with the warp sums of values 32 b + L, b = 0, 1, 2
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      T* a = v + 32 * b;
#pragma unroll
      for (int s = 16; s >= 1; s >>= 1) {
        const bool up = (lane & s) != 0;
#pragma unroll
        for (int k = 0; k < s; ++k) {
          const T send = up ? a[k] : a[k + s];
          const T keep = up ? a[k + s] : a[k];
          a[k] = keep + __shfl_xor_sync(0xffffffffu, send, s);
        }
      }
      const int id = 32 * b + lane, q = q0 + id / NO, t = t0 + id % NO;
      if (q >= nb) continue;
      const T rr = m.f->r[q];
      if (t < H) {
        // du_h = da_h * SiLU'(u_h), u_h = x . W1[:, h] + b1[h], x = [r, delta]
        T u = T(b1[t]) + T(w1[t]) * rr;
#pragma unroll
        for (int k = 0; k < 3; ++k) u += T(w1[(1 + k) * H + t]) * m.f->dv[q][k];
        T f, f1, f2;
        silu3<T>(u, f, f1, f2);
        const T du = a[0] * f1;
        atomicAdd(&m.f->acc[t], du * rr);
#pragma unroll
        for (int k = 0; k < 3; ++k) atomicAdd(&m.f->acc[(1 + k) * H + t], du * m.f->dv[q][k]);
        atomicAdd(&m.f->acc[4 * H + t], du);
      } else {
        // chi_g = f_cut exp(-sigma_g^2 r^2): d chi_g / d sigma_g = -2 sigma_g r^2 chi_g
        const T sgm = T(sigma[t - H]);
        atomicAdd(&m.f->acc[5 * H + t - H], a[0] * (-T(2) * sgm * rr * rr) * m.f->feat[q].f[t][0]);
      }
    }
  }
  __syncthreads();
}

// Gamma's factors of one pair and this thread's column (weights read per
// batch: they are live in the forward part only).
template <typename T, typename W>
struct FilterWeights {
  T w2[kEdgeHidden], we[kGauss];
  __device__ __forceinline__ FilterWeights(const W* pw2, const W* pwe, int d, int c) {
#pragma unroll
    for (int h = 0; h < kEdgeHidden; ++h) w2[h] = T(pw2[h * d + c]);
#pragma unroll
    for (int g = 0; g < kGauss; ++g) we[g] = T(pwe[g * d + c]);
  }
  __device__ __forceinline__ void factors(const PairFeat<T, 1>& f, T& gv, T& ev) const {
    T a[1] = {T(0)}, b[1] = {T(0)};
    feat_dot<kEdgeHidden, 1, T>(f, 0, w2, a);
    feat_dot<kGauss, 1, T>(f, kEdgeHidden, we, b);
    gv = a[0];
    ev = b[0];
  }
};

// Message-passing backward.  One CTA per epc consecutive electrons of a walker
// (the pairs of all of them in one list), blockDim == d.  Inputs: dH1 =
// d/dh^1_i; recomputes each edge.  Outputs: dP [nb][2d] (own rows), dQ [nb][2d]
// (atomics at j), parameter gradients of the e-e filter, W^alpha_c and b^alpha.
constexpr int kGradElectrons = 8;   // largest epc
template <typename T, typename W>
__global__ void __launch_bounds__(kGradThreads, sizeof(T) == 4 ? 2 : 1) msg_bwd_kernel(
    int Wc, int n, int n_up, int d, int K, int epc, const double* __restrict__ r, double cut, Params<W> p,
    const int32_t* __restrict__ idx, const int32_t* __restrict__ cnt, const T* __restrict__ PQ,
    const T* __restrict__ dH1, T* __restrict__ dP, T* __restrict__ dQ, T* __restrict__ grad, int64_t P,
    const int64_t* __restrict__ po) {
  constexpr int H = kEdgeHidden, G = kGauss;
  extern __shared__ __align__(16) unsigned char fg_smem[];
  __shared__ int s_off[kGradElectrons + 1], s_par[kGradElectrons];
  __shared__ int s_e[kGradPairs], s_j[kGradPairs], s_a[kGradPairs];
  const int groups = (n + epc - 1) / epc;
  const int w = blockIdx.x / groups, i0 = (blockIdx.x % groups) * epc;
  const int ne = min(epc, n - i0);
  const int c = threadIdx.x;
  const FilterGradMem<T> m(fg_smem, d);
  const int64_t ld4 = 4 * (int64_t)d;
  T* gw = grad + (int64_t)w * P;
  const double* rw = r + (int64_t)w * n * 3;
  if (c == 0) {
    int o = 0;
    for (int e = 0; e < ne; ++e) {
      const int32_t* ce = cnt + ((int64_t)w * n + i0 + e) * 2;
      s_off[e] = o;
      s_par[e] = ce[0];
      o += ce[0] + ce[1];
    }
    s_off[ne] = o;
  }
  __syncthreads();
  const int total = s_off[ne];
  T gWc[2][4], gB[2], dPa[2];
#pragma unroll
  for (int a = 0; a < 2; ++a) {
    gB[a] = dPa[a] = T(0);
#pragma unroll
    for (int k = 0; k < 4; ++k) gWc[a][k] = T(0);
  }
  int cur = -1;   // the electron whose dP is being summed
  auto flush = [&](int e) {   // dP rows of electrons cur .. e - 1 (those without pairs stay zero)
    for (; cur < e; ++cur) {
      if (cur < 0) continue;
      const int64_t bi = block_index(w, i0 + cur, Wc, n, n_up);
      dP[bi * 2 * d + c] = dPa[0];
      dP[bi * 2 * d + d + c] = dPa[1];
      dPa[0] = dPa[1] = T(0);
    }
  };
  flush(0);
  for (int b0 = 0; b0 < total; b0 += kGradPairs) {
    const int nb = min(kGradPairs, total - b0);
    if (c < nb) {
      int e = 0;
      while (b0 + c >= s_off[e + 1]) ++e;
      const int s = b0 + c - s_off[e], i = i0 + e;
      const int j = idx[((int64_t)w * n + i) * K + s];
      const double dd[3] = {rw[3 * i] - rw[3 * j], rw[3 * i + 1] - rw[3 * j + 1], rw[3 * i + 2] - rw[3 * j + 2]};
      s_e[c] = e;
      s_j[c] = block_index(w, j, Wc, n, n_up);
      s_a[c] = s < s_par[e] ? 0 : 1;
#pragma unroll
      for (int t = 0; t < 3; ++t) m.f->dv[c][t] = T(dd[t]);
      m.f->r[c] = T(sqrt(dd[0] * dd[0] + dd[1] * dd[1] + dd[2] * dd[2]));
    }
    __syncthreads();
    for (int e = c; e < nb * kPairFeat; e += blockDim.x) {
      int q, k;
      feature_item(e, nb, q, k);
      m.f->feat[q].f[k][0] =
          pair_feature<T, W>(k, m.f->dv[q], m.f->r[q], p.ee_w1, p.ee_b1, p.ee_sigma, T(cut)).v;
    }
    __syncthreads();
    {
      const FilterWeights<T, W> fw(p.ee_w2, p.ee_wenv, d, c);
      for (int q = 0; q < nb; ++q) {
        const int e = s_e[q], a = s_a[q];
        if (e != cur) flush(e);
        const int64_t bi = block_index(w, i0 + e, Wc, n, n_up), bj = s_j[q];
        const T delta = dH1[bi * d + c];
        T gv, ev;
        fw.factors(m.f->feat[q], gv, ev);
        T z = PQ[bi * ld4 + (int64_t)a * d + c] + PQ[bj * ld4 + 2 * (int64_t)d + (int64_t)a * d + c] +
              T(p.msg_b[a * d + c]);
        T fk[4];
        ld_vec<T, 4>(fk, &m.f->feat[q].f[H + G][0]);
#pragma unroll
        for (int k = 0; k < 4; ++k) z += fk[k] * T(p.msg_w[((int64_t)a * (2 * d + 4) + 2 * d + k) * d + c]);
        T f, f1, f2;
        silu3<T>(z, f, f1, f2);
        const T gam = gv * ev, dgam = delta * f, dz = delta * gam * f1;
        m.se[q * d + c] = dgam * ev;
        m.sg[q * d + c] = dgam * gv;
        atomicAdd(&dQ[bj * 2 * d + (int64_t)a * d + c], dz);
        const T d0 = a ? T(0) : dz, d1 = a ? dz : T(0);
        dPa[0] += d0;
        dPa[1] += d1;
        gB[0] += d0;
        gB[1] += d1;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          gWc[0][k] += fk[k] * d0;
          gWc[1][k] += fk[k] * d1;
        }
      }
    }
    filter_grad_batch<T, W>(m, nb, d, p.ee_w1, p.ee_b1, p.ee_w2, p.ee_wenv, p.ee_sigma);
  }
  flush(ne);
  if (total > 0) {
    for (int t = c; t < 5 * H + G; t += blockDim.x) {
      if (t < 4 * H) atomicAdd(&gw[po[P_EE_W1] + t], m.f->acc[t]);
      else if (t < 5 * H) atomicAdd(&gw[po[P_EE_B1] + t - 4 * H], m.f->acc[t]);
      else atomicAdd(&gw[po[P_EE_SIGMA] + t - 5 * H], m.f->acc[t]);
    }
    for (int h = 0; h < H; ++h) atomicAdd(&gw[po[P_EE_W2] + h * d + c], m.col[h * d + c]);
    for (int g = 0; g < G; ++g) atomicAdd(&gw[po[P_EE_WENV] + g * d + c], m.col[(H + g) * d + c]);
#pragma unroll
    for (int a = 0; a < 2; ++a) {
      atomicAdd(&gw[po[P_MSG_B] + a * d + c], gB[a]);
#pragma unroll
      for (int k = 0; k < 4; ++k)
        atomicAdd(&gw[po[P_MSG_W] + ((int64_t)a * (2 * d + 4) + 2 * d + k) * d + c], gWc[a][k]);
    }
  }
}

// Electron-nucleus filter backward: ds = d/ds_i (the filter sum).  One CTA per
// (walker, nucleus, segment of seg <= kGradSeg electrons), blockDim == d: the
// nucleus's own weights (h^nuc_m, W_1m, b_1m) are summed within the CTA.
constexpr int kGradSeg = 256;
template <typename T, typename W>
__global__ void __launch_bounds__(kGradThreads, sizeof(T) == 4 ? 2 : 1) en_bwd_kernel(
    int Wc, int n, int n_up, int N, int d, int seg, const double* __restrict__ r, const double* __restrict__ R,
    double cnuc, Params<W> p, const T* __restrict__ dS, T* __restrict__ grad, int64_t P,
    const int64_t* __restrict__ po) {
  constexpr int H = kEdgeHidden, G = kGauss;
  extern __shared__ __align__(16) unsigned char fg_smem[];
  __shared__ int s_list[kGradSeg], s_cnt, s_b[kGradPairs];
  const int nseg = (n + seg - 1) / seg;
  const int m_ = (int)(blockIdx.x / nseg % N), w = (int)(blockIdx.x / nseg / N);
  const int i0 = (int)(blockIdx.x % nseg) * seg, i1 = min(n, i0 + seg);
  const int c = threadIdx.x;
  const FilterGradMem<T> m(fg_smem, d);
  T* gw = grad + (int64_t)w * P;
  const double Rm[3] = {R[3 * m_], R[3 * m_ + 1], R[3 * m_ + 2]};
  const double* rw = r + (int64_t)w * n * 3;
  const W *w1 = p.en_w1 + (int64_t)m_ * 4 * H, *b1 = p.en_b1 + (int64_t)m_ * H;
  if (c < 32) {   // electrons of the segment within the cutoff, ascending
    int have = 0;
    for (int j0 = i0; j0 < i1; j0 += 32) {
      const int i = j0 + c;
      bool in = false;
      if (i < i1) {
        const double d0 = rw[3 * i] - Rm[0], d1 = rw[3 * i + 1] - Rm[1], d2 = rw[3 * i + 2] - Rm[2];
        in = sqrt(d0 * d0 + d1 * d1 + d2 * d2) < cnuc;
      }
      const unsigned bal = __ballot_sync(0xffffffffu, in);
      if (in) s_list[have + __popc(bal & ((1u << c) - 1u))] = i;
      have += __popc(bal);
    }
    if (c == 0) s_cnt = have;
  }
  __syncthreads();
  const int total = s_cnt;
  if (total == 0) return;
  T gWf[4], gE = T(0);
#pragma unroll
  for (int k = 0; k < 4; ++k) gWf[k] = T(0);
  const T emb = T(p.nuc_emb[(int64_t)m_ * d + c]);
  for (int b0 = 0; b0 < total; b0 += kGradPairs) {
    const int nb = min(kGradPairs, total - b0);
    if (c < nb) {
      const int i = s_list[b0 + c];
      const double dd[3] = {rw[3 * i] - Rm[0], rw[3 * i + 1] - Rm[1], rw[3 * i + 2] - Rm[2]};
      s_b[c] = block_index(w, i, Wc, n, n_up);
#pragma unroll
      for (int t = 0; t < 3; ++t) m.f->dv[c][t] = T(dd[t]);
      m.f->r[c] = T(sqrt(dd[0] * dd[0] + dd[1] * dd[1] + dd[2] * dd[2]));
    }
    __syncthreads();
    for (int e = c; e < nb * kPairFeat; e += blockDim.x) {
      int q, k;
      feature_item(e, nb, q, k);
      m.f->feat[q].f[k][0] = pair_feature<T, W>(k, m.f->dv[q], m.f->r[q], w1, b1, p.en_sigma, T(cnuc)).v;
    }
    __syncthreads();
    {
      const FilterWeights<T, W> fw(p.en_w2, p.en_wenv, d, c);
      T wf[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) wf[k] = T(p.en_wfeat[k * d + c]);
      for (int q = 0; q < nb; ++q) {
        const T ds = dS[(int64_t)s_b[q] * d + c];
        T gv, ev, fk[4], fv = emb;
        fw.factors(m.f->feat[q], gv, ev);
        ld_vec<T, 4>(fk, &m.f->feat[q].f[H + G][0]);
#pragma unroll
        for (int k = 0; k < 4; ++k) fv += fk[k] * wf[k];
        const T dgam = ds * fv, dfv = ds * (gv * ev);
        m.se[q * d + c] = dgam * ev;
        m.sg[q * d + c] = dgam * gv;
        gE += dfv;
#pragma unroll
        for (int k = 0; k < 4; ++k) gWf[k] += fk[k] * dfv;
      }
    }
    filter_grad_batch<T, W>(m, nb, d, w1, b1, p.en_w2, p.en_wenv, p.en_sigma);
  }
  atomicAdd(&gw[po[P_NUC_EMB] + (int64_t)m_ * d + c], gE);
  for (int t = c; t < 5 * H + G; t += blockDim.x) {
    if (t < 4 * H) atomicAdd(&gw[po[P_EN_W1] + (int64_t)m_ * 4 * H + t], m.f->acc[t]);
    else if (t < 5 * H) atomicAdd(&gw[po[P_EN_B1] + (int64_t)m_ * H + t - 4 * H], m.f->acc[t]);
    else atomicAdd(&gw[po[P_EN_SIGMA] + t - 5 * H], m.f->acc[t]);
  }
  for (int h = 0; h < H; ++h) atomicAdd(&gw[po[P_EN_W2] + h * d + c], m.col[h * d + c]);
  for (int g = 0; g < G; ++g) atomicAdd(&gw[po[P_EN_WENV] + g * d + c], m.col[(H + g) * d + c]);
#pragma unroll
  for (int k = 0; k < 4; ++k) atomicAdd(&gw[po[P_EN_WFEAT] + k * d + c], gWf[k]);
}

// GLU gate backward: dZg = dP * zv * SiLU'(zg), dZv = dP * SiLU(zg).
template <typename T>
__global__ void gate_bwd_kernel(int64_t rows, int d, const T* __restrict__ Z, const T* __restrict__ dPg,
                                T* __restrict__ dZ) {
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= rows * d) return;
  const int64_t rr = e / d;
  const int c = (int)(e % d);
  const T zg = Z[rr * 2 * d + c], zv = Z[rr * 2 * d + d + c];
  T f, f1, f2;
  silu3<T>(zg, f, f1, f2);
  const T g = dPg[rr * d + c];
  dZ[rr * 2 * d + c] = g * zv * f1;
  dZ[rr * 2 * d + d + c] = g * f;
}

// LayerNorm backward for one row per CTA (blockDim == d): y = gamma xhat + beta,
// dxhat = dy gamma, ds = (dxhat - mean(dxhat) - xhat mean(dxhat xhat)) / sigma.
// Also writes dy * xhat (for d gamma).
template <typename T, typename W>
__global__ void ln_bwd_kernel(int d, const T* __restrict__ S, const T* __restrict__ dY, const W* gamma,
                              T* __restrict__ dS, T* __restrict__ dyx) {
  __shared__ T red[32];
  const int64_t row = blockIdx.x;
  const int c = threadIdx.x;
  const T inv_d = T(1) / T(d);
  const T x = S[row * d + c];
  const T mu = block_sum(x, red) * inv_d;
  const T cc = x - mu;
  const T var = block_sum(cc * cc, red) * inv_d;
  const T sg = dsqrt<T>(var + T(kLnEps));
  const T xh = cc / sg;
  const T dy = dY[row * d + c];
  const T dxh = dy * T(gamma[c]);
  const T m1 = block_sum(dxh, red) * inv_d;
  const T m2 = block_sum(dxh * xh, red) * inv_d;
  dS[row * d + c] = (dxh - m1 - xh * m2) / sg;
  dyx[row * d + c] = dy * xh;
}

// Cusp Jastrow parameter gradient: u = w a^2 / (a + r):
// du/dw = a^2/(a+r), du/da = w a (a + 2r) / (a + r)^2.  One CTA per walker.
template <typename T>
__global__ void cusp_bwd_kernel(int n, int n_up, const double* __restrict__ r, const T* __restrict__ cusp,
                                T* __restrict__ grad, int64_t P, int64_t off) {
  __shared__ T red[32];
  const int w = blockIdx.x;
  const double* rw = r + (int64_t)w * n * 3;
  T g[4] = {T(0), T(0), T(0), T(0)};
  for (int e = threadIdx.x; e < n * n; e += blockDim.x) {
    const int i = e / n, j = e % n;
    if (j <= i) continue;
    const T dx = T(rw[3 * i] - rw[3 * j]), dy = T(rw[3 * i + 1] - rw[3 * j + 1]), dz = T(rw[3 * i + 2] - rw[3 * j + 2]);
    const T rr = dsqrt<T>(dx * dx + dy * dy + dz * dz);
    const bool same = ((i < n_up) == (j < n_up));
    const T om = same ? cusp[0] : cusp[1], al = same ? cusp[2] : cusp[3];
    const T den = al + rr;
    const T dw = al * al / den;
    const T da = om * al * (al + T(2) * rr) / (den * den);
    if (same) { g[0] += dw; g[2] += da; } else { g[1] += dw; g[3] += da; }
  }
  for (int k = 0; k < 4; ++k) {
    T v = g[k];
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
      T s = T(0);
      for (int q = 0; q < (int)(blockDim.x >> 5); ++q) s += red[q];
      grad[(int64_t)w * P + off + k] += s;
    }
  }
}

}  // namespace fire
