// Differentiable FD equalization: forward with per-cluster regularizers and
// free fusion weights, and its hand-written adjoint.
//
// Forward (per subcarrier k, cluster c; n_sym right-hand sides):
//   X_c = (G_c + rho_c I)^{-1} B_c,  B_c = H_c^H Y_c       (L-MMSE, Sec. III-A, with rho_c free)
//   z_u = sum_c nu[c][u] X_c[u]                            (Eq. fusionrule with free weights)
// Adjoint of a real loss with g_z = dL/dRe z + i dL/dIm z:
//   G_x,c = diag(nu_c) G_z,   G_b,c = (G_c + rho_c I)^{-1} G_x,c
//   dL/dH_c   = Y_c G_b^H - H_c W_c,   W_c = G_b X_c^H + X_c G_b^H
//   dL/dY_c   = H_c G_b
//   dL/drho_c = -sum_k Re tr(G_b^H X_c),  dL/dnu[c][u] = sum_k sum_n Re(conj(g_z,u,n) X_c,u,n)
// (dX = M^{-1}(dB - dM X), dM = dH^H H + H^H dH + drho I, dB = dH^H Y + H^H dY.)
// The factorization is recomputed in the backward pass (a Gauss-Jordan sweep on
// [G_c + rho_c I | G_x,c]); the forward keeps the local estimates X_c in the workspace.
//
// Two forms.  FP32 plans whose subcarrier fits in one CTA run the fused kernels, which
// form the local Gram matrices as register tiles and sweep them there
// (ffeq_formed.cuh).  The others run the contraction first, which leaves the Gram
// matrices in the workspace, and the paired-FMA sweep of ffeq_gj.cuh on the augmented
// row [G_c + rho I | R] of UP + NR columns, NR the right-hand-side columns rounded up
// from n_sym (4 when n_sym <= 4, else 16), so a one-symbol problem does not sweep 16
// columns of padding.
//
// Workspace: D [n_sc][C][U+n_sym][U] (contraction output, as ffeq_equalize),
// X [n_sc][C][n_sym][U], Gb [n_sc][C][n_sym][U], W [n_sc][C][U][U] (complex) and
// per-subcarrier partial sums P [C][1+U][n_sc] (float).
#include <cmath>

#include "ffeq_device.cuh"
#include "ffeq_formed.cuh"
#include "ffeq_gj.cuh"
#include "ffeq_internal.h"

namespace ffeq {
namespace {

// Right-hand-side columns of the augmented sweep for n_sym symbols.
inline int rhs_columns(int n_sym) { return n_sym <= 4 ? 4 : kNsymMax; }
// Right-hand sides per lane of the formed tiles (four column lanes).
inline int formed_rhs(int n_sym) { return n_sym <= 4 ? 1 : (n_sym <= 8 ? 2 : 4); }

template <int UP, int NR>
struct TrainLayout {
  static constexpr int kW = UP + NR;              // augmented row width
  static constexpr int kRow = 2 * kW + 4;         // the sweep's two pivot-row buffers (float2 units)
  // Per group: pivot-row buffers + two [NR][UP] blocks.
  static constexpr int kGroup = kRow + 2 * NR * UP + 8;
};

// Row i of [G_c + rho I | R] from the workspace D (padding: identity / zero), as
// pairs of adjacent columns (rp: re of columns 2m, 2m + 1; ip: im).  rhs(n)
// supplies R[i][n] for n < NS.
template <int UP, int NR, typename Rhs>
__device__ __forceinline__ void load_row(float2 (&rp)[(UP + NR) / 2], float2 (&ip)[(UP + NR) / 2],
                                         const float2* Dg, int U, int NS, int i, bool valid, float rho, Rhs rhs) {
  constexpr int W = UP + NR;
  const int ic = i < U ? i : 0;
  float2 aug[W];
#pragma unroll
  for (int j = 0; j < UP; ++j) aug[j] = Dg[(j < U ? j : 0) * U + ic];
#pragma unroll
  for (int j = 0; j < UP; ++j) {
    const bool real = valid && i < U && j < U;
    float2 v = real ? aug[j] : make_float2(i == j ? 1.f : 0.f, 0.f);
    if (real && i == j) v = make_float2(v.x + rho, 0.f);
    aug[j] = v;
  }
#pragma unroll
  for (int n = 0; n < NR; ++n) aug[UP + n] = (n < NS && valid && i < U) ? rhs(n) : make_float2(0.f, 0.f);
#pragma unroll
  for (int m = 0; m < W / 2; ++m) {
    rp[m] = make_float2(aug[2 * m].x, aug[2 * m + 1].x);
    ip[m] = make_float2(aug[2 * m].y, aug[2 * m + 1].y);
  }
}

// Column t of the swept row (after the sweep: t < NR the solution for right-hand
// side t, NR + j column j of the inverse), times the deferred scale 1 / p_i.
template <int W>
__device__ __forceinline__ float2 swept(const float2 (&rp)[W / 2], const float2 (&ip)[W / 2], int t, float rs) {
  return make_float2((t % 2 ? rp[t / 2].y : rp[t / 2].x) * rs, (t % 2 ? ip[t / 2].y : ip[t / 2].x) * rs);
}

// Forward: one CTA per subcarrier, one group of UP lanes per cluster.
template <int UP, int NR>
__global__ void __launch_bounds__(512) train_forward_kernel(const TrainParams p) {
  extern __shared__ __align__(16) unsigned char smem[];
  using Lay = TrainLayout<UP, NR>;
  constexpr int W = Lay::kW;
  const int U = p.U, NS = p.n_sym, C = p.C;
  const int g = threadIdx.x / UP, i = threadIdx.x % UP;
  const int k = blockIdx.x;
  const int gm = g < C ? g : C - 1;
  const bool valid = g < C;
  float2* rowbuf = reinterpret_cast<float2*>(smem + 16) + gm * Lay::kGroup;
  float2* F = rowbuf + Lay::kRow;              // [NR][UP]: nu * X of this cluster
  int* fail_any = reinterpret_cast<int*>(smem);
  if (threadIdx.x == 0) *fail_any = 0;
  __syncthreads();

  const size_t matSize = static_cast<size_t>(U + NS) * U;
  const float2* Dg = p.D + (static_cast<size_t>(k) * C + gm) * matSize;
  float2 rp[W / 2], ip[W / 2];
  const float rho = p.rho_c[gm];
  load_row<UP, NR>(rp, ip, Dg, U, NS, i, valid, rho, [&](int n) { return Dg[(U + n) * U + i]; });
  float rs = 1.f;
  const int fail = gj_sweep_pairs<UP, W>(rp, ip, reinterpret_cast<float*>(rowbuf), i, valid, rs);
  if (valid && i == 0 && fail) atomicOr(fail_any, 1);

  const float w = (valid && i < U) ? p.nu[gm * U + i] : 0.f;
  if (valid && i < U) {
    float2* Xk = p.X + (static_cast<size_t>(k) * C + gm) * NS * U;
#pragma unroll
    for (int n = 0; n < NR; ++n) {
      if (n < NS) {
        const float2 x = swept<W>(rp, ip, n, rs);
        Xk[n * U + i] = x;
        F[n * UP + i] = cscale(x, w);
      }
    }
  }
  __syncthreads();
  const bool bad = *fail_any != 0;
  for (int e = threadIdx.x; e < U * NS; e += blockDim.x) {
    const int u = e % U, n = e / U;
    float2 acc = make_float2(0.f, 0.f);
    for (int c = 0; c < C; ++c)
      acc = cadd(acc, (reinterpret_cast<float2*>(smem + 16) + c * Lay::kGroup + Lay::kRow)[n * UP + u]);
    p.z[(static_cast<size_t>(k) * NS + n) * U + u] = bad ? make_float2(NAN, NAN) : acc;
  }
}

// Backward, per cluster: G_b = (G_c + rho_c I)^{-1} diag(nu_c) G_z, the partial
// sums of dL/drho_c and dL/dnu[c][.] for this subcarrier, and W_c.
template <int UP, int NR>
__global__ void __launch_bounds__(512) train_backward_solve_kernel(const TrainParams p) {
  extern __shared__ __align__(16) unsigned char smem[];
  using Lay = TrainLayout<UP, NR>;
  constexpr int W = Lay::kW;
  const int U = p.U, NS = p.n_sym, C = p.C;
  const int g = threadIdx.x / UP, i = threadIdx.x % UP;
  const int k = blockIdx.x;
  const int gm = g < C ? g : C - 1;
  const bool valid = g < C;
  float2* rowbuf = reinterpret_cast<float2*>(smem + 16) + gm * Lay::kGroup;
  float2* Gs = rowbuf + Lay::kRow;              // [NR][UP]  G_b of this cluster
  float2* Xs = Gs + NR * UP;                    // [NR][UP]  X of this cluster

  const size_t matSize = static_cast<size_t>(U + NS) * U;
  const float2* Dg = p.D + (static_cast<size_t>(k) * C + gm) * matSize;
  const float2* gz = p.gz + static_cast<size_t>(k) * NS * U;
  const float w = (valid && i < U) ? p.nu[gm * U + i] : 0.f;
  float2 rp[W / 2], ip[W / 2];
  load_row<UP, NR>(rp, ip, Dg, U, NS, i, valid, p.rho_c[gm], [&](int n) { return cscale(gz[n * U + i], w); });
  float rs = 1.f;
  gj_sweep_pairs<UP, W>(rp, ip, reinterpret_cast<float*>(rowbuf), i, valid, rs);

  // Row i of G_b; X row i from the forward pass.
  const size_t off = (static_cast<size_t>(k) * C + gm) * NS * U;
  float2 gb[NR], x[NR];
  float prho = 0.f, pnu = 0.f;
#pragma unroll
  for (int n = 0; n < NR; ++n) {
    gb[n] = swept<W>(rp, ip, n, rs);
    x[n] = (n < NS && valid && i < U) ? p.X[off + n * U + i] : make_float2(0.f, 0.f);
    const float2 gzv = (n < NS && valid && i < U) ? gz[n * U + i] : make_float2(0.f, 0.f);
    if (n < NS) {
      prho -= gb[n].x * x[n].x + gb[n].y * x[n].y;          // Re(conj(G_b) X)
      pnu += gzv.x * x[n].x + gzv.y * x[n].y;               // Re(conj(g_z) X)
    }
  }
#pragma unroll
  for (int o = UP / 2; o > 0; o >>= 1) prho += __shfl_xor_sync(kFullMask, prho, o, UP);
  float* P = p.P + static_cast<size_t>(gm) * (1 + U) * p.n_sc + k;   // [C (1 + U)][n_sc]
  if (valid) {
    if (i == 0) P[0] = prho;
    if (i < U) P[static_cast<size_t>(1 + i) * p.n_sc] = pnu;
  }
  if (valid && i < U) {
#pragma unroll
    for (int n = 0; n < NR; ++n) {
      if (n < NS) {
        p.Gb[off + n * U + i] = gb[n];
        Gs[n * UP + i] = gb[n];
        Xs[n * UP + i] = x[n];
      }
    }
  }
  __syncwarp();
  // W row i: W[i][v] = sum_n G_b[i][n] conj(X[v][n]) + X[i][n] conj(G_b[v][n]).
  if (valid && i < U) {
    float2* Wk = p.Wm + (static_cast<size_t>(k) * C + gm) * U * U + i * U;
    for (int v = 0; v < U; ++v) {
      float2 acc = make_float2(0.f, 0.f);
#pragma unroll
      for (int n = 0; n < NR; ++n) {
        if (n < NS) {
          const float2 xv = Xs[n * UP + v], gv = Gs[n * UP + v];
          // G_b[i] conj(X[v]) + X[i] conj(G_b[v])
          acc = cfma(gb[n], make_float2(xv.x, -xv.y), acc);
          acc = cfma(x[n], make_float2(gv.x, -gv.y), acc);
        }
      }
      Wk[v] = acc;
    }
  }
}

// Adjoint through the optimal-weight rule (the FD estimate ffeq_equalize
// computes with unbiased pairs: Lemma 1's weights from diag(A_c) and mu),
// per subcarrier, from the contraction output D and dL/dz.  With M_c = G_c +
// rho I, A_c = M_c^{-1}, X_c = A_c B_c, a_c = diag(A_c), w_c = 1 / a_c,
// D_u = sum_c (w_{c,u} - rho) and z_u = sum_c w_{c,u} X_{c,u} / D_u (Eq. fusionrule
// with nu = mu / (N0 a) / sum, N0 cancelled):
//   G_x = diag(w_c / D) G_z,   G_b = A_c G_x,
//   q_u = -Re(sum_n conj(g_z,u,n) (X_{c,u,n} - z_{u,n})) / (D_u a_{c,u}^2),
//   W_c = X_c G_b^H + G_b X_c^H + 2 A_c diag(q) A_c,
// after which train_backward_contract_kernel forms dL/dH_c = Y_c G_b^H - H_c W_c
// and dL/dY_c = H_c G_b.  (dz_u = sum_c (w dX + (X - z) dw) / D with dw = -da / a^2,
// dX = A (dB - dM X), da_u = -[A dM A]_uu.)  One CTA per subcarrier, one group of
// UP lanes per cluster; lane i = user i.  The sweep runs on [M_c | B_c] and
// leaves row i of X_c and of A_c.  A user no cluster can see (D_u <= 0) has
// z = 0 and contributes nothing.  A subcarrier with a system that is not
// positive definite gets NaN gradients.
template <int UP, int NR>
struct OptimalLayout {
  static constexpr int kW = UP + NR;
  static constexpr int kRow = 2 * kW + 4;   // the sweep's pivot-row buffers; then row broadcasts of A
  // Per group: pivot-row buffers, X [NR][UP], G_x then G_b [NR][UP], and q
  // (UP floats as UP / 2 complex).
  static constexpr int kGroup = kRow + 2 * NR * UP + UP / 2 + 8;
};

template <int UP, int NR>
__global__ void __launch_bounds__(512) train_optimal_solve_kernel(const TrainParams p) {
  extern __shared__ __align__(16) unsigned char smem[];
  using Lay = OptimalLayout<UP, NR>;
  constexpr int W = Lay::kW;
  const int U = p.U, NS = p.n_sym, C = p.C;
  const int g = threadIdx.x / UP, i = threadIdx.x % UP;
  const int k = blockIdx.x;
  const int gm = g < C ? g : C - 1;
  const bool valid = g < C;
  int* fail_any = reinterpret_cast<int*>(smem);
  float* wv = reinterpret_cast<float*>(smem + 16);                       // [C][UP]: w_{c,u}
  float2* grp = reinterpret_cast<float2*>(smem + 16 + ((static_cast<size_t>(C) * UP * 4 + 15) / 16) * 16);
  float2* rowbuf = grp + gm * Lay::kGroup;
  float2* Xs = rowbuf + Lay::kRow;            // [NR][UP]
  float2* Gs = Xs + NR * UP;                  // [NR][UP]
  float* qv = reinterpret_cast<float*>(Gs + NR * UP);   // [UP]
  if (threadIdx.x == 0) *fail_any = 0;
  __syncthreads();

  const size_t matSize = static_cast<size_t>(U + NS) * U;
  const float2* Dg = p.D + (static_cast<size_t>(k) * C + gm) * matSize;
  const float rho = p.rho;
  float2 rp[W / 2], ip[W / 2];
  load_row<UP, NR>(rp, ip, Dg, U, NS, i, valid, rho, [&](int n) { return Dg[(U + n) * U + i]; });
  float rs = 1.f;
  const int fail = gj_sweep_pairs<UP, W>(rp, ip, reinterpret_cast<float*>(rowbuf), i, valid, rs);
  if (valid && i == 0 && fail) atomicOr(fail_any, 1);
  // Row i of X_c and of A_c.
  float2 xr[NR], ar[UP];
#pragma unroll
  for (int n = 0; n < NR; ++n) xr[n] = swept<W>(rp, ip, n, rs);
#pragma unroll
  for (int j = 0; j < UP; ++j) ar[j] = swept<W>(rp, ip, NR + j, rs);
  float a = 1.f;
#pragma unroll
  for (int j = 0; j < UP; ++j)
    if (j == i) a = ar[j].x;
  const bool real = valid && i < U;
  const float w = real ? 1.f / a : 0.f;
  if (valid) {
    wv[gm * UP + i] = real ? w : rho;         // padding users: w - rho = 0
#pragma unroll
    for (int n = 0; n < NR; ++n) Xs[n * UP + i] = (real && n < NS) ? xr[n] : make_float2(0.f, 0.f);
  }
  __syncthreads();
  const bool bad = *fail_any != 0;
  // D_u and z_u over the clusters in a fixed order (every group for its own users).
  float Du = 0.f;
  for (int cc = 0; cc < C; ++cc) Du += wv[cc * UP + i] - rho;
  const bool seen = Du > 0.f;
  const float invD = seen ? 1.f / Du : 0.f;
  const float2* gzk = p.gz + static_cast<size_t>(k) * NS * U;
  float qn = 0.f;                                 // sum_n Re(conj(g_z) (X - z))
#pragma unroll
  for (int n = 0; n < NR; ++n) {
    if (n < NS) {
      float2 num = make_float2(0.f, 0.f);
      for (int cc = 0; cc < C; ++cc) {
        const float2 xc = (grp + cc * Lay::kGroup + Lay::kRow)[n * UP + i];
        const float wc = wv[cc * UP + i];
        num = make_float2(fmaf(wc, xc.x, num.x), fmaf(wc, xc.y, num.y));
      }
      const float2 zn = cscale(num, invD);
      const float2 gzv = real ? gzk[n * U + i] : make_float2(0.f, 0.f);
      qn = fmaf(gzv.x, xr[n].x - zn.x, fmaf(gzv.y, xr[n].y - zn.y, qn));
      if (valid) Gs[n * UP + i] = cscale(gzv, w * invD);   // G_x
    }
  }
  if (valid) qv[i] = (real && seen) ? -qn * invD * w * w : 0.f;   // 1 / a^2 = w^2
  __syncwarp();
  // G_b row i = sum_j A_ij G_x[j].
  float2 gb[NR];
#pragma unroll
  for (int n = 0; n < NR; ++n) {
    float2 acc = make_float2(0.f, 0.f);
    if (n < NS) {
#pragma unroll
      for (int j = 0; j < UP; ++j) acc = cfma(ar[j], Gs[n * UP + j], acc);
    }
    gb[n] = bad ? make_float2(NAN, NAN) : acc;
  }
  __syncwarp();
  const size_t off = (static_cast<size_t>(k) * C + gm) * NS * U;
  if (valid) {
#pragma unroll
    for (int n = 0; n < NR; ++n) {
      if (n < NS) {
        Gs[n * UP + i] = gb[n];
        if (real) p.Gb[off + n * U + i] = gb[n];
      }
    }
  }
  // W row i, column v: sum_n (G_b[i][n] conj(X[v][n]) + X[i][n] conj(G_b[v][n]))
  // + 2 sum_j A_ij q_j A_jv, with row v of A broadcast by lane v (A_jv = conj(A_vj)).
  float2* Wk = p.Wm + (static_cast<size_t>(k) * C + gm) * U * U + static_cast<size_t>(i) * U;
  for (int v = 0; v < U; ++v) {
    __syncwarp();
    if (valid && i == v) {
#pragma unroll
      for (int j = 0; j < UP; ++j) rowbuf[j] = ar[j];
    }
    __syncwarp();
    float2 acc = make_float2(0.f, 0.f);
#pragma unroll
    for (int n = 0; n < NR; ++n) {
      if (n < NS) {
        const float2 xv = Xs[n * UP + v], gv = Gs[n * UP + v];
        acc = cfma(gb[n], make_float2(xv.x, -xv.y), acc);
        acc = cfma(xr[n], make_float2(gv.x, -gv.y), acc);
      }
    }
    float2 ext = make_float2(0.f, 0.f);
#pragma unroll
    for (int j = 0; j < UP; ++j) {
      const float2 av = rowbuf[j];                                     // A_vj
      ext = cfma(cscale(ar[j], qv[j]), make_float2(av.x, -av.y), ext);
    }
    if (real) Wk[v] = bad ? make_float2(NAN, NAN) : make_float2(fmaf(2.f, ext.x, acc.x), fmaf(2.f, ext.y, acc.y));
  }
}

// Antennas [b0, b1) of cluster c.
__device__ __forceinline__ void cluster_range(const TrainParams& p, int c, int& b0, int& b1) {
  if (p.cl_uniform) {
    const int S = p.B / p.C;
    b0 = c * S;
    b1 = b0 + S;
  } else {
    b0 = p.cl_off[c];
    b1 = p.cl_off[c + 1];
  }
}

// Fused training kernels for FP32 plans whose subcarrier fits in shared memory:
// one CTA per subcarrier stages H_k and Y_k in their natural rows, and a lane
// group per cluster forms [G_c + rho_c I | R] as register tiles and sweeps it
// (ffeq_formed.cuh), so the local Gram matrices never go through the workspace.
// Only the right-hand sides are wanted, so the sweep leaves out the inverse.  The
// backward pass forms and factors again (nothing is stored), and with H and Y
// still staged forms the gradients of H and Y from the low-rank form of W:
//   sum_v H[v][b] W[v][u] = sum_n (H X)_n[b] conj(G_b[n][u]) + (H G_b)_n[b] conj(X[n][u]),
//   dL/dH[u][b] = sum_n (Y[n][b] - (H X)_n[b]) conj(G_b[n][u]) - dL/dY[n][b] conj(X[n][u]),
//   dL/dY[n][b] = (H G_b)_n[b] = sum_u H[u][b] G_b[n][u],
// which needs neither W nor G_b in the workspace.
constexpr int kFormedThreads = 256;   // at most this many threads per CTA

template <int UP, int NRC>
struct FormedTrainLayout {
  static constexpr int NR = 4 * NRC;
  // Bytes: a flag, the staged rows, per cluster [NR][UP] values (forward: nu X
  // complex; backward: X and G_b interleaved, two complex).
  __host__ __device__ static size_t values(int B, int rows) { return 16 + formed_staged_bytes(B, rows); }
  static size_t bytes(int B, int U, int n_sym, int C, bool backward) {
    return values(B, U + n_sym) + static_cast<size_t>(C) * NR * UP * (backward ? 16 : 8);
  }
  // Lane groups of a CTA, and its threads: the groups' lanes, and enough to walk
  // the antennas at once.
  static int groups(int C) {
    const int most = kFormedThreads / FormedShape<UP>::GL;
    return C < most ? C : most;
  }
  static int threads(int B, int C) {
    const int t = groups(C) * FormedShape<UP>::GL, w = B < 128 ? B : 128;
    return (((t > w ? t : w) + 31) / 32) * 32;
  }
};

// Fused forward: X_c to the workspace and z = sum_c nu_c X_c (fixed cluster order).
template <int UP, int NRC>
__global__ void __launch_bounds__(kFormedThreads, 2) train_forward_fused_kernel(const TrainParams p, int groups) {
  extern __shared__ __align__(16) unsigned char smem[];
  using F = FormedShape<UP>;
  using Lay = FormedTrainLayout<UP, NRC>;
  constexpr int NR = Lay::NR;
  const int U = p.U, NS = p.n_sym, C = p.C, B = p.B, RS = formed_stride(B);
  const int k = blockIdx.x;
  int* fail_any = reinterpret_cast<int*>(smem);
  float* Ws = reinterpret_cast<float*>(smem + 16);
  float2* Fs = reinterpret_cast<float2*>(smem + Lay::values(B, U + NS));   // [C][NR][UP]: nu X
  if (threadIdx.x == 0) *fail_any = 0;
  formed_stage(p.H + static_cast<size_t>(k) * U * B, p.y + static_cast<size_t>(k) * NS * B, U, NS, B, Ws);
  formed_wait();

  const int grp = threadIdx.x / F::GL, gl = threadIdx.x % F::GL, r = gl / 4, q = gl % 4;
  if ((threadIdx.x & ~31) / F::GL < groups) {   // whole warps: some lane has a group
    for (int c0 = 0; c0 < C; c0 += groups) {
      const bool valid = grp < groups && c0 + grp < C;
      const int c = valid ? c0 + grp : 0;
      int b0, b1;
      cluster_range(p, c, b0, b1);
      float re[F::RPL][F::CA + NRC], im[F::RPL][F::CA + NRC], rs[F::RPL];
      formed_tile<UP, NRC, true, false>(Ws, RS, U, NS, b0, b1, r, q, valid, p.rho_c[c], re, im);
      const int fail = formed_sweep<UP, NRC, false>(re, im, U, r, q, rs);
      if (valid && gl == 0 && fail) atomicOr(fail_any, 1);
      if (valid) {
        float2* Xk = p.X + (static_cast<size_t>(k) * C + c) * NS * U;
#pragma unroll
        for (int i = 0; i < F::RPL; ++i) {
          const int u = r + F::RL * i;
          if (u < U) {
            const float w = p.nu[c * U + u];
#pragma unroll
            for (int j = 0; j < NRC; ++j) {
              const int n = q + 4 * j;
              if (n < NS) {
                const float2 x = make_float2(re[i][F::CA + j] * rs[i], im[i][F::CA + j] * rs[i]);
                Xk[n * U + u] = x;
                Fs[(c * NR + n) * UP + u] = cscale(x, w);
              }
            }
          }
        }
      }
    }
  }
  __syncthreads();
  const bool bad = *fail_any != 0;
  for (int e = threadIdx.x; e < UP * NS; e += blockDim.x) {
    const int u = e % UP, n = e / UP;
    if (u >= U) continue;
    float2 acc = make_float2(0.f, 0.f);
    for (int c = 0; c < C; ++c) acc = cadd(acc, Fs[(c * NR + n) * UP + u]);
    p.z[(static_cast<size_t>(k) * NS + n) * U + u] = bad ? make_float2(NAN, NAN) : acc;
  }
}

// Row stride (complex) of the UP x UP matrices kept per cluster: 16-byte rows, and
// a group's lanes (row r + 4 i, column q + 4 j) fall in different banks.
template <int UP>
constexpr int FormedKStride = UP + 4;

// Gradients at antennas b .. b + AP - 1 of one cluster, users u0 .. u0 + UN - 1, one
// thread: (H X)_n, (H G_b)_n = dL/dY[n][b] (written by the thread of u0 = 0), then
// dL/dH[.][b] from the low-rank form above and, FULL (the optimal weights), minus
// sum_v H[v][b] K[v][u].  xg: X and G_b of the cluster [n][UP], col: the staged rows
// at antenna b.
template <int UP, int AP, int UN, bool FULL>
__device__ __forceinline__ void antenna_gradients(const float* col, int RS, const float4* xg, const float2* K, int U,
                                                  int u0, int NS, int B, float2* gH, float2* gy) {
  auto load = [&](int row, float2 (&h)[AP]) {
    if constexpr (AP == 2) {
      const float4 t = *reinterpret_cast<const float4*>(col + row * RS);
      h[0] = make_float2(t.x, t.y);
      h[1] = make_float2(t.z, t.w);
    } else {
      h[0] = *reinterpret_cast<const float2*>(col + row * RS);
    }
  };
  auto store = [&](float2* at, const float2 (&v)[AP], bool wide) {
    if constexpr (AP == 2) {
      if (wide) {
        *reinterpret_cast<float4*>(at) = make_float4(v[0].x, v[0].y, v[1].x, v[1].y);
        return;
      }
    }
#pragma unroll
    for (int a = 0; a < AP; ++a) at[a] = v[a];
  };
  const bool wide = AP == 2 && ((reinterpret_cast<uintptr_t>(gH) | reinterpret_cast<uintptr_t>(gy)) & 15) == 0;
  float2 acc[UN][AP];
#pragma unroll
  for (int u = 0; u < UN; ++u)
#pragma unroll
    for (int a = 0; a < AP; ++a) acc[u][a] = make_float2(0.f, 0.f);
  for (int n = 0; n < NS; ++n, xg += UP) {
    float2 hx[AP], hg[AP], h[AP];
#pragma unroll
    for (int a = 0; a < AP; ++a) hx[a] = hg[a] = make_float2(0.f, 0.f);
#pragma unroll
    for (int v = 0; v < UP; ++v) {
      if (v < U) {
        load(v, h);
        const float4 t = xg[v];
#pragma unroll
        for (int a = 0; a < AP; ++a) {
          hx[a] = cfma(h[a], make_float2(t.x, t.y), hx[a]);
          hg[a] = cfma(h[a], make_float2(t.z, t.w), hg[a]);
        }
      }
    }
    load(U + n, h);
#pragma unroll
    for (int a = 0; a < AP; ++a) hx[a] = csub(h[a], hx[a]);   // Y[n][b] - (H X)_n[b]
    if (u0 == 0) store(gy + static_cast<size_t>(n) * B, hg, wide);
#pragma unroll
    for (int u = 0; u < UN; ++u) {
      if (u0 + u < U) {
        const float4 t = xg[u0 + u];
#pragma unroll
        for (int a = 0; a < AP; ++a) {
          acc[u][a] = cfma_conj(make_float2(t.z, t.w), hx[a], acc[u][a]);    // conj(G_b[n][u]) (Y - H X)_n
          acc[u][a] = cfms_bconj(hg[a], make_float2(t.x, t.y), acc[u][a]);   // - dL/dY[n][b] conj(X[n][u])
        }
      }
    }
  }
  if constexpr (FULL) {
    constexpr int KS = FormedKStride<UP>;
    for (int v = 0; v < U; ++v, K += KS) {
      float2 h[AP];
      load(v, h);
#pragma unroll
      for (int u = 0; u < UN; u += 2) {
        const float4 t = *reinterpret_cast<const float4*>(K + u0 + u);
#pragma unroll
        for (int a = 0; a < AP; ++a) {
          acc[u][a] = cfms(h[a], make_float2(t.x, t.y), acc[u][a]);
          acc[u + 1][a] = cfms(h[a], make_float2(t.z, t.w), acc[u + 1][a]);
        }
      }
    }
  }
#pragma unroll
  for (int u = 0; u < UN; ++u)
    if (u0 + u < U) store(gH + static_cast<size_t>(u0 + u) * B, acc[u], wide);
}

// antenna_gradients over every antenna of the subcarrier, one per thread; with the
// full-rank term (FULL) and clusters that start and end on even antennas, a thread
// takes two antennas and half of the users instead, which halves the reads of K.
// XG: per cluster `xgs` float4; K: per cluster UP rows of FormedKStride complex.
template <int UP, bool FULL>
__device__ __forceinline__ void subcarrier_gradients(const TrainParams& p, const float* Ws, int RS, const float4* XG,
                                                     int xgs, const float2* K) {
  const int U = p.U, NS = p.n_sym, C = p.C, B = p.B, k = blockIdx.x;
  float2* gHk = p.gH + static_cast<size_t>(k) * U * B;
  float2* gyk = p.gy + static_cast<size_t>(k) * NS * B;
  const int S = p.cl_uniform ? B / C : 0;
  if constexpr (FULL) {
    if (p.cl_uniform && (S & 1) == 0) {
      const int half = B / 2;
      for (int e = threadIdx.x; e < B; e += blockDim.x) {
        const int b = 2 * (e < half ? e : e - half), u0 = e < half ? 0 : UP / 2, c = b / S;
        antenna_gradients<UP, 2, UP / 2, true>(Ws + 2 * b, RS, XG + c * xgs, K + c * UP * FormedKStride<UP>, U, u0, NS,
                                               B, gHk + b, gyk + b);
      }
      return;
    }
  }
  for (int b = threadIdx.x; b < B; b += blockDim.x) {
    int c = 0;
    if (p.cl_uniform) {
      c = b / S;
    } else {
      while (c + 1 < C && b >= p.cl_off[c + 1]) ++c;
    }
    antenna_gradients<UP, 1, UP, FULL>(Ws + 2 * b, RS, XG + c * xgs, FULL ? K + c * UP * FormedKStride<UP> : nullptr, U,
                                       0, NS, B, gHk + b, gyk + b);
  }
}

// Fused backward: G_b from the recomputed factorization of [G_c + rho_c I |
// diag(nu_c) G_z], the partial sums of dL/drho_c and dL/dnu[c][.] (X_c from the
// forward pass), then the gradients of H and Y per antenna (the low-rank form
// above; sums over users and symbols in a fixed order).
template <int UP, int NRC>
__global__ void __launch_bounds__(kFormedThreads, 2) train_backward_fused_kernel(const TrainParams p, int groups) {
  extern __shared__ __align__(16) unsigned char smem[];
  using F = FormedShape<UP>;
  using Lay = FormedTrainLayout<UP, NRC>;
  constexpr int NR = Lay::NR;
  const int U = p.U, NS = p.n_sym, C = p.C, B = p.B, RS = formed_stride(B);
  const int k = blockIdx.x;
  float* Ws = reinterpret_cast<float*>(smem + 16);
  float4* XG = reinterpret_cast<float4*>(smem + Lay::values(B, U + NS));   // [C][NR][UP]: X, G_b
  formed_stage(p.H + static_cast<size_t>(k) * U * B, p.y + static_cast<size_t>(k) * NS * B, U, NS, B, Ws);
  formed_wait();

  const float2* gz = p.gz + static_cast<size_t>(k) * NS * U;
  const int grp = threadIdx.x / F::GL, gl = threadIdx.x % F::GL, r = gl / 4, q = gl % 4;
  if ((threadIdx.x & ~31) / F::GL < groups) {
    for (int c0 = 0; c0 < C; c0 += groups) {
      const bool valid = grp < groups && c0 + grp < C;
      const int c = valid ? c0 + grp : 0;
      int b0, b1;
      cluster_range(p, c, b0, b1);
      const size_t off = (static_cast<size_t>(k) * C + c) * NS * U;
      // nu, g_z and X of this lane's rows, in flight while the tile is formed
      // (several right-hand sides per lane: read when needed, to save registers).
      constexpr int NP = NRC == 1 ? 1 : 0;
      float nu[F::RPL];
      float2 gzr[F::RPL], xr[F::RPL];
#pragma unroll
      for (int i = 0; i < F::RPL; ++i) {
        const int u = r + F::RL * i;
        nu[i] = valid && u < U ? p.nu[c * U + u] : 0.f;
        const bool real = NP && valid && u < U && q < NS;
        gzr[i] = real ? gz[q * U + u] : make_float2(0.f, 0.f);
        xr[i] = real ? p.X[off + q * U + u] : make_float2(0.f, 0.f);
      }
      float re[F::RPL][F::CA + NRC], im[F::RPL][F::CA + NRC], rs[F::RPL];
      formed_tile<UP, NRC, false, false>(Ws, RS, U, NS, b0, b1, r, q, valid, p.rho_c[c], re, im);
#pragma unroll
      for (int i = 0; i < F::RPL; ++i) {
        const int u = r + F::RL * i;
#pragma unroll
        for (int j = 0; j < NRC; ++j) {
          const int n = q + 4 * j;
          const float2 g = NP ? gzr[i] : (valid && u < U && n < NS ? gz[n * U + u] : make_float2(0.f, 0.f));
          re[i][F::CA + j] = g.x * nu[i];
          im[i][F::CA + j] = g.y * nu[i];
        }
      }
      formed_sweep<UP, NRC, false>(re, im, U, r, q, rs);
      float prho = 0.f;
      // Partial sums of this subcarrier, column c (1 + U) + 1 + u (or + 0) of P
      // [C (1 + U)][n_sc]: the reduction reads each column contiguously.
      float* P = p.P + static_cast<size_t>(c) * (1 + U) * p.n_sc + k;
#pragma unroll
      for (int i = 0; i < F::RPL; ++i) {
        const int u = r + F::RL * i;
        float pnu = 0.f;
#pragma unroll
        for (int j = 0; j < NRC; ++j) {
          const int n = q + 4 * j;
          if (valid && u < U && n < NS) {
            const float2 gb = make_float2(re[i][F::CA + j] * rs[i], im[i][F::CA + j] * rs[i]);
            const float2 x = NP ? xr[i] : p.X[off + n * U + u], g = NP ? gzr[i] : gz[n * U + u];
            prho -= gb.x * x.x + gb.y * x.y;          // Re(conj(G_b) X)
            pnu += g.x * x.x + g.y * x.y;             // Re(conj(g_z) X)
            XG[(c * NR + n) * UP + u] = make_float4(x.x, x.y, gb.x, gb.y);
          }
        }
        pnu += __shfl_xor_sync(kFullMask, pnu, 1);
        pnu += __shfl_xor_sync(kFullMask, pnu, 2);
        if (valid && u < U && q == 0) P[static_cast<size_t>(1 + u) * p.n_sc] = pnu;
      }
#pragma unroll
      for (int o = F::GL / 2; o > 0; o >>= 1) prho += __shfl_xor_sync(kFullMask, prho, o);
      if (valid && gl == 0) P[0] = prho;
    }
  }
  __syncthreads();

  subcarrier_gradients<UP, false>(p, Ws, RS, XG, NR * UP, nullptr);
}

// Fused adjoint through the optimal weights (FP32 plans whose subcarrier fits):
// [M_c | B_c] formed from the staged H and Y as register tiles and swept with the
// inverse (ffeq_formed.cuh), the weights, z, q, G_x and G_b of
// train_optimal_solve_kernel by one lane per user, and the gradients per antenna
// from the low-rank part of W_c and its full-rank term K_c = 2 A_c diag(q) A_c,
// formed once per cluster as tiles (it was applied as two products per antenna
// before, (H A) then times q A, with two shared-memory reads per product), so
// neither D nor W_c nor G_b goes through the workspace.
template <int UP, int NRC>
struct FormedOptimalLayout {
  static constexpr int NR = 4 * NRC;
  static constexpr int AS = FormedKStride<UP>;
  // Bytes: a flag, the staged rows, per cluster A [UP][AS] (then K in its place), X
  // and G_b [NR][UP] interleaved, and w, q [UP].
  __host__ __device__ static size_t values(int B, int rows) { return 16 + formed_staged_bytes(B, rows); }
  static constexpr int CLUSTER = UP * AS * 8 + NR * UP * 16 + 2 * UP * 4;   // bytes
  static size_t bytes(int B, int U, int n_sym, int C) {
    return values(B, U + n_sym) + static_cast<size_t>(C) * CLUSTER;
  }
};

template <int UP, int NRC>
__global__ void __launch_bounds__(kFormedThreads, 2) train_optimal_fused_kernel(const TrainParams p, int groups) {
  extern __shared__ __align__(16) unsigned char smem[];
  using F = FormedShape<UP>;
  using Lay = FormedOptimalLayout<UP, NRC>;
  constexpr int NR = Lay::NR, AS = Lay::AS;
  const int U = p.U, NS = p.n_sym, C = p.C, B = p.B, RS = formed_stride(B);
  const int k = blockIdx.x;
  const float rho = p.rho;
  int* fail_any = reinterpret_cast<int*>(smem);
  float* Ws = reinterpret_cast<float*>(smem + 16);
  float4* XG = reinterpret_cast<float4*>(smem + Lay::values(B, U + NS));   // [C][NR][UP]: X, then G_x, then G_b
  float2* As = reinterpret_cast<float2*>(XG + static_cast<size_t>(C) * NR * UP);   // [C][UP][AS]
  float* wv = reinterpret_cast<float*>(As + static_cast<size_t>(C) * UP * AS);   // [C][UP]: w = 1 / A_uu
  float* qv = wv + C * UP;                                                 // [C][UP]
  if (threadIdx.x == 0) *fail_any = 0;
  formed_stage(p.H + static_cast<size_t>(k) * U * B, p.y + static_cast<size_t>(k) * NS * B, U, NS, B, Ws);
  formed_wait();

  const int grp = threadIdx.x / F::GL, gl = threadIdx.x % F::GL, r = gl / 4, q = gl % 4;
  const bool solver = (threadIdx.x & ~31) / F::GL < groups;   // whole warps: some lane has a group
  if (solver) {
    for (int c0 = 0; c0 < C; c0 += groups) {
      const bool valid = grp < groups && c0 + grp < C;
      const int c = valid ? c0 + grp : 0;
      int b0, b1;
      cluster_range(p, c, b0, b1);
      float re[F::RPL][F::CA + NRC], im[F::RPL][F::CA + NRC], rs[F::RPL];
      formed_tile<UP, NRC, true, true>(Ws, RS, U, NS, b0, b1, r, q, valid, rho, re, im);
      const int fail = formed_sweep<UP, NRC, true>(re, im, U, r, q, rs);
      if (valid && gl == 0 && fail) atomicOr(fail_any, 1);
#pragma unroll
      for (int i = 0; i < F::RPL; ++i) {
        const int u = r + F::RL * i;
        const float Ai = formed_diagonal<UP, F::CA + NRC>(re, i, r) * rs[i];
        if (valid) {
          if (q == (r & 3)) wv[c * UP + u] = u < U ? 1.f / Ai : rho;   // padding users: w - rho = 0
#pragma unroll
          for (int j = 0; j < F::CA; ++j)
            As[(c * UP + u) * AS + q + 4 * j] = make_float2(re[i][j] * rs[i], im[i][j] * rs[i]);
#pragma unroll
          for (int j = 0; j < NRC; ++j)
            *reinterpret_cast<float2*>(XG + (c * NR + q + 4 * j) * UP + u) =
                make_float2(re[i][F::CA + j] * rs[i], im[i][F::CA + j] * rs[i]);   // zero for padding
        }
      }
    }
  }
  __syncthreads();
  const bool bad = *fail_any != 0;
  const float2* gzk = p.gz + static_cast<size_t>(k) * NS * U;
  if (solver) {
    for (int c0 = 0; c0 < C; c0 += groups) {
      const bool valid = grp < groups && c0 + grp < C;
      const int c = valid ? c0 + grp : 0;
      // Lane i = user i: D_u and z_u over the clusters in a fixed order, q and G_x.
      const int i = gl;
      const bool real = valid && i < U;
      float4* xg = XG + c * NR * UP;
      if (real) {
        float Du = 0.f;
        for (int cc = 0; cc < C; ++cc) Du += wv[cc * UP + i] - rho;
        const bool seen = Du > 0.f;
        const float invD = seen ? 1.f / Du : 0.f;
        const float w = wv[c * UP + i];
        float qn = 0.f;                                 // sum_n Re(conj(g_z) (X - z))
        for (int n = 0; n < NS; ++n) {
          float2 num = make_float2(0.f, 0.f);
          for (int cc = 0; cc < C; ++cc) {
            const float2 xc = *reinterpret_cast<const float2*>(XG + (cc * NR + n) * UP + i);
            const float wc = wv[cc * UP + i];
            num = make_float2(fmaf(wc, xc.x, num.x), fmaf(wc, xc.y, num.y));
          }
          const float2 zn = cscale(num, invD);
          const float2 xr = *reinterpret_cast<const float2*>(xg + n * UP + i);
          const float2 gzv = gzk[n * U + i];
          qn = fmaf(gzv.x, xr.x - zn.x, fmaf(gzv.y, xr.y - zn.y, qn));
          reinterpret_cast<float2*>(xg + n * UP + i)[1] = cscale(gzv, w * invD);   // G_x
        }
        qv[c * UP + i] = seen ? -qn * invD * w * w : 0.f;   // 1 / a^2 = w^2
      } else if (valid && i < UP) {
        for (int n = 0; n < NS; ++n) reinterpret_cast<float2*>(xg + n * UP + i)[1] = make_float2(0.f, 0.f);
        qv[c * UP + i] = 0.f;
      }
      __syncwarp();
      // G_b row i = sum_j A_ij G_x[j], A_ij = conj(A_ji) (read along a row: A is Hermitian).
      float2 gb[NR];
      const float2* acol = As + c * UP * AS + (i < UP ? i : 0);
#pragma unroll
      for (int n = 0; n < NR; ++n) {
        gb[n] = make_float2(0.f, 0.f);
        if (n < NS) {
          for (int j = 0; j < U; ++j) gb[n] = cfma_conj(acol[j * AS], reinterpret_cast<const float2*>(xg + n * UP + j)[1], gb[n]);
        }
      }
      __syncwarp();
#pragma unroll
      for (int n = 0; n < NR; ++n)
        if (real && n < NS)
          reinterpret_cast<float2*>(xg + n * UP + i)[1] = bad ? make_float2(NAN, NAN) : gb[n];
      // K = 2 A diag(q) A: rows r + RL i, columns q + 4 j.
      float kr[F::RPL][F::CA], ki[F::RPL][F::CA];
#pragma unroll
      for (int a = 0; a < F::RPL; ++a)
#pragma unroll
        for (int j = 0; j < F::CA; ++j) kr[a][j] = ki[a][j] = 0.f;
      const float2* Ac = As + c * UP * AS;
      for (int w = 0; w < U; ++w) {
        const float q2 = 2.f * qv[c * UP + w];
        float2 left[F::RPL];
#pragma unroll
        for (int a = 0; a < F::RPL; ++a) left[a] = cscale(Ac[(r + F::RL * a) * AS + w], q2);
#pragma unroll
        for (int j = 0; j < F::CA; ++j) {
          const float2 v = Ac[w * AS + q + 4 * j];
#pragma unroll
          for (int a = 0; a < F::RPL; ++a) {
            kr[a][j] = fmaf(left[a].x, v.x, kr[a][j]);
            kr[a][j] = fmaf(-left[a].y, v.y, kr[a][j]);
            ki[a][j] = fmaf(left[a].x, v.y, ki[a][j]);
            ki[a][j] = fmaf(left[a].y, v.x, ki[a][j]);
          }
        }
      }
      __syncwarp();   // the group has read A: K takes its place
      if (valid) {
#pragma unroll
        for (int a = 0; a < F::RPL; ++a)
#pragma unroll
          for (int j = 0; j < F::CA; ++j)
            As[(c * UP + r + F::RL * a) * AS + q + 4 * j] = make_float2(kr[a][j], ki[a][j]);
      }
    }
  }
  __syncthreads();
  subcarrier_gradients<UP, true>(p, Ws, RS, XG, NR * UP, As);
}

// Backward contraction, per subcarrier (G_b and W of its clusters staged in
// shared memory):
//   dL/dH[u][b] = sum_n Y[n][b] conj(G_b[n][u]) - sum_v H[v][b] W[v][u]
//   dL/dY[n][b] = sum_u H[u][b] G_b[n][u]
// A work item of dL/dH is one antenna b and kUq users (kUq independent
// accumulators, so the dependent chains overlap); its column of H is read from
// HBM coalesced over b (the items of one antenna share it through L1).  Antenna
// b belongs to cluster b / S, or to the cluster whose offsets hold it.
constexpr int kUq = 4;

template <int UP>
__global__ void __launch_bounds__(256) train_backward_contract_kernel(const TrainParams p) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int U = p.U, NS = p.n_sym, C = p.C, B = p.B, S = B / C;
  const int k = blockIdx.x;
  float2* Gs = reinterpret_cast<float2*>(smem);            // [C][NS][U]
  float2* Ws = Gs + static_cast<size_t>(C) * NS * U;       // [C][U][U]
  const float2* Gk = p.Gb + static_cast<size_t>(k) * C * NS * U;
  const float2* Wk = p.Wm + static_cast<size_t>(k) * C * U * U;
  for (int e = threadIdx.x; e < C * NS * U; e += blockDim.x) Gs[e] = Gk[e];
  for (int e = threadIdx.x; e < C * U * U; e += blockDim.x) Ws[e] = Wk[e];
  __syncthreads();
  const float2* Hk = p.H + static_cast<size_t>(k) * U * B;
  const float2* Yk = p.y + static_cast<size_t>(k) * NS * B;
  float2* gHk = p.gH + static_cast<size_t>(k) * U * B;
  float2* gyk = p.gy + static_cast<size_t>(k) * NS * B;
  auto cluster_of = [&](int b) {
    if (p.cl_uniform) return b / S;
    int c = 0;
    while (c + 1 < C && b >= p.cl_off[c + 1]) ++c;
    return c;
  };
  const int nq = (U + kUq - 1) / kUq;
  for (int e = threadIdx.x; e < B * nq; e += blockDim.x) {
    const int b = e % B, u0 = (e / B) * kUq;
    const int c = cluster_of(b);
    const float2* Gc = Gs + static_cast<size_t>(c) * NS * U;
    const float2* Wc = Ws + static_cast<size_t>(c) * U * U;
    float2 acc[kUq];
#pragma unroll
    for (int q = 0; q < kUq; ++q) acc[q] = make_float2(0.f, 0.f);
    for (int n = 0; n < NS; ++n) {
      const float2 yv = Yk[static_cast<size_t>(n) * B + b];
#pragma unroll
      for (int q = 0; q < kUq; ++q)
        if (u0 + q < U) acc[q] = cfma_conj(Gc[n * U + u0 + q], yv, acc[q]);   // Y[n][b] conj(G_b[n][u])
    }
#pragma unroll
    for (int v = 0; v < UP; ++v) {
      if (v < U) {
        const float2 hv = Hk[static_cast<size_t>(v) * B + b];
#pragma unroll
        for (int q = 0; q < kUq; ++q)
          if (u0 + q < U) acc[q] = cfms(hv, Wc[v * U + u0 + q], acc[q]);          // - H[v][b] W[v][u]
      }
    }
#pragma unroll
    for (int q = 0; q < kUq; ++q)
      if (u0 + q < U) gHk[static_cast<size_t>(u0 + q) * B + b] = acc[q];
  }
  for (int e = threadIdx.x; e < B * NS; e += blockDim.x) {
    const int b = e % B, n = e / B;
    const float2* Gc = Gs + static_cast<size_t>(cluster_of(b)) * NS * U;
    float2 acc0 = make_float2(0.f, 0.f), acc1 = make_float2(0.f, 0.f);
#pragma unroll
    for (int u = 0; u < UP; u += 2) {
      if (u < U) acc0 = cfma(Hk[static_cast<size_t>(u) * B + b], Gc[n * U + u], acc0);
      if (u + 1 < U) acc1 = cfma(Hk[static_cast<size_t>(u + 1) * B + b], Gc[n * U + u + 1], acc1);
    }
    gyk[static_cast<size_t>(n) * B + b] = cadd(acc0, acc1);
  }
}

// dL/drho_c and dL/dnu[c][u]: fixed-order sums of the per-subcarrier partials
// (block j reduces row j of P [C (1 + U)][n_sc], contiguous: with the columns of
// [n_sc][C (1 + U)] and one load at a time it took 23 us for 8192 subcarriers of 8
// clusters and 16 users).
__global__ void __launch_bounds__(256) train_reduce_kernel(const TrainParams p) {
  __shared__ float red[256];
  const int U = p.U;
  const int j = blockIdx.x;
  float acc = 0.f;
  const float* row = p.P + static_cast<size_t>(j) * p.n_sc;
  for (int k = threadIdx.x; k < p.n_sc; k += 8 * blockDim.x) {   // eight loads in flight, added in order
    float v[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const int at = k + e * blockDim.x;
      v[e] = at < p.n_sc ? row[at] : 0.f;
    }
#pragma unroll
    for (int e = 0; e < 8; ++e) acc += v[e];
  }
  red[threadIdx.x] = acc;
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    const int c = j / (1 + U), q = j % (1 + U);
    if (q == 0) p.grho[c] = red[0];
    else p.gnu[c * U + q - 1] = red[0];
  }
}

template <typename K>
cudaError_t set_smem(K kernel, size_t smem) {
  if (smem > 48 * 1024) return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                    static_cast<int>(smem));
  return cudaSuccess;
}

template <int UP, int NR>
size_t train_smem_up(int C) {
  return 16 + static_cast<size_t>(C) * TrainLayout<UP, NR>::kGroup * sizeof(float2);
}

template <int UP>
cudaError_t launch_contract_up(const TrainParams& p, cudaStream_t st) {
  const size_t smem2 = (static_cast<size_t>(p.C) * p.n_sym * p.U + static_cast<size_t>(p.C) * p.U * p.U) *
                       sizeof(float2);
  const cudaError_t e = set_smem(train_backward_contract_kernel<UP>, smem2);
  if (e != cudaSuccess) return e;
  train_backward_contract_kernel<UP><<<p.n_sc, 256, smem2, st>>>(p);
  return cudaGetLastError();
}

cudaError_t launch_contract(const TrainParams& p, cudaStream_t st) {
  switch (padded_users(p.U)) {
    case 8: return launch_contract_up<8>(p, st);
    case 16: return launch_contract_up<16>(p, st);
    default: return launch_contract_up<32>(p, st);
  }
}

template <int UP, int NR>
cudaError_t launch_forward_up(const TrainParams& p, cudaStream_t st) {
  const int threads = ((p.C * UP + 31) / 32) * 32;
  const size_t smem = train_smem_up<UP, NR>(p.C);
  cudaError_t e = set_smem(train_forward_kernel<UP, NR>, smem);
  if (e != cudaSuccess) return e;
  train_forward_kernel<UP, NR><<<p.n_sc, threads, smem, st>>>(p);
  return cudaGetLastError();
}

template <int UP, int NR>
cudaError_t launch_backward_up(const TrainParams& p, cudaStream_t st) {
  const int threads = ((p.C * UP + 31) / 32) * 32;
  const size_t smem = train_smem_up<UP, NR>(p.C);
  cudaError_t e = set_smem(train_backward_solve_kernel<UP, NR>, smem);
  if (e != cudaSuccess) return e;
  train_backward_solve_kernel<UP, NR><<<p.n_sc, threads, smem, st>>>(p);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  if ((e = launch_contract(p, st)) != cudaSuccess) return e;
  train_reduce_kernel<<<p.C * (1 + p.U), 256, 0, st>>>(p);
  return cudaGetLastError();
}

template <int UP, int NRC>
cudaError_t launch_forward_fused_up(const TrainParams& p, cudaStream_t st) {
  using Lay = FormedTrainLayout<UP, NRC>;
  const size_t smem = Lay::bytes(p.B, p.U, p.n_sym, p.C, false);
  cudaError_t e = set_smem(train_forward_fused_kernel<UP, NRC>, smem);
  if (e != cudaSuccess) return e;
  train_forward_fused_kernel<UP, NRC><<<p.n_sc, Lay::threads(p.B, p.C), smem, st>>>(p, Lay::groups(p.C));
  return cudaGetLastError();
}

template <int UP, int NRC>
cudaError_t launch_backward_fused_up(const TrainParams& p, cudaStream_t st) {
  using Lay = FormedTrainLayout<UP, NRC>;
  const size_t smem = Lay::bytes(p.B, p.U, p.n_sym, p.C, true);
  cudaError_t e = set_smem(train_backward_fused_kernel<UP, NRC>, smem);
  if (e != cudaSuccess) return e;
  train_backward_fused_kernel<UP, NRC><<<p.n_sc, Lay::threads(p.B, p.C), smem, st>>>(p, Lay::groups(p.C));
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  train_reduce_kernel<<<p.C * (1 + p.U), 256, 0, st>>>(p);
  return cudaGetLastError();
}

template <int UP, int NRC>
cudaError_t launch_optimal_fused_up(const TrainParams& p, cudaStream_t st) {
  using Lay = FormedTrainLayout<UP, NRC>;   // lane groups and threads
  const size_t smem = FormedOptimalLayout<UP, NRC>::bytes(p.B, p.U, p.n_sym, p.C);
  cudaError_t e = set_smem(train_optimal_fused_kernel<UP, NRC>, smem);
  if (e != cudaSuccess) return e;
  train_optimal_fused_kernel<UP, NRC><<<p.n_sc, Lay::threads(p.B, p.C), smem, st>>>(p, Lay::groups(p.C));
  return cudaGetLastError();
}

template <int UP, int NR>
size_t optimal_smem_up(int C) {
  return 16 + ((static_cast<size_t>(C) * UP * 4 + 15) / 16) * 16 +
         static_cast<size_t>(C) * OptimalLayout<UP, NR>::kGroup * sizeof(float2);
}

template <int UP, int NR>
cudaError_t launch_optimal_up(const TrainParams& p, cudaStream_t st) {
  const int threads = ((p.C * UP + 31) / 32) * 32;
  const size_t smem = optimal_smem_up<UP, NR>(p.C);
  cudaError_t e = set_smem(train_optimal_solve_kernel<UP, NR>, smem);
  if (e != cudaSuccess) return e;
  train_optimal_solve_kernel<UP, NR><<<p.n_sc, threads, smem, st>>>(p);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  return launch_contract(p, st);
}

}  // namespace

// Dispatch on (padded users, right-hand-side columns of the sweep).
#define FFEQ_TRAIN_DISPATCH(call)                                             \
  switch (padded_users(p.U) * 100 + rhs_columns(p.n_sym)) {                   \
    case 804: return call<8, 4>(p, st);                                       \
    case 816: return call<8, kNsymMax>(p, st);                                \
    case 1604: return call<16, 4>(p, st);                                     \
    case 1616: return call<16, kNsymMax>(p, st);                              \
    case 3204: return call<32, 4>(p, st);                                     \
    default: return call<32, kNsymMax>(p, st);                                \
  }

size_t train_smem_bytes(int U, int C) {
  // The widest form (n_sym > 4) bounds every problem with these U and C.
  switch (padded_users(U)) {
    case 8: return train_smem_up<8, kNsymMax>(C);
    case 16: return train_smem_up<16, kNsymMax>(C);
    default: return train_smem_up<32, kNsymMax>(C);
  }
}

cudaError_t launch_train_forward(const TrainParams& p, cudaStream_t st) { FFEQ_TRAIN_DISPATCH(launch_forward_up) }

cudaError_t launch_train_backward(const TrainParams& p, cudaStream_t st) { FFEQ_TRAIN_DISPATCH(launch_backward_up) }

// Dispatch of the formed kernels on (padded users, right-hand sides per lane).
#define FFEQ_FORMED_DISPATCH(call)                                            \
  switch (padded_users(p.U) * 10 + formed_rhs(p.n_sym)) {                     \
    case 81: return call<8, 1>(p, st);                                        \
    case 82: return call<8, 2>(p, st);                                        \
    case 84: return call<8, 4>(p, st);                                        \
    case 161: return call<16, 1>(p, st);                                      \
    case 162: return call<16, 2>(p, st);                                      \
    case 164: return call<16, 4>(p, st);                                      \
    case 321: return call<32, 1>(p, st);                                      \
    case 322: return call<32, 2>(p, st);                                      \
    default: return call<32, 4>(p, st);                                       \
  }

bool train_fused_fits(int U, int n_sym, int B, int C) {
  const int UP = padded_users(U), NR = 4 * formed_rhs(n_sym);
  return 16 + formed_staged_bytes(B, U + n_sym) + static_cast<size_t>(C) * NR * UP * 16 <= 227 * 1024;
}

cudaError_t launch_train_forward_fused(const TrainParams& p, cudaStream_t st) {
  FFEQ_FORMED_DISPATCH(launch_forward_fused_up)
}

cudaError_t launch_train_backward_fused(const TrainParams& p, cudaStream_t st) {
  FFEQ_FORMED_DISPATCH(launch_backward_fused_up)
}

size_t train_optimal_smem_bytes(int U, int C) {
  switch (padded_users(U)) {
    case 8: return optimal_smem_up<8, kNsymMax>(C);
    case 16: return optimal_smem_up<16, kNsymMax>(C);
    default: return optimal_smem_up<32, kNsymMax>(C);
  }
}

cudaError_t launch_train_optimal_backward(const TrainParams& p, cudaStream_t st) {
  FFEQ_TRAIN_DISPATCH(launch_optimal_up)
}

bool train_optimal_fused_fits(int U, int n_sym, int B, int C) {
  const int UP = padded_users(U), NR = 4 * formed_rhs(n_sym);
  const size_t cluster = UP * (UP + 4) * 8 + NR * UP * 16 + 2 * UP * 4;
  return 16 + formed_staged_bytes(B, U + n_sym) + C * cluster <= 227 * 1024;
}

cudaError_t launch_train_optimal_backward_fused(const TrainParams& p, cudaStream_t st) {
  FFEQ_FORMED_DISPATCH(launch_optimal_fused_up)
}

#undef FFEQ_TRAIN_DISPATCH
#undef FFEQ_FORMED_DISPATCH

}  // namespace ffeq
