// Fused equalization of FD problems in FP32 (L-MMSE and ZF): one launch from H and y
// to z, sigma^2 and LLRs.
//
// A CTA stages one subcarrier and a lane group per cluster forms [G_c + rho I |
// y_c^MRC] in registers (Sec. II-C, ffeq_formed.cuh), sweeps it (Sec. III-A) and
// leaves the cluster's fusion terms in shared memory; the CTA then fuses per user
// (Eq. fusionrule, Lemma 1; Thm. 3) and writes the outputs.  Neither the local
// Gram matrices nor the matched filters go through the workspace, and the CUDA-core
// contraction's staging, its partial sums and the second launch are gone.
// What bounds it: issue and its latencies (U = 16, C = 8, 1200 x 14: issue 56% of the
// time, FMA pipe 43%, 11 warps per SM; one symbol, 8192 x 1: 74%, 44%, 15 warps; the
// contraction and the sweep are about 60 / 40).
#include <cmath>

#include "ffeq_device.cuh"
#include "ffeq_epilogue.cuh"
#include "ffeq_formed.cuh"
#include "ffeq_internal.h"

namespace ffeq {
namespace {

constexpr int kThreads = 256;   // at most

// How a cluster's antennas are added up.  With five clusters or more, in one chain.
// With two to four, in parts, eight for the subcarrier as in the contraction launch,
// because the error of a chain grows with its antennas: rms of z against 64 bits, two
// clusters of 16 / 128 / 512 antennas, contraction launch 1.4e-7 / 1.3e-7 / 1.6e-7,
// one chain 1.7e-7 / 2.5e-7 / 4.4e-7, parts 1.3e-7 / 1.2e-7 / 1.5e-7.  A lane takes its
// parts one after another (kSerial), or each part has a lane group (kGroups).
enum Adding { kOneChain, kSerial, kGroups };

template <int UP, int NRC>
constexpr int kTileFloats = 2 * FormedShape<UP>::RPL * (FormedShape<UP>::CA + NRC);   // a lane holds

template <int UP, int NRC, Adding ADD>
struct FormedEqLayout {
  static constexpr int NR = 4 * NRC;
  static constexpr int AREA = NR * UP + UP / 2;   // float2 per cluster: numerators [NR][UP], denominators [UP]
  static constexpr int TILE = kTileFloats<UP, NRC>;
  __host__ __device__ static int parts(int C) { return ADD == kOneChain ? 1 : 8 / C; }
  __host__ __device__ static int group_parts(int C) { return ADD == kGroups ? parts(C) : 1; }
  static int groups(int C) {
    const int most = kThreads / FormedShape<UP>::GL;
    return C < most ? C : most;
  }
  // The areas take the place of the staged rows where every cluster has a lane
  // group (all tiles are formed before the first term is written): 62 instead of
  // 78 KB for B = 256, U = 16, 14 symbols, three CTAs per SM instead of two.
  __host__ __device__ static size_t areas(int B, int rows, bool at_once) {
    return 16 + (at_once ? 0 : formed_staged_bytes(B, rows));
  }
  // After them the tiles of the parts past the first ([part][cluster][TILE][GL]).
  static size_t bytes(int B, int U, int n_sym, int C) {
    const size_t rows = formed_staged_bytes(B, U + n_sym), terms = static_cast<size_t>(C) * AREA * sizeof(float2);
    const size_t tiles = static_cast<size_t>(group_parts(C) - 1) * C * TILE * FormedShape<UP>::GL * sizeof(float);
    return 16 + (groups(C) == C ? (rows > terms + tiles ? rows : terms + tiles) : rows + terms);
  }
  static int threads(int B, int C) {
    const int t = groups(C) * group_parts(C) * FormedShape<UP>::GL, w = B < 128 ? B : 128;
    return (((t > w ? t : w) + 31) / 32) * 32;
  }
};

// (Parts in one lane of eight users: 80 registers as in one chain; with more, fewer of
// the small CTAs share an SM, U = 8, C = 2, S = 63, 800 x 4: 7.7 us, 11.1 without the cap.)
template <int UP, int NRC, Adding ADD>
__global__ void __launch_bounds__(kThreads, ADD == kSerial && UP == 8 && NRC < 4 ? 3 : 2) equalize_formed_kernel(const FormedParams p, int groups) {
  extern __shared__ __align__(16) unsigned char smem[];
  using F = FormedShape<UP>;
  using Lay = FormedEqLayout<UP, NRC, ADD>;
  constexpr int NC = F::CA + NRC;
  const int U = p.s.U, NS = p.s.n_sym, C = p.s.Ceff, B = p.B, RS = formed_stride(B);
  const int k = blockIdx.x;
  const float rho = p.s.rho;
  int* failed = reinterpret_cast<int*>(smem);
  float* Ws = reinterpret_cast<float*>(smem + 16);
  const bool at_once = groups == C;
  float2* areas = reinterpret_cast<float2*>(smem + Lay::areas(B, U + NS, at_once));
  if (threadIdx.x == 0) *failed = 0;
  formed_stage(p.H + static_cast<size_t>(k) * U * B, p.y + static_cast<size_t>(k) * NS * B, U, NS, B, Ws);
  formed_wait();

  const int grp = threadIdx.x / F::GL, gl = threadIdx.x % F::GL, r = gl / 4, q = gl % 4;
  const int first = (threadIdx.x & ~31) / F::GL;   // the warp's first group
  const int parts = Lay::group_parts(C);           // more than one: groups == C, at_once
  if (first >= groups * parts) {   // whole warps without a group
    if (at_once) __syncthreads();
    if constexpr (ADD == kGroups) __syncthreads();
  } else {
    for (int c0 = 0; c0 < C; c0 += groups) {
      const int part = ADD == kGroups ? grp / groups : (grp >= groups), gc = grp - part * groups;   // part by part
      const bool live = part < parts && c0 + gc < C;
      const int c = live ? c0 + gc : 0;
      const int S = p.cl_uniform ? B / C : 0;
      int b0 = p.cl_uniform ? c * S : p.cl_off[c], b1 = p.cl_uniform ? b0 + S : p.cl_off[c + 1];
      if (ADD == kGroups && live) {
        const int n = b1 - b0, a0 = b0;
        b0 = a0 + part * n / parts;
        b1 = a0 + (part + 1) * n / parts;
      }
      const int step = ADD == kSerial ? ((b1 - b0 + Lay::parts(C) - 1) / Lay::parts(C) + 1) & ~1 : 0;
      float re[F::RPL][NC], im[F::RPL][NC], rs[F::RPL];
      formed_tile<UP, NRC, true, true, ADD == kSerial>(Ws, RS, U, NS, b0, b1, r, q, live, 0.f, re, im, step);
      if (at_once) __syncthreads();   // one pass: the staged rows are no longer read
      if constexpr (ADD == kGroups) {
        // The other parts' tiles, added in order by the lanes of the first.
        float* tiles = reinterpret_cast<float*>(areas + static_cast<size_t>(C) * Lay::AREA);
        if (live && part > 0) {
          float* t = tiles + static_cast<size_t>((part - 1) * C + c) * Lay::TILE * F::GL + gl;
#pragma unroll
          for (int i = 0; i < F::RPL; ++i)
#pragma unroll
            for (int j = 0; j < NC; ++j) {
              t[2 * (i * NC + j) * F::GL] = re[i][j];
              t[(2 * (i * NC + j) + 1) * F::GL] = im[i][j];
            }
        }
        __syncthreads();
        if (first >= C) break;   // whole warps without a cluster of their own
        for (int a = 1; a < parts && live && part == 0; ++a) {
          const float* t = tiles + static_cast<size_t>((a - 1) * C + c) * Lay::TILE * F::GL + gl;
#pragma unroll
          for (int i = 0; i < F::RPL; ++i)
#pragma unroll
            for (int j = 0; j < NC; ++j) {
              re[i][j] += t[2 * (i * NC + j) * F::GL];
              im[i][j] += t[(2 * (i * NC + j) + 1) * F::GL];
            }
        }
      }
      const bool valid = live && part == 0;
      unsigned zero_diag = 0;   // users this cluster cannot see (G_ii = 0), one bit per row of the lane
#pragma unroll
      for (int i = 0; i < F::RPL; ++i) {
        if (formed_diagonal<UP, NC>(re, i, r) == 0.f) zero_diag |= 1u << i;
#pragma unroll
        for (int j = 0; j < F::CA; ++j)
          if (q + 4 * j == r + F::RL * i && valid && r + F::RL * i < U) re[i][j] += rho;
      }
      const int fail = formed_sweep<UP, NRC, true>(re, im, U, r, q, rs);
      float2* Fz = areas + static_cast<size_t>(c) * Lay::AREA;
      float* Dn = reinterpret_cast<float*>(Fz + Lay::NR * UP);
#pragma unroll
      for (int i = 0; i < F::RPL; ++i) {
        const int u = r + F::RL * i;
        const float Ai = __shfl_sync(kFullMask, formed_diagonal<UP, NC>(re, i, r) * rs[i], 4 * r + (r & 3), F::GL);
        const float invA = rcp_approx(Ai);
        if (valid && q == (r & 3)) {
          // mu = [A G]_ii = 1 - rho A_ii; a user the cluster cannot see (G_ii = 0) has
          // mu = 0 exactly, which the subtraction would only reach up to rounding.
          const float mu = (zero_diag >> i) & 1u ? 0.f : fmaxf(1.f - rho * Ai, 0.f);
          Dn[u] = (p.s.unbiased ? mu : 1.f) * invA;
        }
#pragma unroll
        for (int j = 0; j < NRC; ++j) {
          const int n = q + 4 * j;
          if (valid && n < NS)
            Fz[n * UP + u] = make_float2(re[i][F::CA + j] * rs[i] * invA, im[i][F::CA + j] * rs[i] * invA);
        }
      }
      if (valid && gl == 0) {
        if (p.s.info) p.s.info[static_cast<size_t>(k) * C + c] = fail;
        if (fail) atomicOr(failed, 1);
      }
    }
  }
  __syncthreads();
  const bool bad = *failed != 0;
  const int bits = p.s.llr_bits, hb = bits / 2;
  for (int e = threadIdx.x; e < UP * NS; e += blockDim.x) {
    const int n = e / UP, u = e % UP;
    if (u >= U) continue;
    float2 nm = make_float2(0.f, 0.f);
    float dn = 0.f;
    for (int c = 0; c < C; ++c) {
      nm = cadd(nm, areas[c * Lay::AREA + e]);
      dn += reinterpret_cast<const float*>(areas + c * Lay::AREA + Lay::NR * UP)[u];
    }
    float2 zz;
    float s2;
    if (bad) {
      zz = make_float2(NAN, NAN);
      s2 = NAN;
    } else if (dn > 0.f) {
      const float rr = rcp_approx(dn);
      zz = cscale(nm, rr);
      s2 = p.s.N0 * rr;
    } else {
      zz = make_float2(0.f, 0.f);
      s2 = INFINITY;
    }
    const size_t zi = (static_cast<size_t>(k) * NS + n) * U + u;
    p.s.z[zi] = zz;
    if (n == 0) p.s.sigma2[static_cast<size_t>(k) * U + u] = s2;
    if (bits) symbol_llr_wide(zz, s2, p.s.llr_scale, hb, p.s.llr + zi * bits);
  }
}

template <int UP, int NRC, Adding ADD>
cudaError_t launch_up(const FormedParams& p, cudaStream_t stream) {
  using Lay = FormedEqLayout<UP, NRC, ADD>;
  const int C = p.s.Ceff;
  const size_t smem = Lay::bytes(p.B, p.s.U, p.s.n_sym, C);
  static int configured[64] = {0};
  int dev = 0;
  cudaError_t err = cudaGetDevice(&dev);
  if (err != cudaSuccess) return err;
  if (dev < 64 && !configured[dev]) {
    err = cudaFuncSetAttribute(equalize_formed_kernel<UP, NRC, ADD>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               227 * 1024);
    if (err != cudaSuccess) return err;
    configured[dev] = 1;
  }
  equalize_formed_kernel<UP, NRC, ADD><<<p.s.n_sc, Lay::threads(p.B, C), smem, stream>>>(p, Lay::groups(C));
  return cudaGetLastError();
}

// Parts in one lane where the sums fit its registers beside the part's tile (U = 16,
// C = 2, S = 128, 1200 x 14: 91 us, groups 53) and its chains are short; groups where a
// cluster has many antennas (U = 4, C = 2, 1200 x 1: S = 128 14.8 us, groups 12.1; S =
// 16, 2000 x 1 5.7, groups 12.1) or an SM has at most two subcarriers (64 x 1: 3.9, 3.4).
template <int UP, int NRC>
cudaError_t launch_adding(const FormedParams& p, cudaStream_t stream) {
  if (p.s.Ceff > 4) return launch_up<UP, NRC, kOneChain>(p, stream);
  if constexpr (kTileFloats<UP, NRC> <= 48) {
    if (p.B < 64 * p.s.Ceff && p.s.n_sc > 2 * kSms) return launch_up<UP, NRC, kSerial>(p, stream);
  }
  return launch_up<UP, NRC, kGroups>(p, stream);
}

template <int UP>
cudaError_t launch_nrc(const FormedParams& p, cudaStream_t stream) {
  if (p.s.n_sym <= 4) return launch_adding<UP, 1>(p, stream);
  if (p.s.n_sym <= 8) return launch_adding<UP, 2>(p, stream);
  return launch_adding<UP, 4>(p, stream);
}

}  // namespace

// Measured against the contraction and solve launches (us a call, captured; before ->
// after): U = 4, C = 2, S = 16, 2000 x 1: 36.1 -> 5.8; U = 8, C = 16, 3000 x 2: 110 -> 43;
// U = 15, C = 3, S = 85, 1200 x 14: 126 -> 62; U = 16, C = 8, S = 32, 1200 x 14: 63.0 -> 59.2;
// U = 32, C = 4, 1000 x 7: 160 -> 118.  Tiles of 32 users with 16 right-hand sides spill
// registers and keep the separate launches (C = 16, 3300 x 14: 823 -> 1017), as do two
// clusters of 24 users (1200 x 7: 101 -> 124).  Two to four clusters with few warps per CTA
// were left out before their antennas were added in parts; with parts some of them would
// gain (U = 16, C = 2, 64 x 14: 15.0 -> 11.4; U = 32, C = 2, 1200 x 4: 138 -> 111).
//
// TF32x3 and FP16x3 problems run here too where the tensor-core contraction and
// the solve measured slower (FP32 is at least as accurate: every product rounds
// once to 24 bits, and nothing is split).  BF16x3 does not: its results are its own.
//   TF32x3: U = 16, C = 8, 1200 x 3: 54 -> 30; 1200 x 7: 57 -> 38; U = 10, 1200 x 14: 67 -> 44;
//   U = 32, C = 8, 1200 x 3: 176 -> 130; left out by an earlier measurement that a captured
//   one does not bear out: U = 14, C = 5, B = 250, 600 x 14 (37.6 -> 33.4).
//   FP16x3: U = 12, C = 16, 800 x 8: 56 -> 35; U = 5, C = 2, 300 x 7: 23 -> 6; U = 11, C = 5,
//   B = 120, 625 x 13: 31 -> 21; U = 16, C = 8, 1200 x 8: 39.8 -> 39.2; not 1200 x 14 (44 -> 59),
//   nor U = 20, C = 4, 600 x 4 (37 -> 49).
// 260 random FD problems against shapes 1, 2 and 5: no problem taken here was faster there.
bool equalize_formed_fits(int precision, int B, int U, int n_sym, int C, int n_sc) {
  if (C < 2 || (U > 16 && (n_sym > 8 || C < 4))) return false;
  if (U > 8 && n_sym > 8 && C < 4 && n_sc < 2 * kSms) return false;
  if (precision == FFEQ_TF32X3) {
    if (U > 16 ? n_sym > 4 : (U > 12 && n_sym > 8 && B > 128)) return false;
  } else if (precision == FFEQ_FP16X3) {
    if (U > 16 || (n_sym > 8 && B > 128) || (U > 8 && C < 4)) return false;
  } else if (precision != FFEQ_FP32) {
    return false;
  }
  const int UP = padded_users(U), NRC = n_sym <= 4 ? 1 : (n_sym <= 8 ? 2 : 4);
  return 16 + formed_staged_bytes(B, U + n_sym) + static_cast<size_t>(C) * (4 * NRC * UP + UP / 2) * 8 <= 227 * 1024;   // bytes() at most (tiles: 41 KB)
}

cudaError_t launch_equalize_formed(const FormedParams& p, cudaStream_t stream) {
  switch (padded_users(p.s.U)) {
    case 8: return launch_nrc<8>(p, stream);
    case 16: return launch_nrc<16>(p, stream);
    default: return launch_nrc<32>(p, stream);
  }
}

}  // namespace ffeq
