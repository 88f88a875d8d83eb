// Register-tiled Gauss-Jordan sweep of the solve kernels (numbers of users that
// fill no lane group; ffeq_gj.cuh holds the row sweeps of the others).
//
// A group of lanes holds one Hermitian positive definite system [M | R] of UP
// users (a multiple of 8) and up to 4 NRC right-hand sides as register tiles:
// lane (r, q) owns rows 4r .. 4r+3 and, of those, matrix columns CA q .. CA q +
// CA - 1 (CA = UP / 4) and right-hand sides NRC q .. NRC q + NRC - 1.  Step k
// fetches the pivot row (from its four lanes) and the pivot column (from its
// UP / 4 lanes) by warp shuffles, and every lane applies the rank-one update to
// its tile.  The right-hand sides ride along as columns (as many operations as
// A times R afterwards), so that no lane needs a whole row of the inverse, and
// the width follows n_sym (4, 8 or 16).
//
// Why tiles.  A row per lane needs UP lanes with UP columns each for any U, so
// 17 users cost as much as 32; tiles come in steps of 8 users.  A lane fetches
// CA + NRC entries of the row and 4 of the column for 4 (CA + NRC) updates
// instead of one per update.  What bounds it: the FMA pipe (57% busy) and issue
// (55%), a paired FMA taking two cycles of the pipe (52,800 systems of 32 users
// and 14 symbols: 550 us).
//
// Arithmetic: the deferred-scaling elimination.  The pivot row is broadcast
// unscaled, its pivot entry replaced by 1 (the identity column it turns into),
// every other row does new = base - g q with g = f / p_k (f its entry in the
// pivot column, base 0 there), and the pivot row keeps its values.  A row that
// has been the pivot row is thereby stored times its pivot; the caller scales
// the entries it uses by 1 / p_i (`rs`).
#pragma once

#include "ffeq_device.cuh"

namespace ffeq {

template <int UP, int NRC>
struct TileShape {
  static_assert(UP % 8 == 0 && UP <= 32 && NRC >= 1 && NRC <= 4, "tile shapes");
  static constexpr int CA = UP / 4;                       // matrix columns per lane
  static constexpr int NC = CA + NRC;                     // columns per lane
  static constexpr int GL = UP == 24 ? 32 : UP;           // lanes per system (24 users: 8 lanes of a warp idle)
  static constexpr int UN = UP == 24 ? 12 : (CA < 4 ? 4 : CA);   // steps per trip: whole row and column owners
};
// Floats of shared memory a system's solve needs (1 / A_ii of its users).
constexpr int tile_smem_floats(int UP) { return UP; }

// new = base - g q on a row of N columns (g = (gr, gi), two columns per paired FMA).
template <int N>
__device__ __forceinline__ void tile_row_update(float (&re)[N], float (&im)[N], const float (&qr)[N],
                                                const float (&qi)[N], float gr, float gi) {
  const float2 nr = make_float2(-gr, -gr), pi = make_float2(gi, gi), ni = make_float2(-gi, -gi);
#pragma unroll
  for (int c = 0; c + 1 < N; c += 2) {
    const float2 a = make_float2(qr[c], qr[c + 1]), b = make_float2(qi[c], qi[c + 1]);
    float2 x = __ffma2_rn(nr, a, make_float2(re[c], re[c + 1]));
    x = __ffma2_rn(pi, b, x);
    float2 y = __ffma2_rn(nr, b, make_float2(im[c], im[c + 1]));
    y = __ffma2_rn(ni, a, y);
    re[c] = x.x;
    re[c + 1] = x.y;
    im[c] = y.x;
    im[c + 1] = y.y;
  }
  if constexpr (N % 2 == 1) {
    constexpr int c = N - 1;
    re[c] = fmaf(gi, qi[c], fmaf(-gr, qr[c], re[c]));
    im[c] = fmaf(-gi, qr[c], fmaf(-gr, qi[c], im[c]));
  }
}

// The sweep.  re[i][c], im[i][c]: row 4r + i, column c of the lane (matrix
// columns first).  Returns the 1-based index of the first pivot that is not
// positive, or 0; rs[i] = 1 / p of row 4r + i.  Every lane of the warp must take
// part (lanes past a 24-user group hold copies and change nothing else).
template <int UP, int NRC>
__device__ __forceinline__ int tile_sweep(float (&re)[4][UP / 4 + NRC], float (&im)[4][UP / 4 + NRC], int U, int r,
                                          int q, float (&rs)[4]) {
  using T = TileShape<UP, NRC>;
  constexpr int CA = T::CA, NC = T::NC, UN = T::UN, GL = T::GL;
  int fail = 0;
#pragma unroll
  for (int i = 0; i < 4; ++i) rs[i] = 1.f;
#pragma unroll 1
  for (int t = 0; t < UP / UN && UN * t < U; ++t) {   // padding pivots change nothing
    static_for<UN>([&](auto sc) {
      constexpr int s = decltype(sc)::value;
      constexpr int I = s % 4, JC = s % CA;                    // the pivot's row and column in its tile
      const int kr = (UN / 4) * t + s / 4, kc = (UN / CA) * t + s / CA;
      const bool rowk = r == kr, colk = q == kc;
      // The pivot row, its pivot entry replaced by 1.
      float qr[NC], qi[NC];
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        qr[c] = __shfl_sync(kFullMask, re[I][c], 4 * kr + q, GL);
        qi[c] = __shfl_sync(kFullMask, im[I][c], 4 * kr + q, GL);
      }
      const float piv = __shfl_sync(kFullMask, re[I][JC], 4 * kr + kc, GL);
      const bool ok = piv > 0.f;
      if (!ok && fail == 0) fail = UN * t + s + 1;
      const float rc = rcp_approx(ok ? piv : 1.f);
      if (colk) {
        qr[JC] = 1.f;
        qi[JC] = 0.f;
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        float sc2 = rc;
        const float fr = __shfl_sync(kFullMask, re[i][JC], 4 * r + kc, GL);
        const float fi = __shfl_sync(kFullMask, im[i][JC], 4 * r + kc, GL);
        if (i == I && rowk) {   // the pivot row keeps its values
          sc2 = 0.f;
          rs[i] = rc;
        }
        if (colk) {             // the pivot column turns into the identity column
          re[i][JC] = (i == I && rowk) ? 1.f : 0.f;
          im[i][JC] = 0.f;
        }
        tile_row_update<NC>(re[i], im[i], qr, qi, fr * sc2, fi * sc2);
      }
    });
  }
  return fail;
}

// One local system on its lane group (lane (r, q)): loads its tile of [G + rho I |
// y^MRC] from D (row stride U), runs the sweep and leaves the fusion terms in the
// system's shared area, numerators z_{c,u}(n) / A_uu in Fz [n][UP] and
// denominators g_{c,u} / A_uu (g = mu or 1) in Dn; or (Xs != nullptr: refinement
// follows) writes the estimates Xs [n][U] and the inverse As [j][i] = A[i][j] to
// global memory.  A group without a system (valid = false) sweeps an identity;
// nothing is left where `writer` is false, and cond is the condition estimate
// ||G + rho I||_1 ||A||_1.  Every lane of the warp takes part;
// returns the sweep's failure index.
template <int UP, int NRC>
__device__ __forceinline__ int tile_solve_system(const float2* __restrict__ Dg, int U, int NS, float rho, bool unbiased,
                                                 bool valid, bool writer, int r, int q, float* buf,
                                                 float2* Fz, float* Dn, float2* Xs, float2* As,
                                                 float& cond) {
  constexpr int CA = UP / 4, NC = CA + NRC;
  float re[4][NC], im[4][NC];
  const int row0 = 4 * r;
  // Columns of D are rows of the system: a lane's four rows are 32 contiguous
  // bytes of each row of D (two 16-byte loads where U is even).
  const bool vec = (U & 1) == 0 && (reinterpret_cast<uintptr_t>(Dg) & 15) == 0;
#pragma unroll
  for (int c = 0; c < NC; ++c) {
    const int col = c < CA ? CA * q + c : NRC * q + (c - CA);
    const bool live = valid && (c < CA ? col < U : col < NS);
    const float2* src = Dg + (c < CA ? col : U + col) * U + row0;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
      if (vec) {
        if (live && row0 + 2 * h < U) v = *reinterpret_cast<const float4*>(src + 2 * h);
      } else if (live) {
        if (row0 + 2 * h < U) {
          const float2 a = src[2 * h];
          v.x = a.x;
          v.y = a.y;
        }
        if (row0 + 2 * h + 1 < U) {
          const float2 a = src[2 * h + 1];
          v.z = a.x;
          v.w = a.y;
        }
      }
      re[2 * h][c] = v.x;
      im[2 * h][c] = v.y;
      re[2 * h + 1][c] = v.z;
      im[2 * h + 1][c] = v.w;
    }
  }
  // The diagonal: G_ii + rho, real; 1 in padding rows.
  unsigned zero_diag = 0;   // users this system cannot see (G_ii = 0), one bit per row of the lane
#pragma unroll
  for (int j = 0; j < CA; ++j) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      if (CA * q + j == row0 + i) {
        if (re[i][j] == 0.f) zero_diag |= 1u << i;
        re[i][j] = (valid && row0 + i < U) ? re[i][j] + rho : 1.f;
        im[i][j] = 0.f;
      }
    }
  }
  constexpr int GL = TileShape<UP, NRC>::GL;
  // max over the group of the rows' absolute sums (rows scaled by s): the 1-norm
  // of a Hermitian matrix.
  auto norm1 = [&](const float (&s)[4]) {
    float most = 0.f;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      float sum = 0.f;
#pragma unroll
      for (int j = 0; j < CA; ++j)
        if (CA * q + j < U && row0 + i < U) sum += sqrt_approx(fmaf(re[i][j], re[i][j], im[i][j] * im[i][j]));
      sum += __shfl_xor_sync(kFullMask, sum, 1);
      sum += __shfl_xor_sync(kFullMask, sum, 2);
      most = fmaxf(most, sum * fabsf(s[i]));
    }
#pragma unroll
    for (int o = GL / 2; o >= 4; o >>= 1) most = fmaxf(most, __shfl_xor_sync(kFullMask, most, o));
    return most;
  };
  float rs[4] = {1.f, 1.f, 1.f, 1.f};
  if (Xs) cond = norm1(rs);
  const int fail = tile_sweep<UP, NRC>(re, im, U, r, q, rs);
  if (Xs) {
    cond *= norm1(rs);
    if (valid && writer) {
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        if (row0 + i < U) {
#pragma unroll
          for (int j = 0; j < NRC; ++j)
            if (NRC * q + j < NS)
              Xs[(NRC * q + j) * U + row0 + i] =
                  make_float2(re[i][CA + j] * rs[i], im[i][CA + j] * rs[i]);
#pragma unroll
          for (int j = 0; j < CA; ++j)
            if (CA * q + j < U)
              As[(CA * q + j) * U + row0 + i] = make_float2(re[i][j] * rs[i], im[i][j] * rs[i]);
        }
      }
    }
    return fail;
  }
  // 1 / A_ii and the denominators, by the lanes that hold the diagonal, then the
  // numerators of every lane's rows ([n][u]: the epilogue reads along u).
#pragma unroll
  for (int j = 0; j < CA; ++j) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      if (CA * q + j == row0 + i && writer) {
        const float Ai = re[i][j] * rs[i];
        const float invA = rcp_approx(Ai);
        // mu = [A G]_ii = 1 - rho A_ii; a user the cluster cannot see (G_ii = 0) has
        // mu = 0 exactly, which the subtraction would only reach up to rounding.
        const float mu = (zero_diag >> i) & 1u ? 0.f : fmaxf(1.f - rho * Ai, 0.f);
        buf[row0 + i] = invA;
        Dn[row0 + i] = (unbiased ? mu : 1.f) * invA;
      }
    }
  }
  __syncwarp();
  const float4 ia = *reinterpret_cast<const float4*>(buf + row0);
  const float invA[4] = {ia.x, ia.y, ia.z, ia.w};
  if (writer) {
#pragma unroll
    for (int j = 0; j < NRC; ++j) {
      if (NRC * q + j < NS) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          float4 v;
          v.x = re[2 * h][CA + j] * rs[2 * h] * invA[2 * h];
          v.y = im[2 * h][CA + j] * rs[2 * h] * invA[2 * h];
          v.z = re[2 * h + 1][CA + j] * rs[2 * h + 1] * invA[2 * h + 1];
          v.w = im[2 * h + 1][CA + j] * rs[2 * h + 1] * invA[2 * h + 1];
          *reinterpret_cast<float4*>(Fz + (NRC * q + j) * UP + row0 + 2 * h) = v;
        }
      }
    }
  }
  __syncwarp();   // buf may be reused
  return fail;
}

}  // namespace ffeq
