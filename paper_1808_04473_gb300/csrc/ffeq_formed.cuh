// Local systems formed in registers from staged inputs, and their sweep: the
// device code shared by the kernels that go from H and Y to solved systems in one
// launch (FP32: training and its adjoints, the fused FP32 equalization).
//
// A CTA stages the U + n_sym rows of a subcarrier in shared memory in their
// natural layout (row = user or symbol, B antennas of interleaved complex, a
// stride of formed_stride(B) floats), and a group of GL lanes forms one
// cluster's system [G_c + rho I | B_c] as register tiles: lane (r, q) holds rows
// r + RL i and columns q + 4 j (then right-hand sides q + 4 j).
//
// Why this layout.  With one row per lane and antenna-major staging, every lane
// read a whole staged row per antenna: 8 bytes of shared memory per complex
// update, where an SM returns 128 bytes per clock to 128 FMA lanes (4 FMAs per
// update), so the loads bound the kernels at 87% of the shared-memory pipe.  A 4 x 5
// tile (16 users, 1 symbol) reads 9 values for 20 updates, 3.6 bytes each.  The
// cyclic rows and the stride (4 floats past a multiple of 32) put the rows one
// load phase reads in different banks, and natural rows stage with 16-byte
// copies (4-byte ones before, to turn the rows around).  Measured on 8192
// subcarriers, B = 128, U = 16, C = 8, one symbol (before -> after): training step
// 407 -> 297 us (forward 175 -> 131, backward 211 -> 155; 282 in all with HALF below),
// optimal adjoint 352 -> 292.  What bounds them now: issue (68-74%), FMA pipe 40-48%,
// 16 warps per SM.
//
// Scalar FMAs: a paired FMA takes two cycles of the pipe (67 against 68 TFLOP/s
// measured), so where the pipe is the limit the scalar form costs nothing and
// needs no duplicated or negated operands.
#pragma once

#include "ffeq_device.cuh"

namespace ffeq {

template <int UP>
struct FormedShape {
  static_assert(UP == 8 || UP == 16 || UP == 32, "padded users");
  static constexpr int RL = UP <= 16 ? 4 : 8;   // row lanes
  static constexpr int RPL = UP / RL;           // rows per lane
  static constexpr int CA = UP / 4;             // matrix columns per lane
  static constexpr int GL = 4 * RL;             // lanes per system
};

// Row stride in floats: a multiple of 4 (16-byte rows), 4 past a multiple of 32.
__host__ __device__ inline int formed_stride(int B) { return ((2 * B + 31) / 32) * 32 + 4; }
__host__ __device__ inline size_t formed_staged_bytes(int B, int rows) {
  return static_cast<size_t>(rows) * formed_stride(B) * sizeof(float);
}

// Copy rows H_k [U][B], Y_k [NS][B] to Ws (every thread of the CTA): 16-byte
// asynchronous copies where B and both addresses allow, else 8-byte ones.
// Completed and made visible by formed_wait.
__device__ __forceinline__ void formed_stage(const float2* Hk, const float2* Yk, int U, int NS, int B, float* Ws) {
  const int RS = formed_stride(B), rows = U + NS;
  const uint32_t dst0 = smem_u32(Ws);
  const bool wide = (B & 1) == 0 && ((reinterpret_cast<uintptr_t>(Hk) | reinterpret_cast<uintptr_t>(Yk)) & 15) == 0;
  const int w = wide ? 2 : 1;                  // antennas per copy
  const int per = B / w;
  // (row, piece) advances by blockDim pieces without a division per copy.
  int row = threadIdx.x / per, e = threadIdx.x - row * per;
  const int drow = blockDim.x / per, de = blockDim.x - drow * per;
  while (row < rows) {
    const float2* src = (row < U ? Hk + static_cast<size_t>(row) * B : Yk + static_cast<size_t>(row - U) * B) + e * w;
    const uint32_t dst = dst0 + 4u * static_cast<uint32_t>(row * RS + 2 * w * e);
    if (wide)
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
    else
      asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(dst), "l"(src) : "memory");
    row += drow;
    e += de;
    if (e >= per) {
      e -= per;
      ++row;
    }
  }
  asm volatile("cp.async.commit_group;" ::: "memory");
}

__device__ __forceinline__ void formed_wait() {
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();
}

// This lane's tile of [G_c + rho I | B_c] over antennas [b0, b1) of the staged
// rows: re/im[i][j] = sum_b conj(H[r + RL i][b]) W[col][b], columns j < CA users,
// then (WITH_Y) NRC symbols, in antenna order.  Padding rows and columns are
// identity; a lane of an invalid group holds an identity system.  Every lane of
// the warp takes part.  G_c is Hermitian, so with four row lanes the entries right
// of the tile diagonal come from lane (q, r): HALF takes their conjugates, whose
// imaginary parts add the two products of an antenna in the other order; otherwise
// only the real parts (the same bits).  The training pair does the latter, so that
// its X and G_b keep their bits: the gradient of the regularizers cancels 25- to
// 45-fold over the subcarriers, and another rounding of the ill-conditioned solves
// moves it by a few 1e-6 either way.  PARTS: every `part` antennas (even) are added up
// by themselves first.
template <int UP, int NRC, bool WITH_Y, bool HALF, bool PARTS = false>
__device__ __forceinline__ void formed_tile(const float* Ws, int RS, int U, int NS, int b0, int b1, int r, int q,
                                            bool valid, float rho,
                                            float (&re)[FormedShape<UP>::RPL][FormedShape<UP>::CA + NRC],
                                            float (&im)[FormedShape<UP>::RPL][FormedShape<UP>::CA + NRC],
                                            int part = 0) {
  using F = FormedShape<UP>;
  constexpr int NC = F::CA + NRC, MC = WITH_Y ? NC : F::CA;
  const float* rowp[F::RPL];
  const float* colp[MC];
#pragma unroll
  for (int i = 0; i < F::RPL; ++i) {
    const int u = r + F::RL * i;
    rowp[i] = Ws + (u < U ? u : 0) * RS;
  }
#pragma unroll
  for (int j = 0; j < MC; ++j) {
    const int c = j < F::CA ? q + 4 * j : q + 4 * (j - F::CA);
    colp[j] = Ws + (j < F::CA ? (c < U ? c : 0) : (c < NS ? U + c : 0)) * RS;
  }
#pragma unroll
  for (int i = 0; i < F::RPL; ++i)
#pragma unroll
    for (int j = 0; j < NC; ++j) re[i][j] = im[i][j] = 0.f;
  constexpr bool kHalf = F::RL == 4;
  float pr[F::RPL][NC], pi[F::RPL][NC];   // PARTS: the part's sums
  auto& ar = PARTS ? pr : re;
  auto& ai = PARTS ? pi : im;
  auto acc = [&](int i, int j, float hr, float hi, float wr, float wi) {   // conj(h) w
    const bool far = kHalf && j < F::CA && j > i;
    if (HALF && far) return;
    if (!far) {
      ar[i][j] = fmaf(hr, wr, ar[i][j]);
      ar[i][j] = fmaf(hi, wi, ar[i][j]);
    }
    ai[i][j] = fmaf(hr, wi, ai[i][j]);
    ai[i][j] = fmaf(-hi, wr, ai[i][j]);
  };
  auto single = [&](int b) {
    float2 h[F::RPL];
#pragma unroll
    for (int i = 0; i < F::RPL; ++i) h[i] = *reinterpret_cast<const float2*>(rowp[i] + 2 * b);
#pragma unroll
    for (int j = 0; j < MC; ++j) {
      const float2 w = *reinterpret_cast<const float2*>(colp[j] + 2 * b);
#pragma unroll
      for (int i = 0; i < F::RPL; ++i) acc(i, j, h[i].x, h[i].y, w.x, w.y);
    }
  };
  auto pair = [&](int b) {   // two antennas per 16-byte load
    float4 h[F::RPL];
#pragma unroll
    for (int i = 0; i < F::RPL; ++i) h[i] = *reinterpret_cast<const float4*>(rowp[i] + 2 * b);
#pragma unroll
    for (int j = 0; j < MC; ++j) {
      const float4 w = *reinterpret_cast<const float4*>(colp[j] + 2 * b);
#pragma unroll
      for (int i = 0; i < F::RPL; ++i) {
        acc(i, j, h[i].x, h[i].y, w.x, w.y);
        acc(i, j, h[i].z, h[i].w, w.z, w.w);
      }
    }
  };
  int b = b0;
  const int b_end = valid ? b1 : b0;
  do {
    const int be = PARTS ? min((b + part) & ~1, b_end) : b_end;
    if constexpr (PARTS) {
#pragma unroll
      for (int i = 0; i < F::RPL; ++i)
#pragma unroll
        for (int j = 0; j < NC; ++j) pr[i][j] = pi[i][j] = 0.f;
    }
    if ((b & 1) && b < be) single(b++);
    if constexpr (PARTS && NRC == 1) {
#pragma unroll 2
      for (; b + 1 < be; b += 2) pair(b);   // (a part is a few pairs)
    } else {
      for (; b + 1 < be; b += 2) pair(b);
    }
    if (b < be) single(b++);
    if constexpr (PARTS) {
#pragma unroll
      for (int i = 0; i < F::RPL; ++i)
#pragma unroll
        for (int j = 0; j < MC; ++j) {
          re[i][j] += pr[i][j];
          im[i][j] += pi[i][j];
        }
    }
  } while (PARTS && b < b_end);
  if constexpr (kHalf) {
#pragma unroll
    for (int i = 0; i < F::RPL; ++i) {
#pragma unroll
      for (int j = i + 1; j < F::CA; ++j) {
        re[i][j] = __shfl_sync(kFullMask, re[j][i], 4 * q + r, F::GL);
        if (HALF) im[i][j] = -__shfl_sync(kFullMask, im[j][i], 4 * q + r, F::GL);
      }
    }
  }
#pragma unroll
  for (int i = 0; i < F::RPL; ++i) {
    const int u = r + F::RL * i;
#pragma unroll
    for (int j = 0; j < F::CA; ++j) {
      const int c = q + 4 * j;
      if (!valid || u >= U || c >= U) {
        re[i][j] = u == c ? 1.f : 0.f;
        im[i][j] = 0.f;
      } else if (u == c) {
        re[i][j] += rho;
        im[i][j] = 0.f;
      }
    }
#pragma unroll
    for (int j = F::CA; j < MC; ++j)
      if (!valid || u >= U || q + 4 * (j - F::CA) >= NS) re[i][j] = im[i][j] = 0.f;
  }
}

// Diagonal entry of tile row i (row r + RL i): held by lane q = r % 4 of row lane r.
template <int UP, int NC>
__device__ __forceinline__ float formed_diagonal(const float (&re)[FormedShape<UP>::RPL][NC], int i, int r) {
  if constexpr (FormedShape<UP>::RL == 4) return re[i][i];
  else return r < 4 ? re[i][2 * i] : re[i][2 * i + 1];
}

// Deferred-scaling Gauss-Jordan sweep on the tiles, pivot row and column fetched
// by warp shuffles: at step k every row but the pivot's does new = base - g q, g =
// f / p_k (f its entry in the pivot column, q the unscaled pivot row); a row that
// has been the pivot row stays multiplied by its pivot, and the caller scales the
// entries it uses by rs[i] = 1 / p.  INV: the pivot column turns into the identity
// column it eliminates, so that the matrix block becomes the inverse.  Without it
// only the right-hand sides are wanted, and the columns already eliminated are
// left alone (half of the matrix updates).  Returns the 1-based index of the
// first pivot that is not positive, or 0.  Every lane of the warp takes part.
template <int UP, int NRC, bool INV>
__device__ __forceinline__ int formed_sweep(float (&re)[FormedShape<UP>::RPL][FormedShape<UP>::CA + NRC],
                                            float (&im)[FormedShape<UP>::RPL][FormedShape<UP>::CA + NRC], int U, int r,
                                            int q, float (&rs)[FormedShape<UP>::RPL]) {
  using F = FormedShape<UP>;
  constexpr int NC = F::CA + NRC;
  int fail = 0;
#pragma unroll
  for (int i = 0; i < F::RPL; ++i) rs[i] = 1.f;
  static_for<F::CA>([&](auto jc) {
    constexpr int J = decltype(jc)::value, I = 4 * J / F::RL, C0 = INV ? 0 : J;
#pragma unroll 1
    for (int s = 0; s < 4; ++s) {
      if (4 * J + s >= U) break;                             // padding pivots change nothing
      const int kr = (4 * J) % F::RL + s;                    // row lane of pivot 4J + s (its column lane is s)
      const bool rowk = r == kr, colk = q == s;
      float qr[NC], qi[NC];
#pragma unroll
      for (int c = C0; c < NC; ++c) {
        qr[c] = __shfl_sync(kFullMask, re[I][c], 4 * kr + q, F::GL);
        qi[c] = __shfl_sync(kFullMask, im[I][c], 4 * kr + q, F::GL);
      }
      const float piv = __shfl_sync(kFullMask, re[I][J], 4 * kr + s, F::GL);
      const bool ok = piv > 0.f;
      if (!ok && fail == 0) fail = 4 * J + s + 1;
      const float rc = rcp_approx(ok ? piv : 1.f);
      if (INV && colk) {
        qr[J] = 1.f;
        qi[J] = 0.f;
      }
#pragma unroll
      for (int i = 0; i < F::RPL; ++i) {
        float gr = __shfl_sync(kFullMask, re[i][J], 4 * r + s, F::GL) * rc;
        float gi = __shfl_sync(kFullMask, im[i][J], 4 * r + s, F::GL) * rc;
        const bool me = i == I && rowk;                      // the pivot row keeps its values
        if (me) {
          gr = gi = 0.f;
          rs[i] = rc;
        }
        if (INV && colk) {
          re[i][J] = me ? 1.f : 0.f;
          im[i][J] = 0.f;
        }
#pragma unroll
        for (int c = C0; c < NC; ++c) {
          re[i][c] = fmaf(-gr, qr[c], re[i][c]);
          re[i][c] = fmaf(gi, qi[c], re[i][c]);
          im[i][c] = fmaf(-gr, qi[c], im[i][c]);
          im[i][c] = fmaf(-gi, qr[c], im[i][c]);
        }
      }
    }
  });
  return fail;
}

}  // namespace ffeq
