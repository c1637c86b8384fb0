// The blocked inverse (I + A)^-1 of a unit lower triangular 128 x 128 matrix by eight warps, shared by the GDN and KDA
// chunk-local kernels (operator #3 of the paper's pipeline).  A is in shared memory: 16 x 16 blocks below the diagonal as fp16 B operands (16 bytes per lane, off_block
// order), the diagonal blocks in fp32.  T = (I + A)^-1 is kept as fp16 blocks of four row-major 8 x 8 matrices (128 bytes
// each, tri_block order), which ldmatrix reads as any operand.
#pragma once

#include "tc_common.cuh"
#include "tc_mma.cuh"

namespace ha_la {
namespace solve {

using namespace ptx;

constexpr int LDD = 20;                                     // row stride (floats) of a 16 x 16 diagonal block of A
constexpr __host__ __device__ int off_block(int I, int J) { return I * (I - 1) / 2 + J; }   // J < I

// Inverse of one 16 x 16 diagonal block I + A_ii by one warp; A_ii in fp32 at sd ([16][LDD]); the result goes to block tb:
//   [[X11, 0], [-X22 A21 X11, X22]],  X11, X22 by forward substitution (16 lanes: half, column), the rest by two products.
__device__ __forceinline__ void invert_diagonal(const float* sd, uint32_t tb, int lane) {
  const int g = lane >> 2, t2 = (lane & 3) * 2;
  const float2 f21 = *reinterpret_cast<const float2*>(sd + (8 + g) * LDD + t2);
  if (lane < 16) {
    const int hb = lane >> 3, c = lane & 7;
    const float* a = sd + hb * 8 * LDD + hb * 8;
    const uint32_t dst = tb + hb * 3 * 128 + c * 2;
    float y[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      float s0 = q == c ? 1.f : 0.f, s1 = 0.f;
#pragma unroll
      for (int r = 0; r < q; ++r) {
        if (r & 1) s1 = fmaf(-a[q * LDD + r], y[r], s1);
        else s0 = fmaf(-a[q * LDD + r], y[r], s0);
      }
      y[q] = s0 + s1;
      sts_u16(dst + q * 16, __half_as_ushort(__float2half_rn(y[q])));
    }
  } else if (lane < 24) {
    const uint32_t z[4] = {0u, 0u, 0u, 0u};
    sts4(tb + 128 + (lane & 7) * 16, z);                 // the quarter above the diagonal
  }
  __syncwarp();
  uint32_t x11t, x22;
  ldsm1t(x11t, tb + (lane & 7) * 16);
  ldsm1(x22, tb + 3 * 128 + (lane & 7) * 16);
  float c1[4] = {0.f, 0.f, 0.f, 0.f}, c2[4] = {0.f, 0.f, 0.f, 0.f};
  const uint32_t a1[4] = {x11t, 0u, 0u, 0u};
  mma_f16(c1, a1, pack_f16(f21.x, f21.y), 0u);           // (A21 X11)^T
  const uint32_t a2[4] = {pack_f16(c1[0], c1[1]), 0u, 0u, 0u};
  mma_f16(c2, a2, x22, 0u);                              // (X22 A21 X11)^T
  stsm1t(tb + 2 * 128 + (lane & 7) * 16, pack_f16(-c2[0], -c2[1]));
  __syncwarp();
}

// X^T += T^T A^T for one pair of 16 x 16 blocks: at = T as a transposed A operand, a = A as a B operand
__device__ __forceinline__ void mma_pair(float (&c)[2][4], const uint32_t (&at)[4], const uint32_t (&a)[4]) {
  mma_f16(c[0], at, a[0], a[1]);
  mma_f16(c[1], at, a[2], a[3]);
}
__device__ __forceinline__ void pack_pair(uint32_t (&a)[4], const float (&c)[2][4]) {
  a[0] = pack_f16(c[0][0], c[0][1]);
  a[1] = pack_f16(c[0][2], c[0][3]);
  a[2] = pack_f16(c[1][0], c[1][1]);
  a[3] = pack_f16(c[1][2], c[1][3]);
}

// Joins two inverted diagonal blocks of N x N (16 x 16 blocks, at block rows lo..lo+N-1 and lo+N..): block column `col` of
// the square below, T_lo = -T_hi (A T_lo'), by one warp.
template <int N>
__device__ __forceinline__ void join_column(uint32_t sT, uint32_t sA, int lo, int col, int lane) {
  float x[N][2][4];
#pragma unroll
  for (int i = 0; i < N; ++i)
#pragma unroll
    for (int h = 0; h < 2; ++h) x[i][h][0] = x[i][h][1] = x[i][h][2] = x[i][h][3] = 0.f;
#pragma unroll
  for (int k = 0; k < N; ++k) {
    if (N > 1 && k < col) continue;                      // (T_lo' is lower triangular)
    uint32_t at[4];
    ldsm4t(at, sT + tri_block(lo + k, lo + col) * 512 + lane * 16);
#pragma unroll
    for (int i = 0; i < N; ++i) {
      uint32_t a[4];
      lds4(a, sA + off_block(lo + N + i, lo + k) * 512 + lane * 16);
      mma_pair(x[i], at, a);
    }
  }
  uint32_t px[N][4];
#pragma unroll
  for (int i = 0; i < N; ++i) pack_pair(px[i], x[i]);
#pragma unroll
  for (int i = 0; i < N; ++i) {
    float r[2][4] = {};
#pragma unroll
    for (int k = 0; k <= i; ++k) {
      uint32_t a[4];
      ldsm4(a, sT + tri_block(lo + N + i, lo + N + k) * 512 + lane * 16);
      mma_pair(r, px[k], a);
    }
    const uint32_t w[4] = {pack_f16(-r[0][0], -r[0][1]), pack_f16(-r[0][2], -r[0][3]), pack_f16(-r[1][0], -r[1][1]),
                           pack_f16(-r[1][2], -r[1][3])};
    stsm4t(sT + tri_block(lo + N + i, lo + col) * 512 + lane * 16, w);
  }
  __syncwarp();
}

// Two rows (g and g + 8 of block (I, J)) of a triangular operand, eight bytes per lane.
__device__ __forceinline__ void store_tri_block(uint8_t* dst, int I, int J, int lane, const uint32_t (&w)[4]) {
  const int g = lane >> 2;
  uint8_t* d = dst + tri_row(16 * I + g, J) + ((((lane & 3) >> 1) ^ (g >> 2)) << 4) + ((lane & 1) << 3);
  *reinterpret_cast<uint2*>(d) = make_uint2(w[0], w[1]);
  *reinterpret_cast<uint2*>(d + 256) = make_uint2(w[2], w[3]);
}

// T block (I, J) diag(beta) -> the record's operand, as bf16.  `bad` becomes NaN if T left the fp16 range: inputs far
// outside the delta rule's stable range (beta |k|^2 <= 2).
__device__ __forceinline__ void emit_block(uint8_t* dst, uint32_t sT, const float* sBeta, int I, int J, int lane, __half2& bad) {
  uint32_t w[4], r[4];
  ldsm4(w, sT + tri_block(I, J) * 512 + lane * 16);
  const int t2 = (lane & 3) * 2;
  const float2 b0 = *reinterpret_cast<const float2*>(sBeta + 16 * J + t2);
  const float2 b1 = *reinterpret_cast<const float2*>(sBeta + 16 * J + 8 + t2);
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const __half2 h = *reinterpret_cast<const __half2*>(&w[e]);
    bad = __hfma2(h, __float2half2_rn(0.f), bad);
    const float2 f = __half22float2(h);
    const float2 bb = (e & 1) ? b1 : b0;
    r[e] = pack_bf16(f.x * bb.x, f.y * bb.y);
  }
  store_tri_block(dst, I, J, lane, r);
}

// The whole solve of one item by eight warps (0..7): T = (I + A)^-1 from the A blocks at sA and the fp32 diagonal blocks at
// sd ([8][16][LDD], dead afterwards: the last level keeps its intermediate there, at address sX), T diag(beta) written to
// the record's operand dst as it becomes final.  `csync` is a barrier of the eight warps; `idle(level)` is called by the
// warps 4..7 where they have nothing to do (level 1, 2).  Returns whether a value left the fp16 range.
template <typename Sync, typename Idle>
__device__ __forceinline__ bool solve_and_emit(uint8_t* dst, uint32_t sT, uint32_t sA, const float* sd, uint32_t sX,
                                               const float* sBeta, int warp, int lane, const Sync& csync, const Idle& idle) {
  const int g8 = lane >> 2;
  __half2 bad = __float2half2_rn(0.f);
  float badf = 0.f;
  invert_diagonal(sd + warp * 16 * LDD, sT + tri_block(warp, warp) * 512, lane);
  emit_block(dst, sT, sBeta, warp, warp, lane, bad);
  csync();
  if (warp < 4) {
    join_column<1>(sT, sA, 2 * warp, 0, lane);
    emit_block(dst, sT, sBeta, 2 * warp + 1, 2 * warp, lane, bad);
  } else {
    idle(1);
  }
  csync();
  if (warp < 4) {
    const int lo = (warp >> 1) * 4, col = warp & 1;
    join_column<2>(sT, sA, lo, col, lane);
    emit_block(dst, sT, sBeta, lo + 2, lo + col, lane, bad);
    emit_block(dst, sT, sBeta, lo + 3, lo + col, lane, bad);
  } else {
    idle(2);
  }
  csync();
  // level 3, the lower left 64 x 64 square, in two balanced halves: X = A T (16 blocks, two of 5 products together per
  // warp), then T_lo = -T_hi X, which goes out straight from the registers
  {
    const int i = warp & 3;
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const int jb = warp < 4 ? 3 * e : 1 + e;
      float x[2][4] = {};
#pragma unroll 1
      for (int k = jb; k < 4; ++k) {
        uint32_t at[4], a[4];
        ldsm4t(at, sT + tri_block(k, jb) * 512 + lane * 16);
        lds4(a, sA + off_block(4 + i, k) * 512 + lane * 16);
        mma_pair(x, at, a);
      }
      uint32_t px[4];
      pack_pair(px, x);
      sts4(sX + (jb * 4 + i) * 512 + lane * 16, px);
    }
  }
  csync();
  {
    const int jb = warp & 3;
    const float b0 = -sBeta[16 * jb + g8], b1 = -sBeta[16 * jb + 8 + g8];
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const int i = warp < 4 ? 3 * e : 1 + e;
      float r[2][4] = {};
#pragma unroll 1
      for (int k = 0; k <= i; ++k) {
        uint32_t at[4], a[4];
        lds4(at, sX + (jb * 4 + k) * 512 + lane * 16);
        ldsm4(a, sT + tri_block(4 + i, 4 + k) * 512 + lane * 16);
        mma_pair(r, at, a);
      }
      uint32_t f[4];                                     // (rows of the accumulators: columns of T)
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        f[2 * c] = transpose8x8(pack_bf16(b0 * r[c][0], b0 * r[c][1]));
        f[2 * c + 1] = transpose8x8(pack_bf16(b1 * r[c][2], b1 * r[c][3]));
        badf = fmaf(r[c][0] + r[c][1] + r[c][2] + r[c][3], 0.f, badf);
      }
      store_tri_block(dst, 4 + i, jb, lane, f);
    }
  }
  return __hisnan(__low2half(bad)) || __hisnan(__high2half(bad)) || badf != badf;
}

}  // namespace solve
}  // namespace ha_la
