// The blocked inverse (I + A)^-1 of a unit lower triangular 128 x 128 matrix by eight warps, shared by the GDN and KDA
// chunk-local kernels (operator #3 of the paper's pipeline).  A is in shared memory: 16 x 16 blocks below the diagonal as fp16 B operands (16 bytes per lane, off_block
// order), the diagonal blocks in fp32.  T = (I + A)^-1 is kept as fp16 blocks of four row-major 8 x 8 matrices (128 bytes
// each, t_block order), which ldmatrix reads as any operand; its lower left 64 x 64 square, which nothing reads again, never is.
// A caller short of shared memory lays buffers over one another: the fp32 diagonal blocks are dead behind the solve's first barrier,
// before any of the last eight blocks of T is written, and the first twelve blocks of A are dead in the last level, when its
// intermediate (16 blocks) is made.
#pragma once

#include "tc_common.cuh"
#include "tc_mma.cuh"

namespace ha_la {
namespace solve {

using namespace ptx;

// A diagonal block in fp32: rows of 16 whose halves are exchanged in rows 2, 3, 6, 7 .., which keeps both the fragment layout's
// writes and the substitution's reads (two blocks, two halves at a time) free of bank conflicts.
constexpr int kDiagStride = 272;                            // floats from one block to the next
constexpr uint32_t kDiagBytes = (7 * kDiagStride + 256) * 4;
constexpr __host__ __device__ int diag_index(int row, int col) { return row * 16 + (col ^ ((row & 2) << 2)); }
// Blocks of 512 bytes.  A (J < I): the six pairs within each 64 x 64 half of the diagonal, then the square between the halves.
// T (J <= I, within a half): the diagonal, then those next to it that level 1 makes, then level 2's.
constexpr __host__ __device__ int off_block(int I, int J) {
  return (I ^ J) < 4 ? (I >> 2) * 6 + (I & 3) * ((I & 3) - 1) / 2 + (J & 3) : 12 + 4 * (I - 4) + J;
}
constexpr __host__ __device__ int t_block(int I, int J) {
  return I == J ? I : (I ^ J) == 1 ? 8 + (I >> 1) : 12 + (I >> 2) * 4 + (I & 1) * 2 + (J & 1);
}
constexpr int kTBlocks = 20, kABlocks = 28, kXBlocks = 16;

// Inverses of the 16 x 16 diagonal blocks 2 w and 2 w + 1 of I + A by one warp, as T's diagonal blocks; A_ii in fp32 at sd:
//   [[X11, 0], [-X22 A21 X11, X22]],  X11, X22 by forward substitution (a lane per block, half and column), the rest by two
// products, which take both blocks at once as a block diagonal operand.
// The coefficients are read ahead and the substitution goes by columns: a serial chain of seven multiply-adds.
__device__ __forceinline__ void invert_diagonal(const float* sd, uint32_t sT, int w, int lane) {
  const int g = lane >> 2, t2 = (lane & 3) * 2;
  const uint32_t tb = sT + 2 * w * 512;
  sd += 2 * w * kDiagStride;
  const float2 f0 = *reinterpret_cast<const float2*>(sd + diag_index(8 + g, t2));
  const float2 f1 = *reinterpret_cast<const float2*>(sd + kDiagStride + diag_index(8 + g, t2));
  const uint32_t mine = tb + (lane >> 4) * 512 + ((lane >> 3) & 1) * 384 + (lane & 7) * 16;
  {
    const int blk = lane >> 4, hb = (lane >> 3) & 1, c = lane & 7;
    const float* base = sd + blk * kDiagStride + hb * 128;
    const float* const same = base + hb * 8;             // this half's columns in rows 0, 1, 4, 5 of it, and in the others
    const float* const swapped = base + (hb ^ 1) * 8;
    auto at = [&](int q) { return ((q & 2) ? swapped : same) + q * 16; };
    const float a10 = *at(1);                            // (no more of a row than is used)
    const float2 a2 = *reinterpret_cast<const float2*>(at(2));
    float4 lo[5];                                        // columns 0 .. 3 of rows 3 .. 7
#pragma unroll
    for (int q = 0; q < 5; ++q) lo[q] = *reinterpret_cast<const float4*>(at(q + 3));
    const float a54 = at(5)[4];
    const float2 a6 = *reinterpret_cast<const float2*>(at(6) + 4);
    const float4 a7 = *reinterpret_cast<const float4*>(at(7) + 4);
    float y[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) y[q] = q == c ? 1.f : 0.f;
    y[1] = fmaf(-a10, y[0], y[1]);
    y[2] = fmaf(-a2.y, y[1], fmaf(-a2.x, y[0], y[2]));
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
      for (int q = r < 3 ? 3 : 4; q < 8; ++q)
        if (q > r) y[q] = fmaf(-(&lo[q - 3].x)[r], y[r], y[q]);
    y[5] = fmaf(-a54, y[4], y[5]);
    y[6] = fmaf(-a6.y, y[5], fmaf(-a6.x, y[4], y[6]));
    y[7] = fmaf(-a7.z, y[6], fmaf(-a7.y, y[5], fmaf(-a7.x, y[4], y[7])));
    const uint32_t col[4] = {pack_f16(y[0], y[1]), pack_f16(y[2], y[3]), pack_f16(y[4], y[5]), pack_f16(y[6], y[7])};
    sts4(mine, col);                                     // (transposed for now)
    if (hb == 0) {
      const uint32_t z[4] = {0u, 0u, 0u, 0u};
      sts4(tb + blk * 512 + 128 + c * 16, z);            // the quarter above the diagonal
    }
  }
  __syncwarp();
  uint32_t xt[4], x[4];                                  // X11, X22 of the first block, of the second
  ldsm4(xt, mine);
  ldsm4t(x, mine);
  __syncwarp();
  stsm4(mine, x);
  float c1[4] = {}, c2[4] = {};
  const uint32_t a1[4] = {xt[0], 0u, 0u, xt[2]};
  mma_f16(c1, a1, pack_f16(f0.x, f0.y), pack_f16(f1.x, f1.y));      // (A21 X11)^T
  const uint32_t a2[4] = {pack_f16(c1[0], c1[1]), 0u, 0u, pack_f16(c1[2], c1[3])};
  mma_f16(c2, a2, x[1], x[3]);                           // (X22 A21 X11)^T
  stsm1t(tb + 256 + (lane & 7) * 16, pack_f16(-c2[0], -c2[1]));
  stsm1t(tb + 512 + 256 + (lane & 7) * 16, pack_f16(-c2[2], -c2[3]));
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

// Joins two inverted diagonal blocks: the square below, T_lo = -T_hi (A T_lo').  Operands are read ahead of the products, and their
// addresses are constants from a base that the caller picks: index arithmetic was most of the solve's instructions.
__device__ __forceinline__ void join_blocks(uint32_t t_lo, uint32_t t_hi, uint32_t a_off, uint32_t t_off) {   // 16 x 16, lane addresses
  uint32_t at[4], a[4], th[4];
  lds4(a, a_off);
  ldsm4t(at, t_lo);
  ldsm4(th, t_hi);
  float x[2][4] = {}, r[2][4] = {};
  uint32_t px[4];
  mma_pair(x, at, a);
  pack_pair(px, x);
  mma_pair(r, px, th);
  const uint32_t w[4] = {pack_f16(-r[0][0], -r[0][1]), pack_f16(-r[0][2], -r[0][3]), pack_f16(-r[1][0], -r[1][1]), pack_f16(-r[1][2], -r[1][3])};
  stsm4t(t_off, w);
}
// ... of 32 x 32, block column COL of the square, by one warp.  td, t1, to: T's diagonal, level 1 and level 2 blocks of this
// 64 x 64 half, ao: A's (lane addresses)
template <int COL>
__device__ __forceinline__ void join_column(uint32_t td, uint32_t t1, uint32_t to, uint32_t ao) {
  uint32_t at[2][4], a[2][2][4], th[2][2][4];            // [k], [i][k]
  if (COL == 0) {
    ldsm4t(at[0], td);
    lds4(a[0][0], ao + 1 * 512);
    lds4(a[1][0], ao + 3 * 512);
  }
  ldsm4t(at[1], COL ? td + 512 : t1);
  lds4(a[0][1], ao + 2 * 512);
  lds4(a[1][1], ao + 4 * 512);
  ldsm4(th[0][0], td + 2 * 512);
  ldsm4(th[1][0], t1 + 512);
  ldsm4(th[1][1], td + 3 * 512);
  uint32_t px[2][4];
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    float x[2][4] = {};
#pragma unroll
    for (int k = COL; k < 2; ++k) mma_pair(x, at[k], a[i][k]);
    pack_pair(px[i], x);
  }
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    float r[2][4] = {};
#pragma unroll
    for (int k = 0; k <= i; ++k) mma_pair(r, px[k], th[i][k]);
    const uint32_t w[4] = {pack_f16(-r[0][0], -r[0][1]), pack_f16(-r[0][2], -r[0][3]), pack_f16(-r[1][0], -r[1][1]),
                           pack_f16(-r[1][2], -r[1][3])};
    stsm4t(to + (2 * i + COL) * 512, w);
  }
}

// A block of a triangular operand: two rows (g and g + 8) of eight bytes per lane, from the lane's place in the block.
__device__ __forceinline__ uint32_t tri_lane(int lane) {
  const int g = lane >> 2;
  return g * 32 + ((((lane & 3) >> 1) ^ (g >> 2)) << 4) + ((lane & 1) << 3);
}
constexpr __host__ __device__ uint32_t tri_offset(int I, int J) { return 512 * I + 256 * J * (15 - J); }   // = tri_row(16 I, J)
static_assert(tri_offset(7, 7) == tri_row(112, 7) && tri_offset(5, 2) == tri_row(80, 2) && tri_offset(3, 0) == tri_row(48, 0), "");
__device__ __forceinline__ void store_tri_block(uint8_t* d, const uint32_t (&w)[4]) {
  *reinterpret_cast<uint2*>(d) = make_uint2(w[0], w[1]);
  *reinterpret_cast<uint2*>(d + 256) = make_uint2(w[2], w[3]);
}

// T block at `block` (lane address), block column J, times diag(beta) -> the record's operand, as bf16.
__device__ __forceinline__ void emit_block(uint8_t* dst, uint32_t block, const float* sBeta, int J, int lane) {
  uint32_t w[4], r[4];
  ldsm4(w, block);
  const int t2 = (lane & 3) * 2;
  const float2 b[2] = {*reinterpret_cast<const float2*>(sBeta + 16 * J + t2), *reinterpret_cast<const float2*>(sBeta + 16 * J + 8 + t2)};
#pragma unroll
  for (int e = 0; e < 4; ++e) r[e] = pack_bf16(mul2(__half22float2(*reinterpret_cast<const __half2*>(&w[e])), b[e & 1]));
  store_tri_block(dst, r);
}

// Level 3, the lower left 64 x 64 square, in two balanced halves: X = A T (16 blocks, two of 5 products together per warp), then
// T_lo = -T_hi X, which goes out straight from the registers.  Warp w4 of the first (UPPER: second) four makes block row w4 of X
// in block columns 0 and 3 (1 and 2), then block column w4 of T_lo in block rows 0 and 3 (1 and 2).  Operands are read three pairs ahead.
template <bool UPPER>
__device__ __forceinline__ void level3_inner(uint32_t sT, uint32_t sA, uint32_t sX, int w4) {      // (lane addresses)
  constexpr int tb[5] = {UPPER ? t_block(1, 1) : t_block(0, 0), UPPER ? t_block(2, 1) : t_block(1, 0), UPPER ? t_block(3, 1) : t_block(2, 0),
                         UPPER ? t_block(2, 2) : t_block(3, 0), UPPER ? t_block(3, 2) : t_block(3, 3)};
  constexpr int ka[5] = {0, 1, 2, UPPER ? 1 : 3, UPPER ? 2 : 3};                 // a[ka]: A's block in column ka (+ 1 if UPPER)
  const uint32_t aw = sA + (12 + 4 * w4) * 512, xw = sX + w4 * 512;
  uint32_t at[5][4], a[4][4], px[4];
  float x[2][2][4] = {};
  auto read = [&](int s) {
    ldsm4t(at[s], sT + tb[s] * 512);
    if (ka[s] == s) lds4(a[s], aw + (s + (UPPER ? 1 : 0)) * 512);
  };
  read(0); read(1); read(2);
#pragma unroll
  for (int s = 0; s < 5; ++s) {
    mma_pair(x[s < (UPPER ? 3 : 4) ? 0 : 1], at[s], a[ka[s]]);
    if (s < 2) read(s + 3);
  }
  pack_pair(px, x[0]);
  sts4(xw + (UPPER ? 1 : 0) * 4 * 512, px);
  pack_pair(px, x[1]);
  sts4(xw + (UPPER ? 2 : 3) * 4 * 512, px);
}
// Returns NaN if a value left the fp16 range anywhere in the solve: every block of T is an operand of the sums here or of X's.
template <bool UPPER>
__device__ __forceinline__ float level3_outer(uint8_t* dst, uint32_t sT, uint32_t sX, const float* sBeta, int w4, int lane) {
  constexpr int i0 = UPPER ? 1 : 0, i1 = UPPER ? 2 : 3;
  constexpr int tb[5] = {UPPER ? t_block(5, 4) : t_block(4, 4), UPPER ? t_block(5, 5) : t_block(7, 4), UPPER ? t_block(6, 4) : t_block(7, 5),
                         UPPER ? t_block(6, 5) : t_block(7, 6), UPPER ? t_block(6, 6) : t_block(7, 7)};
  constexpr int kb[5] = {0, UPPER ? 1 : 0, UPPER ? 0 : 1, UPPER ? 1 : 2, UPPER ? 2 : 3};   // at[kb]: X's block row
  const uint32_t xw = sX + 4 * w4 * 512;
  uint32_t at[4][4], a[5][4];
  float r[2][2][4] = {}, bad = 0.f;
  auto read = [&](int s) {
    if (s == 0 || (UPPER ? s == 1 || s == 4 : s > 1)) lds4(at[kb[s]], xw + kb[s] * 512);
    ldsm4(a[s], sT + tb[s] * 512);
  };
  read(0); read(1); read(2);
  const float b0 = -sBeta[16 * w4 + (lane >> 2)], b1 = -sBeta[16 * w4 + 8 + (lane >> 2)];
#pragma unroll
  for (int s = 0; s < 5; ++s) {
    mma_pair(r[s <= i0 ? 0 : 1], at[kb[s]], a[s]);
    if (s < 2) read(s + 3);
  }
  uint8_t* d = dst + tri_offset(4, w4);
#pragma unroll
  for (int e = 0; e < 2; ++e) {
    uint32_t f[4];                                       // (rows of the accumulators: columns of T)
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      const float2 lo = mul2(make_float2(r[e][c][0], r[e][c][1]), make_float2(b0, b0));
      const float2 hi = mul2(make_float2(r[e][c][2], r[e][c][3]), make_float2(b1, b1));
      f[2 * c] = transpose8x8(pack_bf16(lo));
      f[2 * c + 1] = transpose8x8(pack_bf16(hi));
      bad = fmaf((r[e][c][0] + r[e][c][1]) + (r[e][c][2] + r[e][c][3]), 0.f, bad);
    }
    store_tri_block(d + 512 * (e ? i1 : i0), f);
  }
  return bad;
}

// The whole solve of one item by eight warps (0..7): T = (I + A)^-1 from the A blocks at sA and the fp32 diagonal blocks at
// sd (kDiagStride apart), with room for the last level's intermediate at sX, T diag(beta) written to
// the record's operand dst.  `csync` is a barrier of the eight warps; `idle()` is called by the warps 4..7 where they have
// nothing to do.  Returns whether a value left the fp16 range (inputs far outside the delta rule's stable range, beta |k|^2 <= 2).
template <typename Sync, typename Idle>
__device__ __forceinline__ bool solve_and_emit(uint8_t* dst, uint32_t sT, uint32_t sA, const float* sd, uint32_t sX,
                                               const float* sBeta, int warp, int lane, const Sync& csync, const Idle& idle) {
  const int w4 = warp & 3, half = w4 >> 1, odd = w4 & 1;
  const bool upper = warp >= 4;
  const uint32_t l16 = lane * 16, td = sT + l16, ao = sA + half * 6 * 512 + l16, t1 = td + (8 + half * 2) * 512,
                 to = td + (12 + half * 4) * 512;
  dst += tri_lane(lane);
  if (!upper) {                                          // two diagonal blocks and the one between them: nothing to wait for
    invert_diagonal(sd, sT, warp, lane);
    join_blocks(td + 2 * warp * 512, td + (2 * warp + 1) * 512, ao + 5 * odd * 512, t1 + odd * 512);
  } else {
    idle();
  }
  csync();
  if (!upper) {
    if (odd) join_column<1>(td + half * 4 * 512, t1, to, ao);
    else join_column<0>(td + half * 4 * 512, t1, to, ao);
  } else {                                               // (what is final so far goes out)
    emit_block(dst + tri_offset(2 * w4, 2 * w4), td + 2 * w4 * 512, sBeta, 2 * w4, lane);
    emit_block(dst + tri_offset(2 * w4 + 1, 2 * w4 + 1), td + (2 * w4 + 1) * 512, sBeta, 2 * w4 + 1, lane);
    emit_block(dst + tri_offset(2 * w4 + 1, 2 * w4), t1 + odd * 512, sBeta, 2 * w4, lane);
  }
  csync();
  if (upper) level3_inner<true>(td, sA + l16, sX + l16, w4);
  else level3_inner<false>(td, sA + l16, sX + l16, w4);
  {
    const int I = 4 * half + (upper ? 3 : 2), J = 4 * half + odd;
    emit_block(dst + tri_offset(I, J), to + ((upper ? 2 : 0) + odd) * 512, sBeta, J, lane);
  }
  csync();
  const float bad = upper ? level3_outer<true>(dst, td, sX + l16, sBeta, w4, lane) : level3_outer<false>(dst, td, sX + l16, sBeta, w4, lane);
  return bad != bad;
}

}  // namespace solve
}  // namespace ha_la
