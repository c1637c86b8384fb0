// Layout of the tensor-core path's workspace and what its kernels share.
#pragma once

#include "common.cuh"

namespace ha_la {

// The path works in steps of 128 tokens.  Record of one (step slot, V-head): T diag(beta) and P as bf16 MMA operands, then
// the gate factors (GDN: e^{G_t}[128], e^{G_L-G_t}[128]; KDA: e^{G_L}[128 keys]).  KDA's
// images of a step: K e^G, scale Q e^G, K e^{G_L-G} as tiles, the last with its rows of 16 in step_pos order.
// Triangular operand (128 x 128, lower): eight slabs of 16 columns one after the other, slab J with the rows 16 J .. 127
// only, rows of 32 bytes with the 32-byte swizzle; a product takes slab J as an operand of 128 - 16 J rows.  The 16
// columns of a row are stored in the order 0 1 8 9 2 3 10 11 .. (step_pos), which is the order a lane of a warp-level
// fragment holds them in: eight bytes per lane and row.  The other operand of the product has its K index in that order.
constexpr int kStep = 128;
constexpr uint32_t kTriB = 18432, kStepScB = 1024;
constexpr uint32_t kStepT = 0, kStepP = kTriB, kStepSc = 2 * kTriB, kStepRecB = 2 * kTriB + kStepScB;
constexpr uint32_t kTileBytes = 32768;        // a 128-token, 128-feature bf16 tile, [kb][128 tok][64 feat], 128-byte swizzle
constexpr __host__ __device__ uint32_t tri_slab(int J) { return 32u * (128 * J - 8 * J * (J - 1)); }   // byte offset of slab J
constexpr __host__ __device__ uint32_t tri_row(int row, int J) { return tri_slab(J) + (row - 16 * J) * 32; }
static_assert(tri_slab(8) == kTriB, "eight slabs");
constexpr __host__ __device__ int step_pos(int t) {                // stored position of row / column t
  return (t & ~15) | ((t & 6) << 1) | ((t & 8) >> 2) | (t & 1);
}

struct TcWorkspace {
  uint8_t* img;     // KDA only: [slot][V-head] three tiles
  uint8_t* rec;     // [slot][V-head] records
};

inline __host__ size_t tc_ws_bytes_for(size_t ncj, bool kda) {
  return ncj * (kda ? 3 * kTileBytes : 0) + align_up(ncj * kStepRecB, 1024);
}

inline __host__ TcWorkspace tc_ws_view(void* base, size_t ncj, bool kda) {
  uint8_t* b = reinterpret_cast<uint8_t*>(base);
  return TcWorkspace{b, b + ncj * (kda ? 3 * kTileBytes : 0)};
}

// What HA_LA_TC_SEGMENTS or the 64-token planner's segments add to the workspace (spans forced that way use it): per
// (sequence, V-head) and segment two fp32 and one bf16 128 x 128 matrix, per token-head a bf16 row of 128.
inline __host__ size_t tc_seg_bytes(size_t nj, int nseg, size_t rows, int HV) {
  if (nseg <= 1) return 0;
  return nj * nseg * 128 * 128 * (4 + 4 + 2) + align_up(rows * HV * 128 * 2, 1024);
}

// A transition Phi_s as operand fragments of warp-level products, 64 KiB of words: per 16 output keys w and 16 input keys ks, first
// the high, then (128 words on) the low bf16 parts, 4 words a lane.  Fragment row (and k index) f of a block of 16 is key sigma(f),
// sigma(2 t + e) = 4 t + e, sigma(8 + 2 t + e) = 4 t + 2 + e.  The word of output key 16 w + r and input keys v, v + 1 (v even; an odd
// one gives the same word); rows r and r + 2 (r % 4 < 2) are neighbours.
constexpr __host__ __device__ int phi_word(int w, int r, int v) {
  return ((w * 8 + (v >> 4)) * 2 * 32 + (2 * (r >> 2) + (r & 1)) * 4 + ((v & 15) >> 2)) * 4 + ((v >> 1) & 1) * 2 + ((r >> 1) & 1);
}

// Scratch of a call whose sequences are cut into spans: per (sequence, V-head) and span the offset b_s, which the span's
// true start state h_s replaces (fp32 128 x 128, [key][value channel]), and the transition Phi_s (in phi_word order; span 0 has
// none: its place keeps h0 in a call that works in place).
struct SpanBuffers {
  int nspan;            // 1: off
  float* b;
  float* phi;
};
inline __host__ size_t tc_span_bytes(size_t nj, int nspan) { return nspan <= 1 ? 0 : nj * nspan * 2 * 65536; }
inline __host__ SpanBuffers tc_span_view(void* base, size_t nj, int nspan) {
  if (nspan <= 1) return SpanBuffers{1, nullptr, nullptr};
  float* f = reinterpret_cast<float*>(base);
  return SpanBuffers{nspan, f, f + nj * nspan * 16384};
}

}  // namespace ha_la
