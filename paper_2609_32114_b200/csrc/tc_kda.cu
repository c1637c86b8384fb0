// Chunk-local operators of the delta-rule prefill, KDA (a gate per key channel): what the state-passing kernel needs per
// step of 128 tokens.  Work item = (step slot, V-head).  With G the step-local cumulative log-gates of a channel:
//   #1 Gate   G                                                    (and the operand images K e^G, scale Q e^G, K e^{G_L-G})
//   #2 KKT    A_ij = beta_i sum_c K_ic K_jc e^{G_ic-G_jc}  (j < i)     P_ij = sum_c Q_ic K_jc e^{G_ic-G_jc}  (j <= i)
//   #3 Solve  T = (I + A)^-1 by blocked forward substitution (tc_solve.cuh)
// Out go the three images (tiles as the state-passing kernel's MMAs read them) and the record (tc_common.cuh) T diag(beta),
// scale P, e^{G_L}: 133 KiB per item, 261 KiB with what it reads, which is what bounds the kernel once its two halves
// overlap.  They do: a persistent kernel, one CTA per SM, eight warps that make the gate-scaled operands of one item and
// eight that contract and solve the item before.
//
// The decay sits inside the contraction.  Per block of 16 tokens (block rows I, block columns J) it is split at the gates
// of block boundaries, rounded to whole powers of two, rho_I (log2):
//   K_i 2^{G_i-rho_I} . K_j 2^{rho_{J+1}-G_j} 2^{rho_I-rho_{J+1}}
// Both scaled copies are made once per token, in fp32, with exponents <= 1/2 up to rounding; the factor of the pair of
// blocks is a power of two per channel, so applying it to the bf16 operand in registers rounds nothing.  (A hierarchy of
// reference points with an own copy per level needs twice the shared memory.)  In a diagonal block that factor is >= 1;
// where a channel decays by more than 2^100 over 16 tokens, the block is evaluated entry by entry from the inputs.
// The contraction runs on warp-level MMAs: 36 pairs of blocks of the 64, no work above the diagonal, no operand copies
// per pair; it is a fifth of the kernel's instructions.
//
// Measured on B200 with 32 heads and 8192 tokens: 131 us; with 64-token chunks, a copy of the operands per block row and
// one item at a time per SM it was 262 us.
//
// Tokens past the end of a sequence are made no-ops by beta = 0 and g = 0; whatever the TMA box read for them (the
// next sequence's rows, or zero fill past the end of the tensor) is multiplied by exact zeros.  This relies on the
// inputs being finite.
#include <cuda.h>
#include <cuda_fp16.h>

#include "tc_common.cuh"
#include "tc_mma.cuh"
#include "tc_ptx.cuh"
#include "tc_solve.cuh"

namespace ha_la {

using namespace ptx;
using namespace solve;

namespace {

constexpr int kKdaThreads = 512;                           // eight scaling warps, eight solving warps
// per buffer (items alternate): K then K 2^{G-rho} in place | Q likewise | K 2^{rho-G}, then, once contracted, T (fp16 blocks)
constexpr uint32_t OFF_K = 0, OFF_Q = kTileBytes, OFF_K1 = 2 * kTileBytes, kBufBytes = 3 * kTileBytes;
constexpr uint32_t OFF_A = 2 * kBufBytes;                  // fp16 A below the diagonal blocks: 28 blocks, operand order
constexpr uint32_t OFF_D = OFF_A + kABlocks * 512;         // fp32 diagonal blocks of A, then the solve's last intermediate
constexpr uint32_t OFF_TOT = OFF_D + (kDiagBytes + 127) / 128 * 128;     // float [8][128]: log2 decay of each block
constexpr uint32_t OFF_RHO = OFF_TOT + 4096;               // per buffer: int16 [9][rho_slot(channel pair)][2], rho_J
constexpr uint32_t OFF_BETA = OFF_RHO + 2 * 9 * 256;       // per buffer: float [128]
constexpr uint32_t OFF_FALL = OFF_BETA + 2 * 512;          // per buffer: int [8][2] (channel halves), block needs the evaluation entry by entry
constexpr uint32_t OFF_BAR = OFF_FALL + 2 * 64;
constexpr uint32_t kKdaSmem = OFF_BAR + 32;
static_assert(kKdaSmem <= 227 * 1024, "shared memory budget");
static_assert(kXBlocks * 512 <= OFF_TOT - OFF_D && kTBlocks * 512 <= kTileBytes, "what lies over what (OFF_TOT is the next item's already)");
constexpr float kMaxUp = 100.f;

struct KdaParams {
  const __nv_bfloat16* q;
  const __nv_bfloat16* k;
  const float* g;
  const float* beta;
  const int32_t* chunk_tok0;   // step table of the plan kernel, or NULL for equal-length rows:
  const int32_t* chunk_len;    //   then slot s is step s % cps of row s / cps, T_row tokens per row
  int T_row, cps;
  TcWorkspace ws;
  int HK, HV;
  float scale;
  long long total;             // work items = step slots x V-heads
  int32_t* status;
};

__device__ __forceinline__ float2 ex2(float2 x) { return make_float2(ptx::ex2(x.x), ptx::ex2(x.y)); }
__device__ __forceinline__ uint32_t mul_bf16x2(uint32_t a, uint32_t b) {
  const __nv_bfloat162 r = __hmul2(*reinterpret_cast<const __nv_bfloat162*>(&a), *reinterpret_cast<const __nv_bfloat162*>(&b));
  return *reinterpret_cast<const uint32_t*>(&r);
}
// 2^e for a whole e as bf16 bits (0 below the normal range, the largest power above it)
__device__ __forceinline__ uint32_t pow2_bf16(float e) { return static_cast<uint32_t>(min(max(static_cast<int>(e) + 127, 0), 254)) << 7; }
__device__ __forceinline__ uint32_t pow2_pair(float2 e) { return pow2_bf16(e.x) | (pow2_bf16(e.y) << 16); }
// rho is kept as int16, as the sum of its steps from block to block clamped to +-kMaxStep: a difference of two is either
// exact or, like the true one, far outside the exponents of bf16.
constexpr float kMaxStep = 300.f;
__device__ __forceinline__ uint32_t pack_s16(float2 e) { return (static_cast<uint32_t>(static_cast<int>(e.x)) & 0xffffu) | (static_cast<uint32_t>(static_cast<int>(e.y)) << 16); }
// 2^(a + b) per half as bf16, a with the exponent bias added
__device__ __forceinline__ uint32_t pow2_sum(uint32_t a, uint32_t b) { return __vmins2(__viaddmax_s16x2(a, b, 0u), 0x00fe00feu) << 7; }
__device__ __forceinline__ int rho_slot(int pair) { return (pair & 3) * 16 + (pair >> 2); }   // a lane's sixteen pairs are neighbours

// Diagonal block I of A (fp32, times beta) and scale P (to its operand dst), entry by entry, by one warp: lane l has
// channels 4 l .. 4 l + 3.  (k, q, g: the head's first channel of the step's first token; token strides sk, sg.)
__device__ __noinline__ void slow_diagonal(const __nv_bfloat16* k, const __nv_bfloat16* q, size_t sk, const float* g, size_t sg,
                                           int L, int I, const float* sBeta, float* sd, uint8_t* dst, float scale, int lane) {
  for (int i = 0; i < 16; ++i) {
    const int ti = 16 * I + i;
    float kv[4] = {}, qv[4] = {}, w[4] = {1.f, 1.f, 1.f, 1.f};
    if (ti < L) {
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        kv[c] = __bfloat162float(k[ti * sk + 4 * lane + c]);
        qv[c] = __bfloat162float(q[ti * sk + 4 * lane + c]);
      }
    }
    for (int jj = 15; jj >= 0; --jj) {
      const int tj = 16 * I + jj;
      float a = 0.f, b = 0.f;
      if (ti < L && jj <= i) {
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const float x = __bfloat162float(k[tj * sk + 4 * lane + c]) * w[c];
          a = fmaf(kv[c], x, a);
          b = fmaf(qv[c], x, b);
          w[c] *= __expf(g[tj * sg + 4 * lane + c]);     // decay from tj - 1 to i
        }
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        a += __shfl_xor_sync(0xffffffffu, a, o);
        b += __shfl_xor_sync(0xffffffffu, b, o);
      }
      if (lane == 0) {
        sd[diag_index(i, jj)] = jj < i ? a * sBeta[ti] : 0.f;
        const int t = (jj & 7) >> 1;                     // (store_tri_block's place for column jj)
        *reinterpret_cast<__nv_bfloat16*>(dst + tri_row(ti, I) + (((t >> 1) ^ ((i & 7) >> 2)) << 4) + (t & 1) * 8 + (jj >> 3) * 4 + (jj & 1) * 2) =
            __float2bfloat16_rn(scale * b);
      }
    }
  }
}

__global__ void __launch_bounds__(kKdaThreads, 1)
tc_kda_kernel(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_k, KdaParams p) {
  extern __shared__ __align__(1024) uint8_t sm[];
  uint64_t* full = reinterpret_cast<uint64_t*>(sm + OFF_BAR);         // [2] K and Q tiles
  volatile int* abort_flag = reinterpret_cast<volatile int*>(full + 2);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int R = p.HV / p.HK;
  if (tid == 0) {
    mbar_init(&full[0], 1);
    mbar_init(&full[1], 1);
    *abort_flag = 0;
    mbar_fence_init();
    prefetch_tmap(&map_q); prefetch_tmap(&map_k);
  }
  __syncthreads();
  asm volatile("griddepcontrol.wait;" ::: "memory");     // nothing of this call has been read or written so far
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

  struct Geom { int s, j, L, tok0; };
  auto geom = [&](long long c) {                         // slots that a packed batch does not use come last, with L = 0
    Geom g{0, 0, 0, 0};
    if (c >= p.total) return g;
    if (!p.chunk_len) c = p.total - 1 - c;               // (the steps that are walked first are made last, and are still in L2 then: 1 %)
    g.s = (int)((unsigned)c / (unsigned)p.HV);
    g.j = (int)((unsigned)c - (unsigned)g.s * (unsigned)p.HV);
    if (p.chunk_len) {
      g.L = p.chunk_len[g.s];
      g.tok0 = p.chunk_tok0[g.s];
    } else {
      const int cc = g.s % p.cps;
      g.tok0 = (g.s / p.cps) * p.T_row + cc * kStep;
      g.L = min(kStep, p.T_row - cc * kStep);
    }
    return g;
  };
  auto issue_tiles = [&](const Geom& g, int b) {         // one thread
    mbar_expect_tx(&full[b], 2 * kTileBytes);
    if (R == 1) {                                        // (nothing else reads them: first out of L2, which the images need; 1 %)
      const uint64_t policy = evict_first<100>();
      tma_load_4d(sm + b * kBufBytes + OFF_K, &map_k, &full[b], 0, g.j, g.tok0, 0, policy);
      tma_load_4d(sm + b * kBufBytes + OFF_Q, &map_q, &full[b], 0, g.j, g.tok0, 0, policy);
    } else {
      tma_load_4d(sm + b * kBufBytes + OFF_K, &map_k, &full[b], 0, g.j / R, g.tok0, 0);
      tma_load_4d(sm + b * kBufBytes + OFF_Q, &map_q, &full[b], 0, g.j / R, g.tok0, 0);
    }
  };
  // named barriers: 1, 2 the scaled operands of buffer 0, 1 are ready; 3, 4 the buffer is free again (T read); 5, 6 within
  // the scaling and the solving warps
  auto arrive = [&](int id) { asm volatile("bar.arrive %0, 512;" ::"r"(id) : "memory"); };
  auto sync = [&](int id) { asm volatile("bar.sync %0, 512;" ::"r"(id) : "memory"); };
  auto sync_half = [&](int id) { asm volatile("bar.sync %0, 256;" ::"r"(id) : "memory"); };

  const long long stride = gridDim.x;
  if (warp >= 8) {
    // ------------------------------------------------------------ scaling: a pair of channels and 32 tokens per thread
    const int w = warp - 8, kb = w & 1, tg = w >> 1;
    const int cp = kb * 64 + 2 * lane;                   // channels cp, cp + 1; blocks 2 tg, 2 tg + 1
    const uint32_t o0 = kb * 16384 + ((lane & 3) << 2), ch = (lane >> 2) << 4;
    float* sTot = reinterpret_cast<float*>(sm + OFF_TOT);
    Geom gm = geom(blockIdx.x);
    if (tid == 256 && gm.L > 0) {                        // (later tiles are issued by the solving warps)
      issue_tiles(gm, 0);
      const Geom g1 = geom(blockIdx.x + stride);
      if (g1.L > 0) issue_tiles(g1, 1);
    }
    long long it = 0;
    for (long long item = blockIdx.x; gm.L > 0; ++it) {
      const int b = (int)(it & 1);
      const size_t cj = (size_t)gm.s * p.HV + gm.j;
      float2 l[2][16];                                   // block-local cumulative log2 gates
      {
        const float* gp = p.g + ((size_t)(gm.tok0 + 32 * tg) * p.HV + gm.j) * 128 + cp;
#pragma unroll
        for (int u = 0; u < 2; ++u)
#pragma unroll
          for (int t = 0; t < 16; ++t)
            l[u][t] = 32 * tg + 16 * u + t < gm.L ? __ldcs(reinterpret_cast<const float2*>(gp + (size_t)(16 * u + t) * p.HV * 128)) : make_float2(0.f, 0.f);
      }
      float bt = 0.f;
      if (tg == 0 || tg == 1) {                          // (warps 8 .. 11: a token's beta per thread)
        const int t = w * 32 + lane;
        bt = t < gm.L ? p.beta[(size_t)(gm.tok0 + t) * p.HV + gm.j] : 0.f;
      }
      item += stride;
      const Geom gn = geom(item);
      if (gn.L > 0) {                                    // the next item's gate rows, into L2 (line by line: 128 bulk
        const int t = (tid - 256) >> 1;                  // prefetches of 512 bytes held the copy engine for 6 k cycles)
        const float* g0 = p.g + ((size_t)(gn.tok0 + t) * p.HV + gn.j) * 128 + (tid & 1) * 64;
        if (t < gn.L) {
          prefetch_l2(g0);
          prefetch_l2(g0 + 32);
        }
      }
      const float2 lg = make_float2(1.4426950408889634f, 1.4426950408889634f);
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        l[u][0] = mul2(l[u][0], lg);
#pragma unroll
        for (int t = 1; t < 16; ++t) l[u][t] = fma2(l[u][t], lg, l[u][t - 1]);
        *reinterpret_cast<float2*>(sTot + (2 * tg + u) * 128 + cp) = l[u][15];
      }
      sync_half(5);
      float2 B[2], GL = make_float2(0.f, 0.f);           // gates at the start of this thread's blocks, and the last
      float2 rho[3];                                     // rounded, at the boundaries
      uint32_t rc[3];
      {
        float2 r = GL, x = GL;                           // ... and as they are kept
#pragma unroll
        for (int I = 0; I < 8; ++I) {
          if (I == 2 * tg) { B[0] = GL; rho[0] = r; rc[0] = pack_s16(x); }
          if (I == 2 * tg + 1) B[1] = GL;
          const float2 y = *reinterpret_cast<const float2*>(sTot + I * 128 + cp);
          GL.x += y.x; GL.y += y.y;
          const float2 rn = make_float2(rintf(GL.x), rintf(GL.y));
          x.x += fminf(fmaxf(rn.x - r.x, -kMaxStep), kMaxStep);
          x.y += fminf(fmaxf(rn.y - r.y, -kMaxStep), kMaxStep);
          r = rn;
          if (I == 2 * tg) { rho[1] = r; rc[1] = pack_s16(x); }
          if (I == 2 * tg + 1) { rho[2] = r; rc[2] = pack_s16(x); }
        }
      }
      if (it > 1) sync(3 + b);                           // the solving warps are done with the item two before
      else sync_half(5);                                 // (either way: the totals have been read)
      mbar_wait(&full[b], (uint32_t)(it >> 1) & 1, abort_flag);
      uint8_t* buf = sm + b * kBufBytes;
      uint32_t* kept = reinterpret_cast<uint32_t*>(sm + OFF_RHO + b * 2304) + 128 * tg + rho_slot(cp >> 1);
      if (tg == 0) kept[0] = rc[0];
      kept[64] = rc[1];
      kept[128] = rc[2];
      if (tg < 2) reinterpret_cast<float*>(sm + OFF_BETA + b * 512)[w * 32 + lane] = bt;
      uint8_t* img = p.ws.img + cj * 3 * kTileBytes;
      if (tg == 0) *reinterpret_cast<float2*>(p.ws.rec + cj * kStepRecB + kStepSc + cp * 4) = ex2(GL);
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int I = 2 * tg + u;
        const float2 dn = make_float2(rho[u + 1].x - rho[u].x, rho[u + 1].y - rho[u].y);
        const bool far = __any_sync(0xffffffffu, dn.x < -kMaxUp || dn.y < -kMaxUp);
        if (lane == 0) reinterpret_cast<int*>(sm + OFF_FALL + b * 64)[2 * I + kb] = far;
        const float2 a0 = make_float2(B[u].x - rho[u].x, B[u].y - rho[u].y);
        const float2 a1 = make_float2(rho[u + 1].x - B[u].x, rho[u + 1].y - B[u].y);
        const uint32_t pw = pow2_pair(rho[u]);
        const float2 sq = mul2(ex2(rho[u]), make_float2(p.scale, p.scale));
        const float2 cd = ex2(make_float2(GL.x - rho[u + 1].x, GL.y - rho[u + 1].y));
#pragma unroll
        for (int t = 0; t < 16; ++t) {
          const uint32_t o = o0 + (16 * I + t) * 128 + (ch ^ ((t & 7) << 4));
          const int td = step_pos(t);
          const uint32_t od = o0 + (16 * I + td) * 128 + (ch ^ ((td & 7) << 4));
          const float2 e0 = ex2(make_float2(l[u][t].x + a0.x, l[u][t].y + a0.y));
          const float2 e1 = ex2(make_float2(a1.x - l[u][t].x, a1.y - l[u][t].y));
          const float2 kf = unpack_bf16(*reinterpret_cast<const uint32_t*>(buf + OFF_K + o));
          const float2 qe = mul2(unpack_bf16(*reinterpret_cast<const uint32_t*>(buf + OFF_Q + o)), e0);
          const uint32_t k0 = pack_bf16(mul2(kf, e0));
          const float2 k1 = mul2(kf, e1);
          *reinterpret_cast<uint32_t*>(buf + OFF_K + o) = k0;
          *reinterpret_cast<uint32_t*>(buf + OFF_Q + o) = pack_bf16(qe);
          *reinterpret_cast<uint32_t*>(buf + OFF_K1 + o) = pack_bf16(k1);
          *reinterpret_cast<uint32_t*>(img + o) = mul_bf16x2(k0, pw);
          *reinterpret_cast<uint32_t*>(img + kTileBytes + o) = pack_bf16(mul2(qe, sq));
          *reinterpret_cast<uint32_t*>(img + 2 * kTileBytes + od) = pack_bf16(mul2(k1, cd));
        }
      }
      arrive(1 + b);
      gm = gn;
    }
    for (long long i = it > 2 ? it - 2 : 0; i < it; ++i) sync(3 + (int)(i & 1));   // pair with the last arrivals
  } else {
    // ------------------------------------------------------------ contraction and solve
    // Runs of blocks, (block row, first and last block column) per warp: at most five of the 36 each.
    const int I0 = (0x34556677 >> (4 * warp)) & 7, hi0 = (0x34152637 >> (4 * warp)) & 7, lo0 = (0x00020304 >> (4 * warp)) & 7;
    const int I1 = warp == 3 ? 1 : warp == 5 ? 2 : warp == 7 ? 0 : -1;
    const uint32_t sA = smem_u32(sm + OFF_A);
    float* sD = reinterpret_cast<float*>(sm + OFF_D);
    const int g8 = lane >> 2, t2 = (lane & 3) * 2;
    const int lrow = lane & 15, lch = lane >> 4;         // ldmatrix: row of a 16-row tile, 16-byte piece of a k-step
    Geom gm = geom(blockIdx.x);
    long long it = 0;
    for (long long item = blockIdx.x; gm.L > 0; ++it) {
      const int b = (int)(it & 1);
      const size_t cj = (size_t)gm.s * p.HV + gm.j;
      uint8_t* rec = p.ws.rec + cj * kStepRecB;
      const uint32_t sbuf = smem_u32(sm + b * kBufBytes);
      const float* sBeta = reinterpret_cast<const float*>(sm + OFF_BETA + b * 512);
      const uint32_t* srho = reinterpret_cast<const uint32_t*>(sm + OFF_RHO + b * 2304) + (lane & 3) * 16;
      const int* fall = reinterpret_cast<const int*>(sm + OFF_FALL + b * 64);
      auto frag = [&](uint32_t (&r)[4], uint32_t tile, int I, int k) {    // 16 rows of block I, 16 channels of k-step k
        ldsm4(r, tile + (k >> 2) * 16384 + sw128_offset(16 * I + lrow, (k & 3) * 2 + lch));
      };
      sync(1 + b);
#pragma unroll 1
      for (int sg = 0; sg < 2; ++sg) {
        const int I = sg ? I1 : I0, hi = sg ? I1 : hi0, lo = sg ? 0 : lo0;
        if (I < 0) break;
        uint32_t rI[16];                                 // 127 + rho_I of this lane's channels
#pragma unroll
        for (int x = 0; x < 16; x += 4) {
          const uint4 y = *reinterpret_cast<const uint4*>(srho + 64 * I + x);
          rI[x] = __vadd2(y.x, 0x007f007fu); rI[x + 1] = __vadd2(y.y, 0x007f007fu);
          rI[x + 2] = __vadd2(y.z, 0x007f007fu); rI[x + 3] = __vadd2(y.w, 0x007f007fu);
        }
        const float b0 = sBeta[16 * I + g8], b1 = sBeta[16 * I + 8 + g8];
#pragma unroll 1
        for (int J = hi; J >= lo; --J) {
          float a[2][4] = {}, pq[2][4] = {};
#pragma unroll
          for (int k = 0; k < 8; k += 2) {               // (k-steps in pairs: one 16-byte read of the block's gates)
            const uint4 y = *reinterpret_cast<const uint4*>(srho + 64 * (J + 1) + 2 * k);
            const uint32_t yy[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
            for (int i = 0; i < 2; ++i) {
              uint32_t r[4], kf[4], qf[4];
              frag(r, sbuf + OFF_K1, J, k + i);
              frag(kf, sbuf + OFF_K, I, k + i);
              frag(qf, sbuf + OFF_Q, I, k + i);
#pragma unroll
              for (int e = 0; e < 2; ++e) {              // 2^(rho_I - rho_{J+1})
                const uint32_t m = pow2_sum(rI[2 * (k + i) + e], __vneg2(yy[2 * i + e]));
                r[2 * e] = mul_bf16x2(r[2 * e], m);
                r[2 * e + 1] = mul_bf16x2(r[2 * e + 1], m);
              }
              mma_bf16(a[0], kf, r[0], r[2]);
              mma_bf16(a[1], kf, r[1], r[3]);
              mma_bf16(pq[0], qf, r[0], r[2]);
              mma_bf16(pq[1], qf, r[1], r[3]);
            }
          }
          if (J == I) {
            float* sd = sD + I * kDiagStride;
            if (fall[2 * I] | fall[2 * I + 1]) {
              const size_t jq = gm.j / R;
              slow_diagonal(p.k + ((size_t)gm.tok0 * p.HK + jq) * 128, p.q + ((size_t)gm.tok0 * p.HK + jq) * 128, (size_t)p.HK * 128,
                            p.g + ((size_t)gm.tok0 * p.HV + gm.j) * 128, (size_t)p.HV * 128, gm.L, I, sBeta, sd, rec + kStepP, p.scale, lane);
              continue;
            }
#pragma unroll
            for (int n = 0; n < 2; ++n) {                // (the substitution reads the strictly lower entries only)
              *reinterpret_cast<float2*>(sd + diag_index(g8, 8 * n + t2)) = make_float2(b0 * a[n][0], b0 * a[n][1]);
              *reinterpret_cast<float2*>(sd + diag_index(g8 + 8, 8 * n + t2)) = make_float2(b1 * a[n][2], b1 * a[n][3]);
#pragma unroll
              for (int e = 0; e < 4; ++e)
                if (8 * n + t2 + (e & 1) > g8 + (e >> 1) * 8) pq[n][e] = 0.f;
            }
          } else {
            const uint32_t f[4] = {pack_f16(b0 * a[0][0], b0 * a[0][1]), pack_f16(b0 * a[1][0], b0 * a[1][1]),
                                   pack_f16(b1 * a[0][2], b1 * a[0][3]), pack_f16(b1 * a[1][2], b1 * a[1][3])};
            sts4(sA + off_block(I, J) * 512 + lane * 16, f);
          }
          const uint32_t f[4] = {pack_bf16(p.scale * pq[0][0], p.scale * pq[0][1]), pack_bf16(p.scale * pq[1][0], p.scale * pq[1][1]),
                                 pack_bf16(p.scale * pq[0][2], p.scale * pq[0][3]), pack_bf16(p.scale * pq[1][2], p.scale * pq[1][3])};
          store_tri_block(rec + kStepP + tri_offset(I, J) + tri_lane(lane), f);
        }
      }
      sync_half(6);
      if (tid == 0) {                                    // the tiles of this buffer have been read: the item after next
        const Geom g2 = geom(item + 2 * stride);
        if (g2.L > 0) {
          fence_proxy_async_smem();
          issue_tiles(g2, b);
        }
      }
      const bool bad = solve_and_emit(rec + kStepT, sbuf + OFF_K1, sA, sD, smem_u32(sD), sBeta, warp, lane,
                                      [&]() { sync_half(6); }, []() {});
      if (bad) report_status(p.status, HA_LA_ERR_DEVICE_CHECK);
      arrive(3 + b);
      item += stride;
      gm = geom(item);
    }
  }
  if (tid == 256 && *abort_flag) {
    report_status(p.status, HA_LA_ERR_TIMEOUT);
    settle_copies();
  }
}

}  // namespace

cudaError_t configure_tc_kda() {
  cudaError_t e = cudaFuncSetAttribute(tc_kda_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kKdaSmem);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(tc_kda_kernel, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
}

cudaError_t launch_tc_kda(const Problem& p, const ha_la_prefill_args& a, PlanView plan, const TcWorkspace& ws,
                          const CUtensorMap& mq, const CUtensorMap& mk, int ctas, cudaStream_t stream) {
  KdaParams kp;
  kp.q = reinterpret_cast<const __nv_bfloat16*>(a.q);
  kp.k = reinterpret_cast<const __nv_bfloat16*>(a.k);
  kp.g = a.g; kp.beta = a.beta;
  kp.chunk_tok0 = plan.chunk_tok0; kp.chunk_len = plan.chunk_len;
  kp.T_row = p.T_row; kp.cps = p.max_seq_chunks > 0 ? p.max_seq_chunks : 1;
  kp.ws = ws; kp.HK = p.HK; kp.HV = p.HV; kp.scale = p.scale; kp.status = a.status_word;
  kp.total = (long long)p.max_chunks * p.HV;
  if (kp.total == 0) return cudaSuccess;
  timer_mark(stream, "tc_prep");
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(kp.total < ctas ? kp.total : ctas));
  cfg.blockDim = dim3(kKdaThreads);
  cfg.dynamicSmemBytes = kKdaSmem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = g_timer ? 0 : 1;                        // (per-kernel timing wants one kernel at a time)
  return cudaLaunchKernelEx(&cfg, tc_kda_kernel, mq, mk, kp);
}

}  // namespace ha_la
