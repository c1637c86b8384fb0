// Chunk-local operators of the delta-rule prefill, GDN (scalar gate): what the state-passing kernel needs per step of 128
// tokens.  Unit of work = (step slot, V-head); per unit (paper Section 2.1, "Chunkwise
// Map-Reduce-Map Execution", with steps of 128 tokens in place of chunks of 64):
//   #1 Gate   G = step-local cumulative log-gate
//   #2 KKT    A_ij = beta_i e^{G_i-G_j} (k_i . k_j)  (j < i)      P_ij = e^{G_i-G_j} (q_i . k_j)  (j <= i)
//   #3 Solve  T = (I + A)^-1 by blocked forward substitution
// and the record (tc_common.cuh) T diag(beta), P, e^{G_t}, e^{G_L-G_t} goes to the workspace: 37 KiB per step and head.
// Operator #4 (W/U) is not formed: the state-passing kernel applies T to V - e^G K h directly, which is fewer
// multiply-adds, a quarter less workspace traffic, and rounds fewer intermediates.
//
// A persistent kernel, one CTA per SM with three independent groups of eight warps (own shared memory and named barrier) that
// take the CTA's units in turn, so that one group's dependent phases run under the others', and a warp that loads tiles and issues
// the products ahead of them: two stages of tiles, two halves of tensor memory, each free again when its unit's products
// have been read.  V-heads that share a q/k head are units of their own: the second reading of the tiles hits L2, and the
// products are a fifth of a unit's time on an idle pipe.  The raw products K K^T and Q K^T
// are tcgen05 MMAs (M = N = K = 128: the full tensor rate); a warp reads its accumulators in 16 x 16 blocks, on and
// below the diagonal only, in the lane layout of warp-level matrix fragments (tcgen05.ld 16x256b).  A warp reaches only
// its quarter of the lanes, and the last quarter of K K^T has 15 of the 36 blocks, the first three; the other product
// is therefore formed transposed, K Q^T, where it is the other way round: 18 blocks to each pair of warps.  In that layout a
// block packed to 16 bits is at once the operand of the solve's warp-level products and four 128-byte rows of an 8 x 8
// core of the result operand, so results go from registers to global memory as whole 128-byte lines without staging.
//
// The solve: the 16 x 16 diagonal blocks, two by one warp (8 x 8 halves by forward substitution in fp32, joined by a
// product), then three levels of joining, T_lo = -T_hi (A_lo T_lo'), evaluated transposed so that the accumulators of
// the first product are the A operand of the second.  A and T are held as fp16 there (T is rounded to bf16 for the next
// operator anyway); this assumes the delta rule's usual normalisation (beta |k|^2 of order one), far inside the fp16
// range, and a result outside it is reported.
//
// What bounds it: with a q/k head per V-head and long calls HBM, 101 KiB a unit (8 sequences of 136 k tokens, 16 heads, 17 k units:
// 278 us, 98 % of the measured copy rate); with tiles out of L2, and in short calls, the shared-memory accesses and dependent
// phases of the solve and the masks: 8.5 k warp instructions and 4.8 k SM-cycles a unit with two V-heads per q/k head, the LSU
// data pipe 51 % busy.  This kernel by itself on B200, launch included: 16 heads, T = 333 13.6 us, T = 4096 23; 32 heads,
// T = 16384 86, on 16 q/k heads 80, on 8 77.  (Two groups that shared a unit's loads and products among V-heads: 14.5, 27,
// -, 93 and, on the 136 k tokens, 388.)
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

constexpr int kGroups = 3, kTpThreads = kGroups * 256 + 32;  // three groups of eight warps, and one warp that loads and issues MMAs
// Two stages of TMA tiles (K, Q: [kb][128 tok][64 feat]), then per group, in blocks of 512 bytes: fp16 T | spare | fp16 A.  The
// fp32 diagonal blocks of A lie over T's last eight and the spare ones, the solve's last intermediate over the spare ones
// and A's first (tc_solve.cuh says when which is dead).
constexpr uint32_t kStageB = 2 * kTileBytes;
constexpr int kSpare = 9;
constexpr uint32_t OFF_T = 0, OFF_D = 12 * 512, OFF_X = kTBlocks * 512, OFF_A = OFF_X + kSpare * 512;
// Two sets (used alternately) of G log2(e) [128], beta [128], and with R_I = G at the first token of block I of 16 tokens
// 2^(G_i - R_I) [128], 2^(R_{J+1} - G_j) [128].
constexpr uint32_t kGateB = 4 * 512;
constexpr uint32_t OFF_G = OFF_A + kABlocks * 512;
constexpr uint32_t kGroupB = OFF_G + 2 * kGateB;
static_assert(OFF_D + kDiagBytes <= OFF_A && (kXBlocks - kSpare) <= 12, "what lies over what");
constexpr uint32_t OFF_BAR = 2 * kStageB + kGroups * kGroupB;
constexpr uint32_t kTpSmem = OFF_BAR + (4 + kGroups) * 8 + 16;
static_assert(kTpSmem <= 227 * 1024, "shared memory budget");

struct TpParams {
  const float* g;
  const float* beta;
  const int32_t* chunk_tok0;   // step table of the plan kernel, or NULL for equal-length rows:
  const int32_t* chunk_len;    //   then slot s is step s % cps of row s / cps, T_row tokens per row
  int T_row, cps;
  TcWorkspace ws;
  int HK, HV;
  float scale;                 // of the outputs: P comes times `scale`
  long long total;             // units of work = step slots x V-heads
  int32_t* status;
};

__global__ void __launch_bounds__(kTpThreads, 1)
tc_tp_kernel(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_k, TpParams p) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  const int grp = threadIdx.x >> 8, warp = (threadIdx.x >> 5) & 7, lane = threadIdx.x & 31;   // (group kGroups: the issuing warp)
  uint64_t* full = reinterpret_cast<uint64_t*>(smem_raw + OFF_BAR);   // [2] tiles of a stage
  uint64_t* taken = full + 2;                            // [2] products in half h of tensor memory read by their unit's eight warps
  uint64_t* made = full + 4;                             // [kGroups] products of the group's unit complete
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(made + kGroups);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  const int R = p.HV / p.HK;
  if (threadIdx.x == 0) {
    for (int i = 0; i < 4 + kGroups; ++i) mbar_init(&full[i], i == 2 || i == 3 ? 8 : 1);
    *abort_flag = 0;
    mbar_fence_init();
    prefetch_tmap(&map_q); prefetch_tmap(&map_k);
  }
  if (threadIdx.x < 32) tmem_alloc(tmem_slot, 512);      // two halves: K K^T | K Q^T of one unit each
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  constexpr uint32_t tmem0 = 0;                          // (the whole of tensor memory)
  // This kernel is launched as a programmatic dependent of whatever precedes it in the stream; when that is the previous
  // call's state-passing kernel, which lets its dependents go a few steps before its end, everything above ran under
  // that kernel's tail.  Nothing of this call has been read or written so far: wait for the stream's earlier work here.
  asm volatile("griddepcontrol.wait;" ::: "memory");
  // Every CTA of this grid is running now: a dependent launch (the state-passing kernel) may be scheduled.  It
  // waits for this grid to finish.
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

  // A unit's step slot, V-head, tokens, first token row; slots that a packed batch does not use come last, with L = 0.  Unit u of
  // this CTA is unit blockIdx.x + u gridDim.x of the call; its group is u % kGroups, its stage and half u % 2.
  struct Geom { int s, j, L, tok0; };
  auto geom = [&](long long c) {
    Geom g{0, 0, 0, 0};
    if (c >= p.total) return g;
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
  if (grp == kGroups) {
    // ------------------------------------------------------------ tiles and products (one thread)
    if (elect_one()) {
      auto issue_tiles = [&](const Geom& g, int st) {
        uint8_t* t = smem_raw + st * kStageB;
        mbar_expect_tx(&full[st], kStageB);
        tma_load_4d(t, &map_k, &full[st], 0, g.j / R, g.tok0, 0);
        tma_load_4d(t + kTileBytes, &map_q, &full[st], 0, g.j / R, g.tok0, 0);
      };
      long long item = blockIdx.x;
      Geom g0 = geom(item), g1 = geom(item + gridDim.x);
      if (g0.L > 0) issue_tiles(g0, 0);
      if (g0.L > 0 && g1.L > 0) issue_tiles(g1, 1);
      for (uint32_t u = 0; g0.L > 0; ++u, item += gridDim.x) {
        const uint32_t st = u & 1, ph = (u >> 1) & 1;
        const Geom g2 = g1.L > 0 ? geom(item + 2LL * gridDim.x) : g1;   // (its look-ups under the waits)
        if (u > 1) mbar_wait(&taken[st], ph ^ 1, abort_flag);
        mbar_wait(&full[st], ph, abort_flag);
        tc_fence_after_sync();
        constexpr uint32_t id = idesc_bf16(128, 128, false, false);     // op #2, raw: [K K^T | K Q^T]
        const uint32_t sk = smem_u32(smem_raw + st * kStageB);
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
          for (int ks = 0; ks < 8; ++ks) {
            const uint32_t o = (ks >> 2) * 16384 + (ks & 3) * 32;
            umma_ss(tmem0 + st * 256 + h * 128, smem_desc(sk + o, 16, 1024, kSwizzle128B),
                    smem_desc(sk + h * kTileBytes + o, 16, 1024, kSwizzle128B), id, ks > 0);
          }
        umma_commit(&made[u % kGroups]);
        if (g2.L > 0) {
          mbar_wait(&made[u % kGroups], u / kGroups & 1, abort_flag);   // (the products have read the tiles)
          if (!*abort_flag) issue_tiles(g2, st);
        }
        g0 = g1;
        g1 = g2;
      }
    }
    __syncwarp();
  } else {
    uint8_t* sm = smem_raw + 2 * kStageB + grp * kGroupB;
    auto csync = [&]() { asm volatile("bar.sync %0, %1;" ::"r"(grp + 1), "r"(256) : "memory"); };   // the group's eight warps
    // gates of one (step, V-head), four consecutive tokens per lane; loaded one unit ahead, scanned at its end
    float gx[4], bx[4];
    auto load_gates = [&](int j_, int L_, int tok0_) {
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int t = 4 * lane + e;
        const size_t a = (size_t)(tok0_ + t) * p.HV + j_;
        gx[e] = t < L_ ? p.g[a] : 0.f;
        bx[e] = t < L_ ? p.beta[a] : 0.f;
      }
    };
    auto scan_gates = [&](float* set, uint8_t* rec) {      // op #1 Gate: inclusive scan over the step
      float x[4];
      x[0] = gx[0]; x[1] = x[0] + gx[1]; x[2] = x[1] + gx[2]; x[3] = x[2] + gx[3];
      float s = x[3];
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const float y = __shfl_up_sync(0xffffffffu, s, o);
        if (lane >= o) s += y;
      }
      const float before = s - x[3], gl = __shfl_sync(0xffffffffu, s, 31);
      float4 g2, e1, e2;
      float* pg = &g2.x; float* p1 = &e1.x; float* p2 = &e2.x;
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const float G = before + x[e];
        pg[e] = G * 1.4426950408889634f;                   // times log2(e), for ex2 in the decay mask
        p1[e] = __expf(G);
        p2[e] = __expf(gl - G);
      }
      *reinterpret_cast<float4*>(set + 4 * lane) = g2;
      *reinterpret_cast<float4*>(set + 128 + 4 * lane) = make_float4(bx[0], bx[1], bx[2], bx[3]);
      const float ref = __shfl_sync(0xffffffffu, g2.x, lane & ~3);
      const float ref1 = __shfl_sync(0xffffffffu, g2.x, min((lane & ~3) + 4, 31));   // (of the last block, which nothing uses: any)
      *reinterpret_cast<float4*>(set + 256 + 4 * lane) = make_float4(ex2(g2.x - ref), ex2(g2.y - ref), ex2(g2.z - ref), ex2(g2.w - ref));
      *reinterpret_cast<float4*>(set + 384 + 4 * lane) = make_float4(ex2(ref1 - g2.x), ex2(ref1 - g2.y), ex2(ref1 - g2.z), ex2(ref1 - g2.w));
      float* sc = reinterpret_cast<float*>(rec + kStepSc);
      *reinterpret_cast<float4*>(sc + 4 * lane) = e1;
      *reinterpret_cast<float4*>(sc + 128 + 4 * lane) = e2;
    };
    const uint32_t sT = smem_u32(sm + OFF_T), sA = smem_u32(sm + OFF_A);
    const int g8 = lane >> 2, t2 = (lane & 3) * 2;

    const long long vstride = (long long)gridDim.x * kGroups;
    long long item = (long long)grp * gridDim.x + blockIdx.x;
    Geom gm = geom(item);
    if (warp == 6 && gm.L > 0) {
      load_gates(gm.j, gm.L, gm.tok0);
      scan_gates(reinterpret_cast<float*>(sm + OFF_G), p.ws.rec + ((size_t)gm.s * p.HV + gm.j) * kStepRecB);
    }
    csync();
    uint32_t set = 0;
    for (uint32_t u = grp; gm.L > 0; u += kGroups) {
      item += vstride;
      const Geom gn = geom(item);
      const bool more = gn.L > 0;
      uint8_t* rec = p.ws.rec + ((size_t)gm.s * p.HV + gm.j) * kStepRecB;
      const float* sG2 = reinterpret_cast<const float*>(sm + OFF_G + set * kGateB);
      const float* sBeta = sG2 + 128;
      if (warp == 6 && more) load_gates(gn.j, gn.L, gn.tok0);
      mbar_wait(&made[grp], u / kGroups & 1, abort_flag);
      tc_fence_after_sync();

      // ---- op #2: decay and masks.  The first four warps have the lower, the others the upper 16 of their quarter of tensor-memory lanes: block row
      // rb of A (rb + 1 blocks) and of P^T (8 - rb blocks: block column rb of P).  Off the diagonal the decay from block J to block
      // I factors through the gates at their edges, e^{G_i-R_I} e^{R_I-R_{J+1}} e^{R_{J+1}-G_j}, all exponents <= 0.
      {
        const float* sER = sG2 + 256;                    // 2^(G_i - R_I)
        const float* sEC = sG2 + 384;                    // 2^(R_{J+1} - G_j)
        const int rb = 2 * (warp & 3) + (warp >> 2);
        const uint32_t ta = tmem0 + (u & 1) * 256 + (static_cast<uint32_t>(16 * rb) << 16);
        const float g0 = sG2[16 * rb + g8], g1 = sG2[16 * rb + 8 + g8];
        // w = accumulator block times row factors f0, f1 (rows g8, g8 + 8) and column factors cf
        auto scale = [&](const uint32_t (&r)[8], float f0, float f1, const float* cf, float2 (&lo)[2], float2 (&hi)[2]) {
#pragma unroll
          for (int c = 0; c < 2; ++c) {
            const float2 x = *reinterpret_cast<const float2*>(cf + 8 * c + t2);
            lo[c] = mul2(as_f2(r[4 * c], r[4 * c + 1]), mul2(x, make_float2(f0, f0)));
            hi[c] = mul2(as_f2(r[4 * c + 2], r[4 * c + 3]), mul2(x, make_float2(f1, f1)));
          }
        };
        uint32_t ra[8], rn[8];
        // -- A: blocks left of the diagonal as fp16 operands; the diagonal block in fp32 for the substitution
        {
          const float b0 = sBeta[16 * rb + g8], b1 = sBeta[16 * rb + 8 + g8];
          const float gr = sG2[16 * rb], f0 = b0 * sER[16 * rb + g8], f1 = b1 * sER[16 * rb + 8 + g8];
          uint32_t dst = sA + off_block(rb, 0) * 512 + lane * 16;
          tmem_ld_16x256b_x2(ta, ra);
          tmem_ld_wait();
#pragma unroll 2
          for (int J = 0; J < rb; ++J) {
            tmem_ld_16x256b_x2(ta + 16 * (J + 1), rn);   // (the next block arrives under this one's arithmetic)
            const float s = ex2(gr - sG2[16 * (J + 1)]);
            float2 lo[2], hi[2];
            scale(ra, s * f0, s * f1, sEC + 16 * J, lo, hi);
            const uint32_t f[4] = {pack_f16(lo[0].x, lo[0].y), pack_f16(lo[1].x, lo[1].y), pack_f16(hi[0].x, hi[0].y), pack_f16(hi[1].x, hi[1].y)};
            sts4(dst, f);
            dst = J == 3 ? sA + off_block(rb, 4) * 512 + lane * 16 : dst + 512;
            tmem_ld_wait();
#pragma unroll
            for (int e = 0; e < 8; ++e) ra[e] = rn[e];
          }
          tmem_ld_16x256b_x2(ta + 128 + 16 * rb, rn);    // (the diagonal block of P^T)
          float* sd = reinterpret_cast<float*>(sm + OFF_D) + rb * kDiagStride;
#pragma unroll
          for (int c = 0; c < 2; ++c) {                  // (the substitution reads the strictly lower entries only)
            const float2 gj = *reinterpret_cast<const float2*>(sG2 + 16 * rb + 8 * c + t2);
            *reinterpret_cast<float2*>(sd + diag_index(g8, 8 * c + t2)) =
                make_float2(b0 * __uint_as_float(ra[4 * c]) * ex2(g0 - gj.x), b0 * __uint_as_float(ra[4 * c + 1]) * ex2(g0 - gj.y));
            *reinterpret_cast<float2*>(sd + diag_index(g8 + 8, 8 * c + t2)) =
                make_float2(b1 * __uint_as_float(ra[4 * c + 2]) * ex2(g1 - gj.x), b1 * __uint_as_float(ra[4 * c + 3]) * ex2(g1 - gj.y));
          }
          tmem_ld_wait();
        }
        // -- P: from the transposed accumulator (rows j, columns i), transposed on the way out
        uint8_t* dst = rec + kStepP + tri_offset(rb, rb) + tri_lane(lane);
        auto put = [&](const float2 (&lo)[2], const float2 (&hi)[2]) {
          const uint32_t f[4] = {transpose8x8(pack_bf16(lo[0])), transpose8x8(pack_bf16(hi[0])),
                                 transpose8x8(pack_bf16(lo[1])), transpose8x8(pack_bf16(hi[1]))};
          store_tri_block(dst, f);
          dst += 512;
        };
        if (rb < 7) tmem_ld_16x256b_x2(ta + 128 + 16 * (rb + 1), ra);
        {
          float2 lo[2], hi[2];
#pragma unroll
          for (int c = 0; c < 2; ++c) {                  // diagonal block: keep i (column) >= j (row)
            const int cc = 8 * c + t2;
            const float2 gi = *reinterpret_cast<const float2*>(sG2 + 16 * rb + cc);
            lo[c].x = cc >= g8 ? __uint_as_float(rn[4 * c]) * (p.scale * ex2(gi.x - g0)) : 0.f;
            lo[c].y = cc + 1 >= g8 ? __uint_as_float(rn[4 * c + 1]) * (p.scale * ex2(gi.y - g0)) : 0.f;
            hi[c].x = cc >= g8 + 8 ? __uint_as_float(rn[4 * c + 2]) * (p.scale * ex2(gi.x - g1)) : 0.f;
            hi[c].y = cc + 1 >= g8 + 8 ? __uint_as_float(rn[4 * c + 3]) * (p.scale * ex2(gi.y - g1)) : 0.f;
          }
          put(lo, hi);
        }
        tmem_ld_wait();
        const float r1 = sG2[min(16 * (rb + 1), 127)], f0 = p.scale * sEC[16 * rb + g8], f1 = p.scale * sEC[16 * rb + 8 + g8];
#pragma unroll 2
        for (int I = rb + 1; I < 8; ++I) {
          if (I < 7) tmem_ld_16x256b_x2(ta + 128 + 16 * (I + 1), rn);
          const float s = ex2(sG2[16 * I] - r1);
          float2 lo[2], hi[2];
          scale(ra, s * f0, s * f1, sER + 16 * I, lo, hi);
          put(lo, hi);
          tmem_ld_wait();
#pragma unroll
          for (int e = 0; e < 8; ++e) ra[e] = rn[e];
        }
        tc_fence_before_sync();
        __syncwarp();
        if (lane == 0) mbar_arrive(&taken[u & 1]);
      }
      csync();
      // ---- op #3 Solve
      const bool bad = solve_and_emit(rec + kStepT, sT, sA, reinterpret_cast<const float*>(sm + OFF_D), smem_u32(sm + OFF_X),
                                      sBeta, warp, lane, csync, [&]() {
        if (warp == 6 && more)             // the gates of the next unit
          scan_gates(reinterpret_cast<float*>(sm + OFF_G + (set ^ 1) * kGateB), p.ws.rec + ((size_t)gn.s * p.HV + gn.j) * kStepRecB);
      });
      if (bad) report_status(p.status, HA_LA_ERR_DEVICE_CHECK);
      set ^= 1;
      csync();
      gm = gn;
    }
  }
  __syncthreads();
  if (threadIdx.x == 0 && *abort_flag) {
    report_status(p.status, HA_LA_ERR_TIMEOUT);
    settle_copies();
  }
  tc_fence_before_sync();
  __syncthreads();
  if (threadIdx.x < 32) tmem_dealloc(*tmem_slot, 512);
}

}  // namespace

cudaError_t configure_tc_tp() {
  cudaError_t e = cudaFuncSetAttribute(tc_tp_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kTpSmem);
  if (e != cudaSuccess) return e;
  // Same carve-out preference as the state-passing kernel: kernels that prefer different L1 / shared splits do not run
  // at the same time.
  return cudaFuncSetAttribute(tc_tp_kernel, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
}

// `ctas`: at most so many CTAs, one per SM
cudaError_t launch_tc_tp(const Problem& p, const ha_la_prefill_args& a, PlanView plan, const TcWorkspace& ws,
                         const CUtensorMap& mq, const CUtensorMap& mk, int ctas, cudaStream_t stream) {
  TpParams pp;
  pp.g = a.g; pp.beta = a.beta;
  pp.chunk_tok0 = plan.chunk_tok0; pp.chunk_len = plan.chunk_len;
  pp.T_row = p.T_row; pp.cps = p.max_seq_chunks > 0 ? p.max_seq_chunks : 1;
  pp.ws = ws; pp.HK = p.HK; pp.HV = p.HV; pp.scale = p.scale; pp.status = a.status_word;
  pp.total = (long long)p.max_chunks * p.HV;
  if (pp.total == 0) return cudaSuccess;
  timer_mark(stream, "tc_prep");
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(pp.total < ctas ? pp.total : ctas));
  cfg.blockDim = dim3(kTpThreads);
  cfg.dynamicSmemBytes = kTpSmem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = g_timer ? 0 : 1;                        // (per-kernel timing wants one kernel at a time)
  return cudaLaunchKernelEx(&cfg, tc_tp_kernel, mq, mk, pp);
}

}  // namespace ha_la
