// Chunk-local operators of the delta-rule prefill, GDN (scalar gate): what the state-passing kernel needs per step of 128
// tokens.  Work item = (step slot, q/k head); the V-heads of the group share the tiles and the two products.  For each
// V-head (paper Section 2.1, "Chunkwise Map-Reduce-Map Execution", with steps of 128 tokens in place of chunks of 64):
//   #1 Gate   G = step-local cumulative log-gate
//   #2 KKT    A_ij = beta_i e^{G_i-G_j} (k_i . k_j)  (j < i)      P_ij = e^{G_i-G_j} (q_i . k_j)  (j <= i)
//   #3 Solve  T = (I + A)^-1 by blocked forward substitution
// and the record (tc_common.cuh) T diag(beta), P, e^{G_t}, e^{G_L-G_t} goes to the workspace: 37 KiB per step and head.
// Operator #4 (W/U) is not formed: the state-passing kernel applies T to V - e^G K h directly, which is fewer
// multiply-adds, a quarter less workspace traffic, and rounds fewer intermediates.
//
// A persistent kernel, one CTA per SM with two independent groups of eight warps (own shared memory, named barrier and
// half of tensor memory), so that one group's dependent phases run under the other's.  The raw products K K^T and Q K^T
// are tcgen05 MMAs (M = N = K = 128: the full tensor rate); a warp reads its accumulators in 16 x 16 blocks, on and
// below the diagonal only, in the lane layout of warp-level matrix fragments (tcgen05.ld 16x256b).  A warp reaches only
// its quarter of the lanes, and the last quarter of K K^T has 15 of the 36 blocks, the first three; the other product
// is therefore formed transposed, K Q^T, where it is the other way round: 18 blocks to each pair of warps.  In that layout a
// block packed to 16 bits is at once the operand of the solve's warp-level products and four 128-byte rows of an 8 x 8
// core of the result operand, so results go from registers to global memory as whole 128-byte lines without staging.
//
// The solve: the 16 x 16 diagonal blocks by one warp each (8 x 8 halves by forward substitution in fp32, joined by a
// product), then three levels of joining, T_lo = -T_hi (A_lo T_lo'), evaluated transposed so that the accumulators of
// the first product are the A operand of the second.  A and T are held as fp16 there (T is rounded to bf16 for the next
// operator anyway); this assumes the delta rule's usual normalisation (beta |k|^2 of order one), far inside the fp16
// range, and a result outside it is reported.
//
// What bounds it: the solve's dependent phases and the instructions of the masks (10 k warp instructions per unit, 5.6 k
// SM-cycles with two units in flight).  Measured on B200, with the W, U, Q~ and O_loc images of 64-token chunks before: 16
// heads, T = 4096 36 -> 21 us; 32 heads, T = 16384 188 -> 91; 8 sequences of 136 k tokens, 16 heads 800 -> 384.
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

constexpr int kGroups = 2, kGroupThreads = 288;             // per group: eight warps, and one that loads and issues MMAs
constexpr uint32_t OFF_K = 0, OFF_Q = kTileBytes;           // TMA tiles [kb][128 tok][64 feat]
constexpr uint32_t OFF_T = 2 * kTileBytes;                  // fp16 T, 36 16 x 16 blocks (tri_block order), 512 B each
constexpr uint32_t OFF_A = OFF_T + 36 * 512;                // fp16 A below the diagonal blocks: 28 blocks, operand order
constexpr uint32_t OFF_D = OFF_A + 28 * 512;                // fp32 diagonal blocks of A
constexpr uint32_t OFF_G = OFF_D + 8 * 16 * LDD * 4;        // two sets (used alternately) of G log2(e)[128], beta[128], 2^(G-R)[128]
constexpr uint32_t OFF_BAR = OFF_G + 2 * 1536;
constexpr uint32_t kGroupSmem = (OFF_BAR + 32 + 1023) / 1024 * 1024;
constexpr uint32_t kTpSmem = kGroups * kGroupSmem;
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
  long long total;             // work items = step slots x q/k heads
  int32_t* status;
};

__global__ void __launch_bounds__(kGroups * kGroupThreads, 1)
tc_tp_kernel(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_k, TpParams p) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  const int grp = threadIdx.x / kGroupThreads, tid = threadIdx.x % kGroupThreads;
  const int warp = tid >> 5, lane = tid & 31;
  uint8_t* sm = smem_raw + grp * kGroupSmem;
  uint64_t* bar_load = reinterpret_cast<uint64_t*>(sm + OFF_BAR);
  uint64_t* bar_mma = bar_load + 1;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem_raw + OFF_BAR + 16);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(sm + OFF_BAR + 20);
  auto gsync = [&]() { asm volatile("bar.sync %0, %1;" ::"r"(grp + 1), "r"(kGroupThreads) : "memory"); };
  auto csync = [&]() { asm volatile("bar.sync %0, %1;" ::"r"(grp + 3), "r"(256) : "memory"); };   // its eight compute warps
  const int R = p.HV / p.HK;
  if (tid == 0) {
    mbar_init(bar_load, 1);
    mbar_init(bar_mma, 1);
    *abort_flag = 0;
    mbar_fence_init();
    prefetch_tmap(&map_q); prefetch_tmap(&map_k);
  }
  if (threadIdx.x < 32) tmem_alloc(tmem_slot, 512);      // 256 columns for each group: K K^T | K Q^T
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tmem = *tmem_slot + grp * 256;
  // This kernel is launched as a programmatic dependent of whatever precedes it in the stream; when that is the previous
  // call's state-passing kernel, which lets its dependents go a few steps before its end, everything above ran under
  // that kernel's tail.  Nothing of this call has been read or written so far: wait for the stream's earlier work here.
  asm volatile("griddepcontrol.wait;" ::: "memory");
  // Every CTA of this grid is running now: a dependent launch (the state-passing kernel) may be scheduled.  It
  // waits for this grid to finish.
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

  // an item's step slot, q/k head, tokens, first token row; slots that a packed batch does not use come last
  auto item_geom = [&](long long c, int& s_, int& jq_, int& L_, int& tok0_) {
    s_ = (int)((unsigned)c / (unsigned)p.HK);
    jq_ = (int)((unsigned)c - (unsigned)s_ * (unsigned)p.HK);
    if (p.chunk_len) {
      L_ = p.chunk_len[s_];
      tok0_ = p.chunk_tok0[s_];
    } else {
      const int cc_ = s_ % p.cps;
      tok0_ = (s_ / p.cps) * p.T_row + cc_ * kStep;
      L_ = min(kStep, p.T_row - cc_ * kStep);
    }
  };
  auto issue_tiles = [&](int jq_, int tok0_) {
    mbar_expect_tx(bar_load, 2 * kTileBytes);
    tma_load_4d(sm + OFF_K, &map_k, bar_load, 0, jq_, tok0_, 0);
    tma_load_4d(sm + OFF_Q, &map_q, bar_load, 0, jq_, tok0_, 0);
  };
  uint32_t lph = 0;
  auto issue_products = [&]() {                          // one thread: op #2, raw: [K K^T | K Q^T] once the tiles are there
    mbar_wait(bar_load, lph, abort_flag);
    tc_fence_after_sync();
    constexpr uint32_t id = idesc_bf16(128, 128, false, false);
    const uint32_t sk = smem_u32(sm + OFF_K), sq = smem_u32(sm + OFF_Q);
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
      for (int ks = 0; ks < 8; ++ks) {
        const uint32_t o = (ks >> 2) * 16384 + (ks & 3) * 32;
        umma_ss(tmem + h * 128, smem_desc(sk + o, 16, 1024, kSwizzle128B),
                smem_desc((h ? sq : sk) + o, 16, 1024, kSwizzle128B), id, ks > 0);
      }
    umma_commit(bar_mma);
  };
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
    const float ref = __shfl_sync(0xffffffffu, g2.x, lane & ~3);   // R: the gate at the first token of the 16-token block
    *reinterpret_cast<float4*>(set + 256 + 4 * lane) = make_float4(ex2(g2.x - ref), ex2(g2.y - ref), ex2(g2.z - ref), ex2(g2.w - ref));
    float* sc = reinterpret_cast<float*>(rec + kStepSc);
    *reinterpret_cast<float4*>(sc + 4 * lane) = e1;
    *reinterpret_cast<float4*>(sc + 128 + 4 * lane) = e2;
  };
  const uint32_t sT = smem_u32(sm + OFF_T), sA = smem_u32(sm + OFF_A);
  const int g8 = lane >> 2, t2 = (lane & 3) * 2;

  const long long vstride = (long long)gridDim.x * kGroups;
  long long item = (long long)grp * gridDim.x + blockIdx.x;   // group-major: a last partial round spreads over the SMs
  int s = 0, jq = 0, L = 0, tok0 = 0;
  bool have = item < p.total;
  if (have) { item_geom(item, s, jq, L, tok0); have = L > 0; }
  if (have) {
    if (tid == 256) { issue_tiles(jq, tok0); issue_products(); }
    if (warp == 6) {
      load_gates(jq * R, L, tok0);
      scan_gates(reinterpret_cast<float*>(sm + OFF_G), p.ws.rec + ((size_t)s * p.HV + jq * R) * kStepRecB);
    }
    gsync();
  }
  uint32_t mph = 0, set = 0;
  while (have) {
    item += vstride;
    int sn = 0, jqn = 0, Ln = 0, tok0n = 0;
    bool haven = item < p.total;
    if (haven) { item_geom(item, sn, jqn, Ln, tok0n); haven = Ln > 0; }
    mbar_wait(bar_mma, mph, abort_flag);
    mph ^= 1;
    lph ^= 1;
    tc_fence_after_sync();
    if (tid == 256 && haven) issue_tiles(jqn, tok0n);    // the products have read the tiles
    for (int v = 0; v < R; ++v) {
      const int j = jq * R + v;
      const size_t cj = (size_t)s * p.HV + j;
      uint8_t* rec = p.ws.rec + cj * kStepRecB;
      const float* sG2 = reinterpret_cast<const float*>(sm + OFF_G + set * 1536);
      const float* sBeta = sG2 + 128;
      const bool more = v + 1 < R;                       // the unit after this one
      if (warp == 6 && (more || haven)) load_gates(more ? j + 1 : jqn * R, more ? L : Ln, more ? tok0 : tok0n);

      // ---- op #2: decay and masks.  The first four warps have the lower, the others the upper 16 of their quarter of tensor-memory lanes: block row
      // rb of A (rb + 1 blocks) and of P^T (8 - rb blocks: block column rb of P).  Off the diagonal the decay factors through
      // the gate R_I at block row I's first token, e^{G_i-R_I} e^{R_I-G_j}, both exponents <= 0.
      if (warp < 8) {
        const float* sER = sG2 + 256;                    // 2^(G_i - R_I)
        const int rb = 2 * ((threadIdx.x >> 5) & 3) + (warp >> 2);   // (lanes go by the warp's place in the CTA)
        const uint32_t ta = tmem + (static_cast<uint32_t>(16 * rb) << 16);
        const float g0 = sG2[16 * rb + g8], g1 = sG2[16 * rb + 8 + g8];
        const float b0 = sBeta[16 * rb + g8], b1 = sBeta[16 * rb + 8 + g8];
        // w = accumulator block times row factors f0, f1 (rows g8, g8 + 8) and column factors cf
        auto scale = [&](const uint32_t (&r)[8], float f0, float f1, const float2 (&cf)[2], float (&w)[2][4]) {
#pragma unroll
          for (int c = 0; c < 2; ++c) {
            const float2 lo = mul2(make_float2(__uint_as_float(r[4 * c]), __uint_as_float(r[4 * c + 1])), mul2(cf[c], make_float2(f0, f0)));
            const float2 hi = mul2(make_float2(__uint_as_float(r[4 * c + 2]), __uint_as_float(r[4 * c + 3])), mul2(cf[c], make_float2(f1, f1)));
            w[c][0] = lo.x; w[c][1] = lo.y; w[c][2] = hi.x; w[c][3] = hi.y;
          }
        };
        uint32_t ra[8], rn[8];
        // -- A: blocks left of the diagonal as fp16 operands; the diagonal block in fp32 for the substitution
        {
          const float gr = sG2[16 * rb], f0 = b0 * sER[16 * rb + g8], f1 = b1 * sER[16 * rb + 8 + g8];
          tmem_ld_16x256b_x2(ta, ra);
          tmem_ld_wait();
#pragma unroll 1
          for (int J = 0; J < rb; ++J) {
            tmem_ld_16x256b_x2(ta + 16 * (J + 1), rn);   // (the next block arrives under this one's arithmetic)
            float2 cf[2];
#pragma unroll
            for (int c = 0; c < 2; ++c) {
              const float2 gj = *reinterpret_cast<const float2*>(sG2 + 16 * J + 8 * c + t2);
              cf[c] = make_float2(ex2(gr - gj.x), ex2(gr - gj.y));
            }
            float w[2][4];
            scale(ra, f0, f1, cf, w);
            const uint32_t f[4] = {pack_f16(w[0][0], w[0][1]), pack_f16(w[1][0], w[1][1]), pack_f16(w[0][2], w[0][3]),
                                   pack_f16(w[1][2], w[1][3])};
            sts4(sA + off_block(rb, J) * 512 + lane * 16, f);
            tmem_ld_wait();
#pragma unroll
            for (int e = 0; e < 8; ++e) ra[e] = rn[e];
          }
          tmem_ld_16x256b_x2(ta + 128 + 16 * rb, rn);    // (the diagonal block of P^T)
          float* sd = reinterpret_cast<float*>(sm + OFF_D) + rb * 16 * LDD;
#pragma unroll
          for (int c = 0; c < 2; ++c) {                  // (the substitution reads the strictly lower entries only)
            const float2 gj = *reinterpret_cast<const float2*>(sG2 + 16 * rb + 8 * c + t2);
            *reinterpret_cast<float2*>(sd + g8 * LDD + 8 * c + t2) =
                make_float2(b0 * __uint_as_float(ra[4 * c]) * ex2(g0 - gj.x), b0 * __uint_as_float(ra[4 * c + 1]) * ex2(g0 - gj.y));
            *reinterpret_cast<float2*>(sd + (g8 + 8) * LDD + 8 * c + t2) =
                make_float2(b1 * __uint_as_float(ra[4 * c + 2]) * ex2(g1 - gj.x), b1 * __uint_as_float(ra[4 * c + 3]) * ex2(g1 - gj.y));
          }
          tmem_ld_wait();
        }
        // -- P: from the transposed accumulator (rows j, columns i), transposed on the way out
        auto put = [&](int I, const float (&w)[2][4]) {
          const uint32_t f[4] = {transpose8x8(pack_bf16(w[0][0], w[0][1])), transpose8x8(pack_bf16(w[0][2], w[0][3])),
                                 transpose8x8(pack_bf16(w[1][0], w[1][1])), transpose8x8(pack_bf16(w[1][2], w[1][3]))};
          store_tri_block(rec + kStepP, I, rb, lane, f);
        };
        if (rb < 7) tmem_ld_16x256b_x2(ta + 128 + 16 * (rb + 1), ra);
        {
          float w[2][4];
#pragma unroll
          for (int c = 0; c < 2; ++c) {                  // diagonal block: keep i (column) >= j (row)
            const int cc = 8 * c + t2;
            const float2 gi = *reinterpret_cast<const float2*>(sG2 + 16 * rb + cc);
            w[c][0] = cc >= g8 ? __uint_as_float(rn[4 * c]) * (p.scale * ex2(gi.x - g0)) : 0.f;
            w[c][1] = cc + 1 >= g8 ? __uint_as_float(rn[4 * c + 1]) * (p.scale * ex2(gi.y - g0)) : 0.f;
            w[c][2] = cc >= g8 + 8 ? __uint_as_float(rn[4 * c + 2]) * (p.scale * ex2(gi.x - g1)) : 0.f;
            w[c][3] = cc + 1 >= g8 + 8 ? __uint_as_float(rn[4 * c + 3]) * (p.scale * ex2(gi.y - g1)) : 0.f;
          }
          put(rb, w);
        }
        tmem_ld_wait();
#pragma unroll 1
        for (int I = rb + 1; I < 8; ++I) {
          if (I < 7) tmem_ld_16x256b_x2(ta + 128 + 16 * (I + 1), rn);
          const float gr = sG2[16 * I];
          const float2 cf[2] = {*reinterpret_cast<const float2*>(sER + 16 * I + t2), *reinterpret_cast<const float2*>(sER + 16 * I + 8 + t2)};
          float w[2][4];
          scale(ra, p.scale * ex2(gr - g0), p.scale * ex2(gr - g1), cf, w);
          put(I, w);
          tmem_ld_wait();
#pragma unroll
          for (int e = 0; e < 8; ++e) ra[e] = rn[e];
        }
        tc_fence_before_sync();
      }
      gsync();
      // ---- op #3 Solve
      if (warp < 8) {
        const bool bad = solve_and_emit(rec + kStepT, sT, sA, reinterpret_cast<const float*>(sm + OFF_D), smem_u32(sm + OFF_D),
                                        sBeta, warp, lane, csync, [&](int level) {
          if (level == 1 && warp == 6 && (more || haven))       // the gates of the next unit
            scan_gates(reinterpret_cast<float*>(sm + OFF_G + (set ^ 1) * 1536),
                       p.ws.rec + (more ? cj + 1 : (size_t)sn * p.HV + jqn * R) * kStepRecB);
        });
        if (bad) report_status(p.status, HA_LA_ERR_DEVICE_CHECK);
      } else if (!more && haven && lane == 0) {          // this item's accumulators have been read by everyone
        tc_fence_after_sync();
        issue_products();
      }
      set ^= 1;
      gsync();
    }
    s = sn; jq = jqn; L = Ln; tok0 = tok0n; have = haven;
  }
  if (tid == 0 && *abort_flag) {
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
  pp.total = (long long)p.max_chunks * p.HK;
  if (pp.total == 0) return cudaSuccess;
  timer_mark(stream, "tc_prep");
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(pp.total < ctas ? pp.total : ctas));
  cfg.blockDim = dim3(kGroups * kGroupThreads);
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
