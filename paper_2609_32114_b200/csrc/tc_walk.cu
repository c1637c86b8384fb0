// Sequential part of the delta-rule prefill on tcgen05 tensor cores: operator #5 (state passing) with operator #4
// applied and operator #6 (output) fused in the paper's chunk-first order.
//
// One CTA owns all 128 value channels of a (sequence, V-head) and walks its sequence, or one span of it, in steps of 128
// tokens.  The state is kept TRANSPOSED: fp32 in registers, and as bf16 pairs in tensor memory (lane = value channel,
// columns = key channels), where it is the A operand of the products; every other state-dependent operand is made there
// too, so nothing that threads write goes through shared memory on its way to the tensor cores (no proxy fences), and
// shared memory is left to the B operands, which arrive ready-made by bulk copy.  Per step (GDN; tc_tp.cu supplies
// T diag(beta), P and the gate factors):
//   X^T  = h^T K^T                          R^T = V^T - e^{G_j} X^T                 bf16 pairs
//   U~^T = R^T (T diag(beta))^T                                                     bf16 pairs, plain and times e^{G_L-G_j}
//   h^T <- e^{G_L} h^T + (U~ e^{G_L-G})^T K                                          op #5
//   o^T  = scale [e^{G_i} (h^T Q^T) + U~^T P^T]   (old h; off the sequential path)   op #6
// KDA: K e^G, Q e^G and K e^{G_L-G} come as images from tc_kda.cu, so no column factors are needed and the decay is
// per key channel.
//
// What bounds a step: the serial path of three products and their epilogues (a product: N / 2 cycles per instruction of 16 deep,
// ~180 cycles to a visible result; an epilogue of the compute warps 350 - 900 cycles of tensor-memory round trips), with outputs
// the compute warps themselves (2.5 k of 3.7 k cycles), and on large calls HBM (165 KiB per step and head, KDA 197).  T and P are
// lower triangular: step ks of their products runs with N = 128 - 16 ks rows.  U and D2 run in token halves, so that an epilogue
// starts when half of its input is final; Y goes behind X and P U~ behind D2, where the sequential path leaves the tensor
// cores idle.
// Measured on B200, a launch by itself: 2.2 us per step of 128 tokens with outputs and 1.4 without (between 6 and 43 steps, most SMs
// at work) and 11 for its start and end; 8 sequences of 136 k tokens, 16 heads 537 us, 5.4 TB/s.
//
// Warp roles: sixteen compute warps (tensor-memory lanes 32 (w % 4).., group w / 4 of the columns), four output warps, two
// producer warps, two warps that issue MMAs (the sequential path; the outputs).  Every wait is bounded.
#include <cuda.h>

#include "tc_common.cuh"
#include "tc_mma.cuh"
#include "tc_ptx.cuh"

namespace ha_la {

using namespace ptx;

namespace {

constexpr int kCompute = 512;                              // compute threads: four warps for each of four column groups
constexpr int walk_threads(bool out) { return kCompute + 32 * (out ? 8 : 3); }

// Shared memory: 32-KiB tiles, then the triangular operands.  The slots go where a copy would otherwise start too late: out of HBM
// and behind the other copies an operand takes up to 3.8 k cycles.
template <bool KDA, bool OUT>
struct WalkCfg {
  static constexpr int kNK = OUT ? (KDA ? 1 : 2) : (KDA ? 2 : 3);   // slots of K (KDA: of K e^G); step c has slot c % kNK
  static constexpr int kND = KDA ? (OUT ? 1 : 2) : 0;      // ... of KDA's K e^{G_L-G}
  static constexpr int kNV = 2;                            // ... of V, [2][128 tok][64 ch]
  static constexpr int kNT = KDA || OUT ? 1 : 2;           // ... of T diag(beta)
  static constexpr uint32_t OFF_K = 0, OFF_D = kNK * kTileBytes, OFF_Q = OFF_D + kND * kTileBytes;   // Q (KDA: Q e^G)
  static constexpr uint32_t OFF_V = OFF_Q + (OUT ? kTileBytes : 0), OFF_T = OFF_V + kNV * kTileBytes;
  static constexpr uint32_t OFF_P = OFF_T + kNT * kTriB;
  static constexpr uint32_t OFF_OUT = OFF_P + (OUT ? kTriB : 0);   // output staging: [4 warps][64 tok][32 ch]
  static constexpr uint32_t OFF_SC = OFF_OUT + (OUT ? 16384 : 0);  // two sets of gate factors
  static constexpr uint32_t OFF_BAR = OFF_SC + 2 * kStepScB;
  static constexpr int kBars = 28;
  static constexpr uint32_t kSmem = OFF_BAR + kBars * 8 + 16;
  static_assert(kSmem <= 227 * 1024, "shared memory budget");
  // tensor-memory columns (all 512 are allocated, so the base is column 0): X, then D2 | U, then (GDN) plain U~ as operand | Y, then o | h operand | R, then U~ operand
  static constexpr uint32_t TM_X = 0, TM_U = 128, TM_UP = 128, TM_Y = 256, TM_H = 384, TM_R = 448;
};

struct WalkParams {
  const float* h0;             // start states, h0_stride floats from one (sequence, V-head) to the next, or NULL (zeros)
  size_t h0_stride;
  float* hT;
  void* o;
  const int32_t* seq_tok0;     // per-sequence table of the plan kernel, or NULL for equal-length rows
  const int32_t* seq_len;      //   (then sequence n is tokens [n*T_row, (n+1)*T_row), cps steps each)
  const int32_t* seq_chunk0;
  const int32_t* seq_order;    // launch order of the sequences (longest first), or NULL
  int T_row, cps;
  TcWorkspace ws;
  int HK, HV;
  float scale;
  bool withhold;               // test hook: the producers copy nothing, so that the waits for their tiles run out
  uint32_t spin_limit;         // polls before a bounded wait gives up (a few thousand in that test)
  // Spans: a sequence's steps are cut into `nspan` runs that are walked at the same time (1: off), in two launches with
  // span_fix_kernel (tc_span.cu) between them.  The state recurrence is affine in the start state, so
  //   first launch, state only (OUT = false): spans 0 .. nspan-2 from their own start (span 0: h0, others: zero) into
  //     span_b, and spans 1 .. nspan-2 from the IDENTITY with V = 0 (the transition) into span_phi;
  //     in place (hT = h0), span 0 also leaves h0 in span_phi[0], which no transition uses, for the second launch to
  //     start from: its last span may have stored hT before a CTA of its span 0 gets an SM;
  //   fix: h_1 = b_0, h_{s+1} = Phi_s h_s + b_s,  in place of b_{s+1};
  //   second launch (OUT = true): every span from its true start, outputs and final state.
  int nspan;
  bool keep_h0;
  float* span_b;               // [N*HV][nspan][128 keys][128 channels] fp32
  float* span_phi;
  int32_t* status;
};

// named barriers (0 is __syncthreads)
constexpr int BAR_H = 1;       // compute arrive, W_MMA syncs: h operand stored
constexpr int BAR_R = 2;       // ... R operand, first (2) and second (3) half of the tokens
constexpr int BAR_U = 4;       // ... operand of the state update, likewise (4, 5)
constexpr int BAR_UP = 6;      // (GDN) ... plain U~ operand, and Y times e^{G_i}; syncs the second MMA warp
constexpr int BAR_GY = 7;      // the first MMA warp arrives, the second syncs: X issued
constexpr int BAR_GP = 8;      // ... D2 issued
// A CTA lets the stream's next programmatic dependent be scheduled when it has this many steps left (CTAs with fewer:
// when they exit).  That kernel then gets through its launch and set-up under the tail of this one and waits at its
// griddepcontrol.wait for this grid to complete.
constexpr int kTailSteps = 3;
__device__ __forceinline__ void named_arrive(int id, int count) {
  asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(count) : "memory");
}
__device__ __forceinline__ void named_sync(int id, int count) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(count) : "memory");
}

template <bool KDA, bool OUT>
__global__ void __launch_bounds__(walk_threads(OUT), 1)
tc_walk_kernel(const __grid_constant__ CUtensorMap map_k, const __grid_constant__ CUtensorMap map_q,
               const __grid_constant__ CUtensorMap map_v, WalkParams p) {
  using Cfg = WalkCfg<KDA, OUT>;
  constexpr int NK = Cfg::kNK, ND = Cfg::kND, NV = Cfg::kNV, NT = Cfg::kNT;
  extern __shared__ __align__(1024) uint8_t sm[];       // no static shared memory in this kernel: 1024-aligned
  uint64_t* bar = reinterpret_cast<uint64_t*>(sm + Cfg::OFF_BAR);
  uint64_t* full_k = bar;            // [NK] K tile (KDA: K e^G)
  uint64_t* empty_k = bar + 3;       // [NK] D2 of the slot's step complete (its T diag(beta) has been read as well)
  uint64_t* full_d = bar + 6;        // [ND] (KDA) K e^{G_L-G}
  uint64_t* full_q = bar + 8;
  uint64_t* bar_y = bar + 9;         // Y complete (Q and the old h operand have been read)
  uint64_t* full_v = bar + 10;       // [NV]
  uint64_t* empty_v = bar + 12;      // [NV] V read by the compute warps
  uint64_t* full_t = bar + 14;       // [NT]
  uint64_t* full_p = bar + 16;       // (P is free again when the step's output product is complete)
  uint64_t* full_sc = bar + 17;      // [2]
  uint64_t* empty_sc = bar + 19;     // [2] gate factors read by everyone
  uint64_t* bar_x0 = bar + 21;       // X complete for the first 64 tokens
  uint64_t* bar_x = bar + 27;        // ... for the others
  uint64_t* bar_u0 = bar + 22;       // U complete for the first 64 tokens
  uint64_t* bar_u1 = bar + 23;       // ... for the others
  uint64_t* bar_d2 = bar + 24;
  uint64_t* bar_o = bar + 25;        // o complete in tensor memory
  uint64_t* out_free = bar + 26;     // ... and read by the output warps
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bar + Cfg::kBars);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  constexpr int W_OUT = kCompute / 32, W_P0 = W_OUT + (OUT ? 4 : 0), W_P1 = W_P0 + 1, W_MMA = W_P1 + 1;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int units = p.nspan == 1 ? 1 : (OUT ? p.nspan : 2 * p.nspan - 3);   // runs per (sequence, V-head)
  const int unit = blockIdx.x % units;
  const int nj = blockIdx.x / units;
  const bool trans = !OUT && unit >= p.nspan - 1;        // a transition run
  const int span = trans ? unit - p.nspan + 2 : unit;
  const int j = nj % p.HV, jq = j / (p.HV / p.HK);
  const bool packed = p.seq_tok0 != nullptr;
  int n = nj / p.HV, tok0 = packed ? 0 : n * p.T_row, len = p.T_row, slot0 = packed ? 0 : n * p.cps, nsteps;
  auto take_span = [&]() {                               // this CTA's span of the sequence, walked like a sequence of its own
    const int nst = (len + kStep - 1) / kStep;
    const int spspan = (nst + p.nspan - 1) / p.nspan;
    tok0 += span * spspan * kStep;
    slot0 += span * spspan;
    len = max(0, min(len - span * spspan * kStep, spspan * kStep));
    nsteps = (len + kStep - 1) / kStep;
  };
  take_span();

  if (tid == 0) {
    for (int i = 0; i < Cfg::kBars; ++i) {
      const uint64_t* b = bar + i;
      const bool by_compute = b == empty_v || b == empty_v + 1 || b == empty_sc || b == empty_sc + 1;
      mbar_init(&bar[i], by_compute ? kCompute / 32 : b == out_free ? 4 : 1);
    }
    *abort_flag = 0;
    mbar_fence_init();
    prefetch_tmap(&map_v);
    if (!KDA) { prefetch_tmap(&map_k); prefetch_tmap(&map_q); }
  }
  if (warp == 0) tmem_alloc(tmem_slot, 512);
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  constexpr uint32_t tmem = 0;                           // (the whole of tensor memory)
  // Launched as a programmatic dependent: everything above ran under the tail of the kernel before; wait for it here.
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (packed) {
    // (These tables too are read behind the wait only: in a batch without a token there is no chunk-local kernel between the
    // plan kernel, which lets its dependents go before it writes them, and this one.)
    if (p.seq_order) n = p.seq_order[n];                 // CTAs of the longest sequences come first
    tok0 = p.seq_tok0[n];
    len = p.seq_len[n];
    slot0 = p.seq_chunk0[n];
    take_span();
  }

  const int ncopied = p.withhold ? 0 : nsteps;
  auto aborted = [&]() { return __any_sync(0xffffffffu, *abort_flag) != 0; };
  // (mbarrier.try_wait costs the caller ~150 cycles even when the phase is over: test first)
  auto wait1 = [&](uint64_t* b, uint32_t parity) {
    if (!mbar_test_wait(b, parity & 1)) mbar_wait(b, parity & 1, abort_flag, p.spin_limit);
  };

  // KDA's images, records and V do not fit L2 with what comes after them: what this launch is the last to read goes first, and of what the launch with outputs
  // reads again a third, so that the rest is still there then.  HBM bytes of a call without these policies -> with them (and those of tc_kda.cu): 16 heads, T = 4096 235 -> 201 MB,
  // T = 8192 572 -> 502; 32 heads, T = 8192 1123 -> 1093.  Why a third: it loses nowhere.  None, 35, 50, 65, 100 % of what the states-only launch reads, us for a call: 16 heads,
  // T = 8192 130.4 128.5 127.8 128.1 129.3; 8 heads, T = 16000 135.7 133.6 132.8 132.7 134.0; 32 heads on 16 q/k heads, T = 6000 177.4 175.6 175.5 177.6 179.8;
  // 32 heads, T = 4096 126.4 126.0 126.7 127.7 128.3; two rows of 3000, 16 heads on 8 102.3 102.6 102.9 103.3 103.7; T = 8192 with 4 or 32 heads within 0.4 %.
  // GDN's tiles the same way: 803 -> 836 us for 136 k tokens.  The outputs are the caller's, who reads them next: streamed as well, a call takes up to 0.9 % less (32 heads, T = 8192
  // 234 -> 232) and a kernel that reads them 2 - 4 us more (22.5 -> 26.6; call and reader, 32 heads, T = 4096 140.8 -> 143.4; 8 x 500 tokens 62.3 -> 63.7; only outputs
  // larger than L2 gain, T = 16000 483 -> 481).
  uint64_t policy = 0;
  if (KDA) policy = OUT ? evict_first<100>() : evict_first<35>();
  auto copy = [&](void* dst, const void* src, uint32_t bytes, uint64_t* b) {
    if constexpr (KDA) bulk_load(dst, src, bytes, b, policy);
    else bulk_load(dst, src, bytes, b);
  };
  if (warp == W_P0) {
    // ------------------------------------------------------------ producer of the tiles: X / D2 operands, Q, V
    int st = 0;                                          // c % NK
    uint32_t ph = 0;                                     // (c / NK) & 1
    for (int c = 0; c < ncopied; ++c) {
      if (elect_one()) {
        const int t0 = tok0 + c * kStep;
        const uint8_t* img = KDA ? p.ws.img + ((size_t)(slot0 + c) * p.HV + j) * 3 * kTileBytes : nullptr;
        if (c >= NK) {
          if constexpr (KDA && NK == 1) wait1(bar_x, c - 1);             // (X has read it: earlier than D2)
          else wait1(&empty_k[st], ph ^ 1);
        }
        if (!*abort_flag) {
          mbar_expect_tx(&full_k[st], kTileBytes);
          if constexpr (KDA) copy(sm + Cfg::OFF_K + st * kTileBytes, img, kTileBytes, &full_k[st]);
          else tma_load_4d(sm + Cfg::OFF_K + st * kTileBytes, &map_k, &full_k[st], 0, jq, t0, 0);
        }
        if (!trans) {                                    // (transition: V = 0)
          if (c >= NV) wait1(&empty_v[c & 1], (c >> 1) - 1);
          if (!*abort_flag) {
            mbar_expect_tx(&full_v[c & 1], kTileBytes);
            if constexpr (KDA) tma_load_4d(sm + Cfg::OFF_V + (c & 1) * kTileBytes, &map_v, &full_v[c & 1], 0, j, t0, 0, policy);
            else tma_load_4d(sm + Cfg::OFF_V + (c & 1) * kTileBytes, &map_v, &full_v[c & 1], 0, j, t0, 0);
          }
        }
        if constexpr (OUT) {
          if (c > 0) wait1(bar_y, c - 1);
          if (!*abort_flag) {
            mbar_expect_tx(full_q, kTileBytes);
            if constexpr (KDA) copy(sm + Cfg::OFF_Q, img + kTileBytes, kTileBytes, full_q);
            else tma_load_4d(sm + Cfg::OFF_Q, &map_q, full_q, 0, jq, t0, 0);
          }
        }
        if constexpr (KDA) {
          const int ds = ND == 2 ? st : 0;
          if (ND == 1 && c > 0) wait1(&empty_k[0], c - 1);               // (two slots: waited for above)
          if (!*abort_flag) {
            mbar_expect_tx(&full_d[ds], kTileBytes);
            copy(sm + Cfg::OFF_D + ds * kTileBytes, img + 2 * kTileBytes, kTileBytes, &full_d[ds]);
          }
        }
      }
      if (++st == NK) { st = 0; ph ^= 1; }
      if (aborted()) break;
    }
  } else if (warp == W_P1) {
    // ------------------------------------------------------------ producer of the chunk-local kernel's records
    int s2 = 0;                                          // (c - 2) % NK
    uint32_t ph2 = 0;                                    // ((c - 2) / NK) & 1
    for (int c = 0; c < ncopied; ++c) {
      const uint8_t* rec = p.ws.rec + ((size_t)(slot0 + c) * p.HV + j) * kStepRecB;
      if (elect_one()) {
        if (c > 1) wait1(&empty_sc[c & 1], (c >> 1) - 1);
        if (!*abort_flag) {
          mbar_expect_tx(&full_sc[c & 1], kStepScB);
          copy(sm + Cfg::OFF_SC + (c & 1) * kStepScB, rec + kStepSc, kStepScB, &full_sc[c & 1]);
        }
        const int ts = NT == 2 ? c & 1 : 0;
        if (NT == 1 && c > 0) wait1(bar_u1, c - 1);
        if (NT == 2 && c > 1) wait1(&empty_k[s2], ph2);  // (that slot's next step comes after this one: no phase is missed)
        if (!*abort_flag) {
          mbar_expect_tx(&full_t[ts], kTriB);
          copy(sm + Cfg::OFF_T + ts * kTriB, rec + kStepT, kTriB, &full_t[ts]);
        }
        if constexpr (OUT) {
          if (c > 0) wait1(bar_o, c - 1);
          if (!*abort_flag) {
            mbar_expect_tx(full_p, kTriB);
            copy(sm + Cfg::OFF_P, rec + kStepP, kTriB, full_p);
          }
        }
      }
      if (c > 1 && ++s2 == NK) { s2 = 0; ph2 ^= 1; }
      if (aborted()) break;
    }
  } else if (warp >= W_MMA) {
    // ------------------------------------------------------------ MMA issue (one thread issues; the warp waits and keeps the barriers:
    // bar.sync, bar.arrive and elect.sync are for converged warps.  Waits by the elected thread and __syncwarp: 1.5 % more per step)
    // One warp issues the products of the sequential path, another those of the outputs.  The tensor cores work
    // in order of issue, so the second warp goes when the first one tells it to: Y behind X, under X's epilogue, and P U~
    // behind D2, under the epilogue of the state.  Descriptors advance by constants.
    constexpr uint32_t id_kk = idesc_bf16(128, 128, false, false);   // B K-major: X, Y (rows = tokens)
    constexpr uint32_t id_half = idesc_bf16(128, 64, false, false);
    constexpr uint32_t id_km = idesc_bf16(128, 128, false, true);    // B MN-major: D2 (rows = the K index, tokens)
    auto tile_product = [&](uint32_t d, uint64_t b, uint32_t id) {   // rows (tokens) of a K-major B tile, 16 features per instruction
#pragma unroll
      for (int ks = 0; ks < 8; ++ks)
        umma_ts(d, Cfg::TM_H + 8 * ks, b + ((uint32_t)((ks >> 2) * 16384 + (ks & 3) * 32) >> 4), id, ks > 0);
    };
    // A [128 x 128] (triangular operand)^T, k-steps 4 half ..: slab ks is the operand of the result's columns 16 ks ..
    auto tri_half = [&](int half, uint32_t d, uint32_t a, uint32_t astep, uint64_t tri, uint32_t acc) {
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int ks = 4 * half + i;
        umma_ts(d + 16 * ks, a + ks * astep, tri + (tri_slab(ks) >> 4), idesc_bf16(128, 128 - 16 * ks, false, false), acc | (ks > 0));
      }
    };
    if (warp == W_MMA) {
      const uint64_t dK0 = smem_desc(smem_u32(sm + Cfg::OFF_K), 16, 1024, kSwizzle128B);
      const uint64_t dD0 = smem_desc(smem_u32(sm + (KDA ? Cfg::OFF_D : Cfg::OFF_K)), 16384, 1024, kSwizzle128B);
      const uint64_t dT0 = smem_desc(smem_u32(sm + Cfg::OFF_T), 16, 256, kSwizzle32B);
      int st = 0;                                        // c % NK
      uint32_t ph = 0;                                   // (c / NK) & 1
      for (int c = 0; c < nsteps; ++c) {
        const int ts = NT == 2 ? c & 1 : 0;
        const uint64_t dK = dK0 + st * (kTileBytes >> 4);
        const uint64_t dD = dD0 + (ND == 1 ? 0 : st) * (kTileBytes >> 4);
        const uint64_t dT = dT0 + ts * (kTriB >> 4);
        wait1(&full_k[st], ph);
        __syncwarp();
        named_sync(BAR_H, kCompute + 32);                // h operand of the previous step
        if (elect_one()) {
          tc_fence_after_sync();
          tile_product(Cfg::TM_X, dK, id_half);
          umma_commit(bar_x0);
          tile_product(Cfg::TM_X + 64, dK + (64 * 128 >> 4), id_half);
          umma_commit(bar_x);
        }
        __syncwarp();
        if (OUT) named_arrive(BAR_GY, 64);
        wait1(&full_t[ts], NT == 2 ? c >> 1 : c);
        if (OUT && c > 0) wait1(bar_o, c - 1);         // (its operand lies in U's columns)
        __syncwarp();
#pragma unroll
        for (int half = 0; half < 2; ++half) {           // (tokens 0 .. 63 of U are final after the first four k-steps)
          named_sync(BAR_R + half, kCompute + 32);
          if (elect_one()) {
            tc_fence_after_sync();
            tri_half(half, Cfg::TM_U, Cfg::TM_R, 8, dT, 0u);
            umma_commit(half ? bar_u1 : bar_u0);
          }
          __syncwarp();
        }
        if (KDA) wait1(&full_d[ND == 2 ? st : 0], ND == 2 ? ph : c);
        __syncwarp();
#pragma unroll
        for (int half = 0; half < 2; ++half) {
          named_sync(BAR_U + half, kCompute + 32);
          if (elect_one()) {
            tc_fence_after_sync();
#pragma unroll
            for (int ks = 4 * half; ks < 4 * half + 4; ++ks)   // K index = tokens: 16 rows of 128 bytes per step
              umma_ts(Cfg::TM_X, Cfg::TM_R + 8 * ks, dD + ks * (2048u >> 4), id_km, ks > 0);
            if (half) {
              umma_commit(bar_d2);
              umma_commit(&empty_k[st]);
            }
          }
          __syncwarp();
        }
        if (++st == NK) { st = 0; ph ^= 1; }
        if (OUT) named_arrive(BAR_GP, 64);
      }
      named_sync(BAR_H, kCompute + 32);                  // pairs with the compute warps' last arrival
    } else {
      const uint64_t dQ = smem_desc(smem_u32(sm + Cfg::OFF_Q), 16, 1024, kSwizzle128B);
      const uint64_t dP = smem_desc(smem_u32(sm + Cfg::OFF_P), 16, 256, kSwizzle32B);
      for (int c = 0; c < nsteps; ++c) {
        wait1(full_q, c);
        if (c > 0) wait1(out_free, c - 1);
        __syncwarp();
        named_sync(BAR_GY, 64);
        if (elect_one()) {
          tc_fence_after_sync();
          tile_product(Cfg::TM_Y, dQ, id_kk);
          umma_commit(bar_y);
        }
        __syncwarp();
        wait1(full_p, c);
        __syncwarp();
        if (!KDA) named_sync(BAR_UP, kCompute + 32);
        named_sync(BAR_GP, 64);
        if (elect_one()) {
          tc_fence_after_sync();
          tri_half(0, Cfg::TM_Y, KDA ? Cfg::TM_R : Cfg::TM_UP, KDA ? 8 : 16, dP, 1u);
          tri_half(1, Cfg::TM_Y, KDA ? Cfg::TM_R : Cfg::TM_UP, KDA ? 8 : 16, dP, 1u);
          umma_commit(bar_o);
        }
        __syncwarp();
      }
    }
  } else if (warp >= W_OUT) {
    // ------------------------------------------------------------ output warps: o, transposed
    if constexpr (OUT) {
      const int q = warp - W_OUT;
      const int lm = lane >> 3, lr = lane & 7;
      const uint32_t ty = tmem + Cfg::TM_Y + (static_cast<uint32_t>(q * 32) << 16);
      const uint32_t tile = smem_u32(sm + Cfg::OFF_OUT) + q * 4096;       // [64 tok][32 ch], 64-byte rows
      const uint32_t tile0[2] = {tile + sw64_offset((lm >> 1) * 8 + lr, lm & 1), tile + sw64_offset((lm >> 1) * 8 + lr, 2 + (lm & 1))};
      __nv_bfloat16* obase = reinterpret_cast<__nv_bfloat16*>(p.o) + (size_t)j * 128 + q * 32;
      for (int c = 0; c < nsteps; ++c) {
        wait1(bar_o, c);
        tc_fence_after_sync();
        uint32_t r[2][2][16];
        auto load_o = [&](int tb) {
#pragma unroll
          for (int hl = 0; hl < 2; ++hl) tmem_ld_16x256b_x4(ty + (static_cast<uint32_t>(16 * hl) << 16) + 32 * tb, r[tb & 1][hl]);
        };
        // 32 tokens x 16 channels, packed: [m] is 16 tokens
        auto pack_o = [&](int tb, int hl, uint32_t (&w)[2][4]) {
#pragma unroll
          for (int m = 0; m < 2; ++m)
#pragma unroll
            for (int x = 0; x < 4; ++x) w[m][x] = pack_bf16(as_f2(r[tb & 1][hl][8 * m + 2 * x], r[tb & 1][hl][8 * m + 2 * x + 1]));
        };
        auto stage = [&](int tb, int hl, const uint32_t (&w)[2][4]) {     // transposed on the way
#pragma unroll
          for (int m = 0; m < 2; ++m) stsm4t(tile0[hl] + (32 * (tb & 1) + 16 * m) * 64, w[m]);
        };
        const int left = len - c * kStep;
        __nv_bfloat16* orow = obase + (size_t)(tok0 + c * kStep) * p.HV * 128 + (lane & 3) * 8;
        auto send = [&](int half) {
          __syncwarp();
#pragma unroll 4
          for (int it = 0; it < 8; ++it) {
            const int t = it * 8 + (lane >> 2);
            uint32_t w[4];
            lds4(w, tile + sw64_offset(t, lane & 3));
            if (64 * half + t < left) *reinterpret_cast<uint4*>(orow + (size_t)(64 * half + t) * p.HV * 128) = make_uint4(w[0], w[1], w[2], w[3]);
          }
          __syncwarp();
        };
        uint32_t later[2][2][2][4];                      // the second 64 tokens, out of tensor memory before the first are sent
        load_o(0);
#pragma unroll
        for (int tb = 0; tb < 4; ++tb) {
          tmem_ld_wait();
          if (tb < 3) load_o(tb + 1);
          else {
            tc_fence_before_sync();
            __syncwarp();
            if (lane == 0) mbar_arrive(out_free);        // (the next Y may go there)
          }
#pragma unroll
          for (int hl = 0; hl < 2; ++hl) {
            if (tb < 2) {
              uint32_t w[2][4];
              pack_o(tb, hl, w);
              stage(tb, hl, w);
            } else {
              pack_o(tb, hl, later[tb - 2][hl]);
            }
          }
        }
        send(0);
#pragma unroll
        for (int tb = 2; tb < 4; ++tb)
#pragma unroll
          for (int hl = 0; hl < 2; ++hl) stage(tb, hl, later[tb - 2][hl]);
        send(1);
      }
    }
  } else {
    // ------------------------------------------------------------ compute
    // tensor-memory lanes 32 q ..; columns: keys 32 g .. of the state, tokens 16 g .. of each half of the step
    const int q = warp & 3, g = warp >> 2;
    const int v = q * 32 + lane;                         // value channel of the 32x32b accesses
    const int lm = lane >> 3, lr = lane & 7, t2 = (lane & 3) * 2;
    const uint32_t tq = tmem + (static_cast<uint32_t>(q * 32) << 16);
    float h[32];                                         // h^T[v][32 g ..]
    {
      const float* src = nullptr;
      if (span == 0 && !trans) src = p.h0 ? p.h0 + ((size_t)n * p.HV + j) * p.h0_stride : nullptr;
      else if (OUT) src = p.span_b + (((size_t)n * p.HV + j) * p.nspan + span) * 16384;
#pragma unroll
      for (int k = 0; k < 32; ++k) h[k] = src ? src[(size_t)(32 * g + k) * 128 + v] : (trans && 32 * g + k == v ? 1.f : 0.f);
      if (!OUT && p.keep_h0 && span == 0 && !trans) {
        float* keep = p.span_phi + ((size_t)n * p.HV + j) * p.nspan * 16384;
#pragma unroll
        for (int k = 0; k < 32; ++k) keep[(size_t)(32 * g + k) * 128 + v] = h[k];
      }
    }
    auto step_h = [&](int k, float2 decay, float2 add) {
      const float2 x = fma2(decay, make_float2(h[k], h[k + 1]), add);
      h[k] = x.x;
      h[k + 1] = x.y;
    };
    auto store_h = [&]() {                               // bf16 pairs of this thread's key channels -> A operand
      uint32_t r[16];
#pragma unroll
      for (int k = 0; k < 16; ++k) r[k] = pack_bf16(h[2 * k], h[2 * k + 1]);
      tmem_st16(tq + Cfg::TM_H + 16 * g, r);
      tmem_st_wait();
    };
    store_h();
    tc_fence_before_sync();
    named_arrive(BAR_H, kCompute + 32);

    const uint32_t hi = 16u << 16;                       // sixteen lanes further
    uint32_t va0 = smem_u32(sm + Cfg::OFF_V) + ((4 * q) >> 3) * 16384;    // (of the step's slot)
    uint32_t vv[2][4], x[2][8];
    auto load_v = [&](int tk) {                          // V^T of 16 tokens, 2 x 16 channels (transposed by ldmatrix)
#pragma unroll
      for (int hl = 0; hl < 2; ++hl)
        ldsm4t(vv[hl], va0 + sw128_offset(tk + (lm >> 1) * 8 + lr, (4 * q + 2 * hl + (lm & 1)) & 7));
    };
    auto load_x = [&](int tk) {
#pragma unroll
      for (int hl = 0; hl < 2; ++hl) tmem_ld_16x256b_x2(tq + hl * hi + Cfg::TM_X + tk, x[hl]);
    };
    if (trans) {
#pragma unroll
      for (int i = 0; i < 8; ++i) vv[i >> 2][i & 3] = 0u;
    }
    for (int c = 0, to_go = nsteps; to_go > 0; ++c, --to_go) {
      if (to_go == kTailSteps) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
      wait1(&full_sc[c & 1], c >> 1);
      // GDN: e^{G_t}[128], e^{G_L-G_t}[128]; KDA: e^{G_L} per key
      const float* sc = reinterpret_cast<const float*>(sm + Cfg::OFF_SC + (c & 1) * kStepScB);
      if (!trans) {
        wait1(&full_v[c & 1], c >> 1);
        load_v(16 * g);
      }
      wait1(bar_x0, c);
      tc_fence_after_sync();
      load_x(16 * g);
      if (KDA && OUT && c > 0) wait1(bar_o, c - 1);      // P U~ of the previous step has read its operand there
      // ---- R^T = V^T - e^{G_j} X^T, in fragment layout
#pragma unroll
      for (int half = 0; half < 2; ++half) {
        const int tk = 64 * half + 16 * g;
        float2 e[2];                                     // -e^{G_j} of tokens tk + 8 k + t2, + 1
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          e[k] = make_float2(-1.f, -1.f);
          if (!KDA) {
            const float2 f = *reinterpret_cast<const float2*>(sc + tk + 8 * k + t2);
            e[k] = make_float2(-f.x, -f.y);
          }
        }
        tmem_ld_wait();
#pragma unroll
        for (int hl = 0; hl < 2; ++hl) {
          uint32_t w[4];
#pragma unroll
          for (int y = 0; y < 2; ++y)                    // rows g8, g8 + 8
#pragma unroll
            for (int k = 0; k < 2; ++k)                  // tokens 8 k + t2, + 1; columns in step_pos order
              w[2 * y + k] = pack_bf16(fma2(e[k], as_f2(x[hl][4 * k + 2 * y], x[hl][4 * k + 2 * y + 1]), unpack_bf16(vv[hl][2 * k + y])));
          tmem_st_16x256b_x1(tq + hl * hi + Cfg::TM_R + tk / 2, w);
        }
        tmem_st_wait();
        tc_fence_before_sync();
        named_arrive(BAR_R + half, kCompute + 32);
        if (half == 0) {
          wait1(bar_x, c);
          tc_fence_after_sync();
          load_x(64 + 16 * g);
          if (!trans) load_v(64 + 16 * g);
        }
      }
      __syncwarp();
      if (!trans && lane == 0) mbar_arrive(&empty_v[c & 1]);
      va0 += (c & 1) ? -(int)kTileBytes : (int)kTileBytes;

      // ---- U~^T as operands.  GDN: times e^{G_L-G_t} for the state update, and plain for the outputs, over columns of U
      // that this warp has read already (columns in step_pos order).  KDA: the latter for both.
#pragma unroll
      for (int half = 0; half < 2; ++half) {
        const int tk = 64 * half + 16 * g;
        float4 e[4];                                     // e^{G_L-G_t}
        if (!KDA) {
#pragma unroll
          for (int k = 0; k < 4; ++k) e[k] = *reinterpret_cast<const float4*>(sc + 128 + tk + 4 * k);
        }
        wait1(half ? bar_u1 : bar_u0, c);
        tc_fence_after_sync();
        uint32_t u[16], w[8];
        tmem_ld16(tq + Cfg::TM_U + tk, u);
        tmem_ld_wait();
        if constexpr (!KDA) {
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            w[2 * k] = pack_bf16(mul2(as_f2(u[4 * k], u[4 * k + 1]), make_float2(e[k].x, e[k].y)));
            w[2 * k + 1] = pack_bf16(mul2(as_f2(u[4 * k + 2], u[4 * k + 3]), make_float2(e[k].z, e[k].w)));
          }
          tmem_st8(tq + Cfg::TM_R + tk / 2, w);
          tmem_st_wait();
          tc_fence_before_sync();
          named_arrive(BAR_U + half, kCompute + 32);
        }
        if constexpr (KDA || OUT) {
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            w[2 * k] = pack_bf16(__uint_as_float(u[2 * k]), __uint_as_float(u[2 * k + 1]));
            w[2 * k + 1] = pack_bf16(__uint_as_float(u[8 + 2 * k]), __uint_as_float(u[9 + 2 * k]));
          }
          tmem_st8(tq + (KDA ? Cfg::TM_R + tk / 2 : Cfg::TM_UP + tk), w);
          if (KDA) {
            tmem_st_wait();
            tc_fence_before_sync();
            named_arrive(BAR_U + half, kCompute + 32);
          }
        }
      }

      if (OUT) wait1(bar_y, c);
      if constexpr (OUT && !KDA) {                       // Y <- scale e^{G_i} Y in place while D2 runs; then (scale P) U~ is added to it
        tc_fence_after_sync();
#pragma unroll
        for (int half = 0; half < 2; ++half) {
          const int tk = 64 * half + 16 * g;
#pragma unroll
          for (int hl = 0; hl < 2; ++hl) tmem_ld_16x256b_x2(tq + hl * hi + Cfg::TM_Y + tk, x[hl]);
          float2 e[2];
#pragma unroll
          for (int k = 0; k < 2; ++k) e[k] = mul2(*reinterpret_cast<const float2*>(sc + tk + 8 * k + t2), make_float2(p.scale, p.scale));
          tmem_ld_wait();
#pragma unroll
          for (int hl = 0; hl < 2; ++hl) {
#pragma unroll
            for (int k = 0; k < 4; ++k) {
              const float2 y = mul2(as_f2(x[hl][2 * k], x[hl][2 * k + 1]), e[k >> 1]);
              x[hl][2 * k] = __float_as_uint(y.x);
              x[hl][2 * k + 1] = __float_as_uint(y.y);
            }
            tmem_st_16x256b_x2(tq + hl * hi + Cfg::TM_Y + tk, x[hl]);
          }
        }
        tmem_st_wait();
        tc_fence_before_sync();
        named_arrive(BAR_UP, kCompute + 32);
      }
      wait1(bar_d2, c);
      tc_fence_after_sync();
      // ---- h^T <- decay h^T + D2
      {
        uint32_t d[32];
        tmem_ld32(tq + Cfg::TM_X + 32 * g, d);
        tmem_ld_wait();
        if constexpr (KDA) {
#pragma unroll
          for (int k = 0; k < 32; k += 4) {
            const float4 gm = *reinterpret_cast<const float4*>(sc + 32 * g + k);   // decay per key channel
            step_h(k, make_float2(gm.x, gm.y), as_f2(d[k], d[k + 1]));
            step_h(k + 2, make_float2(gm.z, gm.w), as_f2(d[k + 2], d[k + 3]));
          }
        } else {
          const float gm = sc[127];                      // one decay for the whole step
#pragma unroll
          for (int k = 0; k < 32; k += 2) step_h(k, make_float2(gm, gm), as_f2(d[k], d[k + 1]));
        }
      }
      store_h();                                         // (Y has read the old operand)
      tc_fence_before_sync();
      named_arrive(BAR_H, kCompute + 32);
      __syncwarp();
      if (lane == 0) mbar_arrive(&empty_sc[c & 1]);
    }

    // where the end state goes: hT (from the last span), or the span's offset b_s / transition Phi_s
    float* dst = nullptr;
    if (!OUT) dst = (trans ? p.span_phi : p.span_b) + (((size_t)n * p.HV + j) * p.nspan + span) * 16384;
    else if (p.hT && span == p.nspan - 1) dst = p.hT + ((size_t)n * p.HV + j) * 16384;
    if (!OUT && trans) {
      // Phi_s as the start states' products take it (phi_word): split into two bf16, the halves of a pair of neighbouring columns v
      // from neighbouring lanes.  An even lane writes the first 16 of this thread's rows, an odd one the others.
      uint32_t* word = reinterpret_cast<uint32_t*>(dst) + phi_word(2 * g + (lane & 1), 0, v);
      const bool odd = lane & 1;
      float x[16], y[16];
#pragma unroll
      for (int k = 0; k < 16; ++k) {
        const float got = __shfl_xor_sync(0xffffffffu, odd ? h[k] : h[16 + k], 1);
        x[k] = odd ? got : h[k];
        y[k] = odd ? h[16 + k] : got;
      }
#pragma unroll
      for (int k = 0; k < 16; k += (k & 1) ? 3 : 1) {    // rows k and k + 2 are neighbours there
        uint2 hi, lo;
        split_bf16(x[k], y[k], hi.x, lo.x);
        split_bf16(x[k + 2], y[k + 2], hi.y, lo.y);
        *reinterpret_cast<uint2*>(word + phi_word(0, k, 0)) = hi;
        *reinterpret_cast<uint2*>(word + phi_word(0, k, 0) + 128) = lo;
      }
    } else if (dst) {
#pragma unroll
      for (int k = 0; k < 32; ++k) dst[(size_t)(32 * g + k) * 128 + v] = h[k];
    }
  }

  tc_fence_before_sync();
  __syncthreads();
  if (*abort_flag) {
    // A wait ran out: the producers have stopped.
    if (tid == 0) report_status(p.status, HA_LA_ERR_TIMEOUT);
    settle_copies();
  }
  if (warp == 0) tmem_dealloc(*tmem_slot, 512);
}

template <bool KDA, bool OUT>
cudaError_t run_walk(const WalkParams* wp, const CUtensorMap* mk, const CUtensorMap* mq, const CUtensorMap* mv, int grid,
                     bool dependent, cudaStream_t stream) {
  auto kern = tc_walk_kernel<KDA, OUT>;
  constexpr int smem = WalkCfg<KDA, OUT>::kSmem;
  if (!wp) {                                             // configure only (this also loads the kernel)
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
  }
  timer_mark(stream, OUT ? "tc_chain" : "tc_span");
  // `dependent`: programmatic dependent launch behind the kernel before it (same stream): the CTAs may start as soon
  // as every CTA of that one is running, instead of after its grid has drained.
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3(walk_threads(OUT));
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = dependent ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kern, *mk, *mq, *mv, *wp);
}

}  // namespace

// `states_only`: the first of the two launches of a call whose sequences are cut into spans.
cudaError_t launch_tc_walk(const Problem& p, const ha_la_prefill_args& a, PlanView plan, const TcWorkspace& ws,
                           const CUtensorMap& mk, const CUtensorMap& mq, const CUtensorMap& mv, bool withhold,
                           bool dependent, uint32_t spin_limit, const SpanBuffers& sb, bool states_only,
                           cudaStream_t stream) {
  WalkParams wp;
  const bool in_place = sb.nspan > 1 && a.h0 && a.h0 == a.hT;
  wp.keep_h0 = in_place && states_only;
  wp.h0 = in_place && !states_only ? sb.phi : a.h0;
  wp.h0_stride = in_place && !states_only ? (size_t)sb.nspan * 16384 : 16384;
  wp.hT = a.hT; wp.o = a.o;
  wp.seq_tok0 = plan.seq_tok0; wp.seq_len = plan.seq_len; wp.seq_chunk0 = plan.seq_chunk0;
  wp.seq_order = plan.seq_tok0 ? plan.seq_order : nullptr;
  wp.T_row = p.T_row; wp.cps = p.max_seq_chunks > 0 ? p.max_seq_chunks : 1;
  wp.ws = ws; wp.HK = p.HK; wp.HV = p.HV; wp.scale = p.scale; wp.status = a.status_word;
  wp.withhold = withhold;
  wp.spin_limit = spin_limit;
  wp.nspan = sb.nspan; wp.span_b = sb.b; wp.span_phi = sb.phi;
  const int grid = p.N * p.HV * (states_only ? 2 * sb.nspan - 3 : sb.nspan);
  if (grid == 0) return cudaSuccess;
  const bool kda = p.variant == HA_LA_KDA;
  if (states_only) return kda ? run_walk<true, false>(&wp, &mk, &mq, &mv, grid, dependent, stream)
                              : run_walk<false, false>(&wp, &mk, &mq, &mv, grid, dependent, stream);
  return kda ? run_walk<true, true>(&wp, &mk, &mq, &mv, grid, dependent, stream)
             : run_walk<false, true>(&wp, &mk, &mq, &mv, grid, dependent, stream);
}

// Attributes (and loading) of the instances a launch can use.
cudaError_t configure_tc_walk(const Problem& p) {
  const bool kda = p.variant == HA_LA_KDA;
  cudaError_t e = kda ? run_walk<true, false>(nullptr, nullptr, nullptr, nullptr, 0, false, nullptr)
                      : run_walk<false, false>(nullptr, nullptr, nullptr, nullptr, 0, false, nullptr);
  if (e != cudaSuccess) return e;
  return kda ? run_walk<true, true>(nullptr, nullptr, nullptr, nullptr, 0, false, nullptr)
             : run_walk<false, true>(nullptr, nullptr, nullptr, nullptr, 0, false, nullptr);
}

}  // namespace ha_la
