// Tensor-core (tcgen05) path, host side: tensor maps, workspace carving, spans, launches.
//
// The chunk-local kernel (tc_tp.cu, KDA: tc_kda.cu) and the state-passing kernel (tc_walk.cu) go on the caller's stream one
// behind the other, both in steps of 128 tokens; where sequences are cut into spans, the latter runs twice with the spans'
// start states (tc_span.cu) between.  Each is a programmatic dependent of the one before: it is set up under its tail.
#include <cuda.h>
#include <stdlib.h>

#include <atomic>

#include "tc_common.cuh"

namespace ha_la {

cudaError_t launch_tc_tp(const Problem& p, const ha_la_prefill_args& a, PlanView plan, const TcWorkspace& ws,
                         const CUtensorMap& mq, const CUtensorMap& mk, int ctas, cudaStream_t stream);
cudaError_t launch_tc_kda(const Problem& p, const ha_la_prefill_args& a, PlanView plan, const TcWorkspace& ws,
                          const CUtensorMap& mq, const CUtensorMap& mk, int ctas, cudaStream_t stream);
cudaError_t launch_tc_walk(const Problem& p, const ha_la_prefill_args& a, PlanView plan, const TcWorkspace& ws,
                           const CUtensorMap& mk, const CUtensorMap& mq, const CUtensorMap& mv, bool withhold,
                           bool dependent, uint32_t spin_limit, const SpanBuffers& sb, bool states_only,
                           cudaStream_t stream);
cudaError_t launch_span_fix(const Problem& p, PlanView plan, const SpanBuffers& sb, int32_t* status, cudaStream_t stream);
cudaError_t configure_span_fix();
cudaError_t configure_tc_tp();
cudaError_t configure_tc_walk(const Problem& p);
cudaError_t configure_tc_kda();

int sm_count() {
  static int n = [] {
    int dev = 0, v = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 148;
    if (cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || v <= 0) return 148;
    return v;
  }();
  return n;
}

namespace {

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// The driver entry point is looked up through the runtime, so the library does not link libcuda.
EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = [] {
    void* f = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &f, cudaEnableDefault, &q) != cudaSuccess) f = nullptr;
    return reinterpret_cast<EncodeTiledFn>(f);
  }();
  return fn;
}

// [T][H][128] bf16 token-major tensor, in tiles of 128 features x 1 head x 128 tokens, as two 64-feature halves of 128-byte rows one after the
// other ([kb][128 tok][64 feat], 128-byte swizzle): the feature halves are the outermost dimension of the map.
bool make_map_tile(CUtensorMap* m, const void* base, int T, int H) {
  EncodeTiledFn enc = encode_fn();
  if (!enc) return false;
  const cuuint64_t dims[4] = {64, (cuuint64_t)H, (cuuint64_t)(T > 0 ? T : 1), 2};
  const cuuint64_t strides[3] = {128 * 2, (cuuint64_t)H * 128 * 2, 64 * 2};
  const cuuint32_t box[4] = {64, 1, (cuuint32_t)kStep, 2};
  const cuuint32_t es[4] = {1, 1, 1, 1};
  return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(base), dims, strides, box, es,
             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

constexpr int kMaxDevices = 64;
constexpr uint32_t kDefaultSpinLimit = 4u << 20;      // polls before a device-side bounded wait gives up

// HA_LA_TC_SEGMENTS, or 0
int forced_segments() {
  const char* e = getenv("HA_LA_TC_SEGMENTS");
  const int v = e ? atoi(e) : 0;
  return v == 1 || v == 2 || v == 4 || v == 8 ? v : 0;
}

// Spans per sequence of the step path (tc_walk.cu): with few (sequence, head) pairs a sequence is cut into S runs that
// are walked at the same time, in two launches, 2 S - 3 state-only runs and then S runs with outputs, with S - 2
// products of 128^3 between them.  The rule's costs: 2.0 us per state-only step, 2.45 per step with outputs, 5 for
// a CTA's start and end, 1.25 per product (0.75 where the products' CTAs take 8 columns, 5 where CTAs of 16 do not all have an SM: tc_span.cu) and about 8 for
// the two further launches.  The steps take less now (tc_walk.cu), but with 1.65 and 2.25 here the choice gets no better: it
// changes in 5 % of calls, and 44 of those timed both ways went from 13 % longer (one row of 1300 tokens, 4 heads, in order instead of 6
// runs 28.8 -> 32.6 us) to 7 % shorter (three sequences of 3 k tokens, 4 heads, 13 runs -> 9 68.4 -> 63.4), 0.1 % longer on average.  A CTA fills an SM: equal lengths go in whole rounds, others pack (the longest first) to
// within some 15 %.  And no launch beats HBM, at 6 TB/s, once its operands do not stay in L2: a packed batch of 8 sequences
// with 136 k tokens cut in two took 220 + 15 us for the first launch and the products and 452 for the second, 444 of them
// HBM's, against 570 us uncut (1160 against 1021 for the call).
int plan_spans(const Problem& p) {
  const long long chains = (long long)p.N * p.HV;
  const int sms = sm_count(), longest = (p.max_len + kStep - 1) / kStep;
  const double avg_len = p.N > 0 ? (double)p.T_total / p.N : 0.0;
  const bool even = p.max_len < 1.5 * avg_len;
  const double total = (double)p.max_chunks * p.HV;
  const bool kda = p.variant == HA_LA_KDA;
  auto launch_us = [&](int runs, int spans, bool out) {
    const double step_us = out ? 2.45 : 2.0;
    const int cps = (longest + spans - 1) / spans;
    const long long ctas = chains * runs;
    double t = cps * step_us + 5.0;
    if (ctas > sms && even) {
      t *= (double)((ctas + sms - 1) / sms);
    } else if (ctas > sms) {
      const double spread = 1.15 * total * runs / spans / sms;
      t = (spread > cps ? spread : cps) * step_us + 5.0 * (double)ctas / sms;
    }
    // bytes of a step: the tiles (GDN: K and Q once per group of heads), V, the record, the outputs
    const double qk = kda ? 1.0 : (double)p.HK / p.HV;
    const double bytes = kTileBytes * (qk * (kda ? 2 + out : 1 + out) + 1 + out) + kTriB * (1 + out) + kStepScB;
    const double moved = total * runs / spans * bytes;
    return moved > 126e6 && moved / 6e6 > t ? moved / 6e6 : t;
  };
  int best_s = 1;
  double best = launch_us(1, 1, true);
  for (int S = 2; S <= 32 && S <= longest; ++S) {
    const double t = launch_us(2 * S - 3, S, false) + launch_us(S, S, true) + (16 * chains <= sms ? 0.75 : 8 * chains <= sms ? 1.25 : 5.0) * (S - 2) + 8.0;
    if (t < best) { best = t; best_s = S; }
  }
  return best_s;
}

// What ha_la_prefill_launch_plan and ha_la_prefill_num_segments answer, and what a forced HA_LA_TC_SEGMENTS must fit.  No
// launch follows it: it is the cost model of a pair of kernels in chunks of 64 tokens that stood before the step kernels, kept
// because callers may have built on the answers and on the workspace size.  The pair was a chunk-local kernel, which ran at
// 3.45 (GDN) / 9.8 (KDA) SM-microseconds per (chunk, head), never faster than its rounds of 9 / 10.5 us, and a state-passing
// kernel of 0.9 / 1.23 / 1.5 us per chunk for slices of 32 / 64 / 128 value channels, a CTA and an SM each; it could run
// beside the first one where it left that one half of the SMs, or cut a sequence into segments.
struct TcPlan { int nv; bool concurrent; int nseg; };

TcPlan plan_tc(const Problem& p) {
  const int sms = sm_count();
  const long long chains = (long long)p.N * p.HV;
  const double longest = (double)((p.max_len + kChunk - 1) / kChunk);
  const long long chunks = p.varlen ? ((long long)p.T_total + (kChunk - 1LL) * p.N) / kChunk : (long long)p.N * ((p.max_len + kChunk - 1) / kChunk);
  const double items = (double)chunks * p.HV;
  const int widths[3] = {32, 64, 128};
  const double per_chunk_us[3] = {0.90, 1.23, 1.50};
  const bool kda = p.variant == HA_LA_KDA;
  auto prep_time = [&](int on_sms) {                     // the chunk-local kernel on `on_sms` SMs
    const double thru = items * (kda ? 9.8 : 3.45) / on_sms;
    const double groups = (double)on_sms * (kda ? 1 : 3);
    const double rounds = (double)(long long)((items + groups - 1) / groups) * (kda ? 10.5 : 9.0);
    return thru > rounds ? thru : rounds;
  };
  const double prep_us = prep_time(sms);
  // sequences of about the same length (batch rows, or a packed batch whose longest is close to its average)
  // cannot be packed any better than in rounds of one CTA per SM
  const double avg_len = p.N > 0 ? (double)p.T_total / p.N : 0.0;
  const bool even = avg_len <= 0.0 || p.max_len < 1.5 * avg_len;
  bool may_overlap = chunks > 1;
  bool force_overlap = false;                            // "2": side by side whenever that is legal (tests)
  if (const char* e = getenv("HA_LA_TC_OVERLAP")) {
    may_overlap = may_overlap && e[0] != '0';
    force_overlap = may_overlap && e[0] == '2';
  }
  int forced_nv = 0;
  if (const char* e = getenv("HA_LA_TC_NV")) {
    const int v = atoi(e);
    if (v == 32 || v == 64 || v == 128) forced_nv = v;
  }
  TcPlan plan{32, false, 1};
  double best = 1e30;
  for (int w = 0; w < 3; ++w) {
    if (forced_nv && widths[w] != forced_nv) continue;
    const long long ctas = chains * (128 / widths[w]);
    const double serial = longest * per_chunk_us[w];
    double chain_us = serial;
    if (ctas > sms) {
      const double spread = 1.15 * items * (128 / widths[w]) * per_chunk_us[w] / sms;
      chain_us = even ? serial * (double)((ctas + sms - 1) / sms) : (serial > spread ? serial : spread);
    }
    const double back_to_back = prep_us + chain_us + (force_overlap ? 1e9 : 0.0);
    if (back_to_back < best) { best = back_to_back; plan = TcPlan{widths[w], false, 1}; }
    if (may_overlap && ctas * 2 <= sms) {
      const double prep_beside = 1.1 * prep_time(sms - (int)ctas);
      double overlapped = (chain_us > prep_beside ? chain_us : prep_beside) + 12.0;
      if (p.N > 1) {
        const double last = prep_beside * (1.0 - 1.0 / p.N) + chain_us + 12.0;
        if (last > overlapped) overlapped = last;
      }
      if (overlapped < best) { best = overlapped; plan = TcPlan{widths[w], true, 1}; }
    }
  }
  // Segments: a later one cost three times the columns of the first, 3.1 us for its start state and 15 ns per chunk-head for
  // the correction of its outputs, and they paid only while all CTAs had an SM each.
  const int forced_seg = forced_segments();
  if ((!p.varlen || forced_seg > 1) && forced_seg != 1 && longest >= 2) {
    for (int w = 0; w < 2; ++w) {                          // 32- and 64-channel slices
      if (forced_nv && widths[w] != forced_nv) continue;
      for (int nseg = 2; nseg <= 8; nseg *= 2) {
        if (forced_seg && nseg != forced_seg) continue;
        if (nseg > longest) continue;
        const long long ctas = chains * (128 / widths[w]) * (2 * nseg - 1);
        if (ctas > sms && !forced_seg) continue;
        const double cpseg = (double)(long long)((longest + nseg - 1) / nseg);
        const double waves = (double)((ctas + sms - 1) / sms);
        const double later = items * (1.0 - 1.0 / nseg);
        const double t = prep_us + waves * cpseg * per_chunk_us[w] + (7.0 + 3.1 * (nseg - 1)) + (9.0 + 0.015 * later);
        if (t < best || (forced_seg && plan.nseg != forced_seg)) { best = t; plan = TcPlan{widths[w], false, nseg}; }
      }
    }
  }
  return plan;
}

}  // namespace

bool tc_supported(const Problem& p) {
  return p.dtype == HA_LA_BF16 && p.dk == 128 && p.dv == 128;
}

void tc_plan(Problem* p) {
  const int forced = forced_segments();
  const bool fits = forced > 1 && forced <= (p->max_len + kChunk - 1) / kChunk;
  p->planned_runs = plan_spans(*p);
  p->segments = fits ? forced : plan_tc(*p).nseg;
  p->runs = forced == 1 ? 1 : fits ? forced : p->planned_runs;
}

// Step records (and images), the scratch of the planned runs, and, when the planner above answers with segments, scratch
// for that many, which only runs that are forced use.  (The call checks the caller's size against this same function, so an
// environment switch that is changed between sizing and calling ends in HA_LA_ERR_WORKSPACE, not in an overrun.)
static size_t tc_base_bytes(const Problem& p) {
  return tc_ws_bytes_for((size_t)p.max_chunks * p.HV, p.variant == HA_LA_KDA) + tc_span_bytes((size_t)p.N * p.HV, p.planned_runs);
}

size_t tc_workspace_bytes(const Problem& p) {
  return tc_base_bytes(p) + tc_seg_bytes((size_t)p.N * p.HV, p.segments, (size_t)p.T_total, p.HV);
}

static SpanBuffers call_spans(const Problem& p, void* tc_ws) {
  uint8_t* b = reinterpret_cast<uint8_t*>(tc_ws);
  const size_t nj = (size_t)p.N * p.HV;
  if (p.runs > 1 && p.runs == p.segments) return tc_span_view(b + tc_base_bytes(p), nj, p.runs);   // (forced, or the same either way)
  return tc_span_view(b + tc_ws_bytes_for((size_t)p.max_chunks * p.HV, p.variant == HA_LA_KDA), nj, p.runs);
}

void tc_launch_plan(const Problem& p, int* slice_width, int* concurrent) {
  const TcPlan tp = plan_tc(p);
  *slice_width = tp.nv;
  *concurrent = tp.concurrent ? 1 : 0;
}

cudaError_t launch_tc(const Problem& p, const ha_la_prefill_args& a, PlanView plan, void* tc_ws, cudaStream_t stream) {
  const bool kda = p.variant == HA_LA_KDA;
  const TcWorkspace ws = tc_ws_view(tc_ws, (size_t)p.max_chunks * p.HV, kda);
  const SpanBuffers sb = call_spans(p, tc_ws);
  CUtensorMap mq, mk, mv;
  if (!make_map_tile(&mq, a.q, p.T_total, p.HK) || !make_map_tile(&mk, a.k, p.T_total, p.HK) ||
      !make_map_tile(&mv, a.v, p.T_total, p.HV))
    return cudaErrorInvalidValue;
  // Once per device: the attributes stick, and the calls are not free on the host.
  static std::atomic<uint32_t> configured[kMaxDevices];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return cudaErrorInvalidDevice;
  const uint32_t bit = kda ? 2u : 1u;
  if (dev < 0 || dev >= kMaxDevices || !(configured[dev].load() & bit)) {
    cudaError_t ce = kda ? configure_tc_kda() : configure_tc_tp();
    if (ce == cudaSuccess) ce = configure_tc_walk(p);
    if (ce == cudaSuccess) ce = configure_span_fix();
    if (ce != cudaSuccess) return ce;
    if (dev >= 0 && dev < kMaxDevices) configured[dev].fetch_or(bit);
  }
  const bool dependent = g_timer == nullptr;             // (per-kernel timing wants one kernel at a time)
  cudaError_t e = kda ? launch_tc_kda(p, a, plan, ws, mq, mk, sm_count(), stream) : launch_tc_tp(p, a, plan, ws, mq, mk, sm_count(), stream);
  if (e == cudaSuccess && sb.nspan > 1) {
    e = launch_tc_walk(p, a, plan, ws, mk, mq, mv, false, dependent, kDefaultSpinLimit, sb, true, stream);
    if (e == cudaSuccess) e = launch_span_fix(p, plan, sb, a.status_word, stream);
  }
  return e != cudaSuccess ? e : launch_tc_walk(p, a, plan, ws, mk, mq, mv, false, dependent, kDefaultSpinLimit, sb, false, stream);
}

// Test hook behind ha_la_debug_wait_timeout: the state-passing kernel alone, with its copies withheld and a small poll limit.
// Its waits for the tiles run out, it records the time-out and runs its barriers to a normal exit.
cudaError_t launch_tc_withheld(const Problem& p, const ha_la_prefill_args& a, void* tc_ws, uint32_t spin_limit,
                               cudaStream_t stream) {
  CUtensorMap mq, mk, mv;
  if (!make_map_tile(&mq, a.q, p.T_total, p.HK) || !make_map_tile(&mk, a.k, p.T_total, p.HK) ||
      !make_map_tile(&mv, a.v, p.T_total, p.HV))
    return cudaErrorInvalidValue;
  const TcWorkspace ws = tc_ws_view(tc_ws, (size_t)p.max_chunks * p.HV, p.variant == HA_LA_KDA);
  cudaError_t e = configure_tc_walk(p);
  if (e != cudaSuccess) return e;
  return launch_tc_walk(p, a, PlanView{}, ws, mk, mq, mv, true, false, spin_limit, SpanBuffers{1, nullptr, nullptr}, false, stream);
}

}  // namespace ha_la
