// Start states of the spans of a sequence that is cut into runs walked at the same time (tc_walk.cu):
//   h_1 = b_0,   h_{s+1} = Phi_s h_s + b_s,   s = 1 .. nspan-2        (128 x 128 each, [key][value channel], fp32)
// The columns (value channels) are independent: a CTA takes 16 of them, a warp 16 rows of every product.  What a product
// costs is Phi_s on its way out of L2, 64 KiB per CTA, so that is copied in bulk one product ahead (operand fragments
// read straight from global memory touch every line several times: 2.2 us per product).  The product itself is 48 warp-level
// MMAs a warp on values split into two bf16 each (hi hi + hi lo + lo hi, fp32 accumulation: 2^-16 of the factors).  The
// state's fragments go round the warps through 8 KiB of shared memory, transposed in registers.  What bounds it is the chain:
// 1.2 us per product with every CTA on an SM (2 heads, ten products 18.4 us by themselves, twenty 30.8).  Fragment row r of a warp is key sigma(r), sigma(2 t + e) = 4 t + e, sigma(8 + 2 t + e)
// = 4 t + 2 + e: the four columns of Phi that a lane needs are then neighbours.
#include "tc_common.cuh"
#include "tc_mma.cuh"

namespace ha_la {

using namespace ptx;

namespace {

constexpr int kFixCols = 16, kFewPairs = 4;

__device__ __forceinline__ void split_bf16(float x, float y, uint32_t& hi, uint32_t& lo) {
  hi = pack_bf16(x, y);
  const float2 h = unpack_bf16(hi);
  lo = pack_bf16(x - h.x, y - h.y);
}

constexpr uint32_t kPhiBytes = 65536;
constexpr uint32_t OFF_FRAG = 2 * kPhiBytes, OFF_FBAR = OFF_FRAG + 2 * 8 * 2 * 32 * 16, kSpanSmem = OFF_FBAR + 32;

// Two instances that differ in who issues the copies, a thread elected by elect.sync or thread 0, and for that in the code that the
// compiler makes of the whole kernel (79 registers against 66).  Which is faster goes by the number of CTAs.  Calls, thread 0's first: up to
// four (sequence, V-head) pairs, 32 CTAs, gain at any number of runs and packed or not (1 head, T = 12000, 19 runs 55.7 -> 53.2 us; 2 heads,
// T = 3000, 8 runs 34.0 -> 33.3, T = 16000, 21 runs 65.9 -> 63.6; 4 heads, T = 3000 35.1 -> 34.7, T = 24000, 19 runs 90.1 -> 88.0; two sequences
// of 11 k tokens, 2 heads 68.9 -> 67.7); five and six pairs are within 1 % either way; more lose (7 heads, T = 3000 38.3 -> 39.2; 8 heads, T = 6000
// 52.5 -> 54.4; four rows of 4000, 2 heads 43.7 -> 46.1; 16 heads, T = 4096 55.9 -> 59.0).  The reason is not known: measure again after
// an edit of this kernel or with another compiler.
template <bool ELECT>
__global__ void __launch_bounds__(256) span_fix_kernel(SpanBuffers sb, int T_row, int HV, const int32_t* seq_len, int32_t* status) {
  extern __shared__ __align__(128) uint8_t sm[];
  uint4 (*frag)[8][2][32] = reinterpret_cast<uint4(*)[8][2][32]>(sm + OFF_FRAG);   // [s & 1][k-step][n-tile][lane]: hi b0, b1, lo b0, b1
  uint64_t* full = reinterpret_cast<uint64_t*>(sm + OFF_FBAR);                     // [2]
  volatile int* abort_flag = reinterpret_cast<volatile int*>(full + 2);
  const int nj = blockIdx.x, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int g8 = lane >> 2, t = lane & 3;
  const int r0 = 16 * warp + 4 * (g8 >> 1) + (g8 & 1);   // sigma(g8); sigma(g8 + 8) is two further
  const size_t stride = 128 * 128;
  const float* phi = sb.phi + (size_t)nj * sb.nspan * stride;
  const size_t tile = (size_t)nj * sb.nspan * stride + (size_t)r0 * 128 + blockIdx.y * kFixCols + 2 * t;
  float* b = sb.b + tile;                                // h_s replaces b_s: the same thread reads the one and writes the other
  const int32_t* my_len = seq_len ? seq_len + nj / HV : nullptr;
  if (threadIdx.x == 0) {
    mbar_init(&full[0], 1);
    mbar_init(&full[1], 1);
    *abort_flag = 0;
    mbar_fence_init();
  }
  __syncthreads();
  asm volatile("griddepcontrol.wait;" ::: "memory");     // (launched as a programmatic dependent of the states-only walk)
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  // spans past the end of a short sequence are empty: the state passes through untouched, bit for bit
  const int len = my_len ? *my_len : T_row;              // (another kernel's table: read behind the wait)
  const int nst = (len + kStep - 1) / kStep;
  const int spspan = (nst + sb.nspan - 1) / sb.nspan;
  auto fetch = [&](int s) {                              // one thread
    if (s + 1 >= sb.nspan) return;
    mbar_expect_tx(&full[s & 1], kPhiBytes);
#pragma unroll
    for (int i = 0; i < 4; ++i)
      bulk_load(sm + (s & 1) * kPhiBytes + i * 16384, phi + (size_t)s * stride + i * 4096, 16384, &full[s & 1]);
  };
  auto issuing = [&]() { return ELECT ? warp == 0 && elect_one() : threadIdx.x == 0; };
  if (issuing()) {
    fetch(1);
    fetch(2);
  }
  float2 h[2][2], o[2][2];                               // h_s and b_s: [n-tile][sigma(g8), sigma(g8 + 8)]
  auto load_tile = [&](const float* src, float2 (&d)[2][2]) {
#pragma unroll
    for (int n = 0; n < 2; ++n)
#pragma unroll
      for (int e = 0; e < 2; ++e) d[n][e] = *reinterpret_cast<const float2*>(src + e * 2 * 128 + 8 * n);
  };
  load_tile(b, h);
  for (int s = 1; s < sb.nspan; ++s) {
    if (s + 1 < sb.nspan) load_tile(b + (size_t)s * stride, o);
#pragma unroll
    for (int n = 0; n < 2; ++n) {
#pragma unroll
      for (int e = 0; e < 2; ++e) *reinterpret_cast<float2*>(b + (size_t)s * stride + e * 2 * 128 + 8 * n) = h[n][e];
      uint4 w;
      split_bf16(h[n][0].x, h[n][0].y, w.x, w.z);
      split_bf16(h[n][1].x, h[n][1].y, w.y, w.w);
      w.x = transpose8x8(w.x); w.y = transpose8x8(w.y); w.z = transpose8x8(w.z); w.w = transpose8x8(w.w);
      frag[s & 1][warp][n][lane] = w;
    }
    __syncthreads();                                     // (and everyone is done with the product before)
    if (s + 1 == sb.nspan) break;
    if (s > 1 && issuing()) fetch(s + 1);
    mbar_wait(&full[s & 1], ((s - 1) >> 1) & 1, abort_flag);
    if (s * spspan >= nst) continue;                     // (the same for every thread of the CTA)
    // Rows lie 512 bytes apart, so lanes of an odd row take the other k-step of a pair first: other banks.
    const float* sp = reinterpret_cast<const float*>(sm + (s & 1) * kPhiBytes) + r0 * 128 + 4 * t;
    const bool odd = g8 & 1;
    float c[2][3][4] = {};
#pragma unroll
    for (int k = 0; k < 8; k += 2) {
      float4 x[2], y[2];
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const int o16 = 16 * k + 16 * (odd ? i ^ 1 : i);
        x[i] = *reinterpret_cast<const float4*>(sp + o16);
        y[i] = *reinterpret_cast<const float4*>(sp + 2 * 128 + o16);
      }
      if (odd) {
        const float4 tx = x[0], ty = y[0];
        x[0] = x[1]; x[1] = tx;
        y[0] = y[1]; y[1] = ty;
      }
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        uint32_t hi[4], lo[4];
        split_bf16(x[i].x, x[i].y, hi[0], lo[0]);
        split_bf16(y[i].x, y[i].y, hi[1], lo[1]);
        split_bf16(x[i].z, x[i].w, hi[2], lo[2]);
        split_bf16(y[i].z, y[i].w, hi[3], lo[3]);
#pragma unroll
        for (int n = 0; n < 2; ++n) {
          const uint4 w = frag[s & 1][k + i][n][lane];
          mma_bf16(c[n][0], hi, w.x, w.y);
          mma_bf16(c[n][1], hi, w.z, w.w);
          mma_bf16(c[n][2], lo, w.x, w.y);
        }
      }
    }
#pragma unroll
    for (int n = 0; n < 2; ++n)
#pragma unroll
      for (int e = 0; e < 2; ++e)
        h[n][e] = make_float2(o[n][e].x + (c[n][0][2 * e] + (c[n][1][2 * e] + c[n][2][2 * e])),
                              o[n][e].y + (c[n][0][2 * e + 1] + (c[n][1][2 * e + 1] + c[n][2][2 * e + 1])));
  }
  if (threadIdx.x == 0 && *abort_flag) {
    report_status(status, HA_LA_ERR_TIMEOUT);
    settle_copies();
  }
}

}  // namespace

cudaError_t configure_span_fix() {
  cudaError_t e = cudaFuncSetAttribute(span_fix_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSpanSmem);
  return e != cudaSuccess ? e : cudaFuncSetAttribute(span_fix_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSpanSmem);
}

cudaError_t launch_span_fix(const Problem& p, PlanView plan, const SpanBuffers& sb, int32_t* status, cudaStream_t stream) {
  timer_mark(stream, "tc_span_fix");
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(p.N * p.HV), 128 / kFixCols);
  cfg.blockDim = dim3(256);
  cfg.dynamicSmemBytes = kSpanSmem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = g_timer ? 0 : 1;                        // (per-kernel timing wants one kernel at a time)
  auto kern = p.N * p.HV <= kFewPairs ? span_fix_kernel<true> : span_fix_kernel<false>;
  return cudaLaunchKernelEx(&cfg, kern, sb, p.T_row, p.HV, (const int32_t*)plan.seq_len, status);
}

}  // namespace ha_la
