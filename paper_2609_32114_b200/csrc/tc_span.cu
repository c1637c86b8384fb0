// Start states of the spans of a sequence that is cut into runs walked at the same time (tc_walk.cu):
//   h_1 = b_0,   h_{s+1} = Phi_s h_s + b_s,   s = 1 .. nspan-2        (128 x 128 each, [key][value channel], fp32)
// The columns (value channels) are independent: a CTA takes 8 NT of them, a warp 16 rows of a product.  A product is warp-level MMAs on
// values split into two bf16 each (hi hi + hi lo + lo hi, fp32 accumulation: 2^-16 of the factors), Phi_s copied in bulk ahead of it.  The
// state's fragments go round the warps through shared memory, transposed by stmatrix.
// What bounds it is the chain of products, and in a product the warp-level MMAs (24 NT a warp; a scheduler takes 14 - 16 cycles for each).
// So few columns to a CTA while every CTA has an SM, and everything else kept out of the chain: Phi_s comes split and in fragment
// order from the walk (phi_word), two groups of warps take the products in turn, one reading Phi_{s+1} into its registers under the other's product, and
// b_s is fetched two products ahead (its latency alone was half of a product's time).  Per product, on B200: 8 columns 0.72 us, 16 columns 1.1; 16 columns by one group that
// split Phi_s itself 1.2.  Calls: 2 heads, T = 16384 65.5 us in 22 runs -> 55.1 in 26; 16 heads, T = 4096, 6 runs 55.2 either way.
#include "tc_common.cuh"
#include "tc_mma.cuh"

namespace ha_la {

using namespace ptx;

namespace {

constexpr uint32_t kPhiBytes = 65536;
template <int NT> constexpr uint32_t kFragBytes = 2 * 8 * NT * 512;     // [set][k-step][n-tile]: hi, lo
template <int NT, int BUFS> constexpr uint32_t kSpanSmem = BUFS * kPhiBytes + kFragBytes<NT> + BUFS * 8 + 8;

// 8 NT columns.  Two groups of eight warps take the products in turn (TURNS), so that one reads Phi_{s+1} into its registers under the
// other's product; or a single group.  BUFS: matrices in shared memory.
template <int NT, bool TURNS, int BUFS>
__global__ void __launch_bounds__(TURNS ? 512 : 256, 1) span_fix_kernel(SpanBuffers sb, int T_row, int HV, const int32_t* seq_len, int32_t* status) {
  extern __shared__ __align__(128) uint8_t sm[];
  uint64_t* full = reinterpret_cast<uint64_t*>(sm + BUFS * kPhiBytes + kFragBytes<NT>);              // [BUFS]
  volatile int* abort_flag = reinterpret_cast<volatile int*>(full + BUFS);
  const int nj = blockIdx.x, grp = threadIdx.x >> 8, warp = (threadIdx.x >> 5) & 7, lane = threadIdx.x & 31;
  const int g8 = lane >> 2, t = lane & 3;
  const int r0 = 16 * warp + 4 * (g8 >> 1) + (g8 & 1);   // sigma(g8); sigma(g8 + 8) is two further
  const size_t stride = 128 * 128;
  const float* phi = sb.phi + (size_t)nj * sb.nspan * stride;
  float* b = sb.b + (size_t)nj * sb.nspan * stride + (size_t)r0 * 128 + blockIdx.y * 8 * NT + 2 * t;
  const int32_t* my_len = seq_len ? seq_len + nj / HV : nullptr;
  if (threadIdx.x == 0) {
    for (int i = 0; i < BUFS; ++i) mbar_init(&full[i], 1);
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
  const int last = nst > 0 ? min(sb.nspan - 2, (nst - 1) / spspan) : 0;   // products 1 .. last
  auto fetch = [&](int s) {                              // one thread
    if (s > last) return;
    const int f = s % BUFS;
    mbar_expect_tx(&full[f], kPhiBytes);
#pragma unroll
    for (int i = 0; i < 2; ++i)
      bulk_load(sm + f * kPhiBytes + i * 32768, phi + (size_t)s * stride + i * 8192, 32768, &full[f]);
  };
  if (threadIdx.x == 0)
    for (int s = 1; s <= BUFS; ++s) fetch(s);
  __syncwarp();                                          // (what comes is for converged warps: barriers, matrix instructions)
  struct Tile { float2 x[NT][2]; };                      // [n-tile][sigma(g8), sigma(g8 + 8)]
  auto load_tile = [&](int s) {
    Tile d;
#pragma unroll
    for (int n = 0; n < NT; ++n)
#pragma unroll
      for (int e = 0; e < 2; ++e) d.x[n][e] = *reinterpret_cast<const float2*>(b + (size_t)s * stride + e * 2 * 128 + 8 * n);
    return d;
  };
  auto save = [&](const Tile& d, int s) {
#pragma unroll
    for (int n = 0; n < NT; ++n)
#pragma unroll
      for (int e = 0; e < 2; ++e) *reinterpret_cast<float2*>(b + (size_t)s * stride + e * 2 * 128 + 8 * n) = d.x[n][e];
  };
  const uint32_t frag = smem_u32(sm + BUFS * kPhiBytes) + lane * 16;
  auto put = [&](const Tile& d, int s) {                 // as operand of product s
#pragma unroll
    for (int n = 0; n < NT; ++n) {
      uint32_t w[4];
      split_bf16(d.x[n][0].x, d.x[n][0].y, w[0], w[2]);
      split_bf16(d.x[n][1].x, d.x[n][1].y, w[1], w[3]);
      stsm4t(frag + (((s & 1) * 8 + warp) * NT + n) * 512, w);
    }
  };
  uint32_t hi[8][4], lo[8][4];                           // this warp's rows of Phi_s
  auto take = [&](int s) {
    const int f = s % BUFS, ph = (s - 1) / BUFS & 1;
    if (!mbar_test_wait(&full[f], ph)) mbar_wait(&full[f], ph, abort_flag);
    __syncwarp();                                        // (threads leave the wait one by one)
    const uint32_t sp = smem_u32(sm) + f * kPhiBytes + warp * 8192 + lane * 16;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      lds4(hi[k], sp + k * 1024);
      lds4(lo[k], sp + k * 1024 + 512);
    }
  };
  // Product s is group s % 2's, which holds h_s behind it as h_{s+1}.  Where b_s was, h_s goes, but only when product s has read that:
  // behind the barrier ahead of product s + 1.
  const int step = TURNS ? 2 : 1, first = TURNS && grp == 0 ? 2 : 1;
  Tile h, o;                                             // h_s; b_s of the product to come
  if (first <= last) {
    o = load_tile(first);
    take(first);
  }
  if (first == 1) {
    h = load_tile(0);
    if (last > 0) {
      put(h, 1);
      save(h, 1);                                        // (this thread has read b_1)
    }
  }
  for (int s = first; s <= last; s += step) {
    if (!TURNS) __syncthreads();
    else if (s == 1) asm volatile("bar.sync 3, 256;" ::: "memory");
    else if (grp == 0) asm volatile("bar.sync 1, 512;" ::: "memory");
    else asm volatile("bar.sync 2, 512;" ::: "memory");
    if ((threadIdx.x & 255) == 0) fetch(s + BUFS);        // (Phi_s is in registers)
    __syncwarp();
    if (s > first) save(h, TURNS ? s - 1 : s);
    float c[NT][3][4] = {};
#pragma unroll
    for (int k = 0; k < 8; ++k)
#pragma unroll
      for (int n = 0; n < NT; ++n) {
        uint32_t w[4];
        ldsm4(w, frag + (((s & 1) * 8 + k) * NT + n) * 512);
        mma_bf16(c[n][0], hi[k], w[0], w[1]);
        mma_bf16(c[n][1], hi[k], w[2], w[3]);
        mma_bf16(c[n][2], lo[k], w[0], w[1]);
      }
#pragma unroll
    for (int n = 0; n < NT; ++n)
#pragma unroll
      for (int e = 0; e < 2; ++e)
        h.x[n][e] = make_float2(o.x[n][e].x + (c[n][0][2 * e] + (c[n][1][2 * e] + c[n][2][2 * e])),
                                o.x[n][e].y + (c[n][0][2 * e + 1] + (c[n][1][2 * e + 1] + c[n][2][2 * e + 1])));
    if (s < last) {
      put(h, s + 1);
      if (TURNS && grp == 0) asm volatile("bar.arrive 2, 512;" ::: "memory");
      else if (TURNS) asm volatile("bar.arrive 1, 512;" ::: "memory");
    }
    if (s + step <= last) {
      o = load_tile(s + step);
      take(s + step);
    }
  }
  __syncthreads();
  if (!TURNS || grp == (last > 0 ? last & 1 : 1)) {      // the state behind the last product, also that of empty spans
    for (int s = last + 1; s < sb.nspan; ++s) save(h, s);
  } else if (last > 1) {
    save(h, last);
  }
  if (threadIdx.x == 0 && *abort_flag) {
    report_status(status, HA_LA_ERR_TIMEOUT);
    settle_copies();
  }
}

struct Instance {
  void (*kern)(SpanBuffers, int, int, const int32_t*, int32_t*);
  int cols, threads;
  uint32_t smem;
};
template <int NT, bool TURNS, int BUFS> constexpr Instance kInstance{span_fix_kernel<NT, TURNS, BUFS>, 8 * NT, TURNS ? 512 : 256, kSpanSmem<NT, BUFS>};

}  // namespace

cudaError_t configure_span_fix() {
  for (const Instance& i : {kInstance<1, true, 3>, kInstance<2, true, 3>, kInstance<2, false, 2>}) {
    static_assert(kSpanSmem<2, 3> <= 227 * 1024, "shared memory budget");
    const cudaError_t e = cudaFuncSetAttribute(i.kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)i.smem);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t launch_span_fix(const Problem& p, PlanView plan, const SpanBuffers& sb, int32_t* status, cudaStream_t stream) {
  timer_mark(stream, "tc_span_fix");
  cudaLaunchConfig_t cfg = {};
  // As few columns to a CTA as leave every CTA an SM.  More CTAs than SMs: a group of warps alone (two rounds of those CTAs with one product, 32 heads:
  // 245.6 us for a call, 246.0 with two groups, 249.9 with two such CTAs to an SM).
  const int pairs = p.N * p.HV, sms = sm_count();
  const Instance i = pairs * 16 <= sms ? kInstance<1, true, 3> : pairs * 8 <= sms ? kInstance<2, true, 3> : kInstance<2, false, 2>;
  cfg.gridDim = dim3((unsigned)pairs, (unsigned)(128 / i.cols));
  cfg.blockDim = dim3(i.threads);
  cfg.dynamicSmemBytes = i.smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = g_timer ? 0 : 1;                        // (per-kernel timing wants one kernel at a time)
  return cudaLaunchKernelEx(&cfg, i.kern, sb, p.T_row, p.HV, (const int32_t*)plan.seq_len, status);
}

}  // namespace ha_la
