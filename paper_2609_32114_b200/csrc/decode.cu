// One decoding step of the delta-rule layer (one new token per sequence): see ha_la_decode in ha_la.h.
//
// The step reads and rewrites the whole fp32 state (d_k x d_v per sequence and V-head, 64 KiB at d = 128) for
// about 6 d_k d_v flops, so it is bound by HBM traffic: 2 x 4 d_k d_v bytes per (sequence, V-head).  One CTA of four warps
// per (sequence, V-head) and 64 value channels: a thread keeps four channels of 16 (d = 64: 8) state rows in registers, so
// the state crosses the memory system exactly once in each direction in 16-byte accesses, all loads of a thread in flight
// together, with streaming hints (it is used once per step and exceeds L2).  Small CTAs, five or more to an SM, keep some
// loading while others store and make the last wave short.  The kernel is a programmatic dependent of the step before it:
// launched and set up under that one's tail, it waits on the device before its first access.
// Measured (256 sequences x 16 heads, d = 128): one CTA per head with 4-byte accesses 90.4 us, this 80.6 us = 6.7 TB/s
// (64 channels 80.6, 32 channels 81.5, 128 channels 84.1); 37 sequences x 32 heads: 30.7 -> 25.5 us.
#include "common.cuh"

namespace ha_la {

namespace {

struct DecodeParams {
  const void* q; const void* k; const void* v;
  const float* g; const float* beta; const float* h_in;
  float* h_out; void* o;
  int HK, HV;
  float scale;
};

constexpr int kCols = 64;                                // value channels per CTA
constexpr int kThreads = 128;
constexpr int kRows = kThreads / (kCols / 4);            // state rows in flight per load instruction of the CTA

template <typename In, int D, bool KDA>
__global__ void __launch_bounds__(kThreads, 4) decode_kernel(DecodeParams p) {
  constexpr int NR = D / kRows;                          // rows per thread
  __shared__ __align__(16) float sk[D];
  __shared__ __align__(16) float sq[D];
  __shared__ float sdec[D];
  __shared__ __align__(16) float spart[kRows][kCols];
  const int tid = threadIdx.x;
  const int row0 = tid / (kCols / 4), c4 = (blockIdx.x % (D / kCols)) * kCols + tid % (kCols / 4) * 4;
  const size_t nj = blockIdx.x / (D / kCols);            // (sequence, V-head)
  const int j = (int)(nj % p.HV);
  const size_t n = nj / p.HV;
  const int jq = j / (p.HV / p.HK);
  asm volatile("griddepcontrol.wait;" ::: "memory");     // everything before this step in the stream is complete

  // rows row0, row0 + kRows, ..; the loads do not depend on anything and are read exactly once
  float4 h[NR];
  const size_t base = nj * D * D + (size_t)row0 * D + c4;
#pragma unroll
  for (int i = 0; i < NR; ++i)
    h[i] = p.h_in ? __ldcs(reinterpret_cast<const float4*>(p.h_in + base + (size_t)i * kRows * D)) : make_float4(0.f, 0.f, 0.f, 0.f);
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");   // (the next step waits for this grid's end as above)
  if (tid < D) {
    const size_t qk = (n * p.HK + jq) * D + tid;
    sk[tid] = to_f32(reinterpret_cast<const In*>(p.k)[qk]);
    sq[tid] = to_f32(reinterpret_cast<const In*>(p.q)[qk]);
    sdec[tid] = __expf(KDA ? p.g[nj * D + tid] : p.g[nj]);
  }
  const float4 vv = load4(reinterpret_cast<const In*>(p.v) + nj * D + c4);
  const float beta = p.beta[nj];
  __syncthreads();

  float4 r = make_float4(0.f, 0.f, 0.f, 0.f);            // (decayed h)^T k, this thread's rows
#pragma unroll
  for (int i = 0; i < NR; ++i) {
    const float dec = sdec[row0 + i * kRows], k = sk[row0 + i * kRows];
    h[i].x *= dec; h[i].y *= dec; h[i].z *= dec; h[i].w *= dec;
    r.x = fmaf(h[i].x, k, r.x); r.y = fmaf(h[i].y, k, r.y); r.z = fmaf(h[i].z, k, r.z); r.w = fmaf(h[i].w, k, r.w);
  }
  float4* mine = reinterpret_cast<float4*>(&spart[row0][c4 % kCols]);
  *mine = r;
  __syncthreads();
  r = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
  for (int q = 0; q < kRows; ++q) {
    const float4 x = *reinterpret_cast<const float4*>(&spart[q][c4 % kCols]);
    r.x += x.x; r.y += x.y; r.z += x.z; r.w += x.w;
  }
  __syncthreads();
  const float4 u = make_float4(beta * (vv.x - r.x), beta * (vv.y - r.y), beta * (vv.z - r.z), beta * (vv.w - r.w));
  float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
  for (int i = 0; i < NR; ++i) {
    const float k = sk[row0 + i * kRows], q = sq[row0 + i * kRows];
    h[i].x = fmaf(k, u.x, h[i].x); h[i].y = fmaf(k, u.y, h[i].y); h[i].z = fmaf(k, u.z, h[i].z); h[i].w = fmaf(k, u.w, h[i].w);
    acc.x = fmaf(h[i].x, q, acc.x); acc.y = fmaf(h[i].y, q, acc.y); acc.z = fmaf(h[i].z, q, acc.z); acc.w = fmaf(h[i].w, q, acc.w);
    __stcs(reinterpret_cast<float4*>(p.h_out + base + (size_t)i * kRows * D), h[i]);
  }
  *mine = acc;
  __syncthreads();
  if (tid < kCols) {
    float o = 0.f;
#pragma unroll
    for (int q = 0; q < kRows; ++q) o += spart[q][tid];
    reinterpret_cast<In*>(p.o)[nj * D + (blockIdx.x % (D / kCols)) * kCols + tid] = from_f32<In>(p.scale * o);
  }
}

template <typename In, int D, bool KDA>
cudaError_t launch(const DecodeParams& dp, size_t heads, cudaStream_t stream) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(heads * (D / kCols)));
  cfg.blockDim = dim3(kThreads);
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, decode_kernel<In, D, KDA>, dp);
}

}  // namespace

}  // namespace ha_la

using namespace ha_la;

extern "C" int ha_la_decode(const ha_la_decode_args* a, void* cuda_stream) {
  if (!a) return HA_LA_ERR_INVALID_ARG;
  if (a->variant != HA_LA_GDN && a->variant != HA_LA_KDA) return HA_LA_ERR_INVALID_ARG;
  if (a->dtype != HA_LA_BF16 && a->dtype != HA_LA_FP32) return HA_LA_ERR_INVALID_ARG;
  if (a->num_seqs < 0 || a->num_qk_heads < 1 || a->num_v_heads < 1 || a->num_v_heads % a->num_qk_heads != 0)
    return HA_LA_ERR_INVALID_ARG;
  if (a->d_k < 1 || a->d_v < 1) return HA_LA_ERR_INVALID_ARG;
  if (a->d_k != a->d_v || (a->d_k != 64 && a->d_k != 128)) return HA_LA_ERR_UNSUPPORTED;
  if (!(a->scale == a->scale)) return HA_LA_ERR_INVALID_ARG;
  const unsigned long long grid = (unsigned long long)a->num_seqs * a->num_v_heads;   // CTAs: twice that at d = 128
  if (grid > 0x7fffffffULL / (a->d_k / 64)) return HA_LA_ERR_UNSUPPORTED;
  if (grid == 0) return HA_LA_OK;
  if (!a->q || !a->k || !a->v || !a->g || !a->beta || !a->h_out || !a->o) return HA_LA_ERR_INVALID_ARG;
  const uintptr_t al16 = (uintptr_t)a->q | (uintptr_t)a->k | (uintptr_t)a->v | (uintptr_t)a->o |
                         (uintptr_t)a->h_in | (uintptr_t)a->h_out;
  if (al16 & 15) return HA_LA_ERR_INVALID_ARG;
  if (((uintptr_t)a->g | (uintptr_t)a->beta) & 3) return HA_LA_ERR_INVALID_ARG;

  DecodeParams dp{a->q, a->k, a->v, a->g, a->beta, a->h_in, a->h_out, a->o, a->num_qk_heads, a->num_v_heads, a->scale};
  cudaStream_t stream = reinterpret_cast<cudaStream_t>(cuda_stream);
  const bool kda = a->variant == HA_LA_KDA, bf = a->dtype == HA_LA_BF16, big = a->d_k == 128;
  cudaError_t e;
  if (bf) {
    if (big) e = kda ? launch<__nv_bfloat16, 128, true>(dp, grid, stream) : launch<__nv_bfloat16, 128, false>(dp, grid, stream);
    else e = kda ? launch<__nv_bfloat16, 64, true>(dp, grid, stream) : launch<__nv_bfloat16, 64, false>(dp, grid, stream);
  } else {
    if (big) e = kda ? launch<float, 128, true>(dp, grid, stream) : launch<float, 128, false>(dp, grid, stream);
    else e = kda ? launch<float, 64, true>(dp, grid, stream) : launch<float, 64, false>(dp, grid, stream);
  }
  return e == cudaSuccess ? HA_LA_OK : HA_LA_ERR_CUDA;
}
