// What the kernels of the fp32 path share: parameters, four-wide arithmetic, the launch.
#pragma once

#include "common.cuh"
#include "tc_ptx.cuh"

#include <atomic>

namespace ha_la {

struct Fp32Params {
  const void* q; const void* k; const void* v;
  const float* g; const float* beta; const float* h0;
  void* o; float* hT;
  float* rec;
  const int32_t* chunk_tok0;   // chunk table of the plan kernel, or NULL for equal-length rows:
  const int32_t* chunk_len;    //   slot s is chunk s % cps of row s / cps, T_row tokens per row
  const int32_t* seq_tok0; const int32_t* seq_len; const int32_t* seq_chunk0; const int32_t* seq_order;
  int T_row, cps;
  int HK, HV;
  float scale;
  int32_t* status;
};

template <int N> struct Int { static constexpr int value = N; };

__device__ __forceinline__ float4 ld4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ float dot4(const float4& a, const float4& b, float c) {
  return fmaf(a.w, b.w, fmaf(a.z, b.z, fmaf(a.y, b.y, fmaf(a.x, b.x, c))));
}
__device__ __forceinline__ void store4(float* p, const float4& v) { *reinterpret_cast<float4*>(p) = v; }
__device__ __forceinline__ void store4(__nv_bfloat16* p, const float4& v) {
  *reinterpret_cast<uint2*>(p) = make_uint2(ptx::pack_bf16(v.x, v.y), ptx::pack_bf16(v.z, v.w));
}

// A thread's wait ran out: its kernel's copies land before the CTA's shared memory is given back.
__device__ __forceinline__ void report_timeout(int32_t* status) {
  report_status(status, HA_LA_ERR_TIMEOUT);
  ptx::settle_copies();
}

// Launch as a programmatic dependent: set up under the tail of the kernel before it, waiting on the device.
template <auto kern>
cudaError_t launch_fp32_kernel(unsigned grid, unsigned threads, size_t smem, cudaStream_t stream, const Fp32Params& fp) {
  static std::atomic<uint64_t> configured{0};            // (of this kernel: a bit per device)
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return cudaErrorInvalidDevice;
  if (dev >= 64 || !(configured.load() >> dev & 1)) {
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    if (dev < 64) configured.fetch_or(1ull << dev);
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = g_timer ? 0 : 1;                        // (per-kernel timing wants one kernel at a time)
  return cudaLaunchKernelEx(&cfg, kern, fp);
}

}  // namespace ha_la
