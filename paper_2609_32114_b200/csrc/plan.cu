// Plan kernel: turns (batch, seqlen) or a packed cu_seqlens array into the chunk table that the
// compute kernels index by chunk slot.  Runs on the device so that a packed batch needs no host
// synchronisation.  Chunks restart at every sequence start; the last chunk of a sequence may be
// partial (paper Section 2.1, "Chunkwise Map-Reduce-Map Execution": inputs are partitioned into
// chunks; chunk length 64 in the paper's experimental setup).
#include "common.cuh"

namespace ha_la {

namespace {

struct PlanParams {
  int N, T_total, T_row, max_len, max_chunks, step;
};

// What bounds it is the chain of dependent look-ups, so for up to kOnChip sequences the tables that later phases read are
// kept in shared memory as well; and it is a programmatic dependent of the stream's earlier work, whose own dependents
// may be set up while it runs.  With every look-up in global memory a call with 24 sequences took 3 us more (of 200).
constexpr int kThreads = 512, kOnChip = 1024;

__global__ void __launch_bounds__(kThreads) plan_kernel(PlanParams p, const int32_t* __restrict__ cu, PlanView v,
                                                   int32_t* status) {
  __shared__ int s_warp[kThreads / 32];
  __shared__ int s_carry;
  __shared__ int s_tok0[kOnChip], s_len[kOnChip], s_chunk0[kOnChip];
  const int tid = threadIdx.x;
  const bool on_chip = p.N <= kOnChip;
  int* const tok0 = on_chip ? s_tok0 : v.seq_tok0;
  int* const lens = on_chip ? s_len : v.seq_len;
  int* const chunk0 = on_chip ? s_chunk0 : v.seq_chunk0;
  asm volatile("griddepcontrol.wait;" ::: "memory");     // (nothing has been read or written so far)
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

  // 1. per-sequence start and length, checked
  for (int n = tid; n < p.N; n += blockDim.x) {
    int t0, len;
    if (cu) {
      const int a = cu[n], b = cu[n + 1];
      bool ok = a >= 0 && b >= a && b <= p.T_total && (b - a) <= p.max_len;
      if (n == 0 && a != 0) ok = false;
      if (n == p.N - 1 && b != p.T_total) ok = false;
      if (!ok) report_status(status, HA_LA_ERR_DEVICE_CHECK);
      t0 = ok ? a : 0;
      len = ok ? (b - a) : 0;
    } else {
      t0 = n * p.T_row;
      len = p.T_row;
    }
    v.seq_tok0[n] = t0;
    v.seq_len[n] = len;
    if (on_chip) {
      s_tok0[n] = t0;
      s_len[n] = len;
    }
  }
  if (tid == 0) s_carry = 0;
  __syncthreads();

  // 1b. sequences by descending length (ties: by index), so that a kernel with one CTA per sequence can start
  // the longest ones first.  Rank by counting; beyond a few thousand sequences the order is left as it is
  // (they are then short, and the count would be quadratic).
  for (int n = tid; n < p.N; n += blockDim.x) {
    int rank = n;
    if (p.N <= 4096) {
      const int len = lens[n];
      rank = 0;
      for (int k = 0; k < p.N; ++k) {
        const int lk = lens[k];
        rank += (lk > len || (lk == len && k < n)) ? 1 : 0;
      }
    }
    v.seq_order[rank] = n;
  }

  // 2. exclusive prefix sum of chunk counts over sequences, kThreads at a time
  for (int base = 0; base < p.N; base += blockDim.x) {
    const int n = base + tid;
    const int cnt = n < p.N ? (lens[n] + p.step - 1) / p.step : 0;
    int x = cnt;
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, x, o);
      if ((tid & 31) >= o) x += y;
    }
    if ((tid & 31) == 31) s_warp[tid >> 5] = x;
    __syncthreads();
    int woff = 0;
    for (int w = 0; w < (tid >> 5); ++w) woff += s_warp[w];
    const int incl = x + woff + s_carry;
    if (n < p.N) {
      v.seq_chunk0[n] = incl - cnt;
      if (on_chip) s_chunk0[n] = incl - cnt;
    }
    __syncthreads();
    if (tid == blockDim.x - 1) s_carry = incl;
    __syncthreads();
  }
  int total = s_carry;
  if (total > p.max_chunks) {   // cannot happen for checked lengths; guard the table anyway
    if (tid == 0) report_status(status, HA_LA_ERR_DEVICE_CHECK);
    total = 0;
  }
  if (tid == 0) {
    v.seq_chunk0[p.N] = total;
    v.hdr[0] = total;
    v.hdr[1] = p.N;
  }
  __syncthreads();

  // 3. one entry per chunk slot (binary search for the owning sequence)
  for (int s = tid; s < p.max_chunks; s += blockDim.x) {
    if (s >= total) {
      v.chunk_seq[s] = -1;
      v.chunk_tok0[s] = 0;
      v.chunk_len[s] = 0;
      continue;
    }
    int lo = 0, hi = p.N - 1;   // last n with seq_chunk0[n] <= s
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (chunk0[mid] <= s) lo = mid; else hi = mid - 1;
    }
    const int c = s - chunk0[lo];
    const int L = lens[lo];
    v.chunk_seq[s] = lo;
    v.chunk_tok0[s] = tok0[lo] + c * p.step;
    v.chunk_len[s] = min(p.step, L - c * p.step);
  }
}

}  // namespace

cudaError_t launch_plan(const Problem& p, const int32_t* cu_seqlens, PlanView plan, int32_t* status,
                        cudaStream_t stream) {
  PlanParams pp{p.N, p.T_total, p.T_row, p.max_len, p.max_chunks, p.step};
  timer_mark(stream, "plan");
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(1);
  cfg.blockDim = dim3(kThreads);
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = g_timer ? 0 : 1;                        // (per-kernel timing wants one kernel at a time)
  return cudaLaunchKernelEx(&cfg, plan_kernel, pp, cu_seqlens, plan, status);
}

}  // namespace ha_la
