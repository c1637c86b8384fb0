// fp32 chunkwise delta-rule prefill (GDN and KDA) for head dimension 64: fp32 and bf16 inputs, arithmetic fp32 on the CUDA cores but for the raw products of
// bf16 GDN.  (d = 128 in fp32.cu.)
//
// The step of a chunk is affine in the state that enters it, and at d = 64 its matrices are small enough to be made chunk-locally:
//   h' = M h + b,   o = scale (N h + c),   with  R = T diag(beta),
//   M = e^{G_L} - KD^T R (K e^G)    b = KD^T R V    N = Q e^G - P R (K e^G)    c = P R V         (KD = K e^{G_L-G}, P = decay-masked Q K^T)
// so the sequential kernel has one product and one barrier per chunk (W, U, KD and P out of the chunk-local kernel take it two of each).
//   fp32_prep64_kernel   one CTA per (chunk, V-head) and share of the columns [K e^G | V]: operators #1 - #3 and the products above.
//   fp32_walk64_kernel   one CTA per (sequence, V-head, 4, 8 or 16 value channels) walks the chunks in order: operators #5 and #6.
//
// What bounds it.  The sequential kernel: shared-memory reads (32 KB of M and N per chunk and CTA) and the latency of one product, 0.57 us per chunk
// with 4 channels.  The chunk-local kernel, 11 - 15 us for one unit per SM, is a chain of phases: raw products 3 us (bf16, GDN: 1, on the matrix instructions: each
// product is exact there, their sums of 64 are the matrix unit's fp32), the inverse 2, L = [KD^T; P] T 1.9, L [K e^G | V] 4.4 of which fp32 multiply-adds are 3.4.
// Measured on B200, calls, against one phase more per chunk and a substitution in the chunk-local kernel (us): 1 head, T = 256, fp32 16.8 -> 14.3; 8 heads, T = 1000,
// bf16 34.5 -> 23.8, KDA 41.9 -> 30.7; two rows of 1000, 16 heads 88.2 -> 77.9; eight sequences of 100 to 512, 16 heads, fp32 144.3 -> 139.3; one chunk 12.7 -> 12.4.
// Errors against 64 bits (rms of hT and of o) are 0.69 to 1.00 of what they were with gates of -0.18 per token and less on average.  With hardly any decay the new state is the sum of two large terms, M h and b,
// where it was e^{G_L} h and a small one, and errors are 0.67 to 1.12 of what they were at -0.004 per token and 0.70 to 1.28 without any decay: 2.5e-7 instead of 2.1e-7 for independent keys,
// 8.4e-7 instead of 6.7e-7 for eight keys over and over, less for keys that lean one way (T = 1000, 8 heads, GDN and KDA).
#include "common.cuh"
#include "fp32_common.cuh"
#include "tc_mma.cuh"
#include "tc_ptx.cuh"

namespace ha_la {

using namespace ptx;

namespace {

constexpr int C = kChunk, D = 64;
constexpr int LD = D + 4;                                // row stride of a 64 x 64 matrix: rows 16 bytes apart in the banks
constexpr int LDW = 2 * D + 4;                           // ... of one with 128 columns
constexpr int LDB = D + 8;                               // ... of a bf16 tile (ldmatrix rows 16 bytes apart)
constexpr int kSlice = 4;                                // value channels per slice of b and c in a record
constexpr int kPrepThreads = 512;

// record of one (chunk slot, V-head), in floats: [M; N] rows (in odd ones columns 16 n .. + 15 and 16 n + 16 .. + 31 exchanged, n even: see the
// sequential kernel's reads), then per slice of channels the rows of [b; c]
struct Rec64 {
  static constexpr int MN = 0;                           // [2 C][D]
  static constexpr int BC = 2 * C * D;                   // [D / kSlice][2 C][kSlice]
  static constexpr int size = BC + 2 * C * D;
};

// ------------------------------------------------------------------------------------------------ chunk-local part
template <typename In, bool KDA> struct Prep64Smem {
  static constexpr bool kMma = !KDA && sizeof(In) == 2;
  static constexpr int K = 0;                            // [C][LD]; GDN: KD in its place once it has been read
  static constexpr int Q = K + C * LD;                   // [C][LD]
  static constexpr int A = Q + C * LD;                   // [column][row] -A
  static constexpr int P = A + C * LD;                   // [column][row]
  static constexpr int T = P + C * LD;                   // [row][column]
  static constexpr int R = T + C * LD;                   // [C][LDW]: beta K e^G | beta V (KDA: first K e^{R_I-G}, block rows 1, 2, 3)
  static constexpr int L = R + C * LDW;                  // [column][row]: KD^T T, P T
  static constexpr int X = L + C * LDW;                  // [32][36]
  static constexpr int G = X + 32 * 36;                  // GDN [C]; KDA [C][LD]: cumulative log-gate
  static constexpr int KD = KDA ? G + C * LD : K;        // [C][LD]
  static constexpr int B = (KDA ? KD + C * LD : G + C);  // [C] beta
  static constexpr int BF = B + C;                       // bf16 [2][C][LDB]: K, Q for the matrix instructions
  static constexpr int size = BF + (kMma ? C * LDB : 0);
};
static_assert(96 * LD <= C * LDW, "what lies over what");

// v[N] summed over lanes that differ in the bits FROM, FROM / 2, .. TO: halves are kept by the bit, lanes end with N / (2 FROM / TO) sums
template <int N, int FROM, int TO> __device__ __forceinline__ void scatter_lanes(float (&v)[N], int lane) {
#pragma unroll
  for (int b = FROM, n = N / 2; b >= TO; b >>= 1, n /= 2) {
    const bool up = lane & b;
#pragma unroll
    for (int i = 0; i < N / 2; ++i) {
      if (i >= n) break;
      const float keep = up ? v[i + n] : v[i], send = up ? v[i] : v[i + n];
      v[i] = keep + __shfl_xor_sync(0xffffffffu, send, b);
    }
  }
}
__device__ __forceinline__ float2 dot_pairs(const float4& a, const float4& b, float2 c) {     // even and odd products apart
  return fma2(make_float2(a.z, a.w), make_float2(b.z, b.w), fma2(make_float2(a.x, a.y), make_float2(b.x, b.y), c));
}
__device__ __forceinline__ float4 scale4(const float4& a, float s) { return make_float4(a.x * s, a.y * s, a.z * s, a.w * s); }
__device__ __forceinline__ float4 mul4(const float4& a, const float4& b) { return make_float4(a.x * b.x, a.y * b.y, a.z * b.z, a.w * b.w); }
__device__ __forceinline__ float4 exp_diff(const float4& a, const float4& b) {
  return make_float4(expf(a.x - b.x), expf(a.y - b.y), expf(a.z - b.z), expf(a.w - b.w));
}
__device__ __forceinline__ float4 exp4(const float4& a) { return make_float4(expf(a.x), expf(a.y), expf(a.z), expf(a.w)); }
__device__ __forceinline__ void st4(float* p, const float4& v) { *reinterpret_cast<float4*>(p) = v; }
// (two multiply-adds to an instruction: the same rate of the units, half the issue slots)
__device__ __forceinline__ void axpy4(float4& y, float a, const float4& x) {
  const float2 aa = make_float2(a, a), lo = fma2(aa, make_float2(x.x, x.y), make_float2(y.x, y.y)),
               hi = fma2(aa, make_float2(x.z, x.w), make_float2(y.z, y.w));
  y = make_float4(lo.x, lo.y, hi.x, hi.y);
}

// SPLIT: CTAs that share a chunk's columns of [K e^G | V]
template <typename In, bool KDA, int SPLIT>
__global__ void __launch_bounds__(kPrepThreads, 1) fp32_prep64_kernel(Fp32Params p) {
  using S = Prep64Smem<In, KDA>;
  extern __shared__ __align__(16) float sf[];
  float* const sK = sf + S::K;
  float* const sQ = sf + S::Q;
  float* const sA = sf + S::A;
  float* const sP = sf + S::P;
  float* const sT = sf + S::T;
  float* const sR = sf + S::R;
  float* const sL = sf + S::L;
  float* const sX = sf + S::X;
  float* const sG = sf + S::G;
  float* const sKD = sf + S::KD;
  float* const sB = sf + S::B;
  __nv_bfloat16* const sBF = reinterpret_cast<__nv_bfloat16*>(sf + S::BF);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int share = blockIdx.x % SPLIT, unit = blockIdx.x / SPLIT;
  const int slot = unit / p.HV, j = unit % p.HV, jq = j / (p.HV / p.HK);
  asm volatile("griddepcontrol.wait;" ::: "memory");     // (nothing has been read so far)
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  int len, t0;
  if (p.chunk_len) {
    len = p.chunk_len[slot];
    t0 = p.chunk_tok0[slot];
  } else {
    const int cc = slot % p.cps;
    t0 = (slot / p.cps) * p.T_row + cc * C;
    len = min(C, p.T_row - cc * C);
  }
  if (len <= 0) return;                                  // a slot that a packed batch does not use
  const In* gq = reinterpret_cast<const In*>(p.q);
  const In* gk = reinterpret_cast<const In*>(p.k);
  const In* gv = reinterpret_cast<const In*>(p.v);

  // ---- load the chunk; rows >= len are no-op tokens (k = q = v = 0, beta = 0, g = 0).  V waits in registers.
  const int li = tid >> 4, lc = (tid & 15) * 4;          // rows li, li + 32, four columns
  float4 v4[2];
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    const int i = li + 32 * u;
    float4 q4 = make_float4(0.f, 0.f, 0.f, 0.f), k4 = q4, g4 = q4;
    v4[u] = q4;
    if (i < len) {
      const size_t off = ((size_t)(t0 + i) * p.HK + jq) * D + lc, voff = ((size_t)(t0 + i) * p.HV + j) * D + lc;
      q4 = load4(gq + off);
      k4 = load4(gk + off);
      v4[u] = load4(gv + voff);
      if (KDA) g4 = ld4(p.g + voff);
    }
    st4(sQ + i * LD + lc, q4);
    st4(sK + i * LD + lc, k4);
    if (KDA) st4(sG + i * LD + lc, g4);
    if (S::kMma) {                                       // (exact: they were bf16)
      *reinterpret_cast<uint2*>(sBF + i * LDB + lc) = make_uint2(pack_bf16(k4.x, k4.y), pack_bf16(k4.z, k4.w));
      *reinterpret_cast<uint2*>(sBF + (C + i) * LDB + lc) = make_uint2(pack_bf16(q4.x, q4.y), pack_bf16(q4.z, q4.w));
    }
  }
  if (warp == 0) {
    sB[lane] = lane < len ? p.beta[(size_t)(t0 + lane) * p.HV + j] : 0.f;
    sB[lane + 32] = lane + 32 < len ? p.beta[(size_t)(t0 + lane + 32) * p.HV + j] : 0.f;
  }
  // ---- op #1 Gate: chunk-local inclusive cumulative sum of the log-gate
  if (!KDA && warp == 1) {
    float x0 = lane < len ? p.g[(size_t)(t0 + lane) * p.HV + j] : 0.f, x1 = lane + 32 < len ? p.g[(size_t)(t0 + lane + 32) * p.HV + j] : 0.f;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const float y0 = __shfl_up_sync(0xffffffffu, x0, o), y1 = __shfl_up_sync(0xffffffffu, x1, o);
      if (lane >= o) { x0 += y0; x1 += y1; }
    }
    x1 += __shfl_sync(0xffffffffu, x0, 31);
    sG[lane] = x0;
    sG[lane + 32] = x1;
  }
  __syncthreads();
  if (KDA) {
    if (tid < D) {
      float acc = 0.f;
      for (int i = 0; i < C; ++i) { acc += sG[i * LD + tid]; sG[i * LD + tid] = acc; }
    }
    __syncthreads();
  }

  // ---- op #2: -A (strictly lower, beta-scaled) and P (lower incl. diagonal), by columns, in 16 x 16 blocks.
  auto put = [&](int i, int jj, float a, float q) {      // entry (i, jj) of a block on or below the diagonal
    sA[jj * LD + i] = jj < i ? -sB[i] * a : 0.f;
    sP[jj * LD + i] = jj <= i ? q : 0.f;
  };
  if constexpr (S::kMma) {
    // Products of bf16 are exact in fp32, so the raw products go to the matrix instructions (which add them up in fp32): a warp per block.
    if (warp < 10) {
      const int I = warp < 1 ? 0 : warp < 3 ? 1 : warp < 6 ? 2 : 3, J = warp - I * (I + 1) / 2;
      const uint32_t base = smem_u32(sBF), fr = (lane & 15) * (LDB * 2) + (lane >> 4) * 16;
      float a[2][4] = {}, q[2][4] = {};
#pragma unroll
      for (int k = 0; k < D / 16; ++k) {
        uint32_t kf[4], qf[4], r[4];
        ldsm4(r, base + 16 * J * (LDB * 2) + fr + k * 32);
        ldsm4(kf, base + 16 * I * (LDB * 2) + fr + k * 32);
        ldsm4(qf, base + (C + 16 * I) * (LDB * 2) + fr + k * 32);
        mma_bf16(a[0], kf, r[0], r[2]);
        mma_bf16(a[1], kf, r[1], r[3]);
        mma_bf16(q[0], qf, r[0], r[2]);
        mma_bf16(q[1], qf, r[1], r[3]);
      }
#pragma unroll
      for (int n = 0; n < 2; ++n)
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const int i = 16 * I + (lane >> 2) + (e >> 1) * 8, jj = 16 * J + 8 * n + (lane & 3) * 2 + (e & 1);
          const float d = jj <= i ? expf(sG[i] - sG[jj]) : 0.f;
          put(i, jj, a[n][e] * d, q[n][e] * d);
        }
    }
  } else if constexpr (!KDA) {
    // A thread owns one entry of every block, over half of the features.  Neighbouring lanes share columns: their reads are then one.
    const int half = tid >> 8, tr = ((warp & 7) << 1) | (lane & 1), tc = lane >> 1;
    float2 kk[10] = {}, qk[10] = {};                     // (blocks row by row; even and odd features)
#pragma unroll 2
    for (int c = 32 * half; c < 32 * half + 32; c += 4) {
      float4 kj[4];
#pragma unroll
      for (int b = 0; b < 4; ++b) kj[b] = ld4(sK + (16 * b + tc) * LD + c);
#pragma unroll
      for (int a = 0; a < 4; ++a) {
        const float4 ki = ld4(sK + (16 * a + tr) * LD + c), qi = ld4(sQ + (16 * a + tr) * LD + c);
#pragma unroll
        for (int b = 0; b <= a; ++b) {
          kk[a * (a + 1) / 2 + b] = dot_pairs(ki, kj[b], kk[a * (a + 1) / 2 + b]);
          qk[a * (a + 1) / 2 + b] = dot_pairs(qi, kj[b], qk[a * (a + 1) / 2 + b]);
        }
      }
    }
    float* const other = sL + (tid & 255);               // [20][256]
    if (half) {
#pragma unroll
      for (int b = 0; b < 10; ++b) {
        other[b * 256] = kk[b].x + kk[b].y;
        other[(10 + b) * 256] = qk[b].x + qk[b].y;
      }
    }
    __syncthreads();
    if (!half) {
#pragma unroll
      for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b <= a; ++b) {
          const int i = 16 * a + tr, jj = 16 * b + tc, n = a * (a + 1) / 2 + b;
          const float d = jj <= i ? expf(sG[i] - sG[jj]) : 0.f;
          put(i, jj, (kk[n].x + kk[n].y + other[n * 256]) * d, (qk[n].x + qk[n].y + other[(10 + n) * 256]) * d);
        }
    }
  } else {
    // The decay sits inside the contraction.  For i in block row I and j in an EARLIER block it factors through the gate
    // R_I of the block row's first token, e^{G_i-R_I} e^{R_I-G_j}, both exponents <= 0: a plain contraction of rescaled
    // rows.  Inside the diagonal block the second exponent would be >= 0 without bound, so it is evaluated entry by entry.
    float* const sM = sR;                                // (K e^{R_I-G}: 16, 32, 48 rows)
    const int half = tid >> 8, tr = ((warp & 7) << 1) | (lane & 1), tc = lane >> 1;
    for (int idx = tid; idx < 96 * (D / 4); idx += kPrepThreads) {
      const int r = idx / (D / 4), c = (idx % (D / 4)) * 4;
      const int I = r < 16 ? 1 : (r < 48 ? 2 : 3), jj = r - (I == 1 ? 0 : (I == 2 ? 16 : 48));
      st4(sM + r * LD + c, mul4(ld4(sK + jj * LD + c), exp_diff(ld4(sG + 16 * I * LD + c), ld4(sG + jj * LD + c))));
    }
#pragma unroll 1
    for (int a = 2 * half; a < 2 * half + 2; ++a) {
      const int i = 16 * a + tr, jj = 16 * a + tc;
      float s0 = 0.f, s1 = 0.f;
      if (tc <= tr) {
#pragma unroll 2
        for (int c = 0; c < D; c += 4) {
          const float4 x = mul4(ld4(sK + jj * LD + c), exp_diff(ld4(sG + i * LD + c), ld4(sG + jj * LD + c)));
          s0 = dot4(ld4(sK + i * LD + c), x, s0);
          s1 = dot4(ld4(sQ + i * LD + c), x, s1);
        }
      }
      put(i, jj, s0, s1);
    }
    __syncthreads();
    // KD from the raw rows, then the rows rescaled in place: k, q <- k, q e^{G-R_I}
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int i = li + 32 * u;
      const float4 k4 = ld4(sK + i * LD + lc), g4 = ld4(sG + i * LD + lc);
      st4(sKD + i * LD + lc, mul4(k4, exp_diff(ld4(sG + (C - 1) * LD + lc), g4)));
      const float4 e = exp_diff(g4, ld4(sG + (i & 48) * LD + lc));
      st4(sK + i * LD + lc, mul4(k4, e));
      st4(sQ + i * LD + lc, mul4(ld4(sQ + i * LD + lc), e));
    }
    __syncthreads();
    auto contract = [&](auto first, auto end) {          // block rows first .. end - 1
      constexpr int a0 = decltype(first)::value, a1 = decltype(end)::value;
      float kk[4][3] = {}, qk[4][3] = {};
#pragma unroll 2
      for (int c = 0; c < D; c += 4) {
#pragma unroll
        for (int a = a0; a < a1; ++a) {
          const float4 ki = ld4(sK + (16 * a + tr) * LD + c), qi = ld4(sQ + (16 * a + tr) * LD + c);
          const float* m = sM + (a == 1 ? 0 : (a == 2 ? 16 : 48)) * LD + c;
#pragma unroll
          for (int b = 0; b < a; ++b) {
            const float4 kj = ld4(m + (16 * b + tc) * LD);
            kk[a][b] = dot4(ki, kj, kk[a][b]);
            qk[a][b] = dot4(qi, kj, qk[a][b]);
          }
        }
      }
#pragma unroll
      for (int a = a0; a < a1; ++a)
#pragma unroll
        for (int b = 0; b < a; ++b) put(16 * a + tr, 16 * b + tc, kk[a][b], qk[a][b]);
    };
    if (half) contract(Int<3>{}, Int<4>{});
    else contract(Int<1>{}, Int<3>{});
  }
  __syncthreads();

  // ---- op #3 Solve: T = (I + A)^-1 by four warps, blocks of 16 and two levels of joining, T_lo = T_hi (-A_lo T_lo').  Meanwhile the others make the
  // right-hand sides diag(beta) [K e^G | V] and (GDN) KD.
  if (warp < 4) {
    auto sync4 = [&]() {                                 // (lanes come out of stores and loops of their own)
      __syncwarp();
      asm volatile("bar.sync 1, 128;" ::: "memory");
    };
    {                                                    // diagonal block `warp`, a column per lane (the upper lanes repeat the lower)
      const int c = lane & 15, o = 16 * warp;
      float y[16];
#pragma unroll
      for (int i = 0; i < 16; ++i) y[i] = i == c ? 1.f : 0.f;
      const float* at = sA + o * LD + o;
#pragma unroll
      for (int m = 0; m < 15; ++m)
#pragma unroll
        for (int q = (m + 1) / 4; q < 4; ++q) {
          const float4 a = ld4(at + m * LD + 4 * q);
          if (4 * q > m) y[4 * q] = fmaf(a.x, y[m], y[4 * q]);
          if (4 * q + 1 > m) y[4 * q + 1] = fmaf(a.y, y[m], y[4 * q + 1]);
          if (4 * q + 2 > m) y[4 * q + 2] = fmaf(a.z, y[m], y[4 * q + 2]);
          if (4 * q + 3 > m) y[4 * q + 3] = fmaf(a.w, y[m], y[4 * q + 3]);
        }
      if (lane < 16) {
#pragma unroll
        for (int i = 0; i < 16; ++i) sT[(o + i) * LD + o + c] = y[i];
      }
    }
    sync4();
    {                                                    // blocks (1, 0) and (3, 2): a row, four columns per thread
      const int o = 32 * (tid >> 6), i = (tid >> 2) & 15, c = (tid & 3) * 4;
      float* const x = sX + (tid >> 6) * 16 * 20;
      float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 8
      for (int m = 0; m < 16; ++m) axpy4(s, sA[(o + m) * LD + o + 16 + i], ld4(sT + (o + m) * LD + o + c));
      st4(x + i * 20 + c, s);
      sync4();
      s = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int m = 0; m < 16; m += 4) {
        const float4 t4 = ld4(sT + (o + 16 + i) * LD + o + 16 + m);
        axpy4(s, t4.x, ld4(x + m * 20 + c));
        axpy4(s, t4.y, ld4(x + (m + 1) * 20 + c));
        axpy4(s, t4.z, ld4(x + (m + 2) * 20 + c));
        axpy4(s, t4.w, ld4(x + (m + 3) * 20 + c));
      }
      st4(sT + (o + 16 + i) * LD + o + c, s);
    }
    sync4();
    {                                                    // the square between the halves: two rows, four columns per thread
      const int i = (tid >> 3) * 2, c = (tid & 7) * 4;
      float4 s0 = make_float4(0.f, 0.f, 0.f, 0.f), s1 = s0;
#pragma unroll 8
      for (int m = c & 16; m < 32; ++m) {
        const float2 a = *reinterpret_cast<const float2*>(sA + m * LD + 32 + i);
        const float4 t4 = ld4(sT + m * LD + c);
        axpy4(s0, a.x, t4);
        axpy4(s1, a.y, t4);
      }
      st4(sX + i * 36 + c, s0);
      st4(sX + (i + 1) * 36 + c, s1);
      sync4();
      s0 = s1 = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 4
      for (int m = 0; m < (i & 16) + 16; m += 4) {
        const float4 a = ld4(sT + (32 + i) * LD + 32 + m), b = ld4(sT + (33 + i) * LD + 32 + m);
        const float* pa = &a.x;
        const float* pb = &b.x;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const float4 x4 = ld4(sX + (m + e) * 36 + c);
          axpy4(s0, pa[e], x4);
          axpy4(s1, pb[e], x4);
        }
      }
      st4(sT + (32 + i) * LD + c, s0);
      st4(sT + (33 + i) * LD + c, s1);
    }
  } else {
    for (int idx = tid - 128; idx < C * (D / 4); idx += kPrepThreads - 128) {
      const int i = idx / (D / 4), c = (idx % (D / 4)) * 4;
      const float4 k4 = ld4(sK + i * LD + c);
      if (KDA) {                                         // (the rows are scaled up to R_I already)
        st4(sR + i * LDW + c, scale4(mul4(k4, exp4(ld4(sG + (i & 48) * LD + c))), sB[i]));
      } else {
        st4(sR + i * LDW + c, scale4(k4, expf(sG[i]) * sB[i]));
        st4(sKD + i * LD + c, scale4(k4, expf(sG[C - 1] - sG[i])));
      }
      if (c >= (i & 48) + 16) st4(sT + i * LD + c, make_float4(0.f, 0.f, 0.f, 0.f));   // T above its diagonal blocks
    }
  }
#pragma unroll
  for (int u = 0; u < 2; ++u) st4(sR + (li + 32 * u) * LDW + D + lc, scale4(v4[u], sB[li + 32 * u]));
  __syncthreads();

  // ---- L = [KD^T; P] T, by columns, in 4 x 4 tiles
  if (warp < 8) {
    // tokens from the column's on: the warps of one scheduler (w, w + 4) have 72 together
    const int r = (lane >> 1) * 4, m = 4 * (2 * (warp < 4 ? warp : 11 - warp) + (lane & 1));
    float4 s[4] = {};
#pragma unroll 8
    for (int t = m & ~7; t < C; ++t) {
      const float4 k4 = ld4(sKD + t * LD + r), t4 = ld4(sT + t * LD + m);
      axpy4(s[0], t4.x, k4);
      axpy4(s[1], t4.y, k4);
      axpy4(s[2], t4.z, k4);
      axpy4(s[3], t4.w, k4);
    }
#pragma unroll
    for (int e = 0; e < 4; ++e) st4(sL + (m + e) * LDW + r, s[e]);
  } else {
    const int w = warp - 8, i = 8 * (w < 4 ? w : 11 - w) + 4 * (lane & 1), m = (lane >> 1) * 4;
    float4 s[4] = {};
#pragma unroll 8
    for (int t = 0; t < (i & ~7) + 8; ++t) {             // (P is zero above the diagonal of its blocks, T everywhere)
      const float4 p4 = ld4(sP + t * LD + i), t4 = ld4(sT + t * LD + m);
      axpy4(s[0], t4.x, p4);
      axpy4(s[1], t4.y, p4);
      axpy4(s[2], t4.z, p4);
      axpy4(s[3], t4.w, p4);
    }
#pragma unroll
    for (int e = 0; e < 4; ++e) st4(sL + (m + e) * LDW + D + i, s[e]);
  }
  __syncthreads();

  // ---- L [K e^G | V]: eight rows to a warp; a lane has four of them and four columns of either half (of this CTA's share; SPLIT lanes
  // share a sum).  The warps of one scheduler have 64 + 64 + 72 terms.
  {
    const int w = warp & 7, rg = warp < 8 ? w : (w < 4 ? w : 11 - w), i0 = 8 * rg + 4 * (lane & 1);
    constexpr int COLS = 16 / SPLIT;
    const int part = (lane >> 1) / COLS, col = (share * COLS + (lane >> 1) % COLS) * 4, terms = warp < 8 ? C : 8 * rg + 8;
    const float* l = sL + (warp < 8 ? 0 : D) + i0;
    float4 sum[4][2] = {};                               // [row][K e^G, V]
#pragma unroll 4
    for (int m = part; m < terms; m += SPLIT) {
      const float4 x = ld4(l + m * LDW), r0 = ld4(sR + m * LDW + col), r1 = ld4(sR + m * LDW + D + col);
      const float lx[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        axpy4(sum[e][0], lx[e], r0);
        axpy4(sum[e][1], lx[e], r1);
      }
    }
    float acc[32];
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const float4 x = sum[e >> 1][e & 1];
      acc[4 * e] = x.x; acc[4 * e + 1] = x.y; acc[4 * e + 2] = x.z; acc[4 * e + 3] = x.w;
    }
    if (SPLIT > 1) scatter_lanes<32, 16, 32 / SPLIT>(acc, lane);   // (a lane keeps the part-th of SPLIT equal parts)
    float* rec = p.rec + (size_t)unit * Rec64::size;
    constexpr int FOURS = 8 / SPLIT;
#pragma unroll
    for (int e = 0; e < FOURS; ++e) {
      const int f = FOURS * part + e, i = i0 + (f >> 1), row = (warp < 8 ? 0 : C) + i;   // (f even: of K e^G, odd: of V)
      const float4 s = make_float4(acc[4 * e], acc[4 * e + 1], acc[4 * e + 2], acc[4 * e + 3]);
      if (f & 1) {
        st4(rec + Rec64::BC + (col / kSlice * 2 * C + row) * kSlice, s);
      } else {
        float4 base;
        if (warp < 8) {                                  // e^{G_L} on the diagonal
          const float gl = expf(KDA ? sG[(C - 1) * LD + i] : sG[C - 1]);
          base = make_float4(col == i ? gl : 0.f, col + 1 == i ? gl : 0.f, col + 2 == i ? gl : 0.f, col + 3 == i ? gl : 0.f);
        } else {                                         // Q e^G (KDA: from q e^{G-R_I})
          const float4 q4 = ld4(sQ + i * LD + col);
          base = KDA ? mul4(q4, exp4(ld4(sG + (i & 48) * LD + col))) : scale4(q4, expf(sG[i]));
        }
        st4(rec + Rec64::MN + row * D + (col ^ ((row & 1) << 4)), make_float4(base.x - s.x, base.y - s.y, base.z - s.z, base.w - s.w));
      }
    }
  }
}

// ------------------------------------------------------------------------------------------------ sequential part
template <int NV> struct Walk64Smem {
  static constexpr int kStages = NV == 16 ? 3 : 4;
  static constexpr int BC = 2 * C * D;                   // [NV / kSlice][2 C][kSlice]
  static constexpr int kStage = BC + 2 * C * NV;
  static constexpr int H = kStages * kStage;             // state, two copies taken in turn, [NV][LD]
  static constexpr int BAR = H + 2 * NV * LD;
  static constexpr size_t bytes = (size_t)BAR * 4 + kStages * 8 + 8;
};

template <int NV> constexpr int kThreadCols = NV == 16 ? 8 : 4;
template <int NV> constexpr int kWalk64Threads = 128 * (NV / kThreadCols<NV>);
// 128 threads for four channels: a thread makes four rows (of [M; N]) by four channels over a quarter of the depth; the four parts of the sums
// sit in neighbouring lanes, which add them up so that each ends with four channels of one row, lanes 0 and 1 of M (new state), 2 and 3 of N
// (output).  The rows of the next chunk are read under the end of this one.
template <typename In, int NV>
__global__ void __launch_bounds__(kWalk64Threads<NV>, 1) fp32_walk64_kernel(Fp32Params p) {
  using S = Walk64Smem<NV>;
  constexpr int CT = kThreadCols<NV>, CF = CT / 4;       // channels per thread, and their fours
  constexpr int NSL = D / NV, ST = S::kStages;
  extern __shared__ __align__(16) float sf[];
  float* const sH = sf + S::H;
  uint64_t* full = reinterpret_cast<uint64_t*>(sf + S::BAR);   // [stages]
  const int tid = threadIdx.x, cg = tid >> 7, part = tid & 3, grp = (tid & 127) >> 2;
  const int row = grp + 32 * part;                       // of [M; N], once summed up
  const int slice = blockIdx.x % NSL, nj = blockIdx.x / NSL, j = nj % p.HV;
  const bool packed = p.seq_tok0 != nullptr, state = row < D;
  int n = nj / p.HV, tok0 = packed ? 0 : n * p.T_row, slot0 = packed ? 0 : n * p.cps, len = p.T_row, nch = (len + C - 1) / C;
  if (tid == 0) {
    for (int i = 0; i < ST; ++i) mbar_init(&full[i], 1);
    mbar_fence_init();
  }
  __syncthreads();
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (packed) {                                          // (a batch without a token has no kernel between the plan kernel and this one)
    if (p.seq_order) n = p.seq_order[n];
    tok0 = p.seq_tok0[n];
    slot0 = p.seq_chunk0[n];
    len = p.seq_len[n];
    nch = (len + C - 1) / C;
  }
  auto load = [&](int c) {
    const float* rec = p.rec + ((size_t)(slot0 + c) * p.HV + j) * Rec64::size;
    float* st = sf + (c % ST) * S::kStage;
    mbar_expect_tx(&full[c % ST], S::kStage * 4);
    bulk_load(st, rec + Rec64::MN, S::BC * 4, &full[c % ST]);
    bulk_load(st + S::BC, rec + Rec64::BC + slice * (NV / kSlice) * 2 * C * kSlice, 2 * C * NV * 4, &full[c % ST]);
  };
  if (tid == 0) {
    fence_proxy_async_all();
    for (int c = 0; c < ST && c < nch; ++c) load(c);
  }
  const int ch0 = slice * NV + cg * CT;
  const size_t hbase = (((size_t)n * p.HV + j) * D + (state ? row : 0)) * D + ch0;
  float4 h[CF] = {};
  auto put_state = [&](int copy) {
    float* s = sH + (copy * NV + cg * CT) * LD + row;
#pragma unroll
    for (int f = 0; f < CF; ++f) {
      s[4 * f * LD] = h[f].x; s[(4 * f + 1) * LD] = h[f].y; s[(4 * f + 2) * LD] = h[f].z; s[(4 * f + 3) * LD] = h[f].w;
    }
  };
  if (state) {
#pragma unroll
    for (int f = 0; f < CF; ++f)
      if (p.h0) h[f] = ld4(p.h0 + hbase + 4 * f);
    put_state(0);
  }
  In* go = reinterpret_cast<In*>(p.o) + ((size_t)(tok0 + (state ? 0 : row - D)) * p.HV + j) * D + ch0;
  int gave_up = 0;
  volatile int* abort_flag = &gave_up;                   // (every wait is bounded)
  int st = 0;
  uint32_t ph = 0;
  // A row's 64 columns: this thread has 4 part .. + 3 of each 16.  Eight lanes read two rows, 64 bytes each, which the exchange in odd rows puts
  // into different banks.
  constexpr bool kAhead = CT == 4;                       // the next chunk's rows are read under the end of this one
  float4 w[4][4];
  auto ready = [&]() {
    if (!mbar_test_wait(&full[st], ph)) mbar_wait(&full[st], ph, abort_flag);
  };
  auto rows = [&](int k) {
    const float* m = sf + st * S::kStage + grp * D + 4 * part;
#pragma unroll
    for (int i = 0; i < 4; ++i) w[i][k] = ld4(m + 32 * i * D + 16 * (k ^ (grp & 1)));
  };
  if (nch > 0) {
    ready();
#pragma unroll
    for (int k = 0; kAhead && k < 4; ++k) rows(k);
  }
  __syncthreads();
  for (int c = 0; c < nch; ++c) {
    const float* hp = sH + ((c & 1) * NV + cg * CT) * LD + 4 * part;
    float4 add[CF];
#pragma unroll
    for (int f = 0; f < CF; ++f) add[f] = ld4(sf + st * S::kStage + S::BC + ((cg * CF + f) * 2 * C + row) * kSlice);
    float2 y[4][CT] = {};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      if (!kAhead) rows(k);
#pragma unroll
      for (int e = 0; e < CT; ++e) {
        const float4 hv = ld4(hp + e * LD + 16 * k);
#pragma unroll
        for (int i = 0; i < 4; ++i) y[i][e] = dot_pairs(w[i][k], hv, y[i][e]);
      }
    }
    float x[4 * CT];
#pragma unroll
    for (int i = 0; i < 4 * CT; ++i) x[i] = y[i / CT][i % CT].x + y[i / CT][i % CT].y;
    scatter_lanes<4 * CT, 2, 1>(x, part);
    if (++st == ST) { st = 0; ph ^= 1; }
#pragma unroll
    for (int f = 0; f < CF; ++f)
      h[f] = make_float4(x[4 * f] + add[f].x, x[4 * f + 1] + add[f].y, x[4 * f + 2] + add[f].z, x[4 * f + 3] + add[f].w);
    if (state) put_state((c & 1) ^ 1);
    if (c + 1 < nch) {
      ready();
#pragma unroll
      for (int k = 0; kAhead && k < 4; ++k) rows(k);
    }
    if (!state && row - D < len - c * C) {
#pragma unroll
      for (int f = 0; f < CF; ++f) store4(go + (size_t)c * C * p.HV * D + 4 * f, scale4(h[f], p.scale));
    }
    __syncthreads();                                     // the new state is complete, the chunk's operands are free
    if (tid == 0 && c + ST < nch) load(c + ST);
  }
  if (gave_up) report_timeout(p.status);
  if (p.hT && state) {
#pragma unroll
    for (int f = 0; f < CF; ++f) st4(p.hT + hbase + 4 * f, h[f]);
  }
}

template <typename In, bool KDA>
cudaError_t run(const Problem& p, const Fp32Params& fp, cudaStream_t stream) {
  constexpr size_t prep_smem = Prep64Smem<In, KDA>::size * 4;
  static_assert(prep_smem <= 227 * 1024 && Walk64Smem<4>::bytes <= 227 * 1024 && Walk64Smem<8>::bytes <= 227 * 1024 && Walk64Smem<16>::bytes <= 227 * 1024,
                "shared memory budget");
  const long long units = (long long)p.max_chunks * p.HV, sms = sm_count();
  if (units > 0) {
    timer_mark(stream, "simt_prep");
    // Idle SMs share the last product of a chunk, by columns (4.4 us of its time alone, 1.5 by four, 1.0 by eight; all else is made by each).
    cudaError_t e;
    if (units * 8 <= sms) e = launch_fp32_kernel<fp32_prep64_kernel<In, KDA, 8>>((unsigned)units * 8, kPrepThreads, prep_smem, stream, fp);
    else if (units * 4 <= sms) e = launch_fp32_kernel<fp32_prep64_kernel<In, KDA, 4>>((unsigned)units * 4, kPrepThreads, prep_smem, stream, fp);
    else if (units * 2 <= sms) e = launch_fp32_kernel<fp32_prep64_kernel<In, KDA, 2>>((unsigned)units * 2, kPrepThreads, prep_smem, stream, fp);
    else e = launch_fp32_kernel<fp32_prep64_kernel<In, KDA, 1>>((unsigned)units, kPrepThreads, prep_smem, stream, fp);
    if (e != cudaSuccess) return e;
  }
  timer_mark(stream, "simt_prefill");
  // The narrowest slices that leave every CTA an SM; else 16 channels, eight to a thread (fewer reads of the shared operands per channel: two rows of
  // 1000, 16 heads 82.4 us with four).
  const long long heads = (long long)p.N * p.HV;
  if (heads * (D / 4) <= sms)
    return launch_fp32_kernel<fp32_walk64_kernel<In, 4>>((unsigned)(heads * (D / 4)), (unsigned)kWalk64Threads<4>, Walk64Smem<4>::bytes, stream, fp);
  if (heads * (D / 8) <= sms)
    return launch_fp32_kernel<fp32_walk64_kernel<In, 8>>((unsigned)(heads * (D / 8)), (unsigned)kWalk64Threads<8>, Walk64Smem<8>::bytes, stream, fp);
  return launch_fp32_kernel<fp32_walk64_kernel<In, 16>>((unsigned)(heads * (D / 16)), (unsigned)kWalk64Threads<16>, Walk64Smem<16>::bytes, stream, fp);
}

}  // namespace

size_t fp32_d64_record_bytes() { return Rec64::size * sizeof(float); }

cudaError_t launch_fp32_d64(const Problem& p, const Fp32Params& fp, cudaStream_t stream) {
  const bool kda = p.variant == HA_LA_KDA;
  if (p.dtype == HA_LA_BF16) return kda ? run<__nv_bfloat16, true>(p, fp, stream) : run<__nv_bfloat16, false>(p, fp, stream);
  return kda ? run<float, true>(p, fp, stream) : run<float, false>(p, fp, stream);
}

}  // namespace ha_la
