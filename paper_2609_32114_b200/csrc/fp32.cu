// fp32 chunkwise delta-rule prefill (GDN and KDA) on the CUDA cores, in two kernels, for head dimension 128: fp32 inputs (where the
// 1e-4 tolerance rules out 16-bit tensor-core operands).  All arithmetic is fp32.  (d = 64: fp32_d64.cu.)
//
//   fp32_prep_kernel   one CTA per (chunk, V-head): operators #1-#4 of the paper's pipeline (Section 2.1, "Chunkwise
//                      Map-Reduce-Map Execution").  Chunks are independent here, so a single short sequence already
//                      keeps several SMs busy instead of one.
//   fp32_walk_kernel   one CTA per (sequence, V-head, 4, 8 or 16 value channels) walks the chunks in order: operator #5 with #6 in
//                      the paper's chunk-first order.  Value channels are independent ("Computation Splitting"), so the
//                      sequential part of a head is spread over several SMs.
//
// Per chunk the prep kernel leaves, as fp32 rows padded for conflict-free 16-byte shared-memory reads:
//   W = T diag(beta) (K e^G)   QG = Q e^G   KD = K e^{G_L-G}   P = decay-masked Q K^T   U = T diag(beta) V   e^{G_L}
// and the walk does    U~ = U - W h;   o = scale (QG h + P U~);   h <- e^{G_L} h + KD^T U~.
//
// What bounds it: shared-memory reads (a 16-byte read costs four cycles of the SM's 128 bytes, 2.2 where neighbouring lanes share
// addresses), the walk's two barriers per chunk, and for short sequences its chain of chunks: 2.2 us each.  4 heads, T = 400: 31.7 us (32.2 with lanes that share rows
// apart and the gates summed behind a barrier of their own), KDA, T = 300 42.7 (44.2).
#include "fp32_common.cuh"

namespace ha_la {

size_t fp32_d64_record_bytes();                          // fp32_d64.cu
cudaError_t launch_fp32_d64(const Problem& p, const Fp32Params& fp, cudaStream_t stream);

using namespace ptx;

namespace {

constexpr int C = kChunk, D = 128;
constexpr int kNV = 16;                                  // value channels per slice of U in a record
constexpr int LDP = C + 4;                               // row strides in floats: rows 16 bytes apart in the banks

// record of one (chunk slot, V-head), in floats
struct Rec {
  static constexpr int LD = D + 4;
  static constexpr int W = 0;                            // [C][LD]
  static constexpr int QG = W + C * LD;                  // [C][LD]
  static constexpr int KD = QG + C * LD;                 // [C][LD]
  static constexpr int P = KD + C * LD;                  // [C][LDP]
  static constexpr int GAM = P + C * LDP;                // [D]  e^{G_L} per key channel
  static constexpr int U = GAM + D;                      // [D / kNV][C][kNV]
  static constexpr int size = U + C * D;
};

// ------------------------------------------------------------------------------------------------ chunk-local part
template <bool KDA> struct PrepSmem {
  static constexpr int LD = D + 4;
  static constexpr int K = 0;                            // [C][LD]
  static constexpr int Q = K + C * LD;                   // [C][LD]
  static constexpr int A = Q + C * LD;                   // [C][LDP]
  static constexpr int G = A + C * LDP;                  // GDN [C]; KDA [C][LD]: cumulative log-gate
  static constexpr int B = G + (KDA ? C * LD : C);       // [C] beta
  static constexpr int RHS = B + C;                      // [C][2 D]: (W |) U columns of the substitution
  static constexpr int KM = RHS;                         // KDA: K e^{R_I-G}, block rows I = 1, 2, 3 (16, 32, 48 rows), over the
                                                         // columns, which are filled later
  static constexpr int size = RHS + C * 2 * D;
};

template <typename In, bool KDA>
__global__ void __launch_bounds__(256) fp32_prep_kernel(Fp32Params p) {
  using S = PrepSmem<KDA>;
  using R = Rec;
  constexpr int LD = D + 4;
  extern __shared__ __align__(16) float sf[];
  float* sK = sf + S::K;
  float* sQ = sf + S::Q;
  float* sA = sf + S::A;
  float* sG = sf + S::G;
  float* sB = sf + S::B;
  const int tid = threadIdx.x;
  const int slot = blockIdx.x / p.HV, j = blockIdx.x % p.HV, jq = j / (p.HV / p.HK);
  // (this call's kernels are launched as programmatic dependents; nothing has been read so far)
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  int L, t0;
  if (p.chunk_len) {
    L = p.chunk_len[slot];
    t0 = p.chunk_tok0[slot];
  } else {
    const int cc = slot % p.cps;
    t0 = (slot / p.cps) * p.T_row + cc * C;
    L = min(C, p.T_row - cc * C);
  }
  if (L <= 0) return;                                    // a slot that a packed batch does not use
  const In* gq = reinterpret_cast<const In*>(p.q);
  const In* gk = reinterpret_cast<const In*>(p.k);
  const In* gv = reinterpret_cast<const In*>(p.v);
  float* rec = p.rec + (size_t)blockIdx.x * R::size;

  constexpr bool kLateV = KDA;                           // (its room holds the rescaled K rows first)
  auto v_row = [&](int i, int c) {
    return i < L ? load4(gv + ((size_t)(t0 + i) * p.HV + j) * D + c) : make_float4(0.f, 0.f, 0.f, 0.f);
  };
  // ---- load the chunk; rows >= L are no-op tokens (k = q = v = 0, beta = 0, g = 0)
#pragma unroll
  for (int idx = tid; idx < C * (D / 4); idx += 256) {
    const int i = idx / (D / 4), c = (idx % (D / 4)) * 4;
    float4 q4 = make_float4(0.f, 0.f, 0.f, 0.f), k4 = q4, g4 = q4;
    if (i < L) {
      const size_t off = ((size_t)(t0 + i) * p.HK + jq) * D + c;
      q4 = load4(gq + off);
      k4 = load4(gk + off);
      if (KDA) g4 = ld4(p.g + ((size_t)(t0 + i) * p.HV + j) * D + c);
    }
    *reinterpret_cast<float4*>(sQ + i * LD + c) = q4;
    *reinterpret_cast<float4*>(sK + i * LD + c) = k4;
    if (!kLateV) *reinterpret_cast<float4*>(sf + S::RHS + i * 2 * D + D + c) = v_row(i, c);
    if (KDA) *reinterpret_cast<float4*>(sG + i * LD + c) = g4;
  }
  const int warp = tid >> 5, lane = tid & 31;
  if (warp < 2) sB[tid] = tid < L ? p.beta[(size_t)(t0 + tid) * p.HV + j] : 0.f;
  // ---- op #1 Gate: chunk-local inclusive cumulative sum of the log-gate (GDN: by a warp while the tiles are on their way)
  if (!KDA && warp == 2) {
    float x0 = lane < L ? p.g[(size_t)(t0 + lane) * p.HV + j] : 0.f, x1 = lane + 32 < L ? p.g[(size_t)(t0 + lane + 32) * p.HV + j] : 0.f;
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

  // ---- op #2: A (strictly lower, beta-scaled, negated: what the substitution adds) and P (lower incl. diagonal), in
  // 16 x 16 blocks; thread (tr, tc) owns one entry of every block.  Neighbouring lanes share columns: their reads are then one.
  const int tr = (warp << 1) | (lane & 1), tc = lane >> 1;
  float kk[4][4], qk[4][4];                              // [block row][block column <= block row]
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) kk[a][b] = qk[a][b] = 0.f;
  if constexpr (!KDA) {
#pragma unroll 2
    for (int c = 0; c < D; c += 4) {
      float4 kj[4];
#pragma unroll
      for (int b = 0; b < 4; ++b) kj[b] = ld4(sK + (16 * b + tc) * LD + c);
#pragma unroll
      for (int a = 0; a < 4; ++a) {
        const float4 ki = ld4(sK + (16 * a + tr) * LD + c), qi = ld4(sQ + (16 * a + tr) * LD + c);
#pragma unroll
        for (int b = 0; b <= a; ++b) {
          kk[a][b] = dot4(ki, kj[b], kk[a][b]);
          qk[a][b] = dot4(qi, kj[b], qk[a][b]);
        }
      }
    }
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int b = 0; b <= a; ++b) {
        const float e = 16 * b + tc <= 16 * a + tr ? expf(sG[16 * a + tr] - sG[16 * b + tc]) : 0.f;
        kk[a][b] *= e;
        qk[a][b] *= e;
      }
  } else {
    // The decay sits inside the contraction.  For i in block row I and j in an EARLIER block it factors through the gate
    // R_I of the block row's first token, e^{G_i-R_I} e^{R_I-G_j}, both exponents <= 0: a plain contraction of rescaled
    // rows.  Inside the diagonal block the second exponent would be >= 0 without bound, so it is evaluated entry by entry.
    float* sM = sf + S::KM;
    for (int idx = tid; idx < 96 * (D / 4); idx += 256) {
      const int r = idx / (D / 4), c = (idx % (D / 4)) * 4;
      const int I = r < 16 ? 1 : (r < 48 ? 2 : 3), jj = r - (I == 1 ? 0 : (I == 2 ? 16 : 48));
      const float4 k4 = ld4(sK + jj * LD + c), g4 = ld4(sG + jj * LD + c), r4 = ld4(sG + 16 * I * LD + c);
      *reinterpret_cast<float4*>(sM + r * LD + c) = make_float4(k4.x * expf(r4.x - g4.x), k4.y * expf(r4.y - g4.y),
                                                                k4.z * expf(r4.z - g4.z), k4.w * expf(r4.w - g4.w));
    }
#pragma unroll 1
    for (int a = 0; a < 4; ++a) {
      if (tc > tr) continue;
      float s0 = 0.f, s1 = 0.f;
      const int i = 16 * a + tr, jj = 16 * a + tc;
#pragma unroll 2
      for (int c = 0; c < D; c += 4) {
        const float4 ki = ld4(sK + i * LD + c), qi = ld4(sQ + i * LD + c), kj = ld4(sK + jj * LD + c);
        const float4 gi = ld4(sG + i * LD + c), gj = ld4(sG + jj * LD + c);
        const float4 x = make_float4(kj.x * expf(gi.x - gj.x), kj.y * expf(gi.y - gj.y), kj.z * expf(gi.z - gj.z),
                                     kj.w * expf(gi.w - gj.w));
        s0 = dot4(ki, x, s0);
        s1 = dot4(qi, x, s1);
      }
#pragma unroll
      for (int b = 0; b < 4; ++b)
        if (b == a) { kk[b][b] = s0; qk[b][b] = s1; }
    }
    __syncthreads();
    // images for the walk from the raw rows, then the rows rescaled in place: k, q <- k, q e^{G-R_I}
    for (int idx = tid; idx < C * (D / 4); idx += 256) {
      const int i = idx / (D / 4), c = (idx % (D / 4)) * 4;
      float4 k4 = ld4(sK + i * LD + c), q4 = ld4(sQ + i * LD + c);
      const float4 g4 = ld4(sG + i * LD + c), r4 = ld4(sG + (i & 48) * LD + c), l4 = ld4(sG + 63 * LD + c);
      *reinterpret_cast<float4*>(rec + R::KD + i * LD + c) = make_float4(
          k4.x * expf(l4.x - g4.x), k4.y * expf(l4.y - g4.y), k4.z * expf(l4.z - g4.z), k4.w * expf(l4.w - g4.w));
      *reinterpret_cast<float4*>(rec + R::QG + i * LD + c) =
          make_float4(q4.x * expf(g4.x), q4.y * expf(g4.y), q4.z * expf(g4.z), q4.w * expf(g4.w));
      const float4 e = make_float4(expf(g4.x - r4.x), expf(g4.y - r4.y), expf(g4.z - r4.z), expf(g4.w - r4.w));
      *reinterpret_cast<float4*>(sK + i * LD + c) = make_float4(k4.x * e.x, k4.y * e.y, k4.z * e.z, k4.w * e.w);
      *reinterpret_cast<float4*>(sQ + i * LD + c) = make_float4(q4.x * e.x, q4.y * e.y, q4.z * e.z, q4.w * e.w);
    }
    __syncthreads();
#pragma unroll 2
    for (int c = 0; c < D; c += 4) {
#pragma unroll
      for (int a = 1; a < 4; ++a) {
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
  }
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      const int i = 16 * a + tr, jj = 16 * b + tc;
      if (b <= a) sA[jj * LDP + i] = jj < i ? -sB[i] * kk[a][b] : 0.f;   // transposed
      rec[R::P + i * LDP + jj] = jj <= i ? qk[a][b] : 0.f;
    }
  if (kLateV) {
    __syncthreads();
#pragma unroll 4
    for (int idx = tid; idx < C * (D / 4); idx += 256)
      *reinterpret_cast<float4*>(sf + S::RHS + (idx / (D / 4)) * 2 * D + D + (idx % (D / 4)) * 4) = v_row(idx / (D / 4), (idx % (D / 4)) * 4);
  }
  __syncthreads();

  // ---- op #3 Solve + op #4 W/U: forward substitution of (I + A) [W | U] = diag(beta) [K e^G | V], one thread per column,
  // in blocks of 16 rows held in registers.  The coefficients are broadcast reads of A^T.  (Unrolled over all 64 rows the
  // code was 40 KiB run once per launch: 13 us of instruction fetches.)
  {
    const int c = tid % D;
    float* col = sf + S::RHS + tid;                      // [C][2 D]: this thread's column
    float* dst = tid < D ? rec + R::W + c : rec + R::U + (c / kNV) * (C * kNV) + c % kNV;
    const int ld = tid < D ? LD : kNV;
#pragma unroll 1
    for (int I = 0; I < 4; ++I) {
      float y[16];
      if (tid < D) {
        const float eI = KDA ? expf(sG[16 * I * LD + c]) : 1.f;            // (KDA: the rows are scaled up to R_I already)
#pragma unroll
        for (int i = 0; i < 16; ++i)
          y[i] = sB[16 * I + i] * sK[(16 * I + i) * LD + c] * (KDA ? eI : expf(sG[KDA ? 0 : 16 * I + i]));
      } else {
#pragma unroll
        for (int i = 0; i < 16; ++i) y[i] = sB[16 * I + i] * col[(16 * I + i) * 2 * D];
      }
      const float* at = sA + 16 * I;                     // A^T[m][16 I ..]
#pragma unroll 4
      for (int m = 0; m < 16 * I; ++m) {
        const float v = col[m * 2 * D];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const float4 a = ld4(at + m * LDP + 4 * q);
          y[4 * q] = fmaf(a.x, v, y[4 * q]);
          y[4 * q + 1] = fmaf(a.y, v, y[4 * q + 1]);
          y[4 * q + 2] = fmaf(a.z, v, y[4 * q + 2]);
          y[4 * q + 3] = fmaf(a.w, v, y[4 * q + 3]);
        }
      }
      at += 16 * I * LDP;
#pragma unroll
      for (int m = 0; m < 15; ++m)
#pragma unroll
        for (int q = (m + 1) / 4; q < 4; ++q) {
          const float4 a = ld4(at + m * LDP + 4 * q);
          if (4 * q > m) y[4 * q] = fmaf(a.x, y[m], y[4 * q]);
          if (4 * q + 1 > m) y[4 * q + 1] = fmaf(a.y, y[m], y[4 * q + 1]);
          if (4 * q + 2 > m) y[4 * q + 2] = fmaf(a.z, y[m], y[4 * q + 2]);
          if (4 * q + 3 > m) y[4 * q + 3] = fmaf(a.w, y[m], y[4 * q + 3]);
        }
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        col[(16 * I + i) * 2 * D] = y[i];
        dst[(16 * I + i) * ld] = y[i];
      }
    }
  }
  if (!KDA) {                                            // the walk's other images
    const float gl = sG[C - 1];
    for (int idx = tid; idx < C * (D / 4); idx += 256) {
      const int i = idx / (D / 4), c = (idx % (D / 4)) * 4;
      const float4 k4 = ld4(sK + i * LD + c), q4 = ld4(sQ + i * LD + c);
      const float ek = expf(gl - sG[i]), eq = expf(sG[i]);
      *reinterpret_cast<float4*>(rec + R::KD + i * LD + c) = make_float4(k4.x * ek, k4.y * ek, k4.z * ek, k4.w * ek);
      *reinterpret_cast<float4*>(rec + R::QG + i * LD + c) = make_float4(q4.x * eq, q4.y * eq, q4.z * eq, q4.w * eq);
    }
  }
  if (tid < D) rec[R::GAM + tid] = expf(KDA ? sG[(C - 1) * LD + tid] : sG[C - 1]);
}

// ------------------------------------------------------------------------------------------------ sequential part
struct WalkSmem {
  static constexpr int LD = D + 4;
  static constexpr int kStages = 1;                      // chunks whose operands fit (a load takes about as long as a half step)
  static constexpr int WQ = 0;                           // W, QG of the chunk
  static constexpr int KP = WQ + 2 * C * LD;             // KD, P, e^{G_L}
  static constexpr int U = KP + C * LD + C * LDP + D;    // U slice [C][kNV]
  static constexpr int kStage = U + C * kNV;
  static constexpr int HT = kStages * kStage;            // state [kNV][LD]
  static constexpr int UT = HT + kNV * LD;               // U~ [kNV][LDP]
  static constexpr int Y = UT + kNV * LDP;               // QG h [C][kNV + 1]
  static constexpr int BAR = (Y + C * (kNV + 1) + 3) / 4 * 4;
  static constexpr size_t bytes = (size_t)BAR * 4 + 32;
};
// Threads: the first kUpd update the state, then 256 form the outputs; the first 512 compute W h and QG h.  A thread makes
// four rows (tokens, keys) by NV / 2 channels of a product over an eighth of its depth: sixteen and more multiply-adds for
// every two 16-byte reads, where reads bound the kernel.  The eight parts of a sum sit in neighbouring lanes, which add
// them up so that each ends with one row and NV / 4 channels.
constexpr int kUpd = D * 4, kWalkThreads = kUpd + 256;
// v[N] summed over eight neighbouring lanes; lane l keeps the sums N / 8 (l % 8) .. in v[0 .. N / 8)
template <int N> __device__ __forceinline__ void scatter_sum(float (&v)[N], int lane) {
#pragma unroll
  for (int b = 4, n = N / 2; b > 0; b >>= 1, n /= 2) {
    const bool up = lane & b;
#pragma unroll
    for (int i = 0; i < N / 2; ++i) {
      if (i >= n) break;
      const float keep = up ? v[i + n] : v[i], send = up ? v[i] : v[i + n];
      v[i] = keep + __shfl_xor_sync(0xffffffffu, send, b);
    }
  }
}

template <typename In, int NV>
__global__ void __launch_bounds__(kWalkThreads, 1) fp32_walk_kernel(Fp32Params p) {
  using S = WalkSmem;
  using R = Rec;
  constexpr int LD = D + 4, NSL = D / NV, H = NV / 2, E = NV / 4;   // channels of a thread's products; of its sums
  extern __shared__ __align__(16) float sf[];
  constexpr int ST = S::kStages;
  float* sH = sf + S::HT;
  float* sT = sf + S::UT;
  float* sY = sf + S::Y;
  uint64_t* bar1 = reinterpret_cast<uint64_t*>(sf + S::BAR);   // [stages] W, QG, U
  uint64_t* bar3 = bar1 + 2;                                   // [stages] KD, P, e^{G_L}
  const int tid = threadIdx.x, part = tid & 7, ch0 = ((tid >> 3) & 1) * H, grp = tid >> 4;
  const int row = part >> 1, ch = ch0 + (part & 1) * E;   // this thread's row of four and first channel, once summed up
  const int slice = blockIdx.x % NSL, nj = blockIdx.x / NSL, j = nj % p.HV;
  const bool packed = p.seq_tok0 != nullptr;
  int n = nj / p.HV, tok0 = packed ? 0 : n * p.T_row, slot0 = packed ? 0 : n * p.cps, len = p.T_row, nch = (len + C - 1) / C;
  if (tid == 0) {
    for (int i = 0; i < ST; ++i) { mbar_init(&bar1[i], 1); mbar_init(&bar3[i], 1); }
    mbar_fence_init();
  }
  // state: thread -> key 4 grp + row, its E channels of the slice
  const bool upd = tid < kUpd;
  const int key = 4 * grp + row;
  const int uc = slice % (kNV / NV) * NV;       // first channel within the record's U slice
  float h[E];
#pragma unroll
  for (int e = 0; e < E; ++e) h[e] = 0.f;
  __syncthreads();
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (packed) {                                          // (a batch without a token has no kernel between the plan kernel and this one)
    if (p.seq_order) n = p.seq_order[n];
    tok0 = p.seq_tok0[n];
    slot0 = p.seq_chunk0[n];
    len = p.seq_len[n];
    nch = (len + C - 1) / C;
  }
  const size_t hbase = (((size_t)n * p.HV + j) * D + key) * D + slice * NV + ch;
  if (upd) {
#pragma unroll
    for (int e = 0; e < E; ++e) {
      h[e] = p.h0 ? p.h0[hbase + e] : 0.f;
      sH[(ch + e) * LD + key] = h[e];
    }
  }
  auto load1 = [&](int c) {
    const float* rec = p.rec + ((size_t)(slot0 + c) * p.HV + j) * R::size;
    float* st = sf + (c % ST) * S::kStage;
    mbar_expect_tx(&bar1[c % ST], (2 * C * LD + C * kNV) * 4);
    bulk_load(st + S::WQ, rec + R::W, 2 * C * LD * 4, &bar1[c % ST]);
    bulk_load(st + S::U, rec + R::U + (slice * NV / kNV) * (C * kNV), C * kNV * 4, &bar1[c % ST]);
  };
  auto load3 = [&](int c) {
    const float* rec = p.rec + ((size_t)(slot0 + c) * p.HV + j) * R::size;
    constexpr uint32_t bytes = (C * LD + C * LDP + D) * 4;
    mbar_expect_tx(&bar3[c % ST], bytes);
    bulk_load(sf + (c % ST) * S::kStage + S::KP, rec + R::KD, bytes, &bar3[c % ST]);
  };
  if (tid == 0) {
    fence_proxy_async_all();
    for (int c = 0; c < ST && c < nch; ++c) { load1(c); load3(c); }
  }
  int gave_up = 0;
  volatile int* abort_flag = &gave_up;                   // (every wait is bounded)
  __syncthreads();

  for (int c = 0; c < nch; ++c) {
    const float* sW = sf + (c % ST) * S::kStage + S::WQ;
    const float* sK = sf + (c % ST) * S::kStage + S::KP;   // (QG follows W: rows 64 .. 127 of one operand)
    const float* sP = sK + C * LD;
    const float* sGam = sP + C * LDP;
    const float* sU = sf + (c % ST) * S::kStage + S::U;
    // ---- [W; QG] h: 128 rows x NV channels; rows grp + 32 i
    if (tid < 512) {
      if (!mbar_test_wait(&bar1[c % ST], (c / ST) & 1)) mbar_wait(&bar1[c % ST], (c / ST) & 1, abort_flag);
      float x[4 * H] = {};
#pragma unroll 2
      for (int k = 4 * part; k < D; k += 32) {
        float4 w[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) w[i] = ld4(sW + (grp + 32 * i) * LD + k);
#pragma unroll
        for (int e = 0; e < H; ++e) {
          const float4 hv = ld4(sH + (ch0 + e) * LD + k);
#pragma unroll
          for (int i = 0; i < 4; ++i) x[i * H + e] = dot4(w[i], hv, x[i * H + e]);
        }
      }
      scatter_sum(x, part);
      const int t = grp + 32 * (row & 1);
#pragma unroll
      for (int e = 0; e < E; ++e) {
        if (row < 2) sT[(ch + e) * LDP + t] = sU[t * kNV + uc + ch + e] - x[e];
        else sY[t * (kNV + 1) + ch + e] = x[e];
      }
    }
    __syncthreads();                                     // U~ and QG h are complete; W, QG, U and the old state are free
    if (tid == 0 && c + ST < nch) load1(c + ST);
    if (!mbar_test_wait(&bar3[c % ST], (c / ST) & 1)) mbar_wait(&bar3[c % ST], (c / ST) & 1, abort_flag);
    if (upd) {
      // ---- h <- e^{G_L} h + KD^T U~: keys 4 grp .., tokens part + 8 m
      float d[4 * H] = {};
#pragma unroll 4
      for (int t = part; t < C; t += 8) {
        const float4 k4 = ld4(sK + t * LD + 4 * grp);
#pragma unroll
        for (int e = 0; e < H; ++e) {
          const float u = sT[(ch0 + e) * LDP + t];
          d[e] = fmaf(k4.x, u, d[e]);
          d[H + e] = fmaf(k4.y, u, d[H + e]);
          d[2 * H + e] = fmaf(k4.z, u, d[2 * H + e]);
          d[3 * H + e] = fmaf(k4.w, u, d[3 * H + e]);
        }
      }
      scatter_sum(d, part);
      const float gm = sGam[key];
#pragma unroll
      for (int e = 0; e < E; ++e) {
        h[e] = fmaf(gm, h[e], d[e]);
        sH[(ch + e) * LD + key] = h[e];
      }
    } else {
      // ---- o = scale (QG h + P U~): rows rg + 16 i, tokens 4 part + 32 m; P's blocks of 16 above the diagonal are not there
      const int rg = grp - kUpd / 16;
      float s[4 * H] = {};
#pragma unroll
      for (int m = 0; m < 2; ++m) {
        const int t = 4 * part + 32 * m;
        float4 q[4];
#pragma unroll
        for (int i = 2 * m; i < 4; ++i) q[i] = t < 16 * (i + 1) ? ld4(sP + (rg + 16 * i) * LDP + t) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int e = 0; e < H; ++e) {
          const float4 u = ld4(sT + (ch0 + e) * LDP + t);
#pragma unroll
          for (int i = 2 * m; i < 4; ++i) s[i * H + e] = dot4(q[i], u, s[i * H + e]);
        }
      }
      scatter_sum(s, part);
      const int t = rg + 16 * row;
      In* go = reinterpret_cast<In*>(p.o) + ((size_t)(tok0 + c * C + t) * p.HV + j) * D + slice * NV + ch;
      if (t < len - c * C) {
#pragma unroll
        for (int e = 0; e < E; ++e) go[e] = from_f32<In>(p.scale * (sY[t * (kNV + 1) + ch + e] + s[e]));
      }
    }
    __syncthreads();                                     // the new state is complete; KD, P, U~ and QG h are free
    if (tid == 0 && c + ST < nch) load3(c + ST);
  }
  if (gave_up) {
    report_status(p.status, HA_LA_ERR_TIMEOUT);
    settle_copies();
  }
  if (p.hT && upd) {
#pragma unroll
    for (int e = 0; e < E; ++e) p.hT[hbase + e] = h[e];
  }
}

template <typename In, bool KDA>
cudaError_t run(const Problem& p, const Fp32Params& fp, cudaStream_t stream) {
  static_assert(PrepSmem<KDA>::size * 4 <= 227 * 1024 && WalkSmem::bytes <= 227 * 1024, "shared memory budget");
  if (p.max_chunks * p.HV > 0) {
    timer_mark(stream, "simt_prep");
    const cudaError_t e = launch_fp32_kernel<fp32_prep_kernel<In, KDA>>((unsigned)(p.max_chunks * p.HV), 256u, PrepSmem<KDA>::size * 4,
                                                               stream, fp);
    if (e != cudaSuccess) return e;
  }
  timer_mark(stream, "simt_prefill");
  // The narrowest slices that leave every CTA an SM: a chunk takes less with fewer channels; else 16
  // (fewer reads of the shared operands per channel).
  const long long heads = (long long)p.N * p.HV;
  if (heads * (D / 4) <= sm_count())
    return launch_fp32_kernel<fp32_walk_kernel<In, 4>>((unsigned)(heads * (D / 4)), (unsigned)kWalkThreads, WalkSmem::bytes, stream, fp);
  if (heads * (D / 8) <= sm_count())
    return launch_fp32_kernel<fp32_walk_kernel<In, 8>>((unsigned)(heads * (D / 8)), (unsigned)kWalkThreads, WalkSmem::bytes, stream, fp);
  return launch_fp32_kernel<fp32_walk_kernel<In, 16>>((unsigned)(heads * (D / 16)), (unsigned)kWalkThreads, WalkSmem::bytes, stream, fp);
}

template <typename In, bool KDA>
cudaError_t run_dims(const Problem& p, const Fp32Params& fp, cudaStream_t stream) {
  return p.dk == 128 ? run<In, KDA>(p, fp, stream) : launch_fp32_d64(p, fp, stream);
}

Fp32Params make_params(const Problem& p, const ha_la_prefill_args& a, PlanView plan, void* ws) {
  Fp32Params fp;
  fp.q = a.q; fp.k = a.k; fp.v = a.v; fp.g = a.g; fp.beta = a.beta; fp.h0 = a.h0;
  fp.o = a.o; fp.hT = a.hT; fp.rec = reinterpret_cast<float*>(ws);
  fp.chunk_tok0 = plan.chunk_tok0; fp.chunk_len = plan.chunk_len;
  fp.seq_tok0 = plan.seq_tok0; fp.seq_len = plan.seq_len; fp.seq_chunk0 = plan.seq_chunk0;
  fp.seq_order = plan.seq_tok0 ? plan.seq_order : nullptr;
  fp.T_row = p.T_row; fp.cps = p.max_seq_chunks > 0 ? p.max_seq_chunks : 1;
  fp.HK = p.HK; fp.HV = p.HV; fp.scale = p.scale; fp.status = a.status_word;
  return fp;
}

}  // namespace

// The instantiations are spread over translation units (HA_LA_FP32_UNIT = 0..3, one per dtype x variant) so that they
// compile in parallel; unit 4 holds the dispatcher.
#ifndef HA_LA_FP32_UNIT
#error "compile with -DHA_LA_FP32_UNIT=0..4"
#endif

#define HA_LA_FP32_DEFINE(NAME, IN, KDA)                                                                         \
  cudaError_t NAME(const Problem& p, const ha_la_prefill_args& a, PlanView plan, void* ws, cudaStream_t stream) { \
    return run_dims<IN, KDA>(p, make_params(p, a, plan, ws), stream);                                             \
  }

#if HA_LA_FP32_UNIT == 0
HA_LA_FP32_DEFINE(fp32_bf16_gdn, __nv_bfloat16, false)
#elif HA_LA_FP32_UNIT == 1
HA_LA_FP32_DEFINE(fp32_bf16_kda, __nv_bfloat16, true)
#elif HA_LA_FP32_UNIT == 2
HA_LA_FP32_DEFINE(fp32_f32_gdn, float, false)
#elif HA_LA_FP32_UNIT == 3
HA_LA_FP32_DEFINE(fp32_f32_kda, float, true)
#else
cudaError_t fp32_bf16_gdn(const Problem&, const ha_la_prefill_args&, PlanView, void*, cudaStream_t);
cudaError_t fp32_bf16_kda(const Problem&, const ha_la_prefill_args&, PlanView, void*, cudaStream_t);
cudaError_t fp32_f32_gdn(const Problem&, const ha_la_prefill_args&, PlanView, void*, cudaStream_t);
cudaError_t fp32_f32_kda(const Problem&, const ha_la_prefill_args&, PlanView, void*, cudaStream_t);

size_t fp32_workspace_bytes(const Problem& p) {
  return align_up((size_t)p.max_chunks * p.HV * (p.dk == 128 ? Rec::size * sizeof(float) : fp32_d64_record_bytes()), 1024);
}

cudaError_t launch_fp32(const Problem& p, const ha_la_prefill_args& a, PlanView plan, void* ws, cudaStream_t stream) {
  if (p.N * p.HV == 0) return cudaSuccess;
  const bool kda = p.variant == HA_LA_KDA;
  if (p.dtype == HA_LA_BF16) return kda ? fp32_bf16_kda(p, a, plan, ws, stream) : fp32_bf16_gdn(p, a, plan, ws, stream);
  return kda ? fp32_f32_kda(p, a, plan, ws, stream) : fp32_f32_gdn(p, a, plan, ws, stream);
}
#endif

}  // namespace ha_la
