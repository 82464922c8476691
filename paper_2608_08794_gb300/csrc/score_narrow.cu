// score_narrow.cu -- relevance scores of Eq. inner_score (Sec. 3.2) when each KV head group
// has few query rows: the paper's own setting scores with the last query token only
// (Table S-hparams), i.e. G = Hq/Hkv rows per group (7 for the 7B model).
//
// With so few rows the step is bound by reading K once, so the logits are computed once and
// kept:
//   logits kernel:  the dot product of every (logit row, key), stored per logit row with a row
//                   stride padded to 64 keys, and per CTA the (max, sum of exp2) of every logit row
//                   over its multimodal keys, in log2 units.  Two variants:
//                   * Hkv = 1, 2, 4 or 8: the tcgen05 kernel of score_narrow_tc.cu (keys as M = 128,
//                     the group's rows as N = 16 or 32);
//                   * other head counts: one thread per key reads its whole token row and dots it
//                     with the group's query rows held in shared memory;
//   final kernel:   the row normalisers lse2 from the CTA partials, then one thread per key sums
//                   exp2(x log2(e)/sqrt(D) - lse2) over all logit rows in a fixed order and scales
//                   by 1/(Hq n_q).  Above 32 rows or with many partials (kMergeInside) a merge kernel
//                   computes lse2 first.
// The logits of the 10-minute 7B sequence with one query row take 15 MB and stay
// in L2 between the first and the last kernel.
#include <algorithm>
#include <cmath>
#include <type_traits>

#include "internal.cuh"
#include "narrow_plan.cuh"
#include "ptx.cuh"

namespace apack {

namespace {

constexpr int kThreads = 256;          // keys per CTA (general logits kernel)
constexpr int kWarps = kThreads / 32;
constexpr int kFinalThreads = 512;     // threads per CTA (final kernel)
constexpr int kPartTokens = 64;        // a sequence has at most one partial per this many keys (sizes the workspace)
// Rows of a sequence, and rows times its partials, up to which every CTA of the final kernel merges the
// partials by itself instead of a kernel of its own before it: one round of its warps.  Inside / a kernel of
// its own, 28/4 heads: 28 rows of 8,400 keys 9.4 / 9.9 us, 16 sequences of 8,400 33.4 / 35.2; 56 rows of
// 4,000 keys 11.2 / 10.6, 67,500 27.7 / 25.0; 84 rows of 67,500 36.1 / 31.8; but 56 rows of 40 sequences of
// 600 keys 18.9 / 20.7.
constexpr int kMergeRows = 32;
constexpr int kMergeInside = 16384;
// Keys read as the first to leave the 129 MB L2, for the logits to stay in it until the final kernel: where
// the keys are more than the first figure (below it they may stay for what reads them next) and the
// logits less than the second. 28/4 heads, normal -> first to leave: keys 98 MB 29.1 -> 27.9 us, 132 MB
// 36.7 -> 34.7 us and with four query rows 64.4 -> 56.4 us, 488 MB 120.5 -> 114.5 us; 16 sequences, 262 MB
// and 60 MB of logits 104.2 -> 96.5 us; but 66 MB 19.7 -> 19.5 us, and 293 MB beside 134 MB of logits
// 127.8 -> 129.9 us.
constexpr int64_t kStreamKeyBytes = 96 << 20;
constexpr int64_t kStreamLogitBytes = 100 << 20;
constexpr int kLogitPad = 64;          // logit row stride: the key count rounded up to this

__device__ __forceinline__ bool is_mm(uint8_t m) { return m == APACK_MOD_AUDIO || m == APACK_MOD_VISUAL; }

__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

__device__ __forceinline__ void bf16x8_to_f32(const uint4 &v, float (&f)[8]) {
  const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    f[2 * i] = __uint_as_float(w[i] << 16);
    f[2 * i + 1] = __uint_as_float(w[i] & 0xFFFF0000u);
  }
}

// RG = compile-time upper bound of the rows of one KV head group (G * n_q <= RG).
template <int RG>
__global__ void __launch_bounds__(kThreads)
    score_narrow_logits_kernel(const __grid_constant__ NarrowPlan plan, const uint16_t *__restrict__ q,
                               const uint8_t *__restrict__ k, int64_t k_stride, const uint8_t *__restrict__ modality,
                               float *__restrict__ logits, float2 *__restrict__ part) {
  pdl_wait_and_release();
  extern __shared__ __align__(16) float smem_f[];
  const int s = find_unit_seq(plan, blockIdx.x);
  const NSeq &sq = plan.seq[s];
  const int R = sq.rows;
  float *qs = smem_f;                                                  // [R][128]
  float2 *wpart = reinterpret_cast<float2 *>(smem_f + R * 128);       // [kWarps][R]
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int kt = blockIdx.x - sq.unit_begin;
  const int key = sq.t0 + kt * kThreads + tid;
  const bool in = key < sq.t0 + sq.len;
  const bool mm = in && is_mm(modality[key]);
  // query rows of the sequence: logit row rho = token * Hq + head (the order of Q in memory)
  for (int i = tid; i < R * 128; i += kThreads)
    qs[i] = __uint_as_float(static_cast<uint32_t>(q[static_cast<int64_t>(sq.q_off) * plan.hq * 128 + i]) << 16);
  __syncthreads();
  const int G = plan.group, rg = G * sq.n_q;
  const uint8_t *krow = k + static_cast<int64_t>(in ? key : sq.t0) * k_stride;
  const int64_t lbase = sq.logit_base + (key - sq.t0);
  for (int g = 0; g < plan.hkv; ++g) {
    float acc[RG];
    int qoff[RG];                      // logit row rho = token * Hq + g * G + j, as an offset into qs
#pragma unroll
    for (int l = 0; l < RG; ++l) {
      acc[l] = 0.f;
      qoff[l] = l < rg ? ((l / G) * plan.hq + g * G + (l % G)) * 128 : 0;
    }
    const uint4 *kg = reinterpret_cast<const uint4 *>(krow + g * 256);
#pragma unroll 4
    for (int c = 0; c < 16; ++c) {
      float kf[8];
      bf16x8_to_f32(in ? __ldg(kg + c) : make_uint4(0, 0, 0, 0), kf);
#pragma unroll
      for (int l = 0; l < RG; ++l) {
        if (l < rg) {
          const float4 qa = *reinterpret_cast<const float4 *>(qs + qoff[l] + c * 8);
          const float4 qb = *reinterpret_cast<const float4 *>(qs + qoff[l] + c * 8 + 4);
          acc[l] = fmaf(kf[0], qa.x, acc[l]);
          acc[l] = fmaf(kf[1], qa.y, acc[l]);
          acc[l] = fmaf(kf[2], qa.z, acc[l]);
          acc[l] = fmaf(kf[3], qa.w, acc[l]);
          acc[l] = fmaf(kf[4], qb.x, acc[l]);
          acc[l] = fmaf(kf[5], qb.y, acc[l]);
          acc[l] = fmaf(kf[6], qb.z, acc[l]);
          acc[l] = fmaf(kf[7], qb.w, acc[l]);
        }
      }
    }
#pragma unroll
    for (int l = 0; l < RG; ++l) {
      if (l < rg) {
        const int rho = qoff[l] / 128;
        const float y = acc[l] * plan.scale2;
        if (in) logits[lbase + static_cast<int64_t>(rho) * sq.lstride] = acc[l];
        // this warp's (max, sum of exp2) of the row over the keys in its denominator: the
        // multimodal keys, or (causal rows) every key up to the row's own position
        const bool use = plan.causal ? (in && key - sq.t0 <= sq.q_pos + l / G) : mm;
        const float wm = warp_max(use ? y : -INFINITY);
        const float ws = warp_sum(use && wm != -INFINITY ? ex2_approx(y - wm) : 0.f);
        if (lane == 0) wpart[warp * R + rho] = make_float2(wm, ws);
      }
    }
  }
  __syncthreads();
  for (int rho = tid; rho < R; rho += kThreads) {
    float m = -INFINITY;
    for (int w = 0; w < kWarps; ++w) m = fmaxf(m, wpart[w * R + rho].x);
    float sum = 0.f;
    if (m != -INFINITY)
      for (int w = 0; w < kWarps; ++w) {
        const float2 v = wpart[w * R + rho];
        if (v.x != -INFINITY) sum += v.y * ex2_approx(v.x - m);
      }
    part[sq.part_base + static_cast<int64_t>(rho) * sq.nparts + kt] = make_float2(m, sum);
  }
}

// One block per (sequence, logit row): lse2 over the CTA partials.  Each thread
// folds a fixed stride of partials, then a fixed-shape tree combines the
// threads: the order never depends on timing, so lse2 is deterministic.
__global__ void __launch_bounds__(kThreads)
    score_narrow_merge_kernel(const __grid_constant__ NarrowPlan plan, const float2 *__restrict__ part,
                              float *__restrict__ lse2) {
  pdl_wait_and_release();
  __shared__ float red[kWarps];
  __shared__ float mshared;
  const int64_t e = blockIdx.x;
  int s = 0;
  int64_t acc = 0;
  while (s + 1 < plan.nseq && acc + plan.seq[s].rows <= e) acc += plan.seq[s++].rows;
  const NSeq &sq = plan.seq[s];
  const int rho = static_cast<int>(e - acc);
  const int ctas = sq.nparts;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  // up to kHold partials per thread are loaded once, together, and kept for the sum
  constexpr int kHold = 8;
  const bool held = ctas <= kHold * kThreads;
  float2 v[kHold];
  float m = -INFINITY;
  if (held) {
#pragma unroll
    for (int i = 0; i < kHold; ++i) {
      const int c = tid + i * kThreads;
      v[i] = c < ctas ? part[sq.part_base + static_cast<int64_t>(rho) * sq.nparts + c] : make_float2(-INFINITY, 0.f);
      m = fmaxf(m, v[i].x);
    }
  } else {
    for (int c = tid; c < ctas; c += kThreads) m = fmaxf(m, part[sq.part_base + static_cast<int64_t>(rho) * sq.nparts + c].x);
  }
  m = warp_max(m);
  if (lane == 0) red[warp] = m;
  __syncthreads();
  if (tid == 0) {
    float mm = -INFINITY;
    for (int w = 0; w < kWarps; ++w) mm = fmaxf(mm, red[w]);
    mshared = mm;
  }
  __syncthreads();
  m = mshared;
  float sum = 0.f;
  if (m != -INFINITY) {
    if (held) {
#pragma unroll
      for (int i = 0; i < kHold; ++i)   // the same partials in the same order as the loop below
        if (v[i].x != -INFINITY) sum += v[i].y * exp2f(v[i].x - m);
    } else {
      for (int c = tid; c < ctas; c += kThreads) {
        const float2 w = part[sq.part_base + static_cast<int64_t>(rho) * sq.nparts + c];
        if (w.x != -INFINITY) sum += w.y * exp2f(w.x - m);
      }
    }
  }
  sum = warp_sum(sum);
  __syncthreads();
  if (lane == 0) red[warp] = sum;
  __syncthreads();
  if (tid == 0) {
    float tot = 0.f;
    for (int w = 0; w < kWarps; ++w) tot += red[w];
    // no multimodal key: nothing is scored in this sequence
    lse2[sq.lse_base + rho] = m == -INFINITY ? INFINITY : m + log2f(tot);
  }
}

// One warp merges a row's partials p[0..n): the first 32 kHold in registers, so that their loads can be
// issued before the work of another row.  Returns lse2; +inf where no key is in the denominator.
constexpr int kHold = 5;

__device__ __forceinline__ void load_parts(const float2 *p, int n, int lane, float2 (&v)[kHold]) {
#pragma unroll
  for (int i = 0; i < kHold; ++i) v[i] = lane + 32 * i < n ? p[lane + 32 * i] : make_float2(-INFINITY, 0.f);
}

__device__ __forceinline__ float merge_parts(const float2 *p, int n, int lane, const float2 (&v)[kHold]) {
  float m = v[0].x, sum = 0.f;
#pragma unroll
  for (int i = 1; i < kHold; ++i) m = fmaxf(m, v[i].x);
  for (int c = lane + 32 * kHold; c < n; c += 32) m = fmaxf(m, p[c].x);
  m = warp_max(m);
  if (m != -INFINITY) {
#pragma unroll
    for (int i = 0; i < kHold; ++i) sum += v[i].y * exp2f(v[i].x - m);
    for (int c = lane + 32 * kHold; c < n; c += 32) sum += p[c].y * exp2f(p[c].x - m);
  }
  sum = warp_sum(sum);
  return m == -INFINITY ? INFINITY : m + log2f(sum);
}

// The merge with one warp per logit row, where no row has more than 32 kHold partials.  84 rows of each of
// 40 sequences of 600 keys: 24.5 us for the whole call where a CTA per row took 34.5.
__global__ void __launch_bounds__(kThreads)
    score_narrow_merge_rows_kernel(const __grid_constant__ NarrowPlan plan, const float2 *__restrict__ part,
                                   float *__restrict__ lse2, int rows_all) {
  pdl_wait_and_release();
  const int lane = threadIdx.x & 31, e = blockIdx.x * kWarps + (threadIdx.x >> 5);
  if (e >= rows_all) return;
  int s = 0, acc = 0;
  while (s + 1 < plan.nseq && acc + plan.seq[s].rows <= e) acc += plan.seq[s++].rows;
  const NSeq &sq = plan.seq[s];
  const int rho = e - acc;
  const float2 *p = part + sq.part_base + static_cast<int64_t>(rho) * sq.nparts;
  float2 v[kHold];
  load_parts(p, sq.nparts, lane, v);
  const float r = merge_parts(p, sq.nparts, lane, v);
  if (lane == 0) lse2[sq.lse_base + rho] = r;
}

// One thread per key: I = sum over logit rows of exp2(x c2 - lse2) / (Hq n_q), x the stored dot
// product.  MERGE (at most 32 rows): the CTA's warps first merge the sequence's partials into lse2
// while the keys' own logits are in flight (a fixed order).  SPLIT threads share a key's rows, so that
// a thread's loads stay a few rounds.  OCC: CTAs per SM; one where the grid is no more than that, with
// the registers for all loads at once, else two within 64 registers.
// Latency-bound (two or three L2 round trips and the launch).  The whole call with one CTA per SM / two:
// 84 rows of 8,400 keys 11.4 / 12.0 us, 84 rows of 67,500 (264 CTAs) 29.8 / 29.3, 112 rows of 16 x 16,800
// 108 / 101; 28 rows of 67,500 keys (132 CTAs) 18.9 / 20.1, of 135,041 35.7 / 34.7.
template <bool MERGE, int SPLIT, int OCC>
__global__ void __launch_bounds__(kFinalThreads, OCC)
    score_narrow_final_kernel(const __grid_constant__ NarrowPlan plan, const uint8_t *__restrict__ modality,
                              const float *__restrict__ logits, const float2 *__restrict__ part,
                              const float *__restrict__ lse2, float *__restrict__ scores) {
  pdl_wait_and_release();
  extern __shared__ __align__(16) float ls[];            // -lse2 per logit row
  const int s = find_final_seq(plan, blockIdx.x);
  const NSeq &sq = plan.seq[s];
  const int R = sq.rows;
  const int kt = blockIdx.x - sq.final_begin;
  constexpr int kKeys = kFinalThreads / SPLIT;           // keys per CTA
  const int kl = threadIdx.x % kKeys;
  const int key = sq.t0 + kt * kKeys + kl;
  const bool in = key < sq.t0 + sq.len;
  const float *lp = logits + sq.logit_base + (key - sq.t0);
  // this thread's rows [ra, rb); the key's own loads (modality, and the first 32 rows' logits) are
  // issued before the normalisers arrive: one round trip for all of them
  const int share = threadIdx.x / kKeys, per = (R + SPLIT - 1) / SPLIT;
  const int ra = SPLIT == 1 ? 0 : min(R, share * per), rb = SPLIT == 1 ? R : min(R, ra + per);
  const uint8_t mod = in ? modality[key] : static_cast<uint8_t>(0);
  float raw[32];
#pragma unroll
  for (int u = 0; u < 32; ++u) raw[u] = (in && ra + u < rb) ? lp[static_cast<int64_t>(ra + u) * sq.lstride] : 0.f;
  if (MERGE) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    constexpr int kAtOnce = OCC == 1 ? 2 : 1;            // rows of a warp whose loads are issued together
#pragma unroll 1
    for (int r0 = warp; r0 < R; r0 += kAtOnce * (kFinalThreads / 32)) {
      float2 v[kAtOnce][kHold];
      const float2 *p[kAtOnce];
#pragma unroll
      for (int k = 0; k < kAtOnce; ++k) {
        const int rho = r0 + k * (kFinalThreads / 32);
        p[k] = part + sq.part_base + static_cast<int64_t>(rho) * sq.nparts;
        load_parts(p[k], rho < R ? sq.nparts : 0, lane, v[k]);
      }
#pragma unroll
      for (int k = 0; k < kAtOnce; ++k) {
        const int rho = r0 + k * (kFinalThreads / 32);
        if (rho >= R) break;                             // uniform over the warp
        const float r = merge_parts(p[k], sq.nparts, lane, v[k]);
        if (lane == 0) ls[rho] = -r;
      }
    }
  } else {
    for (int i = threadIdx.x; i < R; i += kFinalThreads) ls[i] = -lse2[sq.lse_base + i];
  }
  __syncthreads();
  float out = 0.f;
  const bool scored = in && sq.n_q > 0 && is_mm(mod);
  if (scored) {
    const float c2 = plan.scale2;
    // eight independent sums, the loads of a block of 16 rows issued together
    float a[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    // causal rows: logit row rho = token * Hq + head sees this key when token >= key - q_pos
    const int rho_min = plan.causal ? max(0, key - sq.t0 - sq.q_pos) * plan.hq : 0;
#pragma unroll
    for (int u = 0; u < 32; ++u)
      if (ra + u < rb && ra + u >= rho_min) a[u & 7] += ex2_approx(fmaf(raw[u], c2, ls[ra + u]));
    for (int r0 = ra + 32; r0 < rb; r0 += 16) {
      float x[16];
#pragma unroll
      for (int u = 0; u < 16; ++u) x[u] = r0 + u < rb ? lp[static_cast<int64_t>(r0 + u) * sq.lstride] : 0.f;
#pragma unroll
      for (int u = 0; u < 16; ++u)
        if (r0 + u < rb && r0 + u >= rho_min) a[u & 7] += ex2_approx(fmaf(x[u], c2, ls[r0 + u]));
    }
    out = ((a[0] + a[1]) + (a[2] + a[3])) + ((a[4] + a[5]) + (a[6] + a[7]));
  }
  if (SPLIT > 1) {                                       // the shares of a key meet in share order
    __shared__ float sums[SPLIT > 1 ? kFinalThreads : 1];
    sums[threadIdx.x] = out;
    __syncthreads();
    if (share > 0) return;
#pragma unroll
    for (int i = 1; i < SPLIT; ++i) out += sums[i * kKeys + kl];
  }
  if (in) scores[key] = scored ? out / static_cast<float>(plan.hq * sq.n_q) : 0.f;
}

template <int RG>
cudaError_t launch_logits(int grid, size_t smem, cudaStream_t stream, const NarrowPlan &P, const uint16_t *q,
                          const uint8_t *k, int64_t k_stride, const uint8_t *modality, float *logits, float2 *part) {
  static std::atomic<uint64_t> attr{0};
  const cudaError_t e = once_per_device(attr, [] {
    return cudaFuncSetAttribute(score_narrow_logits_kernel<RG>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                160 * 1024);
  });
  if (e != cudaSuccess) return e;
  // Not a programmatic dependent: up to six of its CTAs fit an SM, and those that start while the previous
  // launch drains pile up on the SMs it leaves first (8 sequences of 5,000 keys, 16/16 heads, four query
  // rows, 160 CTAs: 474 us a call among others as a dependent, 214 us so).
  score_narrow_logits_kernel<RG><<<grid, kThreads, smem, stream>>>(P, q, k, k_stride, modality, logits, part);
  return cudaGetLastError();
}

}  // namespace

bool narrow_score_applies(const apack_seqs *s) {
  const int G = s->num_q_heads / s->num_kv_heads;
  for (int b = 0; b < s->num_seqs; ++b) {
    const int nq = s->cu_qlens_h[b + 1] - s->cu_qlens_h[b];
    if (G * nq > kNarrowGroupRows || s->num_q_heads * nq > kNarrowRows) return false;
  }
  return true;
}

void narrow_layout(const apack_seqs *s, size_t *logit_floats, size_t *part_float2s, size_t *lse_floats) {
  size_t lf = 0, pf = 0, ef = 0;
  for (int b = 0; b < s->num_seqs; ++b) {
    const int64_t len = s->cu_seqlens_h[b + 1] - s->cu_seqlens_h[b];
    const int64_t R = static_cast<int64_t>(s->num_q_heads) * (s->cu_qlens_h[b + 1] - s->cu_qlens_h[b]);
    lf += static_cast<size_t>(R * ((len + kLogitPad - 1) / kLogitPad * kLogitPad));
    pf += static_cast<size_t>(R * ((len + kPartTokens - 1) / kPartTokens));   // enough for either kernel
    ef += static_cast<size_t>(R);
  }
  *logit_floats = lf;
  *part_float2s = pf;
  *lse_floats = ef;
}

apack_status run_score_narrow(const apack_seqs *seqs, const void *q, const void *k, int64_t k_token_stride,
                              float *scores, void *ws, cudaStream_t stream) {
  const WsLayout L = workspace_layout(seqs);
  uint8_t *wsb = static_cast<uint8_t *>(ws);
  float *logits = reinterpret_cast<float *>(wsb + L.nlog_off);
  float2 *part = reinterpret_cast<float2 *>(wsb + L.npart_off);
  float *lse2 = reinterpret_cast<float *>(wsb + L.nlse_off);
  const int B = seqs->num_seqs;
  const int hq = seqs->num_q_heads, hkv = seqs->num_kv_heads, G = hq / hkv;
  int64_t logit_base = 0, part_base = 0, lse_base = 0;
  for (int s0 = 0; s0 < B; s0 += kSeqsPerLaunch) {
    const int ns = (B - s0 < kSeqsPerLaunch) ? (B - s0) : kSeqsPerLaunch;
    NarrowPlan P{};
    P.nseq = ns;
    P.hq = hq;
    P.hkv = hkv;
    P.group = G;
    P.causal = seqs->softmax_domain == APACK_SOFTMAX_CAUSAL_ROW;
    int max_rg = 0;
    for (int i = 0; i < ns; ++i) {
      const int nq = seqs->cu_qlens_h[s0 + i + 1] - seqs->cu_qlens_h[s0 + i];
      max_rg = G * nq > max_rg ? G * nq : max_rg;
    }
    const bool tc = hkv == 1 || hkv == 2 || hkv == 4 || hkv == 8;
    P.scale2 = tc ? kScale2Tc : kScale2;
    // its work: the (tile, KV head) stages of the sequences with query rows, `chunk` of them per CTA,
    // the smallest chunk (within 3 %) that keeps the launch to one CTA per SM
    auto stages_of = [&](int b) -> int64_t {
      const int64_t len = seqs->cu_seqlens_h[b + 1] - seqs->cu_seqlens_h[b];
      return seqs->cu_qlens_h[b + 1] > seqs->cu_qlens_h[b] ? (len + 127) / 128 * hkv : 0;
    };
    auto ctas_of = [&](int b, int64_t chunk) -> int64_t {
      const int64_t len = seqs->cu_seqlens_h[b + 1] - seqs->cu_seqlens_h[b];
      return std::min<int64_t>((stages_of(b) + chunk - 1) / chunk, (len + kPartTokens - 1) / kPartTokens);
    };
    const int64_t sms = device_sm_count();
    int64_t all_stages = 0, max_stages = 1, logit_bytes = 0;
    for (int i = 0; i < ns; ++i) {
      const int64_t len = seqs->cu_seqlens_h[s0 + i + 1] - seqs->cu_seqlens_h[s0 + i];
      logit_bytes += len * hq * (seqs->cu_qlens_h[s0 + i + 1] - seqs->cu_qlens_h[s0 + i]) * 4;
      all_stages += stages_of(s0 + i);
      max_stages = std::max(max_stages, stages_of(s0 + i));
    }
    P.stream_keys = all_stages * (128 * 256) > kStreamKeyBytes && logit_bytes < kStreamLogitBytes;
    int64_t chunk = std::max<int64_t>(1, (all_stages + sms - 1) / sms);
    for (; chunk < max_stages; chunk += std::max<int64_t>(1, chunk / 32)) {
      int64_t ctas = 0;
      for (int i = 0; i < ns; ++i) ctas += ctas_of(s0 + i, chunk);
      if (ctas <= sms) break;
    }
    // The final kernel's threads per key: two above 32 rows and four above 128, so that a thread's loads stay
    // a few rounds.  While all its CTAs still run at once, four above 64 rows (84 rows of 8,400 keys 13.65 ->
    // 12.9 us); when there are more than two CTAs per SM the loads of other CTAs hide a thread's rounds, and
    // one does up to 128 rows (112 rows of 135,041 keys 55.4 -> 51.9 us, 16 sequences of 16,800 keys 120.8 ->
    // 108.3 us; at 264 CTAs, 67,500 keys, both 31.7 us).
    auto final_ctas = [&](int per_key) {
      int64_t n = 0;
      for (int i = 0; i < ns; ++i)
        n += (static_cast<int64_t>(seqs->cu_seqlens_h[s0 + i + 1] - seqs->cu_seqlens_h[s0 + i]) * per_key +
              kFinalThreads - 1) / kFinalThreads;
      return n;
    };
    const int seq_rows = hq * (max_rg / G);
    const int split = seq_rows <= 32                              ? 1
                      : seq_rows > 128                            ? 4
                      : seq_rows > 64 && final_ctas(4) <= sms     ? 4
                      : final_ctas(2) > 2 * sms                   ? 1
                                                                  : 2;
    const int final_keys = kFinalThreads / split;
    int units = 0, units8 = 0, finals = 0, max_rows = 0;
    int64_t rows_all = 0, max_parts = 0;
    int max_nparts = 0;
    for (int i = 0; i < ns; ++i) {
      const int b = s0 + i;
      NSeq &sq = P.seq[i];
      sq.t0 = seqs->cu_seqlens_h[b];
      sq.len = seqs->cu_seqlens_h[b + 1] - sq.t0;
      sq.q_off = seqs->cu_qlens_h[b];
      sq.n_q = seqs->cu_qlens_h[b + 1] - sq.q_off;
      sq.rows = hq * sq.n_q;
      sq.q_pos = query_position(seqs, b);
      sq.unit_begin = units;
      sq.unit8_begin = units8;
      sq.final_begin = finals;
      sq.lstride = (sq.len + kLogitPad - 1) / kLogitPad * kLogitPad;
      sq.logit_base = logit_base;
      sq.part_base = part_base;
      sq.lse_base = lse_base;
      sq.stages = static_cast<int32_t>(stages_of(b));
      const int ctas = (sq.len + kThreads - 1) / kThreads;
      int ctas8 = static_cast<int>(ctas_of(b, chunk));
      sq.chunk = ctas8 > 0 ? (sq.stages + ctas8 - 1) / ctas8 : 1;
      ctas8 = (sq.stages + sq.chunk - 1) / sq.chunk;        // no CTA without a stage
      sq.nparts = tc ? ctas8 : ctas;                        // at most one per kPartTokens keys: fits the workspace
      units += ctas;
      units8 += ctas8;
      finals += (sq.len + final_keys - 1) / final_keys;
      logit_base += static_cast<int64_t>(sq.rows) * sq.lstride;
      part_base += static_cast<int64_t>(sq.rows) * sq.nparts;
      lse_base += sq.rows;
      rows_all += sq.rows;
      max_rows = sq.rows > max_rows ? sq.rows : max_rows;
      max_nparts = std::max(max_nparts, sq.nparts);
      max_parts = std::max(max_parts, static_cast<int64_t>(sq.rows) * sq.nparts);
    }
    if (units == 0) continue;
    const uint16_t *q16 = static_cast<const uint16_t *>(q);
    const uint8_t *k8 = static_cast<const uint8_t *>(k);
    if (tc ? units8 > 0 : units > 0) {
      cudaError_t e;
      if (tc) {
        DeviceError *err = reinterpret_cast<DeviceError *>(wsb + L.err_off);
        CUtensorMap kmap;
        if (!make_kv_tile_map(&kmap, k, hkv, seqs->cu_seqlens_h[B], k_token_stride, 128)) return APACK_ECUDA;
        e = launch_narrow_tc(max_rg, units8, stream, kmap, P, q16, seqs->modality, logits, part, err);
      } else {
        const size_t smem = static_cast<size_t>(max_rows) * 128 * sizeof(float) +
                            static_cast<size_t>(kWarps) * max_rows * sizeof(float2);
        if (max_rg <= 8)
          e = launch_logits<8>(units, smem, stream, P, q16, k8, k_token_stride, seqs->modality, logits, part);
        else if (max_rg <= 16)
          e = launch_logits<16>(units, smem, stream, P, q16, k8, k_token_stride, seqs->modality, logits, part);
        else
          e = launch_logits<32>(units, smem, stream, P, q16, k8, k_token_stride, seqs->modality, logits, part);
      }
      count_launches(1);
      if (check_cuda(e) != APACK_OK) return APACK_ECUDA;
    }
    const bool inside = max_rows <= kMergeRows && max_parts <= kMergeInside;
    if (rows_all > 0 && !inside) {
      const cudaError_t e =
          max_nparts <= 32 * kHold
              ? launch_pdl(score_narrow_merge_rows_kernel, dim3(static_cast<unsigned>((rows_all + kWarps - 1) / kWarps)),
                           dim3(kThreads), 0, stream, P, part, lse2, static_cast<int>(rows_all))
              : launch_pdl(score_narrow_merge_kernel, dim3(static_cast<unsigned>(rows_all)), dim3(kThreads), 0,
                           stream, P, part, lse2);
      if (check_cuda(e) != APACK_OK) return APACK_ECUDA;
      count_launches(1);
    }
    auto pick = [&](auto occ) {
      constexpr int kOcc = decltype(occ)::value;
      return inside       ? score_narrow_final_kernel<true, 1, kOcc>
             : split == 1 ? score_narrow_final_kernel<false, 1, kOcc>
             : split == 2 ? score_narrow_final_kernel<false, 2, kOcc>
                          : score_narrow_final_kernel<false, 4, kOcc>;
    };
    auto *final_kernel = finals <= sms ? pick(std::integral_constant<int, 1>{}) : pick(std::integral_constant<int, 2>{});
    if (check_cuda(launch_pdl(final_kernel, dim3(finals), dim3(kFinalThreads), static_cast<size_t>(max_rows) * sizeof(float),
                              stream, P, seqs->modality, logits, part, lse2, scores)) != APACK_OK)
      return APACK_ECUDA;
    count_launches(1);
  }
  return APACK_OK;
}

}  // namespace apack
