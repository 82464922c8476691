// score_narrow_tc.cu -- logits of the narrow scoring path (few query rows per KV head group,
// e.g. the paper's last query token: Sec. 3.2, Eq. inner_score; Table S-hparams) on the
// tcgen05 tensor cores, for 1, 2, 4 or 8 KV heads and up to 32 query rows per KV head group.
//
// A stage is one KV head of one 128-key tile (32 KB of K).  The stages of a sequence are cut into
// equal contiguous ranges, one per CTA (about one CTA per SM over the launch); for each stage the
// MMA computes D[key][row] = K_h[key] . Q_h[row] with keys as M = 128 and the head group's query
// rows as N = 16 or 32 (zero rows pad them): bf16 operands in 128-byte-swizzled shared memory, fp32
// accumulators in TMEM.
//   warp 0, one lane:  TMA loads of the K stages, the first ones before the query rows are staged
//   warp 1, one lane:  TMEM allocation and the MMAs (8 per stage), commits to mbarriers
//   warps 2..:         epilogue, one warpgroup per KV head (8 heads: two per warpgroup), one key per
//                      thread: reads the stage's columns, stores the logits (row-major per logit
//                      row) and folds the warp's 32 keys into a running (max, sum of exp2) per row.
//                      The 32 keys meet by a reduce-scatter over the lanes: NR rows cost NR - 1
//                      shuffles and leave row r in lane r (NR = 32), so the running state of up to
//                      32 rows is one register pair per lane.
// At the end the CTA merges its warps' states per logit row in warp order and writes one
// (max, sum) partial per row for the final kernel.  Every wait is bounded.
//
// Bound by reading K once; what the CTA adds to that is its prologue and the last stage's
// epilogue.  A per-thread online state over up to 8 rows (two registers a row) carried only the
// shapes of at most 8 rows: the others ran on CUDA cores, one thread per key.
// Three query tokens (21 rows per group) over 67,541 keys: 127 us there, 20 us here.
#include <cmath>

#include "internal.cuh"
#include "narrow_plan.cuh"
#include "ptx.cuh"

namespace apack {
namespace {

constexpr int kTcM = 128;                          // keys per tile (MMA M)
constexpr int kTcHalf = kTcM * 128;                // 64 dims x 128 keys x 2 B = 16 KB
constexpr int kTcStageBytes = 2 * kTcHalf;         // 32 KB
constexpr int kTcMaxStages = 6;

// HKV KV heads, at most NR query rows per KV head group.
template <int HKV, int NR>
struct TcLayout {
  static constexpr int kN = NR < 16 ? 16 : NR;                           // MMA N
  static constexpr int kGroups = HKV < 4 ? HKV : 4;                      // epilogue warpgroups
  static constexpr int kHeads = HKV / kGroups;                           // KV heads per warpgroup
  static constexpr int kThreads = 64 + 128 * kGroups;                    // warp 0 TMA, warp 1 MMA, epilogue
  static constexpr int kQHalf = kN * 128;                                // 64 dims of the kN rows
  static constexpr int kQBytes = HKV * 2 * kQHalf;
  static constexpr int kStages = kTcMaxStages * kTcStageBytes + kQBytes <= 230000 ? kTcMaxStages : kTcMaxStages - 1;
  static constexpr uint32_t kOffQ = kStages * kTcStageBytes;             // 1024-aligned
  static constexpr uint32_t kOffRho = kOffQ + kQBytes;                   // int32 [NR]: logit row of row j, head 0
  static constexpr uint32_t kOffBars = kOffRho + NR * 4;
  static constexpr uint32_t kBytes = kOffBars + 512;
  static constexpr uint32_t kTmemCols = 2 * HKV * kN;                    // a power of two, 32 .. 512
  static constexpr uint32_t kIdesc = idesc_bf16_f32(kTcM, kN);
  static_assert(kBytes <= 232448, "shared memory budget");
};

struct __align__(8) TcBars {
  uint64_t k_full[kTcMaxStages], k_empty[kTcMaxStages], drain;
  uint64_t acc_full[8][2], acc_empty[8][2];          // per KV head and accumulator buffer
  uint32_t tmem_base;
  volatile int32_t abort;
};
static_assert(sizeof(TcBars) <= 512, "barrier block");

__device__ __forceinline__ bool tc_wait(uint64_t *bar, uint32_t parity, TcBars *bars, DeviceError *err, int where) {
  if (mbar_try_wait(bar, parity)) return true;
  const uint64_t t0 = globaltimer_ns();
  for (;;) {
    for (int i = 0; i < 32; ++i)
      if (mbar_try_wait(bar, parity)) return true;
    if (bars->abort) return false;
    if (globaltimer_ns() - t0 > kWaitLimitNs) {
      bars->abort = 1;
      raise_device_error(err, APACK_ETIMEOUT, where);
      return false;
    }
  }
}

__device__ __forceinline__ bool is_mm_tc(uint8_t m) { return m == APACK_MOD_AUDIO || m == APACK_MOD_VISUAL; }

__device__ __forceinline__ void load_rows(uint32_t taddr, uint32_t (&r)[8]) { tmem_ld8_wait(taddr, r); }
__device__ __forceinline__ void load_rows(uint32_t taddr, uint32_t (&r)[16]) { tmem_ld16_wait(taddr, r); }
__device__ __forceinline__ void load_rows(uint32_t taddr, uint32_t (&r)[32]) {
  tmem_ld32(taddr, r);
  tmem_wait32(r);
}

// Combines v[j] of the 32 lanes for every j < NR with op: lane l ends with row l / (32 / NR).
// At each level the lanes of a pair exchange the halves that the other one keeps.
template <int NR, class Op>
__device__ __forceinline__ float reduce_scatter(float (&v)[NR], int lane, Op op) {
  int mask = 16;
#pragma unroll
  for (int half = NR / 2; half >= 1; half /= 2, mask /= 2) {
    const bool up = lane & mask;
#pragma unroll
    for (int e = 0; e < half; ++e) {
      const float keep = up ? v[e + half] : v[e];
      const float send = up ? v[e] : v[e + half];
      v[e] = op(keep, __shfl_xor_sync(0xffffffffu, send, mask));
    }
  }
#pragma unroll
  for (; mask >= 1; mask /= 2) v[0] = op(v[0], __shfl_xor_sync(0xffffffffu, v[0], mask));
  return v[0];
}

template <int HKV, int NR>
__global__ void __launch_bounds__(TcLayout<HKV, NR>::kThreads, 1)
    score_narrow_tc_kernel(const __grid_constant__ CUtensorMap kmap, const __grid_constant__ NarrowPlan plan,
                           const uint16_t *__restrict__ q, const uint8_t *__restrict__ modality,
                           float *__restrict__ logits, float2 *__restrict__ part, DeviceError *err) {
  using Lay = TcLayout<HKV, NR>;
  constexpr int kN = Lay::kN, kStages = Lay::kStages;
  extern __shared__ __align__(1024) uint8_t smem[];
  if ((smem_u32(smem) & 1023u) != 0) {
    if (threadIdx.x == 0) raise_device_error(err, APACK_EDEVICE, 80);
    return;
  }
  uint8_t *ring = smem;
  uint8_t *qs = smem + Lay::kOffQ;
  int32_t *rho_of = reinterpret_cast<int32_t *>(smem + Lay::kOffRho);
  TcBars *bars = reinterpret_cast<TcBars *>(smem + Lay::kOffBars);
  const int s = find_unit8_seq(plan, blockIdx.x);
  const NSeq &sq = plan.seq[s];
  const int G = plan.group;
  const int rg = G * sq.n_q;                           // rows per head group, 1 .. NR (sequences without have no CTA)
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int c = blockIdx.x - sq.unit8_begin;           // this CTA's range of the sequence's stages
  const int u0 = c * sq.chunk;
  const int nstage = min(sq.stages - u0, sq.chunk);

  if (threadIdx.x == 0) {
    for (int i = 0; i < kStages; ++i) {
      mbar_init(&bars->k_full[i], 1);
      mbar_init(&bars->k_empty[i], 1);
    }
    for (int h = 0; h < HKV; ++h)
      for (int i = 0; i < 2; ++i) {
        mbar_init(&bars->acc_full[h][i], 1);
        mbar_init(&bars->acc_empty[h][i], 4);
      }
    mbar_init(&bars->drain, 1);
    bars->abort = 0;
    fence_mbar_init();
    tma_prefetch_desc(&kmap);
  }
  if (warp == 1) {
    tmem_alloc(&bars->tmem_base, Lay::kTmemCols);
    tc_fence_before();
  }
  pdl_wait_and_release();   // the set-up above runs beside the previous launch; q and K are read below
  // many keys are read as the first to leave L2, so that the logits stay for the final kernel
  const uint64_t policy = plan.stream_keys ? l2_evict_first() : l2_evict_normal();
  // stage n of this CTA: unit u0 + n = tile * HKV + head
  auto issue_load = [&](int n) {
    const int slot = n % kStages, t = (u0 + n) / HKV, h = (u0 + n) % HKV;
    uint8_t *dst = ring + slot * kTcStageBytes;
    const int key0 = sq.t0 + t * kTcM;
    mbar_arrive_expect_tx(&bars->k_full[slot], kTcStageBytes);
    tma_load_3d_hint(dst, &kmap, &bars->k_full[slot], 0, h, key0, policy);
    tma_load_3d_hint(dst + kTcHalf, &kmap, &bars->k_full[slot], 64, h, key0, policy);
  };
  const int first = min(nstage, kStages);
  if (threadIdx.x == 0)
    for (int n = 0; n < first; ++n) issue_load(n);
  // query tiles in the 128-byte-swizzled K-major layout: row r, 16-byte chunk cc of a 64-dim
  // half sits at chunk cc ^ (r & 7) of the row's 128 bytes (every ring stage the MMAs read is
  // written whole by its TMA load, rows past the cache as zeros)
  for (int idx = threadIdx.x; idx < HKV * kN * 16; idx += Lay::kThreads) {
    const int h = idx / (kN * 16), rem = idx % (kN * 16);
    const int row = rem / 16, ch = rem % 16;
    const int half = ch >> 3, cc = ch & 7;
    uint4 v = make_uint4(0, 0, 0, 0);
    if (row < rg) {
      const int rho = (row / G) * plan.hq + h * G + row % G;
      v = __ldg(reinterpret_cast<const uint4 *>(q + (static_cast<int64_t>(sq.q_off) * plan.hq + rho) * 128) + ch);
    }
    *reinterpret_cast<uint4 *>(qs + h * 2 * Lay::kQHalf + half * Lay::kQHalf + (row >> 3) * 1024 + (row & 7) * 128 +
                               ((cc ^ (row & 7)) << 4)) = v;
  }
  for (int j = threadIdx.x; j < NR; j += Lay::kThreads) rho_of[j] = (j / G) * plan.hq + j % G;
  fence_proxy_async_smem();   // generic-proxy writes of the query tiles -> visible to the MMA
  __syncthreads();
  tc_fence_after();

  // epilogue warps: running (max, sum of exp2) of the row this lane owns, per KV head
  float m_run[Lay::kHeads], l_run[Lay::kHeads];
#pragma unroll
  for (int i = 0; i < Lay::kHeads; ++i) {
    m_run[i] = -INFINITY;
    l_run[i] = 0.f;
  }

  if (warp == 0) {
    // ------------------------------------------------------------ TMA producer
    if (lane == 0) {
      int n = first;
      for (; n < nstage; ++n) {
        if (!tc_wait(&bars->k_empty[n % kStages], ((n / kStages) - 1) & 1u, bars, err, 81)) break;
        issue_load(n);
      }
      if (bars->abort)   // loads issued but not consumed: let the last of every slot land before the CTA exits
        for (int i = n > kStages ? n - kStages : 0; i < n; ++i)
          mbar_wait(&bars->k_full[i % kStages], (i / kStages) & 1u, kWaitLimitNs / 4);
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issuer
    if (lane == 0) {
      const uint32_t tmem = bars->tmem_base;
      const uint32_t q_base = smem_u32(qs);
      for (int n = 0; n < nstage; ++n) {
        const int h = (u0 + n) % HKV, i = n / HKV, buf = i & 1, slot = n % kStages;   // i: earlier stages of the head
        if (i >= 2 && !tc_wait(&bars->acc_empty[h][buf], ((i >> 1) - 1) & 1u, bars, err, 82)) break;
        if (!tc_wait(&bars->k_full[slot], (n / kStages) & 1u, bars, err, 83)) break;
        tc_fence_after();
        const uint32_t a_base = smem_u32(ring + slot * kTcStageBytes);
        const uint32_t b_base = q_base + h * 2 * Lay::kQHalf;
#pragma unroll
        for (int kk = 0; kk < 8; ++kk) {
          const uint32_t ao = (kk >> 2) * kTcHalf + (kk & 3) * 32;
          const uint32_t bo = (kk >> 2) * Lay::kQHalf + (kk & 3) * 32;
          tc_mma_bf16(tmem + (buf * HKV + h) * kN, smem_desc_sw128(a_base + ao), smem_desc_sw128(b_base + bo),
                      Lay::kIdesc, kk > 0 ? 1u : 0u);
        }
        tc_commit(&bars->k_empty[slot]);
        tc_commit(&bars->acc_full[h][buf]);
      }
      // no commit arrives after the CTA has left: the last one covers every MMA of this thread
      tc_commit(&bars->drain);
      mbar_wait(&bars->drain, 0, kWaitLimitNs / 4);
    }
  } else {
    // ------------------------------------------------------------ epilogue
    const int wg = (warp - 2) >> 2;                   // heads wg, wg + kGroups, ..
    const int quad = warp & 3;                        // TMEM lanes 32 * (warp % 4) ..
    const int kt = quad * 32 + lane;                  // key within the tile
    const uint32_t lane_off = static_cast<uint32_t>(quad * 32) << 16;
    const float c2 = plan.scale2;
    constexpr int kLanes = 32 / NR;                   // lanes per row after the reduce-scatter
    int n = (wg - u0 % Lay::kGroups + Lay::kGroups) % Lay::kGroups;   // this warpgroup's stages: every kGroups-th
    auto key_of = [&](int nn) { return ((u0 + nn) / HKV) * kTcM + kt; };
    auto mod_of = [&](int nn) -> uint8_t {
      const int key = key_of(nn);
      return (nn < nstage && key < sq.len) ? modality[sq.t0 + key] : static_cast<uint8_t>(0);
    };
    uint8_t mod_next = mod_of(n);                     // one stage ahead
    for (; n < nstage; n += Lay::kGroups) {
      const int h = (u0 + n) % HKV, i = n / HKV, buf = i & 1;
      const int key = key_of(n);
      const bool valid = key < sq.len;
      const bool mm = valid && is_mm_tc(mod_next);
      mod_next = mod_of(n + Lay::kGroups);
      // rows j >= j_min have this key in their denominator: every row of a multimodal key, or
      // (causal rows) the rows of the tokens at or after the key, token j / G >= key - q_pos
      const int j_min = plan.causal ? (valid ? max(0, key - sq.q_pos) * G : NR) : (mm ? 0 : NR);
      // warp-uniform: tcgen05.ld below is a warp-collective instruction
      if (!__all_sync(0xffffffffu, tc_wait(&bars->acc_full[h][buf], (i >> 1) & 1u, bars, err, 84))) break;
      tc_fence_after();
      uint32_t r[NR];
      load_rows(bars->tmem_base + lane_off + (buf * HKV + h) * kN, r);
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&bars->acc_empty[h][buf]);   // the values are in registers
      float v[NR];
      float *lp = logits + sq.logit_base + static_cast<int64_t>(h * G) * sq.lstride + key;
#pragma unroll
      for (int j = 0; j < NR; ++j) {
        const float x = __uint_as_float(r[j]);
        if (valid && j < rg) lp[rho_of[j] * sq.lstride] = x;
        v[j] = (j < rg && j >= j_min) ? x : -INFINITY;
      }
      // the row maxima of the warp's keys, then sums relative to the raised maxima
      const int hh = Lay::kHeads == 1 ? 0 : h / Lay::kGroups;
      const float tmax = reduce_scatter<NR>(v, lane, [](float a, float b) { return fmaxf(a, b); });
      float m_old = m_run[0], l_old = l_run[0];
      if (Lay::kHeads > 1 && hh) {
        m_old = m_run[Lay::kHeads - 1];
        l_old = l_run[Lay::kHeads - 1];
      }
      const float m_new = fmaxf(m_old, tmax * c2);    // log2 units; -inf while no key has counted
#pragma unroll
      for (int j = 0; j < NR; ++j) {
        const float mj = __shfl_sync(0xffffffffu, m_new, j * kLanes);
        // no counted key of the row yet: every term is exp2(-inf - 0) = 0
        const float x = (j < rg && j >= j_min) ? __uint_as_float(r[j]) : -INFINITY;
        v[j] = ex2_approx(fmaf(x, c2, mj == -INFINITY ? 0.f : -mj));
      }
      const float tsum = reduce_scatter<NR>(v, lane, [](float a, float b) { return a + b; });
      const float l_new = (m_old == -INFINITY ? 0.f : l_old * ex2_approx(m_old - m_new)) + tsum;
      if (Lay::kHeads > 1 && hh) {
        m_run[Lay::kHeads - 1] = m_new;
        l_run[Lay::kHeads - 1] = l_new;
      } else {
        m_run[0] = m_new;
        l_run[0] = l_new;
      }
    }
  }
  // every stage is consumed (or a wait gave up): the ring holds the warps' states next
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const bool ok = !bars->abort;
  float2 *st = reinterpret_cast<float2 *>(ring);                        // [HKV][4 quads][NR]
  if (ok && warp >= 2 && lane % (32 / NR) == 0) {
    const int wg = (warp - 2) >> 2, quad = warp & 3;
#pragma unroll
    for (int i = 0; i < Lay::kHeads; ++i)
      st[((wg + i * Lay::kGroups) * 4 + quad) * NR + lane / (32 / NR)] = make_float2(m_run[i], l_run[i]);
  }
  __syncthreads();
  if (ok) {
    for (int e = threadIdx.x; e < HKV * NR; e += Lay::kThreads) {
      const int h = e / NR, j = e % NR;
      if (j >= rg) continue;
      float2 w[4];
      float mx = -INFINITY, tot = 0.f;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        w[i] = st[(h * 4 + i) * NR + j];
        mx = fmaxf(mx, w[i].x);
      }
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (w[i].x != -INFINITY) tot += w[i].y * ex2_approx(w[i].x - mx);
      part[sq.part_base + static_cast<int64_t>(rho_of[j] + h * G) * sq.nparts + c] = make_float2(mx, tot);
    }
  }
  if (warp == 1) tmem_dealloc(bars->tmem_base, Lay::kTmemCols);
}

template <int HKV, int NR>
cudaError_t launch(int grid, cudaStream_t stream, const CUtensorMap &kmap, const NarrowPlan &P, const uint16_t *q,
                   const uint8_t *modality, float *logits, float2 *part, DeviceError *err) {
  using Lay = TcLayout<HKV, NR>;
  static std::atomic<uint64_t> attr{0};
  const cudaError_t e = once_per_device(attr, [] {
    return cudaFuncSetAttribute(score_narrow_tc_kernel<HKV, NR>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                static_cast<int>(Lay::kBytes));
  });
  if (e != cudaSuccess) return e;
  return launch_pdl(score_narrow_tc_kernel<HKV, NR>, dim3(grid), dim3(Lay::kThreads), Lay::kBytes, stream, kmap, P, q,
                    modality, logits, part, err);
}

template <int HKV>
cudaError_t launch_rows(int max_rg, int grid, cudaStream_t stream, const CUtensorMap &kmap, const NarrowPlan &P,
                        const uint16_t *q, const uint8_t *modality, float *logits, float2 *part, DeviceError *err) {
  if (max_rg <= 8) return launch<HKV, 8>(grid, stream, kmap, P, q, modality, logits, part, err);
  if (max_rg <= 16) return launch<HKV, 16>(grid, stream, kmap, P, q, modality, logits, part, err);
  return launch<HKV, 32>(grid, stream, kmap, P, q, modality, logits, part, err);
}

}  // namespace

cudaError_t launch_narrow_tc(int max_rg, int grid, cudaStream_t stream, const CUtensorMap &kmap, const NarrowPlan &P,
                             const uint16_t *q, const uint8_t *modality, float *logits, float2 *part,
                             DeviceError *err) {
  switch (P.hkv) {
    case 1: return launch_rows<1>(max_rg, grid, stream, kmap, P, q, modality, logits, part, err);
    case 2: return launch_rows<2>(max_rg, grid, stream, kmap, P, q, modality, logits, part, err);
    case 4: return launch_rows<4>(max_rg, grid, stream, kmap, P, q, modality, logits, part, err);
    case 8: return launch_rows<8>(max_rg, grid, stream, kmap, P, q, modality, logits, part, err);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace apack
