// score.cu -- relevance scores of Eq. inner_score (Sec. 3.2) on the tcgen05 tensor cores.
//
// I_i = 1/(Hq n_q) sum_h sum_r softmax_{j in S}(q_{r,h} . k_{j,g(h)} / sqrt(D))_i
//
// The softmax normaliser of every (query row, head) needs all keys of S before
// any per-key average can be formed, so the scores take two passes over K:
//
//  pass 1 (row statistics): D[row][key] = Q . K^T with query rows in TMEM lanes;
//     each epilogue thread owns one row and keeps an online (reference, sum of
//     exp2) over its keys.  The (row group, key block) space is cut into equal
//     contiguous ranges, one per CTA pair; a pair writes one partial (m, sum) per
//     row for each row group its range touches.
//  merge: per packed query row, the partials combine in pair order into a log2-domain
//     normaliser lse2 = log2 sum_j 2^(x_j log2(e)/sqrt(D)), stored negated.
//  pass 2 (column sums): D[key][row] = K . Q^T with keys in TMEM lanes; each
//     thread owns one key and sums 2^(x c - lse2[row]) over the rows of one KV
//     head group; the Hkv group sums are added in a fixed order and scaled by
//     1/(Hq n_q): by the unit itself when it runs over every group, else by the last
//     unit of a key block (a counter), else (long sequences whose groups are better
//     split, or sequences without query rows in the launch) by a final kernel.
//     Scores are deterministic: the counters only say who adds, not in what order.
//
// Query rows are first repacked per KV head g into linear rows rho = token * G + j
// (query head g*G + j), padded to a multiple of 256, so that tiles hold no holes.
//
// Both passes run on CTA pairs (clusters of two CTAs on two SMs) with
// tcgen05.mma.cta_group::2: one M=256 x N=256 x K=16 instruction per step, issued
// by the even CTA, reads 128 rows of A and 128 rows of B from each CTA's shared
// memory and leaves each CTA's 128 rows of D (256 fp32 columns) in its own TMEM.
// Per SM that moves 64 B of operands from shared memory per clock at the full MMA
// rate, against 128 B for an M=128 x N=128 instruction on one SM, which is what
// bounded the single-CTA version.  Each CTA loads its halves of the operands with
// TMA; the copies of both CTAs complete on the even CTA's barriers
// (cp.async.bulk.tensor ... .cta_group::2), the MMA completions arrive on both CTAs'
// barriers (tcgen05.commit ... .multicast::cluster).  The stationary operand A
// (query rows in pass 1, keys in pass 2) is held for a run of streamed B tiles (key
// blocks in pass 1, query chunks in pass 2), four B stages deep; two 256-column
// accumulators alternate in TMEM.  Warp 0 issues TMA, warp 1 owns TMEM (and on the
// even CTA issues the MMAs), warps 2..17 are four epilogue warpgroups; warpgroups 2b
// and 2b + 1 read the tiles of accumulator b, 128 columns each for the CTA's 128 lanes.  Pass 1
// takes each key block's masks (which keys count) from a bit array that the query repack kernel
// writes once per call.  Operands sit in 128-byte swizzled shared memory.  Persistent pairs, one
// CTA per SM.
#include <algorithm>
#include <cmath>
#include <cstdio>

#include "internal.cuh"
#include "ptx.cuh"

namespace apack {

namespace {

constexpr int kEpiWG = 4;                         // epilogue warpgroups
constexpr int kEpiWarps = 4 * kEpiWG;
// Warpgroups 2b and 2b + 1 own accumulator buffer b (the tiles of one parity): each reads half of
// the buffer's 256 columns, in two loads of kCols, so that one pair computes while the other waits
// for its next tile.
constexpr int kPairWarps = kEpiWarps / 2;        // epilogue warps that read one buffer
constexpr int kSpan = 128;                       // columns of a tile per warpgroup of the owning pair
constexpr int kCols = 64;                        // columns per TMEM load, pass 1
constexpr int kCols2 = 32;                       // columns per TMEM load, pass 2
static_assert(2 * kSpan == 256 && 2 * kCols == kSpan && 4 * kCols2 == kSpan,
              "two warpgroups x (two or four) loads cover a 256-column tile");
// The epilogue bounds both passes, not the MMA: 64 columns loaded and summed by 16 warps take 1,220
// clocks a tile (the exp2 unit 1,024, TMEM loads do not overlap it) against 1,024 for the MMA, and what
// a warp does around its tiles comes on top, since the four warps of a scheduler tend to do it at the
// same time.  So the loops run over a warpgroup's own tiles only, the masks come in one load, and the
// exponentials are scheduled by hand (exp_sum): pass 1 188 -> 173 us, pass 2 170 -> 156 us over
// 135,272 keys and 7,168 rows (6 us of pass 2 from its set-up running before the wait).  Measured
// slower: 8 epilogue warps with 64 or 128 columns in registers (209 / 178 and 258 / 185 us), all 16
// warps on every tile (197 / 187), half tiles of 128 columns as MMAs of their own (200 / 206: N =
// 128 re-reads A from shared memory), and 2 of 16 exponentials as a degree-5 polynomial on the FMA
// pipe (the whole call 380 -> 395 us).
// warp 0: TMA, warp 1: TMEM (+ MMA on the even CTA), then the epilogue warps.
constexpr int kThreads = 32 * (2 + kEpiWarps);
constexpr uint32_t kTmemCols = 512;    // 2 accumulators x 256 fp32 columns
constexpr int kAStages = 2, kBStages = 4;
constexpr uint32_t kRows = 128;                // rows of A and of B per CTA (M/2, N/2 of the pair)
constexpr uint32_t kTileBytes = kRows * 256;   // 128 rows x 128 bf16
constexpr uint32_t kHalf = kRows * 128;        // second 64-element K half of a tile
constexpr uint32_t kIdesc = idesc_bf16_f32(256, 256);
constexpr int kBlock = 256;                    // keys per key block (pass 1) / per key unit (pass 2)
constexpr int kChunk = 256;                    // query rows per chunk (pass 2) / per row pair (pass 1)
constexpr int kPairSlots = kMaxSplits;         // pair ranges per row group (one partial each)

constexpr int kMergeThreads = 64;

struct SeqPlan {
  int32_t t0, len;        // token range of the sequence in the packed batch
  int32_t q_off, n_q;     // query tokens in packed Q
  int32_t qp_base;        // first packed row of head group 0; group g starts at qp_base + g * rows_pad
  int32_t rows_pad;       // G * n_q rounded up to a multiple of 256
  int32_t nb;             // key blocks (256 keys) of the sequence
  int32_t q_pos;          // causal rows: position of query row 0 within the sequence
  int32_t unit_begin;     // pass 2: first work unit of this sequence in the launch
  int32_t flat0;          // pass 1: first flat (row group, key block) index of the sequence
  int32_t blk0;           // pass 1: first key block of the sequence in the launch's mask array
};

struct ScorePlan {
  int32_t nseq;
  int32_t total_units;     // pass 2
  int32_t pairs;           // pass 1: CTA pairs of the launch
  int32_t flat_total;      // pass 1: (row group, key block) items of the launch (< 2^31, checked)
  int32_t hq, hkv, group;
  int32_t total_qrows;     // sum n_q over the whole batch
  int32_t total_tokens;    // T
  int32_t causal;          // APACK_SOFTMAX_CAUSAL_ROW: rows see every token up to their own position
  int32_t unit_groups;     // pass 2: KV head groups per unit, 1 or hkv
  int32_t direct;          // pass 2: a unit holds every group and writes its keys' scores
  int32_t counted;         // pass 2, one of several groups per unit: the last of a key block's units adds them
  float scale2;            // log2(e) / sqrt(D)
  SeqPlan seq[kSeqsPerLaunch];
};

struct __align__(8) Bars {
  uint64_t a_full[kAStages], a_empty[kAStages], b_full[kBStages], b_empty[kBStages];
  uint64_t acc_full[2], acc_empty[2], drain;
  uint64_t l_full[kBStages], l_empty[kBStages];   // pass 2: normaliser slot loaded / released (this CTA)
  uint64_t comb_full[2], comb_empty[2];           // column ranges 1.. -> range 0 hand-off
  uint32_t tmem_base;
  volatile int32_t abort;
  volatile int32_t marked;                        // pass 1: the CTA wrote a partial with a sum out of range
};

// Shared memory: [A x2][B x4][-lse2 x4 (pass 2)][combine 2 x (kEpiWG - 1) x 128 float2][Bars].
// The dynamic shared window is declared 1024-byte aligned (the 128-byte swizzle
// atoms of the operand tiles need it); the kernels verify it before any use.
constexpr uint32_t kOffA = 0;
constexpr uint32_t kOffB = kAStages * kTileBytes;
constexpr uint32_t kOffL = kOffB + kBStages * kTileBytes;
constexpr uint32_t kOffC = kOffL + kBStages * kChunk * sizeof(float);
constexpr uint32_t kOffBars = kOffC + 2 * (kEpiWG - 1) * kRows * sizeof(float2);
constexpr uint32_t kSmemBytes = kOffBars + 512;
static_assert(sizeof(Bars) <= 512, "barrier block");
static_assert(kSmemBytes <= 232448, "shared memory budget");

// Rows of a unit times partials per row up to which pass 2 merges by itself (8,780 keys, 512 rows with 19
// each: 20.5 -> 19.3 us; 13,500 keys, 2,048 rows with 12: 27.0 -> 31.3 us).
constexpr int kMergeInside = 16384;
// pass 2 counters of a launch (one word per key block, 4 bits per 32 keys) in the workspace, between the
// error word and the words of the in-place compaction, which may run beside a scoring on the workspace.
// A counted call has at most as many blocks as half the GPU's CTA pairs (38 with 152 SMs).
constexpr size_t kCounterOff = sizeof(DeviceError);
constexpr int kMaxCounted = (256 - static_cast<int>(kCounterOff)) / 4;   // key blocks
constexpr int kMaxCountedGroups = 15;          // what 4 bits count

__device__ __forceinline__ bool is_mm(uint8_t m) { return m == APACK_MOD_AUDIO || m == APACK_MOD_VISUAL; }

__host__ __device__ __forceinline__ int n_pairs(const SeqPlan &sp) { return sp.rows_pad / kChunk; }
__host__ __device__ __forceinline__ int64_t pass1_items(const SeqPlan &sp, int hkv) {
  return static_cast<int64_t>(sp.nb) * hkv * n_pairs(sp);
}

// Pass 1: pair p of P owns the flat items [start(p), start(p + 1)), start(p) = p W / P,
// and the pair holding item x is ((x + 1) P - 1) / W (64-bit products of 32-bit indices).
__host__ __device__ __forceinline__ int32_t range_start(int64_t p, int64_t P, int64_t W) {
  return static_cast<int32_t>(p * W / P);
}
__host__ __device__ __forceinline__ int32_t pair_of(int64_t x, int64_t P, int64_t W) {
  return static_cast<int32_t>(((x + 1) * P - 1) / W);
}

// ---------------------------------------------------------------- cluster-pair helpers
// Barrier waits and arrivals keep the default (CTA-scope) semantics: what crosses the pair
// through them is ordered by the asynchronous proxies themselves (TMA byte counts, MMA
// commits) and by the tcgen05 fences around TMEM reads, not by generic memory accesses.
// (Cluster-scope acquire and release here made every wait and arrival a memory barrier:
// measured 1.5x slower, with memory-barrier stalls the largest stall reason.)

// Remote (or local) arrive on a barrier given by its shared::cluster address.
__device__ __forceinline__ void arrive_cluster(uint32_t cluster_addr) {
  asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
}

__device__ __forceinline__ void st_cluster_u32(uint32_t cluster_addr, uint32_t v) {
  asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(cluster_addr), "r"(v) : "memory");
}

// 3-D tiled load into this CTA's shared memory, completion counted on a barrier of
// either CTA of the pair (given as a shared::cluster address).
__device__ __forceinline__ void tma_load_3d_pair(void *dst, const CUtensorMap *map, uint32_t bar_cluster, int32_t c0,
                                                 int32_t c1, int32_t c2) {
  asm volatile(
      "cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, "
      "%5}], [%2];" ::"r"(smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(bar_cluster), "r"(c0), "r"(c1), "r"(c2)
      : "memory");
}

__device__ __forceinline__ void mma_pair(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
      "l"(a_desc), "l"(b_desc), "r"(kIdesc), "r"(accumulate)
      : "memory");
}

// Arrive on the barrier at this offset in both CTAs once the issued MMAs complete.
__device__ __forceinline__ void commit_pair(uint64_t *bar) {
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(
          smem_u32(bar)),
      "h"(static_cast<uint16_t>(3))
      : "memory");
}

// Arrive on this CTA's own barrier once the issued MMAs complete.
__device__ __forceinline__ void commit_pair_self(uint64_t *bar) {
  asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
               : "memory");
}

__device__ __forceinline__ void tmem_alloc_pair(uint32_t *dst_smem, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(dst_smem)),
               "r"(ncols)
               : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ void tmem_dealloc_pair(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}

struct PairCtx {
  uint32_t rank;          // 0: the even CTA (issues the MMAs), 1: its peer
  uint32_t lead_bars;     // shared::cluster address of the even CTA's Bars
  uint32_t peer_abort;    // shared::cluster address of the other CTA's abort flag
};

template <typename T>
__device__ __forceinline__ uint32_t lead_addr(const PairCtx &pc, const Bars *bars, const T *member) {
  return pc.lead_bars + static_cast<uint32_t>(reinterpret_cast<const uint8_t *>(member) -
                                              reinterpret_cast<const uint8_t *>(bars));
}

// A wait that also gives up when a role of either CTA has aborted; a timeout aborts both.
__device__ __forceinline__ bool wait_or_abort(uint64_t *bar, uint32_t parity, Bars *bars, const PairCtx &pc,
                                              DeviceError *err, int where) {
  if (mbar_try_wait(bar, parity)) return true;
  const uint64_t t0 = globaltimer_ns();
  for (;;) {
    for (int i = 0; i < 32; ++i)
      if (mbar_try_wait(bar, parity)) return true;
    if (bars->abort) return false;
    if (globaltimer_ns() - t0 > kWaitLimitNs) {
      bars->abort = 1;
      st_cluster_u32(pc.peer_abort, 1u);
      raise_device_error(err, APACK_ETIMEOUT, where);
      return false;
    }
  }
}

// True when the dynamic shared window has the 1024-byte alignment the operand tiles need.
__device__ __forceinline__ bool smem_aligned(const uint8_t *smem) { return (smem_u32(smem) & 1023u) == 0; }

__device__ PairCtx init_pair(uint8_t *smem, Bars *bars, int warp) {
  PairCtx pc;
  pc.rank = cluster_ctarank();
  if (threadIdx.x == 0) {
    for (int i = 0; i < kAStages; ++i) {
      mbar_init(&bars->a_full[i], 1);
      mbar_init(&bars->a_empty[i], 1);
    }
    for (int i = 0; i < kBStages; ++i) {
      mbar_init(&bars->b_full[i], 1);
      mbar_init(&bars->b_empty[i], 1);
      mbar_init(&bars->l_full[i], 1);
      mbar_init(&bars->l_empty[i], kPairWarps);    // stage i is read by the pair owning buffer i % 2
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&bars->acc_full[i], 1);
      mbar_init(&bars->acc_empty[i], 2 * kPairWarps);  // the owning pair's warps in both CTAs
      mbar_init(&bars->comb_full[i], (kEpiWG - 1) * 4);
      mbar_init(&bars->comb_empty[i], 4);
    }
    mbar_init(&bars->drain, 1);
    bars->abort = 0;
    bars->marked = 0;
    fence_mbar_init();
  }
  pc.lead_bars = map_shared_rank(bars, 0);
  pc.peer_abort = map_shared_rank(const_cast<const int32_t *>(&bars->abort), pc.rank ^ 1u);
  cluster_sync();                      // both CTAs' barriers exist before any remote arrive or copy
  if (warp == 1) {
    tmem_alloc_pair(&bars->tmem_base, kTmemCols);
    tc_fence_before();
  }
  __syncthreads();
  tc_fence_after();
  return pc;
}

// Teardown: after an abort the MMA thread makes sure no MMA is in flight; both CTAs
// then meet (every TMEM read and every MMA of the pair is done) and free TMEM.
__device__ void finish_pair(Bars *bars, const PairCtx &pc, int warp, bool mma_thread) {
  if (mma_thread && bars->abort) {
    commit_pair_self(&bars->drain);
    mbar_wait(&bars->drain, 0, kWaitLimitNs / 4);
  }
  if (threadIdx.x == 0 && bars->abort) {
    // copies of this CTA complete on the even CTA's barriers, which this CTA cannot watch:
    // give any still in flight time to land before the pair meets (bounded)
    const uint64_t t0 = globaltimer_ns();
    while (globaltimer_ns() - t0 < 200000ull) {
    }
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync();
  tc_fence_after();
  if (warp == 1) tmem_dealloc_pair(bars->tmem_base, kTmemCols);
}

// Waits (bounded, ignoring the abort flag) for TMA loads that were issued but never
// consumed, so that no copy lands in shared memory after exit (the even CTA's barriers).
__device__ void drain_loads(uint64_t *full, const bool *pending, const uint32_t *parity, int n) {
  for (int i = 0; i < n; ++i)
    if (pending[i]) mbar_wait(&full[i], parity[i], kWaitLimitNs / 4);
}

// kCols consecutive TMEM columns of this warp's 32 lanes -> registers, loaded and waited for
// in one statement (the registers are defined only once the data is there).
__device__ __forceinline__ void tmem_load_cols(uint32_t taddr, uint32_t (&r)[64]) { tmem_ld64_wait(taddr, r); }
__device__ __forceinline__ void tmem_load_cols(uint32_t taddr, uint32_t (&r)[32]) {
  tmem_ld32(taddr, r);
  tmem_wait32(r);
}

// The eight K=16 steps of one 256 x 256 x 128 product into accumulator `ci`.
__device__ __forceinline__ void issue_mma(uint32_t tmem, int ci, uint32_t a_base, uint32_t b_base) {
  const uint64_t a_desc = smem_desc_sw128(a_base), b_desc = smem_desc_sw128(b_base);
#pragma unroll
  for (int kk = 0; kk < 8; ++kk) {   // the address field counts 16 bytes; the tiles lie below 256 KB
    const uint32_t off = ((kk >> 2) * kHalf + (kk & 3) * 32) >> 4;
    mma_pair(tmem + ci * 256, a_desc + off, b_desc + off, kk > 0 ? 1u : 0u);
  }
}

// ------------------------------------------------------------------ pass 1
// A run: the part of a pair's flat range that lies in one row group (sequence s, KV head
// group g, 256-row pair qp): key blocks [b0, b1) of that row group.
struct Run {
  int s, g, qp, b0, b1;
  int x1;          // flat index after the run
  int slot;        // partial slot: pair - first pair of the row group
};

__device__ __forceinline__ int seq_of_flat(const ScorePlan &p, int x) {
  int s = 0;
  while (s + 1 < p.nseq && p.seq[s + 1].flat0 <= x) ++s;
  return s;
}

__device__ __forceinline__ Run next_run(const ScorePlan &p, int x, int x_end, int pair) {
  Run r;
  r.s = seq_of_flat(p, x);
  const SeqPlan &sp = p.seq[r.s];
  const int local = x - sp.flat0;
  const int grp = local / sp.nb;                      // row group index within the sequence
  const int np = n_pairs(sp);
  r.g = grp / np;
  r.qp = grp - r.g * np;
  r.b0 = local - grp * sp.nb;
  const int grp_end = sp.flat0 + (grp + 1) * sp.nb;
  r.x1 = x_end < grp_end ? x_end : grp_end;
  r.b1 = r.b0 + (r.x1 - x);
  r.slot = pair - pair_of(sp.flat0 + grp * sp.nb, p.pairs, p.flat_total);
  return r;
}

// Online (reference, sum) update with a thread's 64 logits of a block, in log2 units.  Keys
// that do not count are first replaced by -inf (exp2 gives 0), so that one code path serves
// every mask.  The reference is the first counted block's maximum and stays fixed for the
// run: no block's sums feed back into the next block's arithmetic.  A block whose sum leaves
// the safe range (a logit more than about 2^99 above the reference, or an overflow) only sets
// `bad`; such a partial is recomputed exactly at the CTA's end (repair_marked).  Four independent
// partial sums keep the add chains short.
constexpr float kSumLimit = 6.338253e29f;   // 2^99

// a[0..3] += 2^(x c2 + add) over the N logits x of a thread, add(i) for logits i and i + 1; x is
// overwritten.  The three steps of a group of kGroup logits (scale, exp2, sum) are written one group
// apart and in place: the exp2 unit's latency is covered without registers for its results.
constexpr int kGroup = 16;

template <int N, class Add>
__device__ __forceinline__ void exp_sum(uint32_t (&x)[N], float c2, Add add, float2 (&a)[4]) {
  const float2 cc = make_float2(c2, c2);
#pragma unroll
  for (int g = 0; g < N / kGroup + 2; ++g) {
    if (g >= 2) {
#pragma unroll
      for (int j = 0; j < kGroup; j += 2) {
        const int i = (g - 2) * kGroup + j;
        a[(i >> 1) & 3] = fadd2(a[(i >> 1) & 3], make_float2(__uint_as_float(x[i]), __uint_as_float(x[i + 1])));
      }
    }
    if (g >= 1 && g - 1 < N / kGroup) {
#pragma unroll
      for (int j = 0; j < kGroup; ++j) {
        const int i = (g - 1) * kGroup + j;
        x[i] = __float_as_uint(ex2_approx(__uint_as_float(x[i])));
      }
    }
    if (g < N / kGroup) {
#pragma unroll
      for (int j = 0; j < kGroup; j += 2) {
        const int i = g * kGroup + j;
        const float2 y = ffma2(make_float2(__uint_as_float(x[i]), __uint_as_float(x[i + 1])), cc, add(i));
        x[i] = __float_as_uint(y.x);
        x[i + 1] = __float_as_uint(y.y);
      }
    }
  }
}

__device__ __forceinline__ void online_block(uint32_t (&r)[64], uint32_t mask0, uint32_t mask1, float c2, float &m,
                                             float &sum, bool &bad) {
  if ((mask0 & mask1) != 0xffffffffu) {
    if ((mask0 | mask1) == 0u) return;
    const uint32_t ninf = __float_as_uint(-INFINITY);
#pragma unroll
    for (int i = 0; i < 32; ++i) {
      r[i] = ((mask0 >> i) & 1u) ? r[i] : ninf;
      r[32 + i] = ((mask1 >> i) & 1u) ? r[32 + i] : ninf;
    }
  }
  if (m == -INFINITY) {
    float mx = __uint_as_float(r[0]);
#pragma unroll
    for (int i = 1; i < 64; ++i) mx = fmaxf(mx, __uint_as_float(r[i]));
    m = mx * c2;
  }
  float2 a[4] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
  const float2 nm = make_float2(-m, -m);
  exp_sum(r, c2, [&](int) { return nm; }, a);
  const float2 s01 = fadd2(a[0], a[1]), s23 = fadd2(a[2], a[3]);
  const float2 s4 = fadd2(s01, s23);
  const float t = s4.x + s4.y;
  bad |= !(t <= kSumLimit);
  sum += t;
}

// The (maximum, sum) in log2 units of one query row qr over the keys of blocks [b0, b1) of a sequence,
// computed by a warp without the tensor cores.  kg: the head group's keys of the sequence; words: its key
// masks; keys past `see` do not count.  One key per lane: dot products in fp32 from the bf16 values, an
// online sum with exact rescaling, the lanes combined in a fixed order.
__device__ __forceinline__ float2 exact_part(const uint4 *__restrict__ qr, const uint8_t *__restrict__ kg, int64_t k_stride,
                                             const uint32_t *__restrict__ words, int b0, int b1, int see) {
  const int lane = threadIdx.x & 31;
  float m = -INFINITY, sum = 0.f;
  for (int w = b0 * (kBlock / 32); w < b1 * (kBlock / 32); ++w) {
    const int key = w * 32 + lane;
    if (!((__ldg(words + w) >> lane) & 1u) || key > see) continue;
    const uint4 *kr = reinterpret_cast<const uint4 *>(kg + key * k_stride);
    float2 a[4] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
#pragma unroll 4
    for (int d = 0; d < 16; ++d) {
      const uint4 q8 = __ldg(qr + d), k8 = __ldg(kr + d);
      const uint32_t qw[4] = {q8.x, q8.y, q8.z, q8.w}, kw[4] = {k8.x, k8.y, k8.z, k8.w};
#pragma unroll
      for (int e = 0; e < 4; ++e)
        a[e] = ffma2(make_float2(__uint_as_float(qw[e] << 16), __uint_as_float(qw[e] & 0xFFFF0000u)),
                     make_float2(__uint_as_float(kw[e] << 16), __uint_as_float(kw[e] & 0xFFFF0000u)), a[e]);
    }
    const float2 t = fadd2(fadd2(a[0], a[1]), fadd2(a[2], a[3]));
    const float y = (t.x + t.y) * kScale2;                // not from the tensor cores
    if (y > m) {
      sum = (m == -INFINITY ? 0.f : sum * exp2f(m - y)) + 1.f;
      m = y;
    } else {
      sum += exp2f(y - m);
    }
  }
  __syncwarp();
  float mm = m;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) mm = fmaxf(mm, __shfl_xor_sync(0xffffffffu, mm, o));
  float tot = m != -INFINITY ? sum * exp2f(m - mm) : sum;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) tot += __shfl_xor_sync(0xffffffffu, tot, o);
  return make_float2(mm, tot);
}

// Computes the partials that a CTA marked (a negative sum) again, its warps a row each.  The work stays in
// the row's run, so it is spread over the GPU like the runs, and the merge finds every partial in range.
// With every row marked, against whole rows recomputed in the merge by a warp per row and by a warp per 32
// rows: 135,272 keys, 256 x 28 rows, 67 ms against 640 and 963; 8,780 keys, 64 x 16 rows, 0.16 ms against 29
// and 232.  As a call at the end of each run it took the tile loop's registers (370 -> 390 us without a mark).
template <bool CAUSAL>
__device__ __noinline__ void repair_marked(const ScorePlan &plan, int pair, int row_half,
                                           const uint32_t *__restrict__ mask_words, const uint4 *__restrict__ qp,
                                           const uint8_t *__restrict__ k, int64_t k_stride, float2 *part) {
  const int G = plan.group;
  const int x_end = range_start(pair + 1, plan.pairs, plan.flat_total);
  for (int x = range_start(pair, plan.pairs, plan.flat_total); x < x_end;) {
    const Run w = next_run(plan, x, x_end, pair);
    const SeqPlan &sp = plan.seq[w.s];
    x = w.x1;
    for (int row = row_half + (threadIdx.x >> 5); row < row_half + kRows; row += kThreads / 32) {
      const int rho = w.qp * kChunk + row;                    // linear row of the head group
      if (rho >= G * sp.n_q) break;
      const int r = rho / G, j = rho - r * G;
      float2 *p = part + (static_cast<size_t>(w.slot) * plan.total_qrows + sp.q_off + r) * plan.hq + w.g * G + j;
      if (!(p->y < 0.f)) continue;
      const float2 v = exact_part(qp + (sp.qp_base + static_cast<int64_t>(w.g) * sp.rows_pad + rho) * 16,
                                  k + sp.t0 * k_stride + w.g * 256, k_stride, mask_words + sp.blk0 * 8, w.b0, w.b1,
                                  CAUSAL ? sp.q_pos + r : sp.len);
      if ((threadIdx.x & 31) == 0) *p = v;
    }
  }
}

template <bool CAUSAL>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreads, 1)
    score_rowstats_kernel(const __grid_constant__ CUtensorMap qmap, const __grid_constant__ CUtensorMap kmap,
                          const __grid_constant__ ScorePlan plan, const uint32_t *__restrict__ mask_words,
                          const uint4 *__restrict__ qp, const uint8_t *__restrict__ k, int64_t k_stride,
                          float2 *__restrict__ part, DeviceError *err) {
  extern __shared__ __align__(1024) uint8_t smem[];
  if (!smem_aligned(smem)) {   // the same in both CTAs of the pair: both leave here
    if (threadIdx.x == 0) raise_device_error(err, APACK_EDEVICE, 10);
    return;
  }
  Bars *bars = reinterpret_cast<Bars *>(smem + kOffBars);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const PairCtx pc = init_pair(smem, bars, warp);
  pdl_wait_and_release();      // the set-up runs beside the previous launch
  const int G = plan.group;
  const int pair = blockIdx.x >> 1;
  const int x_begin = range_start(pair, plan.pairs, plan.flat_total);
  const int x_end = range_start(pair + 1, plan.pairs, plan.flat_total);
  const int row_half = static_cast<int>(pc.rank) * kRows;   // this CTA's rows of the 256-row pair

  if (warp == 0) {
    if (lane == 0) {
      tma_prefetch_desc(&qmap);
      tma_prefetch_desc(&kmap);
      int ai = 0, bi = 0;
      uint32_t aph = 0, bph = 0;
      bool pend[kBStages] = {}, apend[kAStages] = {};
      uint32_t pend_par[kBStages] = {}, apend_par[kAStages] = {};
      bool ok = true;
      for (int x = x_begin; ok && x < x_end;) {
        const Run w = next_run(plan, x, x_end, pair);
        const SeqPlan &sp = plan.seq[w.s];
        x = w.x1;
        if (!wait_or_abort(&bars->a_empty[ai], aph ^ 1, bars, pc, err, 11)) { ok = false; break; }
        uint8_t *A = smem + kOffA + ai * kTileBytes;
        if (pc.rank == 0) mbar_arrive_expect_tx(&bars->a_full[ai], 2 * kTileBytes);
        const uint32_t afull = lead_addr(pc, bars, &bars->a_full[ai]);
        const int arow = sp.qp_base + w.g * sp.rows_pad + w.qp * kChunk + row_half;
        tma_load_3d_pair(A, &qmap, afull, 0, 0, arow);
        tma_load_3d_pair(A + kHalf, &qmap, afull, 64, 0, arow);
        apend[ai] = true;
        apend_par[ai] = aph;
        for (int b = w.b0; b < w.b1; ++b) {
          if (!wait_or_abort(&bars->b_empty[bi], bph ^ 1, bars, pc, err, 12)) { ok = false; break; }
          uint8_t *B = smem + kOffB + bi * kTileBytes;
          if (pc.rank == 0) mbar_arrive_expect_tx(&bars->b_full[bi], 2 * kTileBytes);
          const uint32_t bfull = lead_addr(pc, bars, &bars->b_full[bi]);
          const int key0 = sp.t0 + b * kBlock + row_half;
          tma_load_3d_pair(B, &kmap, bfull, 0, w.g, key0);
          tma_load_3d_pair(B + kHalf, &kmap, bfull, 64, w.g, key0);
          pend[bi] = true;
          pend_par[bi] = bph;
          if (++bi == kBStages) { bi = 0; bph ^= 1; }
        }
        if (++ai == kAStages) { ai = 0; aph ^= 1; }
      }
      if (!ok && pc.rank == 0) {
        drain_loads(bars->b_full, pend, pend_par, kBStages);
        drain_loads(bars->a_full, apend, apend_par, kAStages);
      }
    }
  } else if (warp == 1) {
    if (lane == 0 && pc.rank == 0) {
      int ai = 0, bi = 0, ci = 0;
      uint32_t aph = 0, bph = 0, cph = 0;
      const uint32_t tmem = bars->tmem_base;
      bool ok = true;
      for (int x = x_begin; ok && x < x_end;) {
        const Run w = next_run(plan, x, x_end, pair);
        x = w.x1;
        if (!wait_or_abort(&bars->a_full[ai], aph, bars, pc, err, 13)) { ok = false; break; }
        const uint32_t a_base = smem_u32(smem + kOffA + ai * kTileBytes);
        for (int b = w.b0; b < w.b1; ++b) {
          if (!wait_or_abort(&bars->b_full[bi], bph, bars, pc, err, 14)) { ok = false; break; }
          if (!wait_or_abort(&bars->acc_empty[ci], cph ^ 1, bars, pc, err, 15)) { ok = false; break; }
          tc_fence_after();
          issue_mma(tmem, ci, a_base, smem_u32(smem + kOffB + bi * kTileBytes));
          commit_pair(&bars->b_empty[bi]);
          commit_pair(&bars->acc_full[ci]);
          if (++bi == kBStages) { bi = 0; bph ^= 1; }
          if (++ci == 2) { ci = 0; cph ^= 1; }
        }
        if (!ok) break;
        commit_pair(&bars->a_empty[ai]);
        if (++ai == kAStages) { ai = 0; aph ^= 1; }
      }
    }
  } else {
    // Epilogue: warpgroup q reads the blocks of accumulator buffer q / 2 (every other block), its
    // columns (q % 2) * 128.. (keys of the block) for the CTA's 128 rows; warp w reads TMEM lanes
    // 32*(w%4)..
    const int q = (warp - 2) >> 2;
    const int own = q >> 1;                                  // accumulator buffer of this warpgroup
    const int col_base = (q & 1) * kSpan;
    const int quad = warp & 3;
    const int row = row_half + quad * 32 + lane;            // row of the 256-row pair
    const uint32_t lane_off = static_cast<uint32_t>(quad * 32) << 16;
    const uint32_t acc_empty_own = lead_addr(pc, bars, &bars->acc_empty[own]);
    const uint32_t tmem_q = bars->tmem_base + lane_off + own * 256 + col_base;
    const float c2 = plan.scale2;
    float2 *comb = reinterpret_cast<float2 *>(smem + kOffC);   // [2 parities][kEpiWG - 1 ranges][128 rows]
    uint32_t tile0 = 0, cph = 0, xph = 0;                   // tiles of the runs before; own buffer's phase
    bool ok = true;
    for (int x = x_begin; ok && x < x_end;) {
      const Run w = next_run(plan, x, x_end, pair);
      const SeqPlan &sp = plan.seq[w.s];
      x = w.x1;
      float m = -INFINITY, sum = 0.f;
      bool bad = false;
      // causal rows: this lane's row (token r of the query span) sees keys up to q_pos + r
      const int see = sp.q_pos + (w.qp * kChunk + row) / G;
      // the warpgroup's four 32-key mask words of a block (which keys count), one own block ahead;
      // the blocks alternate between the buffers
      const uint4 *mwords = reinterpret_cast<const uint4 *>(mask_words + sp.blk0 * 8) + (q & 1);
      const int b_first = w.b0 + ((own ^ tile0) & 1);
      tile0 += w.b1 - w.b0;
      uint4 m_next = b_first < w.b1 ? __ldg(mwords + b_first * 2) : make_uint4(0, 0, 0, 0);
      for (int b = b_first; b < w.b1; b += 2) {
        const uint4 mk = m_next;
        if (b + 2 < w.b1) m_next = __ldg(mwords + (b + 2) * 2);
        // the keys of this thread's words that count; and those this lane's row sees
        uint32_t rm[4] = {mk.x, mk.y, mk.z, mk.w};
        if (CAUSAL) {          // keys at local index <= see
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const int lim = see - (b * kBlock + col_base + 32 * i);
            rm[i] &= lim >= 31 ? 0xffffffffu : (lim < 0 ? 0u : (2u << lim) - 1u);
          }
        }
        if (!wait_or_abort(&bars->acc_full[own], cph, bars, pc, err, 16)) { ok = false; break; }
        cph ^= 1;
        tc_fence_after();
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const bool any = (h == 0 ? (mk.x | mk.y) : (mk.z | mk.w)) != 0u;   // uniform over the warp
          uint32_t rr[kCols];
          if (any) tmem_load_cols(tmem_q + h * kCols, rr);
          if (h == 1) {     // both halves are in registers: release the buffer
            tc_fence_before();
            __syncwarp();
            if (lane == 0) arrive_cluster(acc_empty_own);
          }
          if (any) online_block(rr, rm[2 * h], rm[2 * h + 1], c2, m, sum, bad);
        }
      }
      if (!ok) break;
      // the column ranges of each row combine in a fixed order (range 0 writes the pair's
      // partial of the row group; the merge combines the pairs' partials in pair order).  A
      // sum out of range travels as a negative sum: the CTA recomputes the partial at its end.
      if (bad) sum = -1.f;
      float2 *cb = comb + (xph & 1) * (kEpiWG - 1) * kRows;
      const int trow = quad * 32 + lane;
      if (q > 0) {
        if (!wait_or_abort(&bars->comb_empty[xph & 1], ((xph >> 1) & 1) ^ 1, bars, pc, err, 17)) break;
        cb[(q - 1) * kRows + trow] = make_float2(m, sum);
        __syncwarp();
        if (lane == 0) mbar_arrive(&bars->comb_full[xph & 1]);
      } else {
        if (!wait_or_abort(&bars->comb_full[xph & 1], (xph >> 1) & 1, bars, pc, err, 18)) break;
        float2 v[kEpiWG];
        v[0] = make_float2(m, sum);
#pragma unroll
        for (int i = 1; i < kEpiWG; ++i) v[i] = cb[(i - 1) * kRows + trow];
        __syncwarp();
        if (lane == 0) mbar_arrive(&bars->comb_empty[xph & 1]);
        float mm = v[0].x;
        bool flagged = v[0].y < 0.f;
#pragma unroll
        for (int i = 1; i < kEpiWG; ++i) {
          mm = fmaxf(mm, v[i].x);
          flagged |= v[i].y < 0.f;
        }
        float tot = 0.f;
        if (mm != -INFINITY) {
#pragma unroll
          for (int i = 0; i < kEpiWG; ++i)
            if (v[i].x != -INFINITY) tot += v[i].y * exp2f(v[i].x - mm);
        }
        if (flagged) tot = -1.f;
        const int rho = w.qp * kChunk + row;                  // linear row of the head group
        if (rho < G * sp.n_q) {
          const int r = rho / G, j = rho - r * G;
          part[(static_cast<size_t>(w.slot) * plan.total_qrows + sp.q_off + r) * plan.hq + w.g * G + j] =
              make_float2(mm, tot);
          if (flagged) bars->marked = 1;
        }
      }
      ++xph;
    }
  }
  finish_pair(bars, pc, warp, warp == 1 && lane == 0 && pc.rank == 0);
  // the epilogue's stores are visible to the whole CTA after finish_pair's barriers
  if (bars->marked && !bars->abort) repair_marked<CAUSAL>(plan, pair, row_half, mask_words, qp, k, k_stride, part);
}

// ------------------------------------------------------------------ repack
// Packed Q: for each sequence and KV head group g, rows rho = token * G + j hold
// query head g*G + j of that token (16-byte vectors, zero padding to 256 rows).
__global__ void q_pack_kernel(const __grid_constant__ ScorePlan plan, const uint4 *__restrict__ q,
                              uint4 *__restrict__ qp, int64_t row_begin, int64_t n_vec,
                              const uint8_t *__restrict__ modality, uint32_t *__restrict__ mask_words,
                              int64_t n_words, uint32_t *__restrict__ counters) {
  pdl_wait_and_release();
  const int64_t e = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
  if (e >= n_vec) {
    // pass 1's key masks: word c of block b of a sequence has bit k set when key 32c + k of the
    // block is in the sequence and counts in the denominator (in S; every key in the causal
    // domain, whose per-row limit the epilogue applies)
    const int64_t wd = e - n_vec;
    if (wd >= n_words) return;
    const int gb = static_cast<int>(wd >> 3), c = static_cast<int>(wd & 7);
    int s = 0;
    while (s + 1 < plan.nseq && plan.seq[s + 1].blk0 <= gb) ++s;
    const SeqPlan &sp = plan.seq[s];
    const int key0 = sp.t0 + (gb - sp.blk0) * kBlock + c * 32, t_end = sp.t0 + sp.len;
    uint32_t word = 0;
    for (int k = 0; k < 32; ++k) {
      const int key = key0 + k;
      if (key < t_end && (plan.causal || is_mm(modality[key]))) word |= 1u << k;
    }
    mask_words[wd] = word;
    if (c == 0 && plan.counted) counters[gb] = 0u;       // pass 2's count of the block's finished units
    return;
  }
  const int64_t prow = row_begin + e / 16;
  const int v = static_cast<int>(e % 16);
  int s = 0;
  while (s + 1 < plan.nseq && plan.seq[s + 1].qp_base <= prow) ++s;
  const SeqPlan &sp = plan.seq[s];
  const int local = static_cast<int>(prow - sp.qp_base);
  const int g = local / sp.rows_pad, rho = local - g * sp.rows_pad;
  const int G = plan.group;
  uint4 val = make_uint4(0, 0, 0, 0);
  if (rho < G * sp.n_q) {
    const int r = rho / G, j = rho - r * G;
    val = q[(static_cast<int64_t>(sp.q_off + r) * plan.hq + g * G + j) * 16 + v];
  }
  qp[prow * 16 + v] = val;
}

// ------------------------------------------------------------------ merge
// -lse2 of a packed query row (sequence, KV head group, rho), one thread per row (padding rows -inf, so
// that they add exp2(-inf) = 0).  The partials of the pair ranges that touched the row group (at most 32)
// are taken in pair order, kBatch of them loaded together: deterministic.
__device__ __forceinline__ float merged_nlse(const ScorePlan &plan, const float2 *__restrict__ part, int64_t prow) {
  int s = 0;
  while (s + 1 < plan.nseq && plan.seq[s + 1].qp_base <= prow) ++s;
  const SeqPlan &sp = plan.seq[s];
  const int G = plan.group;
  const int local = static_cast<int>(prow - sp.qp_base);
  const int g = local / sp.rows_pad, rho = local - g * sp.rows_pad;
  const bool real = rho < G * sp.n_q;
  const int r = rho / G, j = rho - r * G;
  // the pair ranges that touched this row group, one partial each
  const int x0 = sp.flat0 + (g * n_pairs(sp) + rho / kChunk) * sp.nb;
  const int np = sp.nb > 0 ? pair_of(x0 + sp.nb - 1, plan.pairs, plan.flat_total) -
                                 pair_of(x0, plan.pairs, plan.flat_total) + 1
                           : 0;
  float out = -INFINITY;
  if (real) {
    const float2 *p = part + static_cast<size_t>(sp.q_off + r) * plan.hq + g * G + j;
    const size_t stride = static_cast<size_t>(plan.total_qrows) * plan.hq;
    float m = -INFINITY, tot = 0.f;
    constexpr int kBatch = 8;
    for (int i0 = 0; i0 < np; i0 += kBatch) {
      float2 v[kBatch];
      float mn = m;
#pragma unroll
      for (int i = 0; i < kBatch; ++i) {
        v[i] = i0 + i < np ? p[(i0 + i) * stride] : make_float2(-INFINITY, 0.f);
        mn = fmaxf(mn, v[i].x);
      }
      if (m != -INFINITY) tot *= exp2f(m - mn);
#pragma unroll
      for (int i = 0; i < kBatch; ++i) {
        if (v[i].x != -INFINITY) tot += v[i].y * exp2f(v[i].x - mn);
      }
      m = mn;
    }
    out = m == -INFINITY ? INFINITY : -(m + log2f(tot));   // no key at all (S empty): nothing is scored
  }
  return out;
}

// The merge as a kernel of its own.  Bound by latency: one or two L2 round trips.  A warp per row, one
// partial per lane, took 25 us for 68,608 rows; this takes 4.8 us.
__global__ void __launch_bounds__(kMergeThreads)
    lse_merge_kernel(const __grid_constant__ ScorePlan plan, const float2 *__restrict__ part,
                     float *__restrict__ nlse2, int64_t row_begin) {
  pdl_wait_and_release();
  // the rows of a launch are a multiple of 256: whole CTAs
  const int64_t prow = row_begin + blockIdx.x * static_cast<int64_t>(kMergeThreads) + threadIdx.x;
  nlse2[prow] = merged_nlse(plan, part, prow);
}

// ------------------------------------------------------------------ pass 2
struct Unit2 {
  int s, kp, g;            // sequence, key block, first KV head group (plan.unit_groups of them)
};

__device__ __forceinline__ Unit2 decode_unit2(const ScorePlan &p, int u) {
  Unit2 w;
  int s = 0;
  while (s + 1 < p.nseq && p.seq[s + 1].unit_begin <= u) ++s;
  w.s = s;
  const int local = u - p.seq[s].unit_begin;
  w.g = 0;
  w.kp = local;
  if (p.unit_groups == 1) {
    w.kp = local / p.hkv;
    w.g = local - w.kp * p.hkv;
  }
  return w;
}

// a[0..3] += 2^(x c2 + nl[col]) over the columns of one load (four independent partial sums).
__device__ __forceinline__ void colsum_word(uint32_t (&r)[kCols2], const float *nl, float c2, float2 (&a)[4]) {
  exp_sum(r, c2, [&](int i) { return *reinterpret_cast<const float2 *>(nl + i); }, a);
}

// The same over the columns i >= first only (causal rows that cannot see the key drop out;
// taken only by keys inside the query span).
__device__ __forceinline__ void colsum_word_from(const uint32_t (&r)[kCols2], const float *nl, float c2, int first,
                                                 float2 (&a)[4]) {
#pragma unroll
  for (int i = 0; i < 32; ++i)
    if (i >= first) a[i & 3].x += ex2_approx(fmaf(__uint_as_float(r[i]), c2, nl[i]));
}

// Work unit = (256 keys, KV head group g) or (256 keys, every group): 128 keys per CTA of the pair.
// A unit of every group writes its keys' scores.  A unit of one group writes the group's sums to
// gsum[g][key]; with counters the last of a key block's units then adds the groups (every warp for its
// 32 keys), without them the final kernel does.
// MERGE (at most one unit per pair): there is no merge kernel; the epilogue warps merge the unit's rows
// into shared memory while the tiles load and the first MMA runs.  A launch less in a chain of dependent
// launches: 28/4 heads, 64 query rows, 1,298 keys 16.5 -> 15.0 us, 2,600 keys 18.2 -> 16.7 us; four
// sequences of 600 keys 19.6 -> 17.4 us.
template <bool CAUSAL, bool MERGE>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreads, 1)
    score_colsum_kernel(const __grid_constant__ CUtensorMap qmap, const __grid_constant__ CUtensorMap kmap,
                        const __grid_constant__ ScorePlan plan, const float *__restrict__ nlse2, const float2 *__restrict__ part, float *gsum,
                        uint32_t *counters, const uint8_t *__restrict__ modality, float *__restrict__ scores,
                        DeviceError *err) {
  extern __shared__ __align__(1024) uint8_t smem[];
  if (!smem_aligned(smem)) {   // the same in both CTAs of the pair: both leave here
    if (threadIdx.x == 0) raise_device_error(err, APACK_EDEVICE, 10);
    return;
  }
  Bars *bars = reinterpret_cast<Bars *>(smem + kOffBars);
  float *lse_s = reinterpret_cast<float *>(smem + kOffL);   // [4][256] by B stage; MERGE: by chunk of the unit
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const PairCtx pc = init_pair(smem, bars, warp);
  pdl_wait_and_release();      // the set-up runs beside the previous launch
  const int G = plan.group;
  const int pair = blockIdx.x >> 1, npairs = gridDim.x >> 1;
  const int row_half = static_cast<int>(pc.rank) * kRows;   // this CTA's keys of a unit, rows of a chunk

  if (warp == 0) {
    if (lane == 0) {
      tma_prefetch_desc(&qmap);
      tma_prefetch_desc(&kmap);
      int ai = 0, bi = 0;
      uint32_t aph = 0, bph = 0;
      bool pend[kBStages] = {}, apend[kAStages] = {};
      uint32_t pend_par[kBStages] = {}, apend_par[kAStages] = {};
      bool ok = true;
      for (int u = pair; ok && u < plan.total_units; u += npairs) {
        const Unit2 w = decode_unit2(plan, u);
        const SeqPlan &sp = plan.seq[w.s];
        const int nch = sp.rows_pad / kChunk;
        if (nch == 0) continue;
        for (int g = w.g; ok && g < w.g + plan.unit_groups; ++g) {
          if (!wait_or_abort(&bars->a_empty[ai], aph ^ 1, bars, pc, err, 21)) { ok = false; break; }
          uint8_t *A = smem + kOffA + ai * kTileBytes;
          if (pc.rank == 0) mbar_arrive_expect_tx(&bars->a_full[ai], 2 * kTileBytes);
          const uint32_t afull = lead_addr(pc, bars, &bars->a_full[ai]);
          const int key0 = sp.t0 + w.kp * kBlock + row_half;
          tma_load_3d_pair(A, &kmap, afull, 0, g, key0);
          tma_load_3d_pair(A + kHalf, &kmap, afull, 64, g, key0);
          apend[ai] = true;
          apend_par[ai] = aph;
          for (int c = 0; c < nch; ++c) {
            if (!wait_or_abort(&bars->b_empty[bi], bph ^ 1, bars, pc, err, 22)) { ok = false; break; }
            // normaliser slot bi is free once this CTA's epilogue of the chunk that used it is done
            if (!MERGE && !wait_or_abort(&bars->l_empty[bi], bph ^ 1, bars, pc, err, 29)) { ok = false; break; }
            const int64_t row0 = static_cast<int64_t>(sp.qp_base) + g * sp.rows_pad + c * kChunk;
            if (!MERGE) {
              mbar_arrive_expect_tx(&bars->l_full[bi], kChunk * sizeof(float));
              bulk_load(lse_s + bi * kChunk, nlse2 + row0, kChunk * sizeof(float), &bars->l_full[bi]);
            }
            uint8_t *B = smem + kOffB + bi * kTileBytes;
            if (pc.rank == 0) mbar_arrive_expect_tx(&bars->b_full[bi], 2 * kTileBytes);
            const uint32_t bfull = lead_addr(pc, bars, &bars->b_full[bi]);
            tma_load_3d_pair(B, &qmap, bfull, 0, 0, static_cast<int32_t>(row0) + row_half);
            tma_load_3d_pair(B + kHalf, &qmap, bfull, 64, 0, static_cast<int32_t>(row0) + row_half);
            pend[bi] = true;
            pend_par[bi] = bph;
            if (++bi == kBStages) { bi = 0; bph ^= 1; }
          }
          if (++ai == kAStages) { ai = 0; aph ^= 1; }
        }
      }
      if (!ok) {
        // this CTA's normaliser copies complete on its own barriers
        if (!MERGE) drain_loads(bars->l_full, pend, pend_par, kBStages);
        if (pc.rank == 0) {
          drain_loads(bars->b_full, pend, pend_par, kBStages);
          drain_loads(bars->a_full, apend, apend_par, kAStages);
        }
      }
    }
  } else if (warp == 1) {
    if (lane == 0 && pc.rank == 0) {
      int ai = 0, bi = 0, ci = 0;
      uint32_t aph = 0, bph = 0, cph = 0;
      const uint32_t tmem = bars->tmem_base;
      bool ok = true;
      for (int u = pair; ok && u < plan.total_units; u += npairs) {
        const Unit2 w = decode_unit2(plan, u);
        const int nch = plan.seq[w.s].rows_pad / kChunk;
        if (nch == 0) continue;
        for (int g = 0; ok && g < plan.unit_groups; ++g) {
          if (!wait_or_abort(&bars->a_full[ai], aph, bars, pc, err, 23)) { ok = false; break; }
          const uint32_t a_base = smem_u32(smem + kOffA + ai * kTileBytes);
          for (int c = 0; c < nch; ++c) {
            if (!wait_or_abort(&bars->b_full[bi], bph, bars, pc, err, 24)) { ok = false; break; }
            if (!wait_or_abort(&bars->acc_empty[ci], cph ^ 1, bars, pc, err, 25)) { ok = false; break; }
            tc_fence_after();
            issue_mma(tmem, ci, a_base, smem_u32(smem + kOffB + bi * kTileBytes));
            commit_pair(&bars->b_empty[bi]);
            commit_pair(&bars->acc_full[ci]);
            if (++bi == kBStages) { bi = 0; bph ^= 1; }
            if (++ci == 2) { ci = 0; cph ^= 1; }
          }
          if (!ok) break;
          commit_pair(&bars->a_empty[ai]);
          if (++ai == kAStages) { ai = 0; aph ^= 1; }
        }
      }
    }
  } else {
    // Epilogue: warpgroup q reads the chunks of accumulator buffer q / 2 (every other chunk), its
    // columns (q % 2) * 128.. (rows of the chunk); one key per thread.
    const int q = (warp - 2) >> 2;
    const int own = q >> 1;                                  // accumulator buffer of this warpgroup
    const int col_base = (q & 1) * kSpan;
    const int quad = warp & 3;
    const int tkey = quad * 32 + lane;
    const int klane = row_half + tkey;                  // key of the 256-key unit
    const uint32_t lane_off = static_cast<uint32_t>(quad * 32) << 16;
    const uint32_t acc_empty_own = lead_addr(pc, bars, &bars->acc_empty[own]);
    const uint32_t tmem_q = bars->tmem_base + lane_off + own * 256 + col_base;
    const float c2 = plan.scale2;
    float *comb = reinterpret_cast<float *>(smem + kOffC);   // [2 parities][kEpiWG - 1 ranges][128 keys]
    uint32_t tile0 = 0, cph = 0, xph = 0;                   // chunks of the units before; own buffer's phase
    bool ok = true;
    for (int u = pair; ok && u < plan.total_units; u += npairs) {
      const Unit2 w = decode_unit2(plan, u);
      const SeqPlan &sp = plan.seq[w.s];
      const int nch = sp.rows_pad / kChunk;
      if (nch == 0) continue;
      // causal rows: only packed rows rho >= rho_min (tokens r >= key - q_pos) see this key
      const int rho_min = CAUSAL ? max(0, w.kp * kBlock + klane - sp.q_pos) * G : 0;
      if (MERGE) {                                          // the pair's only unit
        const int64_t row0 = static_cast<int64_t>(sp.qp_base) + w.g * sp.rows_pad;
        for (int i = threadIdx.x - 64; i < plan.unit_groups * sp.rows_pad; i += 32 * kEpiWarps)
          lse_s[i] = merged_nlse(plan, part, row0 + i);
        asm volatile("bar.sync 1, %0;" ::"n"(32 * kEpiWarps) : "memory");
      }
      float mine = 0.f;                                     // the groups' sums, in group order
      for (int g = 0; ok && g < plan.unit_groups; ++g) {
        float2 a[4] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
        // chunks alternate between the buffers; normaliser slot = chunk % kBStages, an even number
        for (int c = (own ^ tile0) & 1; c < nch; c += 2) {
          const uint32_t t = tile0 + c, li = MERGE ? t : t % kBStages;
          if (!MERGE && !wait_or_abort(&bars->l_full[li], (t / kBStages) & 1, bars, pc, err, 30)) { ok = false; break; }
          if (!wait_or_abort(&bars->acc_full[own], cph, bars, pc, err, 26)) { ok = false; break; }
          cph ^= 1;
          tc_fence_after();
#pragma unroll
          for (int h = 0; h < kSpan / kCols2; ++h) {
            const int col0 = col_base + h * kCols2;
            const float *nl = lse_s + li * kChunk + col0;
            uint32_t rr[kCols2];
            tmem_load_cols(tmem_q + h * kCols2, rr);
            if (h == kSpan / kCols2 - 1) {     // every column is in registers: release the buffer
              tc_fence_before();
              __syncwarp();
              if (lane == 0) arrive_cluster(acc_empty_own);
            }
            const int first = rho_min - (c * kChunk + col0);
            if (!CAUSAL || first <= 0)
              colsum_word(rr, nl, c2, a);
            else if (first < kCols2)
              colsum_word_from(rr, nl, c2, first, a);
          }
          __syncwarp();
          if (!MERGE && lane == 0) mbar_arrive(&bars->l_empty[li]);
        }
        tile0 += nch;
        const float2 s01 = fadd2(a[0], a[1]), s23 = fadd2(a[2], a[3]);
        const float2 s4 = fadd2(s01, s23);
        mine += s4.x + s4.y;
      }
      if (!ok) break;
      float *cb = comb + (xph & 1) * (kEpiWG - 1) * kRows;
      if (q < kEpiWG - 1) {
        if (!wait_or_abort(&bars->comb_empty[xph & 1], ((xph >> 1) & 1) ^ 1, bars, pc, err, 27)) break;
        cb[q * kRows + tkey] = mine;
        __syncwarp();
        if (lane == 0) mbar_arrive(&bars->comb_full[xph & 1]);
      } else {
        if (!wait_or_abort(&bars->comb_full[xph & 1], (xph >> 1) & 1, bars, pc, err, 28)) break;
        float tot = cb[tkey];
#pragma unroll
        for (int i = 1; i < kEpiWG - 1; ++i) tot += cb[i * kRows + tkey];   // fixed order
        tot += mine;
        __syncwarp();
        if (lane == 0) mbar_arrive(&bars->comb_empty[xph & 1]);
        const int key = sp.t0 + w.kp * kBlock + klane;
        const bool in = key < sp.t0 + sp.len;
        const float rows = static_cast<float>(plan.hq * sp.n_q);
        if (plan.direct) {
          if (in) scores[key] = is_mm(modality[key]) ? tot / rows : 0.f;
        } else {
          if (in) gsum[static_cast<int64_t>(w.g) * plan.total_tokens + key] = tot;
          if (plan.counted) {
            __threadfence();
            __syncwarp();
            const int shift = 4 * (static_cast<int>(pc.rank) * 4 + quad);   // this warp's 32 keys of the block
            uint32_t before = 0;
            if (lane == 0) before = atomicAdd(counters + sp.blk0 + w.kp, 1u << shift);
            before = (__shfl_sync(0xffffffffu, before, 0) >> shift) & 15u;
            if (before == static_cast<uint32_t>(plan.hkv - 1)) {
              __threadfence();
              if (in) {
                float acc = 0.f;
                for (int g = 0; g < plan.hkv; ++g) acc += __ldcg(gsum + static_cast<int64_t>(g) * plan.total_tokens + key);
                scores[key] = is_mm(modality[key]) ? acc / rows : 0.f;
              }
            }
          }
        }
      }
      ++xph;
    }
  }
  finish_pair(bars, pc, warp, warp == 1 && lane == 0 && pc.rank == 0);
}

// ------------------------------------------------------------------ final
// I_i = (sum over KV head groups, in order) / (Hq n_q) for tokens of S, 0 otherwise.
__global__ void score_finalize_kernel(const __grid_constant__ ScorePlan plan, const uint8_t *__restrict__ modality,
                                      const float *__restrict__ gsum, float *__restrict__ scores, int64_t t_begin,
                                      int64_t n) {
  pdl_wait_and_release();
  const int64_t e = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
  if (e >= n) return;
  const int64_t i = t_begin + e;
  int s = 0;
  while (s + 1 < plan.nseq && plan.seq[s + 1].t0 <= i) ++s;
  const SeqPlan &sp = plan.seq[s];
  float out = 0.f;
  if (sp.n_q > 0 && is_mm(modality[i])) {
    float acc = 0.f;
    for (int g = 0; g < plan.hkv; ++g) acc += gsum[static_cast<int64_t>(g) * plan.total_tokens + i];
    out = acc / static_cast<float>(plan.hq * sp.n_q);
  }
  scores[i] = out;
}

// ------------------------------------------------------------------ host side
using EncodeTiledFn = CUresult (*)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                   const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                   CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
  // looked up once, by a thread-safe static initialiser (the entry point is the same on every device)
  static const EncodeTiledFn fn = [] {
    void *p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      return reinterpret_cast<EncodeTiledFn>(p);
    return static_cast<EncodeTiledFn>(nullptr);
  }();
  return fn;
}

// 3-D bf16 map: dims {128, mid, rows}, byte strides {mid_stride, row_stride}, box {64, box_mid, box_rows}.
bool make_map(CUtensorMap *map, const void *base, uint64_t mid, uint64_t rows, uint64_t mid_stride,
              uint64_t row_stride, uint32_t box_mid, uint32_t box_rows) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  cuuint64_t dims[3] = {128, mid, rows};
  cuuint64_t strides[2] = {mid_stride, row_stride};
  cuuint32_t box[3] = {64, box_mid, box_rows};
  cuuint32_t estr[3] = {1, 1, 1};
  return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void *>(base), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

std::atomic<uint64_t> g_attr_done{0};
std::atomic<int> g_max_pairs[64];   // per device: CTA pairs that can be resident at once (0 = not probed)

// CTA pairs of the scoring kernels that fit the device at once (one CTA per SM).
int max_resident_pairs() {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0) return 1;
  if (dev < 64) {
    const int cached = g_max_pairs[dev].load(std::memory_order_relaxed);
    if (cached > 0) return cached;
  }
  int n = 0;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(2 * (device_sm_count() / 2), 1, 1);
  cfg.blockDim = dim3(kThreads, 1, 1);
  cfg.dynamicSmemBytes = kSmemBytes;
  // the kernels declare their cluster shape (__cluster_dims__), so the configuration leaves it out
  if (cudaOccupancyMaxActiveClusters(&n, score_colsum_kernel<false, false>, &cfg) != cudaSuccess || n <= 0) {
    cudaGetLastError();
    n = device_sm_count() / 2;
  }
  if (n > device_sm_count() / 2) n = device_sm_count() / 2;
  if (n < 1) n = 1;
  if (dev < 64) g_max_pairs[dev].store(n, std::memory_order_relaxed);
  return n;
}

}  // namespace

bool make_kv_tile_map(CUtensorMap *map, const void *k, int hkv, int64_t tokens, int64_t token_stride,
                      uint32_t box_tokens) {
  return make_map(map, k, static_cast<uint64_t>(hkv), static_cast<uint64_t>(tokens), 256,
                  static_cast<uint64_t>(token_stride), 1, box_tokens);
}

apack_status run_score(const apack_seqs *seqs, const void *q, const void *k, int64_t k_token_stride,
                       float *scores, void *ws, cudaStream_t stream) {
  int64_t T = 0, NQ = 0;
  apack_status st = validate_seqs(seqs, &T, &NQ);
  if (st != APACK_OK) return st;
  if (!q || !k || !scores || !ws) return APACK_EINVAL;
  if ((reinterpret_cast<uintptr_t>(q) & 15) || (reinterpret_cast<uintptr_t>(k) & 15) || (k_token_stride & 15) ||
      k_token_stride < static_cast<int64_t>(seqs->num_kv_heads) * 256)
    return APACK_EINVAL;
  const int B = seqs->num_seqs;
  const int hq = seqs->num_q_heads, hkv = seqs->num_kv_heads, G = hq / hkv;
  if (hkv > 256) return APACK_EUNSUPPORTED;
  if (T == 0) return APACK_OK;
  // few query rows per head group (e.g. the last query token only): K-read-bound path
  if (narrow_score_applies(seqs)) return run_score_narrow(seqs, q, k, k_token_stride, scores, ws, stream);
  const WsLayout L = workspace_layout(seqs);
  uint8_t *wsb = static_cast<uint8_t *>(ws);
  DeviceError *err = reinterpret_cast<DeviceError *>(wsb + L.err_off);
  float2 *part = reinterpret_cast<float2 *>(wsb + L.part_off);
  float *nlse2 = reinterpret_cast<float *>(wsb + L.lse_off);
  uint8_t *qp = wsb + L.qp_off;
  float *gsum = reinterpret_cast<float *>(wsb + L.gsum_off);
  uint32_t *mask_words = reinterpret_cast<uint32_t *>(wsb + L.mask_off);
  uint32_t *counters = reinterpret_cast<uint32_t *>(wsb + kCounterOff);

  if (once_per_device(g_attr_done, [] {
        cudaError_t e = cudaFuncSetAttribute(score_rowstats_kernel<false>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes);
        if (e == cudaSuccess)
          e = cudaFuncSetAttribute(score_rowstats_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   kSmemBytes);
        for (auto *f : {score_colsum_kernel<false, false>, score_colsum_kernel<true, false>,
                        score_colsum_kernel<false, true>, score_colsum_kernel<true, true>})
          if (e == cudaSuccess) e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes);
        return e;
      }) != cudaSuccess)
    return APACK_ECUDA;
  CUtensorMap qmap, kmap;
  const uint64_t qp_rows = static_cast<uint64_t>(L.qp_rows > 0 ? L.qp_rows : 256);
  // every operand tile is 128 rows (of packed Q or of one KV head's keys) per CTA
  if (!make_map(&qmap, qp, 1, qp_rows, 256, 256, 1, kRows) || !make_map(&kmap, k, hkv, T, 256, k_token_stride, 1, kRows))
    return APACK_ECUDA;

  const int max_pairs = max_resident_pairs();
  int64_t qp_base = 0;
  for (int s0 = 0; s0 < B; s0 += kSeqsPerLaunch) {
    const int ns = (B - s0 < kSeqsPerLaunch) ? (B - s0) : kSeqsPerLaunch;
    ScorePlan P{};
    P.nseq = ns;
    P.hq = hq;
    P.hkv = hkv;
    P.group = G;
    P.total_qrows = static_cast<int32_t>(NQ);
    P.total_tokens = static_cast<int32_t>(T);
    P.scale2 = kScale2Tc;
    P.causal = seqs->softmax_domain == APACK_SOFTMAX_CAUSAL_ROW;
    int64_t qrows = 0, flat = 0, nb_max = 0;
    int64_t chunks2 = 0;       // pass 2: (key block, query chunk) products of one head group
    int blocks = 0;
    bool unscored = false;     // a sequence without query rows: its scores are zeros that no unit writes
    for (int i = 0; i < ns; ++i) {
      const int b = s0 + i;
      SeqPlan &sp = P.seq[i];
      sp.t0 = seqs->cu_seqlens_h[b];
      sp.len = seqs->cu_seqlens_h[b + 1] - sp.t0;
      sp.q_off = seqs->cu_qlens_h[b];
      sp.n_q = seqs->cu_qlens_h[b + 1] - sp.q_off;
      sp.rows_pad = ((G * sp.n_q + kChunk - 1) / kChunk) * kChunk;
      sp.qp_base = static_cast<int32_t>(qp_base + qrows);
      qrows += static_cast<int64_t>(hkv) * sp.rows_pad;
      sp.nb = sp.n_q > 0 ? (sp.len + kBlock - 1) / kBlock : 0;
      sp.q_pos = query_position(seqs, b);
      sp.flat0 = static_cast<int32_t>(flat);
      sp.blk0 = blocks;
      blocks += sp.nb;
      flat += pass1_items(sp, hkv);
      if (sp.nb > nb_max) nb_max = sp.nb;
      if (sp.rows_pad > 0) chunks2 += static_cast<int64_t>((sp.len + kBlock - 1) / kBlock) * (sp.rows_pad / kChunk);
      if (sp.rows_pad == 0 && sp.len > 0) unscored = true;
    }
    // Pass 1: equal ranges of the flat (row group, key block) items per pair; a range must stay at
    // least ceil(nb_max / (kPairSlots - 1)) items long so that a row group meets at most kPairSlots
    // pairs (its partial slots).
    if (flat >= (int64_t{1} << 31) - 1) return APACK_EUNSUPPORTED;   // flat indices are 32-bit on the device
    P.flat_total = static_cast<int32_t>(flat);
    int64_t pairs1 = max_pairs;
    if (flat > 0) {
      const int64_t min_len = (nb_max + kPairSlots - 2) / (kPairSlots - 1);
      if (pairs1 > flat / min_len) pairs1 = flat / min_len;
      if (pairs1 < 1) pairs1 = 1;
    }
    P.pairs = static_cast<int32_t>(pairs1);
    // Pass 2: units of one head group, or of every group, which saves the group sums' round trip and the
    // hand-over between the warpgroups once per group (about a chunk's time), as long as the longer units
    // do not leave pairs idle in the last round.  10 minutes, 256 query rows (529 blocks, 7 chunks):
    // 28 (7 + 1) = 224 chunk times against 7 (28 + 1) = 203; 2 minutes, 128 rows: 30 against 34.
    const int64_t chunks_avg = blocks > 0 ? (chunks2 + blocks - 1) / blocks : 0;
    const int64_t rounds1 = (static_cast<int64_t>(blocks) * hkv + max_pairs - 1) / max_pairs;
    const int64_t rounds_all = (blocks + max_pairs - 1) / max_pairs;
    const bool all_groups = hkv > 1 && !unscored && rounds_all * (hkv * chunks_avg + 1) <= rounds1 * (chunks_avg + 1);
    P.unit_groups = all_groups ? hkv : 1;
    P.direct = all_groups || (hkv == 1 && !unscored);
    // The count and the re-read take about 2 us of a warpgroup, which is what the final kernel takes:
    // hidden neither way, but a launch saved, when every pair has one unit; with more units per pair it
    // would hold each of them up (two-minute schedule: 499 us with the kernel, 515 us counted).
    P.counted = !P.direct && !unscored && static_cast<int64_t>(blocks) * hkv <= max_pairs && blocks <= kMaxCounted &&
                hkv <= kMaxCountedGroups;
    const bool final_kernel = !P.direct && !P.counted;
    int units2 = 0;
    for (int i = 0; i < ns; ++i) {
      SeqPlan &sp = P.seq[i];
      sp.unit_begin = units2;
      if (sp.rows_pad > 0) units2 += sp.nb * (all_groups ? 1 : hkv);
    }
    // repack the query rows of this launch's sequences, write pass 1's key masks and zero the counters
    const int64_t n_words = static_cast<int64_t>(blocks) * (kBlock / 32);
    if (qrows > 0) {
      const int64_t n_vec = qrows * 16;
      if (check_cuda(launch_pdl(q_pack_kernel, dim3(static_cast<unsigned>((n_vec + n_words + 255) / 256)), dim3(256), 0,
                                stream, P, static_cast<const uint4 *>(q), reinterpret_cast<uint4 *>(qp), qp_base, n_vec,
                                seqs->modality, mask_words, n_words, counters)) != APACK_OK)
        return APACK_ECUDA;
      count_launches(1);
    }
    if (flat > 0) {
      const cudaError_t e = launch_pdl(P.causal ? score_rowstats_kernel<true> : score_rowstats_kernel<false>,
                                       dim3(static_cast<unsigned>(2 * pairs1)), dim3(kThreads), kSmemBytes, stream, qmap,
                                       kmap, P, mask_words, reinterpret_cast<const uint4 *>(qp),
                                       static_cast<const uint8_t *>(k), k_token_stride, part, err);
      count_launches(1);
      if (check_cuda(e) != APACK_OK) return APACK_ECUDA;
    }
    // Pass 2 merges the row statistics by itself where each pair has one unit, the unit's chunks fit its
    // normaliser slots, and the rows and partials that all units read again are few (kMergeInside).
    int64_t tiles_max = 0;
    for (int i = 0; i < ns; ++i) tiles_max = std::max<int64_t>(tiles_max, P.unit_groups * (P.seq[i].rows_pad / kChunk));
    const int64_t parts_max = flat > 0 ? (nb_max - 1) / (flat / pairs1) + 2 : 0;
    const bool merge_inside = units2 <= max_pairs && tiles_max <= kBStages && tiles_max * kChunk * parts_max <= kMergeInside;
    if (qrows > 0 && !merge_inside) {
      const cudaError_t e = launch_pdl(lse_merge_kernel, dim3(static_cast<unsigned>(qrows / kMergeThreads)),
                                       dim3(kMergeThreads), 0, stream, P, part, nlse2, qp_base);
      count_launches(1);
      if (check_cuda(e) != APACK_OK) return APACK_ECUDA;
    }
    // Pass 2 units are dealt round-robin to the pairs.
    P.total_units = units2;
    if (units2 > 0) {
      const int pairs2 = units2 < max_pairs ? units2 : max_pairs;
      auto *colsum = merge_inside ? (P.causal ? score_colsum_kernel<true, true> : score_colsum_kernel<false, true>)
                                  : (P.causal ? score_colsum_kernel<true, false> : score_colsum_kernel<false, false>);
      const cudaError_t e = launch_pdl(colsum, dim3(static_cast<unsigned>(2 * pairs2)), dim3(kThreads), kSmemBytes,
                                       stream, qmap, kmap, P, nlse2, part, gsum, counters, seqs->modality, scores, err);
      count_launches(1);
      if (check_cuda(e) != APACK_OK) return APACK_ECUDA;
    }
    const int64_t t_begin = P.seq[0].t0;
    const int64_t n_tok = static_cast<int64_t>(P.seq[ns - 1].t0) + P.seq[ns - 1].len - t_begin;
    if (n_tok > 0 && final_kernel) {
      const float *gs = gsum;
      if (check_cuda(launch_pdl(score_finalize_kernel, dim3(static_cast<unsigned>((n_tok + 255) / 256)), dim3(256), 0,
                                stream, P, static_cast<const uint8_t *>(seqs->modality), gs, scores, t_begin,
                                n_tok)) != APACK_OK)
        return APACK_ECUDA;
      count_launches(1);
    }
    qp_base += qrows;
  }
  return APACK_OK;
}

}  // namespace apack
