// select.cu -- per-(sequence, modality) top-k of Eq. inner (Sec. 3.2) and the stable keep map.
//
// One thread-block cluster of CL CTAs per sequence (1, 4, 8 or 16 by its length); CTA c owns a
// contiguous slice of the sequence's tokens, each of its 32 warps a contiguous run of the slice.  The
// slice (bit patterns and modality codes) is read from global memory once into shared memory when it
// fits (kMaxCached tokens); a thread only reads back what it wrote itself.
//
//  1. The k-th largest score of every segment.  Scores are >= 0, so the order of their IEEE bit
//     patterns as unsigned integers is their numeric order.  A level cuts the range of bit patterns
//     that still holds the k-th score into 2048 equal bins, counts the tokens per bin and keeps the
//     bin that holds it; the first range is that of the segment's scores themselves, so that the bins
//     lie where the scores are (a fixed first digit puts most of them into a few bins, whose counting
//     is serial).  Each CTA counts in its shared memory and adds its non-zero bins into the bins'
//     owner CTAs (distributed shared memory); after one cluster barrier every CTA reads the sums back
//     and derives the same bin.  Once at most kGather tokens are left (usually after one level), every
//     CTA collects them all (one more barrier) and finishes by itself: it ranks them against one
//     another, or, above kRank of them, goes on with levels of its own.  The result per segment is a
//     threshold bit pattern T and a quota q: keep every score > T and the first q scores == T in token
//     order (ties go to the lower index).
//  2. Counts per warp run and per CTA (kept for sure, == T per segment) are exchanged through
//     distributed shared memory, so that each warp knows its output offset and how many ties precede it.
//  3. Each warp walks its run in token order (ballot prefix counts give the positions) and writes
//     keep_idx (ascending), the compacted modality and dst_of_src.
//
// Bound by latency: the launch, the token loads, and a chain of block and cluster barriers; then by
// issue, one SM working through its slice about five times.  The loops over the tokens stay rolled:
// unrolled over tokens in registers they ran out of the instruction cache (per modality, 2,000 tokens:
// 9.5 us against 6.0).  Four fixed 8-bit digits with a histogram exchange each took 25.3 us jointly
// over 135,000 tokens and 9.2 us over 1,000, on clusters of 16 and 8; this takes 17.3 and 4.4 us.

#include "internal.cuh"
#include "ptx.cuh"

namespace apack {

namespace {

constexpr int kThreads = 1024;
constexpr int kWarps = kThreads / 32;
static_assert(kWarps == 32, "the keep-offset scan gives one lane to each warp of a CTA");
constexpr int kBins = 2048;                     // per segment: four per thread of half the CTA
static_assert(2 * kBins == 4 * kThreads, "one uint4 of the two segments' bins per thread");
constexpr int kBatch = 12;                      // a thread's tokens loaded together
constexpr int kMaxCached = 36864;               // tokens per CTA slice cached in shared memory (180 KB)
constexpr int kGather = 2 * kThreads;           // candidates a CTA finishes by itself: two per thread
constexpr int kRank = 256;                      // candidates ranked against one another
constexpr uint32_t kFirstSpan = (1u << 28) - 1; // the first level resolves 32 binades below the largest score

struct SelSeq {
  int32_t t0, len;
  int32_t out_base, out_len;   // host-computed output offset and kept count
  int32_t n_seg[2];            // host counts per segment
  int32_t k[2];                // keep counts per segment
};

struct SelectPlan {
  int32_t nseq;
  int32_t write_cu0;           // write new_cu_seqlens[0] = 0 (first launch of a batch)
  int32_t seq_base;            // index of seq[0] in the batch
  int32_t cache_tokens;        // slice tokens the dynamic shared memory holds (0: no cache)
  SelSeq seq[kSeqsPerLaunch];
};

__device__ __forceinline__ uint32_t warp_incl_scan(uint32_t v, int lane) {
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, v, off);
    if (lane >= off) v += y;
  }
  return v;
}

// The range of bit patterns that still holds a segment's k-th largest score, as offsets below the
// segment's largest pattern: [o0, o0 + span], `krem` = the rank of the k-th score within it.
struct Range {
  uint32_t top, o0, span, krem;
  uint32_t count;              // tokens in the range (once a level has counted them)
  int shift;                   // this level's bin width, log2
  bool act;                    // still wider than one pattern
};

__device__ __forceinline__ int level_shift(uint32_t span) {
  const int nb = 32 - __clz(static_cast<int>(span));
  return nb > 11 ? nb - 11 : 0;
}

__device__ __forceinline__ int bin_of(const Range &g, uint32_t off) {
  const uint32_t rel = off - g.o0;               // below the range: wraps to above the span
  return rel <= g.span ? static_cast<int>(min(rel >> g.shift, static_cast<uint32_t>(kBins - 1))) : -1;
}

// CL: CTAs of the sequence's cluster.  NSEG: segments (2 per modality, 1 joint).
template <int CL, int NSEG>
__global__ void __cluster_dims__(CL, 1, 1) __launch_bounds__(kThreads, 1)
    select_kernel(const __grid_constant__ SelectPlan plan, const float *__restrict__ scores,
                  const uint8_t *__restrict__ modality, int32_t *__restrict__ keep_idx,
                  uint8_t *__restrict__ modality_out, int32_t *__restrict__ dst_of_src,
                  int32_t *__restrict__ new_cu, DeviceError *err) {
  constexpr int kOwned = CL > 1 ? 2 * kBins / CL : 4;   // summed bins owned by a CTA
  __shared__ __align__(16) uint32_t hist[2 * kBins];
  __shared__ __align__(16) uint32_t sums[3][kOwned];    // levels rotate over three buffers
  __shared__ uint32_t list[kGather];                    // this CTA's candidates
  __shared__ __align__(16) uint32_t rank_of[kRank];     // every CTA's, when they are ranked
  __shared__ uint32_t lcnt;
  __shared__ __align__(16) uint32_t range_s[4];         // this CTA's max, ~min per segment
  __shared__ uint32_t wrange[kWarps][4];
  __shared__ uint32_t wtot[kWarps];
  __shared__ uint32_t res[2][4];                        // per segment: found, bin, count above, count of the bin
  __shared__ uint32_t st_total[2];
  __shared__ uint32_t wcnt[kWarps][3];                  // per warp run: kept for sure, == T0, == T1
  __shared__ uint32_t cnt[3];                           // per CTA (read by the cluster)
  __shared__ uint32_t wbase[kWarps], weqb[kWarps][2];
  extern __shared__ __align__(16) uint8_t cache_raw[];  // the slice: bit patterns, then modality codes
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  // zero the counters beside the previous launch
  reinterpret_cast<uint4 *>(hist)[tid] = make_uint4(0, 0, 0, 0);
  for (int i = tid; i < 3 * kOwned; i += kThreads) (&sums[0][0])[i] = 0u;
  if (tid == 0) lcnt = 0u;
  if (tid < 2) {
    st_total[tid] = 0u;
    res[tid][0] = 0u;
  }
  pdl_wait_and_release();                     // the scores are complete; the compaction may be scheduled

  const SelSeq &sq = plan.seq[blockIdx.y];
  const uint32_t crank = CL > 1 ? cluster_ctarank() : 0u;
  const uint32_t lt_mask = (1u << lane) - 1u;
  const int chunk = (sq.len + CL - 1) / CL;
  const int lo = sq.t0 + min(sq.len, static_cast<int>(crank) * chunk);
  const int hi = sq.t0 + min(sq.len, static_cast<int>(crank + 1) * chunk);
  // each warp owns a contiguous run of the slice (a multiple of 32 tokens)
  const int cw = ((hi - lo) + kWarps * 32 - 1) / (kWarps * 32) * 32;
  const int wlo = min(hi, lo + warp * cw), whi = min(hi, wlo + cw);
  // this warp's part of the shared copy: cw slots, those past its run hold a token outside S
  const int wlen = whi - wlo, wpad = (wlen + 31) / 32 * 32;
  const bool cached = cw * kWarps <= plan.cache_tokens;
  uint32_t *c_bits = reinterpret_cast<uint32_t *>(cache_raw) + warp * cw;
  uint8_t *c_mod = cache_raw + static_cast<size_t>(plan.cache_tokens) * 4 + warp * cw;
  // f(position in the run, bits, modality, in segment 0, in segment 1) for this thread's tokens, one
  // 32-token round of the warp's run at a time, in token order
  auto token = [&](int x, uint32_t b, uint32_t m, auto &&f) {
    f(x, b, m, NSEG > 1 ? m == APACK_MOD_AUDIO : m - 1u < 2u, NSEG > 1 && m == APACK_MOD_VISUAL);
  };
  static_assert(APACK_MOD_AUDIO == 1 && APACK_MOD_VISUAL == 2, "the joint segment's test");
  auto each = [&](auto &&f) {
    if (cached) {
#pragma unroll 4
      for (int x = lane; x < wpad; x += 32) token(x, c_bits[x], c_mod[x], f);
    } else {
#pragma unroll 1
      for (int x = lane; x < wpad; x += 32)
        token(x, x < wlen ? __float_as_uint(scores[wlo + x]) : 0u,
              x < wlen ? static_cast<uint32_t>(modality[wlo + x]) : 0u, f);
    }
  };

  // ---- the segments' ranges of bit patterns (max and the complement of min, so that 0 is neutral)
  {
    uint32_t v[4] = {0u, 0u, 0u, 0u};
    auto take = [&](int, uint32_t b, uint32_t, bool s0, bool s1) {
      v[0] = max(v[0], s0 ? b : 0u);
      v[1] = max(v[1], s0 ? ~b : 0u);
      if (NSEG > 1) {
        v[2] = max(v[2], s1 ? b : 0u);
        v[3] = max(v[3], s1 ? ~b : 0u);
      }
    };
    // kBatch rounds' loads in flight together
    for (int x0 = lane; x0 < wpad; x0 += 32 * kBatch) {
      uint32_t b[kBatch], m[kBatch];
#pragma unroll
      for (int r = 0; r < kBatch; ++r) {
        const int x = x0 + 32 * r;
        b[r] = x < wlen ? __float_as_uint(scores[wlo + x]) : 0u;
        m[r] = x < wlen ? modality[wlo + x] : 0u;
      }
#pragma unroll
      for (int r = 0; r < kBatch; ++r) {
        const int x = x0 + 32 * r;
        if (x - lane >= wpad) break;            // uniform over the warp
        if (cached) {
          c_bits[x] = b[r];
          c_mod[x] = static_cast<uint8_t>(m[r]);
        }
        token(x, b[r], m[r], take);
      }
    }
#pragma unroll
    for (int i = 0; i < 2 * NSEG; ++i) {
      v[i] = __reduce_max_sync(0xffffffffu, v[i]);
      if (lane == 0) wrange[warp][i] = v[i];
    }
    __syncthreads();
    if (warp < 2 * NSEG) {
      const uint32_t x = __reduce_max_sync(0xffffffffu, wrange[lane][warp]);
      if (lane == 0) range_s[warp] = x;
    }
    __syncthreads();
    if (CL > 1) cluster_sync();   // the ranges and the zeroed counters of every CTA
  }
  Range g[NSEG];
  {
    uint32_t v[4] = {0u, 0u, 0u, 0u};
    if (CL == 1) {
#pragma unroll
      for (int i = 0; i < 2 * NSEG; ++i) v[i] = range_s[i];
    } else {
      uint4 x = make_uint4(0, 0, 0, 0);
      if (lane < CL) x = ld_shared_cluster_u32x4(map_shared_rank(range_s, lane));
      v[0] = __reduce_max_sync(0xffffffffu, x.x);
      v[1] = __reduce_max_sync(0xffffffffu, x.y);
      if (NSEG > 1) {
        v[2] = __reduce_max_sync(0xffffffffu, x.z);
        v[3] = __reduce_max_sync(0xffffffffu, x.w);
      }
    }
#pragma unroll
    for (int s = 0; s < NSEG; ++s) {
      const uint32_t mx = v[2 * s], mn = ~v[2 * s + 1];
      g[s].top = mx;
      g[s].o0 = 0u;
      g[s].span = mx > mn ? mx - mn : 0u;
      g[s].krem = static_cast<uint32_t>(sq.k[s]);
      g[s].count = 0u;
      g[s].shift = level_shift(min(g[s].span, kFirstSpan));
      g[s].act = true;                        // the first level also counts the segment
    }
  }
  auto any_active = [&] { return g[0].act || (NSEG > 1 && g[NSEG - 1].act); };

  // Finds the bin of each active segment that holds its k-th score, from the bins (4 per thread:
  // thread t holds bins 4 (t % 512) .. of segment t / 512), and narrows the ranges to it.
  auto pick = [&](const uint4 &c, uint32_t level) {
    const int seg = tid >> 9;
    const uint32_t s4 = c.x + c.y + c.z + c.w;
    const uint32_t incl = warp_incl_scan(s4, lane);
    if (lane == 31) wtot[warp] = incl;
    __syncthreads();
    const uint32_t wsum = warp_incl_scan(lane < 16 ? wtot[(seg << 4) + lane] : 0u, lane);
    const uint32_t before = (warp & 15) ? __shfl_sync(0xffffffffu, wsum, (warp & 15) - 1) : 0u;
    const uint32_t e = before + incl - s4;    // tokens in higher bins
    const Range &r = seg ? g[NSEG - 1] : g[0];
    const uint32_t k = r.krem;
    if (seg < NSEG && r.act && e < k && k <= e + s4) {
      uint32_t run = e, b = 0, in = c.x;
      if (run + in < k) { run += in; b = 1; in = c.y; }
      if (b == 1 && run + in < k) { run += in; b = 2; in = c.z; }
      if (b == 2 && run + in < k) { run += in; b = 3; in = c.w; }
      res[seg][0] = level + 1u;               // found at this level
      res[seg][1] = 4u * static_cast<uint32_t>(tid & 511) + b;
      res[seg][2] = run;
      res[seg][3] = in;
    }
    if (level == 0 && (tid & 511) == 511) st_total[seg] = before + incl;
    __syncthreads();
#pragma unroll
    for (int s = 0; s < NSEG; ++s) {
      if (!g[s].act) continue;
      if (res[s][0] != level + 1u) {          // nothing to keep (or fewer tokens than the host said)
        g[s].act = false;
        continue;
      }
      const uint32_t b = res[s][1], skip = b << g[s].shift;
      g[s].krem -= res[s][2];
      g[s].count = res[s][3];
      g[s].o0 += skip;
      const uint32_t rest = g[s].span - skip;
      // the last bin of the first level also holds every lower pattern
      g[s].span = b == kBins - 1 ? rest : min(rest, (1u << g[s].shift) - 1u);
      g[s].act = g[s].span > 0u;
      g[s].shift = level_shift(g[s].span);
    }
  };

  // ---- 1. narrow the ranges
  uint32_t level = 0;
  for (; any_active(); ++level) {
    if (level > 0) {   // few candidates left: collect them
      uint32_t left = g[0].act ? g[0].count : 0u;
      bool fits = !g[0].act || g[0].span < 0x80000000u;
      if (NSEG > 1 && g[NSEG - 1].act) {
        left += g[NSEG - 1].count;
        fits &= g[NSEG - 1].span < 0x80000000u;
      }
      if (fits && left <= kGather) break;
    }
    each([&](int, uint32_t b, uint32_t, bool s0, bool s1) {
      if (s0 && g[0].act) {
        const int bin = bin_of(g[0], g[0].top - b);
        if (bin >= 0) atomicAdd(&hist[bin], 1u);
      }
      if (NSEG > 1 && s1 && g[NSEG - 1].act) {
        const int bin = bin_of(g[NSEG - 1], g[NSEG - 1].top - b);
        if (bin >= 0) atomicAdd(&hist[kBins + bin], 1u);
      }
    });
    __syncthreads();
    uint4 c = reinterpret_cast<const uint4 *>(hist)[tid];
    reinterpret_cast<uint4 *>(hist)[tid] = make_uint4(0, 0, 0, 0);
    if (CL > 1) {
      uint32_t *buf = sums[level % 3];
      const int w = 4 * tid, owner = w / kOwned;
      const uint32_t dst = map_shared_rank(buf + w % kOwned, owner);
      if (c.x) red_shared_cluster_add(dst, c.x);
      if (c.y) red_shared_cluster_add(dst + 4, c.y);
      if (c.z) red_shared_cluster_add(dst + 8, c.z);
      if (c.w) red_shared_cluster_add(dst + 12, c.w);
      cluster_sync();
      if (tid < NSEG * 512) c = ld_shared_cluster_u32x4(dst);
      // every CTA has read the previous level's sums: its buffer is zeroed for the level after next
      if (level > 0)
        for (int i = tid; i < kOwned; i += kThreads) sums[(level + 2) % 3][i] = 0u;
    }
    pick(c, level);
  }
  if (any_active()) {
    // the candidates, as offsets within their range, the segment in bit 31
    each([&](int, uint32_t b, uint32_t, bool s0, bool s1) {
      uint32_t rel = g[0].top - b - g[0].o0;
      bool in = s0 && g[0].act && rel <= g[0].span;
      if (NSEG > 1 && s1) {
        rel = g[NSEG - 1].top - b - g[NSEG - 1].o0;
        in = g[NSEG - 1].act && rel <= g[NSEG - 1].span;
        rel |= 0x80000000u;
      }
      if (in) list[atomicAdd(&lcnt, 1u)] = rel;
    });
    __syncthreads();
    uint32_t upto = 0, total;
    if (CL > 1) {
      cluster_sync();
      const uint32_t have = lane < CL ? ld_shared_cluster_u32(map_shared_rank(&lcnt, lane)) : 0u;
      upto = warp_incl_scan(have, lane);
      total = __shfl_sync(0xffffffffu, upto, CL - 1);
    } else {
      total = lcnt;
    }
    // candidate x of the CTAs' concatenated lists
    auto candidate = [&](uint32_t x) {
      if (CL == 1) return x < total ? list[x] : 0u;
      uint32_t src = 0, base = 0;
#pragma unroll
      for (int r = 0; r < CL - 1; ++r) {
        const uint32_t u = __shfl_sync(0xffffffffu, upto, r);
        if (x >= u) {
          src = r + 1;
          base = u;
        }
      }
      return x < total ? ld_shared_cluster_u32(map_shared_rank(list + (x - base), src)) : 0u;
    };
    if (total <= kRank) {
      uint32_t mine = 0;
      if (warp < kRank / 32) {
        mine = candidate(tid);
        // beyond the last candidate: above every offset of segment 1 (rank_of is only compared)
        rank_of[tid] = tid < total ? mine : 0xFFFFFFFFu;
      }
      __syncthreads();
      if (tid < total) {
        const uint32_t s = mine >> 31, first = s << 31;
        uint32_t below = 0, same = 0;         // smaller offsets: larger scores
        for (uint32_t j = 0; j < total; j += 4) {
          const uint4 v = *reinterpret_cast<const uint4 *>(rank_of + j);
          below += (v.x >= first && v.x < mine) + (v.y >= first && v.y < mine) + (v.z >= first && v.z < mine) +
                   (v.w >= first && v.w < mine);
          same += (v.x == mine) + (v.y == mine) + (v.z == mine) + (v.w == mine);
        }
        const uint32_t k = s ? g[NSEG - 1].krem : g[0].krem;
        if (below < k && k <= below + same) {   // every equal candidate writes the same values
          res[s][0] = level + 1u;
          res[s][1] = mine & 0x7FFFFFFFu;
          res[s][2] = below;
        }
      }
      __syncthreads();
#pragma unroll
      for (int s = 0; s < NSEG; ++s)
        if (g[s].act && res[s][0] == level + 1u) {
          g[s].o0 += res[s][1];
          g[s].krem -= res[s][2];
        }
    } else {
      uint32_t cand[2];
#pragma unroll
      for (int j = 0; j < 2; ++j) cand[j] = candidate(tid + j * kThreads);
      uint32_t from[NSEG];
#pragma unroll
      for (int s = 0; s < NSEG; ++s) from[s] = g[s].o0;
      for (; any_active(); ++level) {
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          if (tid + j * kThreads >= total) continue;
          const bool s1 = NSEG > 1 && (cand[j] >> 31);
          const Range &r = s1 ? g[NSEG - 1] : g[0];
          const int bin = r.act ? bin_of(r, (s1 ? from[NSEG - 1] : from[0]) + (cand[j] & 0x7FFFFFFFu)) : -1;
          if (bin >= 0) atomicAdd(&hist[(s1 ? kBins : 0) + bin], 1u);
        }
        __syncthreads();
        const uint4 c = reinterpret_cast<const uint4 *>(hist)[tid];
        reinterpret_cast<uint4 *>(hist)[tid] = make_uint4(0, 0, 0, 0);
        pick(c, level);
      }
    }
  }

  // Threshold and tie quota per segment.
  uint32_t T[2] = {0xFFFFFFFFu, 0xFFFFFFFFu}, quota[2] = {0u, 0u};
#pragma unroll
  for (int s = 0; s < NSEG; ++s)
    if (sq.k[s] > 0) {
      T[s] = g[s].top - g[s].o0;
      quota[s] = g[s].krem;
    }

  // ---- 2. counts per warp run, per CTA, exchanged through the cluster
  uint32_t c_keep = 0, c_eq0 = 0, c_eq1 = 0;
  each([&](int x, uint32_t b, uint32_t, bool s0, bool s1) {
    const bool in = x < wlen;
    const uint32_t tt = s1 ? T[1] : T[0];
    c_keep += __popc(__ballot_sync(0xffffffffu, in && ((!s0 && !s1) || b > tt)));
    c_eq0 += __popc(__ballot_sync(0xffffffffu, s0 && b == tt));
    if (NSEG > 1) c_eq1 += __popc(__ballot_sync(0xffffffffu, s1 && b == tt));
  });
  if (lane == 0) {
    wcnt[warp][0] = c_keep;
    wcnt[warp][1] = c_eq0;
    wcnt[warp][2] = c_eq1;
  }
  __syncthreads();
  if (warp < 3) {
    const uint32_t v = __reduce_add_sync(0xffffffffu, wcnt[lane][warp]);
    if (lane == 0) cnt[warp] = v;
  }
  __syncthreads();
  if (CL > 1) cluster_sync();
  if (warp == 0) {
    // Token order runs over the CTAs of the cluster, then over the warps of this CTA: ties are
    // granted in that order until each segment's quota runs out.  Lane r stands for CTA r, then
    // for warp r; exclusive prefix sums over the lanes replace a walk in order.
    auto excl_scan = [&](uint32_t v) -> uint32_t { return warp_incl_scan(v, lane) - v; };
    auto granted = [](uint32_t ties, uint32_t before, uint32_t q) -> uint32_t {
      const uint32_t avail = q > before ? q - before : 0u;
      return ties < avail ? ties : avail;
    };
    // the cluster's CTAs
    uint32_t c[3] = {0u, 0u, 0u};
    if (lane < CL) {
#pragma unroll
      for (int i = 0; i < 3; ++i) c[i] = CL > 1 ? ld_shared_cluster_u32(map_shared_rank(&cnt[i], lane)) : cnt[i];
    }
    const uint32_t eqp0 = excl_scan(c[1]), eqp1 = excl_scan(c[2]);   // ties of the CTAs before
    const uint32_t kept = c[0] + granted(c[1], eqp0, quota[0]) + granted(c[2], eqp1, quota[1]);
    const uint32_t kept_excl = excl_scan(kept);
    const uint32_t kept_all = __shfl_sync(0xffffffffu, kept_excl + kept, 31);
    const uint32_t kept_before = __shfl_sync(0xffffffffu, kept_excl, static_cast<int>(crank));
    const uint32_t eqb0 = __shfl_sync(0xffffffffu, eqp0, static_cast<int>(crank));
    const uint32_t eqb1 = __shfl_sync(0xffffffffu, eqp1, static_cast<int>(crank));
    // this CTA's warps (kWarps == 32: one lane each)
    const uint32_t *wc = wcnt[lane];
    const uint32_t we0 = eqb0 + excl_scan(wc[1]), we1 = eqb1 + excl_scan(wc[2]);
    const uint32_t wk = wc[0] + granted(wc[1], we0, quota[0]) + granted(wc[2], we1, quota[1]);
    wbase[lane] = kept_before + excl_scan(wk);
    weqb[lane][0] = we0;
    weqb[lane][1] = we1;
    if (crank == 0 && lane == 0) {
      // Device-side consistency with the host counts.
      bool bad = kept_all != static_cast<uint32_t>(sq.out_len);
      for (int s = 0; s < NSEG; ++s)   // segment sizes seen by the first level
        if (st_total[s] != static_cast<uint32_t>(sq.n_seg[s])) bad = true;
      if (bad) raise_device_error(err, APACK_EDEVICE, 31, plan.seq_base + static_cast<int>(blockIdx.y),
                                  static_cast<int32_t>(kept_all));
      if (new_cu) {
        if (plan.write_cu0 && blockIdx.y == 0) new_cu[0] = 0;
        new_cu[plan.seq_base + blockIdx.y + 1] = sq.out_base + sq.out_len;
      }
    }
  }
  __syncthreads();
  // this CTA's remote reads are done; it leaves once every CTA's are (waited for below)
  if (CL > 1) asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");

  // ---- 3. ordered writes: each warp walks its run in token order
  uint32_t pos = wbase[warp];
  uint32_t er0 = weqb[warp][0], er1 = weqb[warp][1];
  // ties of this warp's run: all granted, or counted one by one (uniform over the warp)
  const bool all0 = er0 + c_eq0 <= quota[0], all1 = er1 + c_eq1 <= quota[1];
  each([&](int x, uint32_t b, uint32_t m, bool s0, bool s1) {
    const bool in = x < wlen;
    const int i = wlo + x;
    const uint32_t tt = s1 ? T[1] : T[0];
    const bool eq = (s0 || s1) && b == tt;
    bool keep = in && ((!s0 && !s1) || b > tt);
    if (all0 && all1) {
      keep |= eq;
    } else {
      const uint32_t em0 = __ballot_sync(0xffffffffu, eq && s0);
      const uint32_t em1 = NSEG > 1 ? __ballot_sync(0xffffffffu, eq && s1) : 0u;
      if (eq) {
        const uint32_t rank = s1 ? er1 + __popc(em1 & lt_mask) : er0 + __popc(em0 & lt_mask);
        keep = rank < (s1 ? quota[1] : quota[0]);
      }
      er0 += __popc(em0);
      er1 += __popc(em1);
    }
    const uint32_t km = __ballot_sync(0xffffffffu, keep);
    const uint32_t p = pos + __popc(km & lt_mask);
    if (in) {
      if (keep && p < static_cast<uint32_t>(sq.out_len)) {
        const int o = sq.out_base + static_cast<int>(p);
        keep_idx[o] = i;
        if (modality_out) modality_out[o] = static_cast<uint8_t>(m);
        if (dst_of_src) dst_of_src[i] = o;
      } else if (dst_of_src) {
        dst_of_src[i] = -1;
      }
    }
    pos += __popc(km);
  });
  if (CL > 1) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

template <int CL, int NSEG>
cudaError_t launch_select(const SelectPlan &P, int ns, size_t smem, const float *scores, const uint8_t *modality,
                          int32_t *keep_idx, uint8_t *modality_out, int32_t *dst_of_src, int32_t *new_cu,
                          DeviceError *err, cudaStream_t stream) {
  static std::atomic<uint64_t> attr{0};
  const cudaError_t e = once_per_device(attr, [] {
    return cudaFuncSetAttribute(select_kernel<CL, NSEG>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxCached * 5);
  });
  if (e != cudaSuccess) return e;
  return launch_pdl(select_kernel<CL, NSEG>, dim3(CL, ns, 1), dim3(kThreads), smem, stream, P, scores, modality,
                    keep_idx, modality_out, dst_of_src, new_cu, err);
}

}  // namespace

// Clusters of each size that can be resident on the current device at once (16 CTAs are beyond the
// portable cluster size); probed once per device, 0 = that size cannot run.
struct ClusterCaps {
  int of1, of4, of8, of16;
};

template <int CL>
int resident_clusters() {
  if (CL > 8 && (cudaFuncSetAttribute(select_kernel<CL, 1>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) !=
                     cudaSuccess ||
                 cudaFuncSetAttribute(select_kernel<CL, 2>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) !=
                     cudaSuccess))
    return 0;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = CL;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.gridDim = dim3(CL, 1, 1);
  cfg.blockDim = dim3(kThreads, 1, 1);
  cfg.attrs = at;
  cfg.numAttrs = 1;
  int n = 0;
  return cudaOccupancyMaxActiveClusters(&n, select_kernel<CL, 2>, &cfg) == cudaSuccess ? n : 0;
}

ClusterCaps cluster_caps() {
  static std::atomic<uint64_t> probed[64];   // 16 bits per size, biased by one (0 = not probed yet)
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return {device_sm_count(), 0, 0, 0};
  uint64_t v = probed[dev].load(std::memory_order_acquire);
  if (v == 0) {
    const uint64_t c4 = resident_clusters<4>(), c8 = resident_clusters<8>(), c16 = resident_clusters<16>();
    cudaGetLastError();
    v = 1 | ((c4 & 0x7FFF) << 16) | ((c8 & 0x7FFF) << 32) | ((c16 & 0x7FFF) << 48);
    probed[dev].store(v, std::memory_order_release);
  }
  return {device_sm_count(), static_cast<int>((v >> 16) & 0x7FFF), static_cast<int>((v >> 32) & 0x7FFF),
          static_cast<int>((v >> 48) & 0x7FFF)};
}

// CTAs per sequence: the size with the least estimated time, waves x (fixed + tokens per CTA).
// Fitted to GB300 (graph replays, joint top-k, us): 1,000 tokens take 4.2 / 6.5 / 7.2 / 9.6 with 1 / 4
// / 8 / 16 CTAs, each further 1,024 tokens of a CTA 0.6; 8,000 tokens 8.2 / 8.1 / 8.6 / 10.6, 135,000
// tokens 171 / 28 / 19.7 / 17.5; 16 sequences of 37,000 tokens 36 / 14.5 / 23.4 / 38.
int select_cluster_size(int max_len, int ns) {
  const ClusterCaps caps = cluster_caps();
  const int size[4] = {1, 4, 8, 16}, cap[4] = {caps.of1, caps.of4, caps.of8, caps.of16};
  const float fixed[4] = {3.8f, 6.2f, 6.8f, 9.3f};
  int best = 1;
  float best_t = 0.f;
  for (int i = 0; i < 4; ++i) {
    if (cap[i] <= 0) continue;
    const int slice = (max_len + size[i] - 1) / size[i];
    const float per = slice <= kMaxCached ? 0.6f / 1024.f : 1.3f / 1024.f;
    const float t = static_cast<float>((ns + cap[i] - 1) / cap[i]) * (fixed[i] + per * static_cast<float>(slice));
    if (i == 0 || t < best_t) {
      best = size[i];
      best_t = t;
    }
  }
  return best;
}

apack_status run_select(const apack_seqs *seqs, const float *scores, const int32_t *keep_count_h, int32_t mode,
                        int32_t *keep_idx, uint8_t *modality_out, int32_t *dst_of_src, int32_t *new_cu_seqlens,
                        void *ws, cudaStream_t stream) {
  int64_t T = 0, NQ = 0;
  apack_status st = validate_seqs(seqs, &T, &NQ);
  if (st != APACK_OK) return st;
  if (!keep_count_h || !ws || (mode != APACK_SELECT_PER_MODALITY && mode != APACK_SELECT_JOINT)) return APACK_EINVAL;
  if (T > 0 && (!scores || !keep_idx)) return APACK_EINVAL;
  const int B = seqs->num_seqs;
  const int nsegs = mode == APACK_SELECT_JOINT ? 1 : 2;
  // Host-side plan: counts, output offsets.
  int64_t out_total = 0;
  for (int b = 0; b < B; ++b) {
    const int na = seqs->n_audio_h[b], nv = seqs->n_visual_h[b];
    const int len = seqs->cu_seqlens_h[b + 1] - seqs->cu_seqlens_h[b];
    const int k0 = keep_count_h[2 * b], k1 = keep_count_h[2 * b + 1];
    if (nsegs == 2) {
      if (k0 < 0 || k0 > na || k1 < 0 || k1 > nv) return APACK_EINVAL;
      out_total += len - na - nv + k0 + k1;
    } else {
      if (k0 < 0 || k0 > na + nv) return APACK_EINVAL;
      out_total += len - na - nv + k0;
    }
  }
  (void)out_total;
  const WsLayout L = workspace_layout(seqs);
  DeviceError *err = reinterpret_cast<DeviceError *>(static_cast<uint8_t *>(ws) + L.err_off);
  int32_t out_base = 0;
  for (int s0 = 0; s0 < B; s0 += kSeqsPerLaunch) {
    const int ns = (B - s0 < kSeqsPerLaunch) ? (B - s0) : kSeqsPerLaunch;
    SelectPlan P{};
    P.nseq = ns;
    P.write_cu0 = s0 == 0;
    P.seq_base = s0;
    for (int i = 0; i < ns; ++i) {
      const int b = s0 + i;
      SelSeq &q = P.seq[i];
      q.t0 = seqs->cu_seqlens_h[b];
      q.len = seqs->cu_seqlens_h[b + 1] - q.t0;
      const int na = seqs->n_audio_h[b], nv = seqs->n_visual_h[b];
      if (nsegs == 2) {
        q.n_seg[0] = na; q.n_seg[1] = nv;
        q.k[0] = keep_count_h[2 * b]; q.k[1] = keep_count_h[2 * b + 1];
      } else {
        q.n_seg[0] = na + nv; q.n_seg[1] = 0;
        q.k[0] = keep_count_h[2 * b]; q.k[1] = 0;
      }
      q.out_len = q.len - na - nv + q.k[0] + q.k[1];
      q.out_base = out_base;
      out_base += q.out_len;
    }
    int max_len = 0;
    for (int i = 0; i < ns; ++i) max_len = P.seq[i].len > max_len ? P.seq[i].len : max_len;
    const int CL = select_cluster_size(max_len, ns);
    auto *launch = nsegs == 1 ? (CL == 16  ? launch_select<16, 1>
                                 : CL == 8 ? launch_select<8, 1>
                                 : CL == 4 ? launch_select<4, 1>
                                           : launch_select<1, 1>)
                              : (CL == 16  ? launch_select<16, 2>
                                 : CL == 8 ? launch_select<8, 2>
                                 : CL == 4 ? launch_select<4, 2>
                                           : launch_select<1, 2>);
    // cache each CTA's slice in shared memory (32 warps' runs of whole 32-token rounds) when the
    // longest slice of the launch fits
    const int64_t slots = ((static_cast<int64_t>(max_len) + CL - 1) / CL + kThreads - 1) / kThreads * kThreads;
    P.cache_tokens = slots <= kMaxCached ? static_cast<int32_t>(slots) : 0;
    const cudaError_t e = launch(P, ns, static_cast<size_t>(P.cache_tokens) * 5, scores, seqs->modality, keep_idx, modality_out, dst_of_src, new_cu_seqlens, err,
                                 stream);
    if (check_cuda(e) != APACK_OK) return APACK_ECUDA;
    count_launches(1);
    if (check_cuda(cudaGetLastError()) != APACK_OK) return APACK_ECUDA;
  }
  return APACK_OK;
}

}  // namespace apack
