// prellm.cu -- pre-LLM frame alignment of A-PACK (Sec. 3.1, "Coarse pass" and "Gated fine
// pass"; Eq. cka and Eq. gate; Algorithm 1, the first steps of the pre-LLM stage).
//
//  pool kernel:  v_f = mean of frame f's visual tokens, a_f = mean of the audio tokens
//                resampled onto frame f (token j -> frame floor(j F / N_a)); fp32 sums
//                of bf16 rows in token order.  Reads every encoder token once: the
//                HBM-bound part of this stage.
//  cka kernel:   one CTA per frame; over the window W_f (cut to the clip) the rows are
//                centred and the w x w Grams K_A = A A^T, K_V = V V^T accumulated over
//                the feature dimension, which gives Eq. cka exactly since
//                ||V^T A||_F^2 = <K_A, K_V>_F and ||A^T A||_F = ||K_A||_F; also the
//                direct distance d_f = ||v_f - a_f||.
//  gate:         the last CTA of the CKA kernel to finish (a counter in the workspace,
//                zeroed by the pool kernel) computes c-bar, min/max of d, the min-max
//                normalised distance and the gated score s_f of Eq. gate (blend when
//                c-bar < tau) over the whole clip.
//  run kernel:   in place of the pool kernel for long clips and windows 3 and 5 (below): pools a
//                run of frames per CTA and computes the CKA of the frames inside it, so that the
//                cka kernel is left with the frames at the runs' ends.
// All reductions run in a fixed order: results are deterministic.  Two launches per call; the
// CKA kernel is a programmatic dependent of the pool kernel (scheduled while the pool drains,
// waiting for its completion before any read).
#include <algorithm>
#include <type_traits>
#include <cmath>

#include "internal.cuh"
#include "ptx.cuh"

namespace apack {

namespace {

constexpr int kPoolMaxThreads = 512;   // 8 features per thread: up to 4096 features per CTA
constexpr int kCkaThreads = 256;
constexpr int kMaxWindow = 7;
constexpr int kGateHold = 6;            // frames per thread whose c and d the gate keeps in registers

__device__ __forceinline__ void add_bf16x8(const uint4 &v, float (&acc)[8]) {
  const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    acc[2 * i] += __uint_as_float(w[i] << 16);
    acc[2 * i + 1] += __uint_as_float(w[i] & 0xFFFF0000u);
  }
}

__global__ void __launch_bounds__(kPoolMaxThreads, 2)
    frame_pool_kernel(const uint4 *__restrict__ visual, const uint4 *__restrict__ audio, int n_frames, int tpf,
                      int n_audio, int64_t dim, float *__restrict__ v_out, float *__restrict__ a_out,
                      unsigned int *done) {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");   // the CKA kernel may be scheduled
  const int f = blockIdx.x;
  if (f == 0 && blockIdx.y == 0 && threadIdx.x == 0) *done = 0u;   // CTA counter of the CKA kernel
  const int64_t fi = (static_cast<int64_t>(blockIdx.y) * blockDim.x + threadIdx.x) * 8;
  if (fi >= dim) return;
  const int64_t vec_per_row = dim / 8;
  const int64_t col = fi / 8;
  float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
  const int64_t r0 = static_cast<int64_t>(f) * tpf;
#pragma unroll 8
  for (int t = 0; t < tpf; ++t) add_bf16x8(__ldg(visual + (r0 + t) * vec_per_row + col), acc);
  const float inv_v = 1.f / static_cast<float>(tpf);
#pragma unroll
  for (int i = 0; i < 8; ++i) v_out[static_cast<int64_t>(f) * dim + fi + i] = acc[i] * inv_v;
  // audio tokens j with floor(j F / N_a) == f: j in [ceil(f N_a / F), ceil((f+1) N_a / F))
  const int64_t j0 = (static_cast<int64_t>(f) * n_audio + n_frames - 1) / n_frames;
  const int64_t j1 = (static_cast<int64_t>(f + 1) * n_audio + n_frames - 1) / n_frames;
#pragma unroll
  for (int i = 0; i < 8; ++i) acc[i] = 0.f;
#pragma unroll 8
  for (int64_t j = j0; j < j1; ++j) add_bf16x8(__ldg(audio + j * vec_per_row + col), acc);
  const float inv_a = 1.f / static_cast<float>(j1 - j0);
#pragma unroll
  for (int i = 0; i < 8; ++i) a_out[static_cast<int64_t>(f) * dim + fi + i] = acc[i] * inv_a;
}

// ------------------------------------------------------------------ runs of frames
// Long clips: one CTA per SM pools a run of consecutive frames and computes the CKA of the frames whose
// window lies inside the run at once, from the last W pooled rows in registers; only the rows of windows
// that cross the run's ends go to memory, and the CKA kernel is left with those frames.  The encoder
// tokens stream through a shared-memory ring of bulk copies (a producer warp; each consumer thread owns 8
// features and adds the rows in token order), so the sums at a frame's end do not interrupt the reading.
// Bound by HBM: 139 us (6.96 TB/s) for 1,200 frames of 100 tokens, d = 3584, window 3, and 12 us for the
// CKA kernel after it, where the pool took 145 us and the CKA of every frame 19.6 us.
constexpr int kRunStage = 32768;                // bytes of a ring stage, at most
constexpr int kRunStages = 6;
// Consumer threads (the producer is one more warp): rows of 4096 features, or of 3584 with window 5,
// whose rows take more registers than 17 warps leave each thread.
template <int W>
constexpr int run_threads() { return W > 3 ? 448 : 512; }

struct RunShape {
  int n_frames, tpf, n_audio, run;              // run: frames per CTA
  int64_t dim;
};

__device__ __forceinline__ int64_t audio_begin(int f, int n_audio, int n_frames) {
  return (static_cast<int64_t>(f) * n_audio + n_frames - 1) / n_frames;
}

// Sums of one feature's window rows into the Grams' upper triangles (w == W rows).
template <int W>
__device__ __forceinline__ void add_window(const float (&a_rows)[W], const float (&v_rows)[W], float inv_w,
                                           float (&ga)[W * (W + 1) / 2], float (&gv)[W * (W + 1) / 2]) {
  float av[W], vv[W], am = 0.f, vm = 0.f;
#pragma unroll
  for (int r = 0; r < W; ++r) {
    am += a_rows[r];
    vm += v_rows[r];
  }
  am *= inv_w;
  vm *= inv_w;
#pragma unroll
  for (int r = 0; r < W; ++r) {
    av[r] = a_rows[r] - am;
    vv[r] = v_rows[r] - vm;
  }
  int k = 0;
#pragma unroll
  for (int i = 0; i < W; ++i)
#pragma unroll
    for (int j = i; j < W; ++j, ++k) {
      ga[k] = fmaf(av[i], av[j], ga[k]);
      gv[k] = fmaf(vv[i], vv[j], gv[k]);
    }
}

// Eq. cka from the Grams' upper triangles tot[0..kG) (audio) and tot[kG..2 kG) (visual).
template <int W>
__device__ __forceinline__ float cka_of(const float *tot) {
  constexpr int kG = W * (W + 1) / 2;
  // <K_A, K_V>_F, ||K_A||_F^2 and ||K_V||_F^2 (off-diagonal entries twice)
  float dot = 0.f, na = 0.f, nv = 0.f;
  int k = 0;
#pragma unroll
  for (int i = 0; i < W; ++i)
#pragma unroll
    for (int j = i; j < W; ++j, ++k) {
      const float m = (i == j) ? 1.f : 2.f;
      dot = fmaf(m * tot[k], tot[kG + k], dot);
      na = fmaf(m * tot[k], tot[k], na);
      nv = fmaf(m * tot[kG + k], tot[kG + k], nv);
    }
  const float den = sqrtf(na) * sqrtf(nv);
  return den > 0.f ? dot / den : 0.f;
}

// A bounded wait that also gives up when another thread of the CTA has; one that runs out sets the flag.
__device__ __forceinline__ bool run_wait(uint64_t *bar, uint32_t parity, volatile unsigned int *gave_up) {
  if (mbar_try_wait(bar, parity)) return true;
  const uint64_t t0 = globaltimer_ns();
  for (;;) {
    for (int i = 0; i < 32; ++i)
      if (mbar_try_wait(bar, parity)) return true;
    if (*gave_up) return false;
    if (globaltimer_ns() - t0 > kWaitLimitNs) {
      *gave_up = 1;
      return false;
    }
  }
}

// status[run]: 1 when a wait of the run's CTA gave up (its sums are then not to be used), else 0.
template <int W>
__global__ void __launch_bounds__(run_threads<W>() + 32, 1)
    frame_run_kernel(const __grid_constant__ RunShape sh, const uint8_t *__restrict__ visual,
                     const uint8_t *__restrict__ audio, float *__restrict__ v_out, float *__restrict__ a_out,
                     float *__restrict__ c_out, float *__restrict__ d_out, unsigned int *done,
                     unsigned int *__restrict__ status) {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");   // the CKA kernel may be scheduled
  constexpr int kH = W / 2, kG = W * (W + 1) / 2, kN = 2 * kG + 1;
  extern __shared__ __align__(128) uint8_t ring[];
  __shared__ __align__(8) uint64_t full[kRunStages], empty[kRunStages];
  __shared__ float red[run_threads<W>() / 32][kN];
  __shared__ float tot[kN];
  __shared__ volatile unsigned int gave_up;
  const int nthr = blockDim.x - 32, nwarps = nthr / 32;               // consumers
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int64_t row = sh.dim * 2;                                     // bytes of a token row, a multiple of 16
  const int stage_rows = max(1, kRunStage / static_cast<int>(row));
  const int f0 = blockIdx.x * sh.run, f1 = min(sh.n_frames, f0 + sh.run);
  if (tid == 0) {
    for (int i = 0; i < kRunStages; ++i) {
      mbar_init(&full[i], 1);
      mbar_init(&empty[i], nwarps);
    }
    gave_up = 0;
    fence_mbar_init();
    if (blockIdx.x == 0) *done = 0u;                                  // CTA counter of the CKA kernel
  }
  __syncthreads();
  if (warp == nwarps) {
    // ---- producer: the frames' visual rows, then their audio rows, stage_rows at a time
    if (lane == 0) {
      uint32_t n = 0;
      auto stream = [&](const uint8_t *src, int64_t rows) -> bool {
        for (int64_t r = 0; r < rows; r += stage_rows, ++n) {
          const int slot = n % kRunStages;
          if (n >= kRunStages && !run_wait(&empty[slot], (n / kRunStages - 1) & 1u, &gave_up)) return false;
          const uint32_t bytes = static_cast<uint32_t>(min(static_cast<int64_t>(stage_rows), rows - r) * row);
          mbar_arrive_expect_tx(&full[slot], bytes);
          bulk_load(ring + slot * kRunStage, src + r * row, bytes, &full[slot]);
        }
        return true;
      };
      bool ok = true;
      for (int f = f0; ok && f < f1; ++f) {
        ok = stream(visual + static_cast<int64_t>(f) * sh.tpf * row, sh.tpf);
        const int64_t j0 = audio_begin(f, sh.n_audio, sh.n_frames), j1 = audio_begin(f + 1, sh.n_audio, sh.n_frames);
        if (ok) ok = stream(audio + j0 * row, j1 - j0);
      }
      // no copy lands after the CTA has left, whoever gave up: the last of every slot is awaited here (the
      // ones before were consumed)
      for (uint32_t i = n > kRunStages ? n - kRunStages : 0; i < n; ++i)
        if (!mbar_wait(&full[i % kRunStages], (i / kRunStages) & 1u, kWaitLimitNs)) gave_up = 1;
    }
    return;
  }
  // ---- consumers
  const bool mine = tid < sh.dim / 8;                                 // this thread has features 8 tid ..
  uint32_t n = 0;
  bool ok = true;
  auto pool = [&](int64_t rows, float (&acc)[8]) {
#pragma unroll
    for (int i = 0; i < 8; ++i) acc[i] = 0.f;
    for (int64_t r = 0; r < rows; r += stage_rows, ++n) {
      const int slot = n % kRunStages;
      if (ok && !__all_sync(0xffffffffu, run_wait(&full[slot], (n / kRunStages) & 1u, &gave_up))) ok = false;
      if (!ok) continue;                          // no barrier is touched after a wait that failed
      const int cnt = static_cast<int>(min(static_cast<int64_t>(stage_rows), rows - r));
      const uint8_t *p = ring + slot * kRunStage + tid * 16;
      if (mine)
#pragma unroll 4
        for (int i = 0; i < cnt; ++i) add_bf16x8(*reinterpret_cast<const uint4 *>(p + i * row), acc);
      __syncwarp();
      if (lane == 0) mbar_arrive(&empty[slot]);
    }
    const float inv = 1.f / static_cast<float>(rows);
#pragma unroll
    for (int i = 0; i < 8; ++i) acc[i] *= inv;
  };
  float vr[W][8], ar[W][8];                       // the last W pooled rows, oldest first
#pragma unroll
  for (int r = 0; r < W; ++r)
#pragma unroll
    for (int i = 0; i < 8; ++i) vr[r][i] = ar[r][i] = 0.f;
  for (int f = f0; f < f1; ++f) {
#pragma unroll
    for (int r = 0; r + 1 < W; ++r)
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        vr[r][i] = vr[r + 1][i];
        ar[r][i] = ar[r + 1][i];
      }
    pool(sh.tpf, vr[W - 1]);
    pool(audio_begin(f + 1, sh.n_audio, sh.n_frames) - audio_begin(f, sh.n_audio, sh.n_frames), ar[W - 1]);
    // rows that windows across the run's ends read
    if (mine && (f < f0 + 2 * kH || f >= f1 - 2 * kH)) {
      float4 *vo = reinterpret_cast<float4 *>(v_out + static_cast<int64_t>(f) * sh.dim) + 2 * tid;
      float4 *ao = reinterpret_cast<float4 *>(a_out + static_cast<int64_t>(f) * sh.dim) + 2 * tid;
      vo[0] = make_float4(vr[W - 1][0], vr[W - 1][1], vr[W - 1][2], vr[W - 1][3]);
      vo[1] = make_float4(vr[W - 1][4], vr[W - 1][5], vr[W - 1][6], vr[W - 1][7]);
      ao[0] = make_float4(ar[W - 1][0], ar[W - 1][1], ar[W - 1][2], ar[W - 1][3]);
      ao[1] = make_float4(ar[W - 1][4], ar[W - 1][5], ar[W - 1][6], ar[W - 1][7]);
    }
    if (f < f0 + 2 * kH) continue;                // the window of frame f - kH is complete from here on
    float ga[kG], gv[kG], dist = 0.f;
#pragma unroll
    for (int i = 0; i < kG; ++i) ga[i] = gv[i] = 0.f;
#pragma unroll
    for (int i = 0; i < 8; ++i) {                 // features without a thread hold zeros
      float a1[W], v1[W];
#pragma unroll
      for (int r = 0; r < W; ++r) {
        a1[r] = ar[r][i];
        v1[r] = vr[r][i];
      }
      const float dd = v1[kH] - a1[kH];
      dist = fmaf(dd, dd, dist);
      add_window<W>(a1, v1, 1.f / static_cast<float>(W), ga, gv);
    }
    // fixed-order reduction over the consumers: warp trees, then one thread per sum over the warps
#pragma unroll
    for (int i = 0; i < kG; ++i) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        ga[i] += __shfl_xor_sync(0xffffffffu, ga[i], o);
        gv[i] += __shfl_xor_sync(0xffffffffu, gv[i], o);
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) dist += __shfl_xor_sync(0xffffffffu, dist, o);
    if (lane == 0) {
#pragma unroll
      for (int i = 0; i < kG; ++i) {
        red[warp][i] = ga[i];
        red[warp][kG + i] = gv[i];
      }
      red[warp][2 * kG] = dist;
    }
    asm volatile("bar.sync 1, %0;" ::"r"(nthr) : "memory");
    if (warp == 0) {
      for (int i = lane; i < kN; i += 32) {
        float t = 0.f;
        for (int w = 0; w < nwarps; ++w) t += red[w][i];
        tot[i] = t;
      }
      __syncwarp();
      if (lane == 0) {
        c_out[f - kH] = cka_of<W>(tot);
        d_out[f - kH] = sqrtf(tot[2 * kG]);
      }
    }
    asm volatile("bar.sync 1, %0;" ::"r"(nthr) : "memory");   // red is free again
  }
  asm volatile("bar.sync 1, %0;" ::"r"(nthr) : "memory");     // every consumer's last wait is over
  if (tid == 0) status[blockIdx.x] = gave_up;
}

// Per-frame windowed CKA (Eq. cka) and direct distance; the last CTA to finish also
// runs the gate (Eq. gate) over all frames.  One CTA per frame, or with RUNS per frame at the ends
// of runs of `run` frames (W - 1 CTAs per run), whose windows cross them.  W is the window size (odd,
// <= kMaxWindow); windows cut by the clip's ends hold w < W rows and the missing rows are zeros that
// never enter a Gram entry with i or j >= w.
// With RUNS the grid is about two CTAs per SM and its latency the call's: twice the loads in flight, and
// the gate's inputs in registers (two CTAs per SM stated: left open, the compiler takes 64 registers for
// window 3 in place of 96, and the call of 1,200 frames 158 us in place of 155.5).  Otherwise as many CTAs per SM as the window's rows leave registers
// for (window 7 at 136 registers and one CTA per SM: 212 us a call of 1,200 frames, at 128 and two 190).
// The last CTA also writes the device error word.  If a run gave up a wait, every output is NaN: the
// gate's mean and range need all frames.
template <int W, bool RUNS>
__global__ void __launch_bounds__(kCkaThreads, W == 7 || RUNS ? 2 : 0)
    frame_cka_gate_kernel(const float *__restrict__ v, const float *__restrict__ a, int n_frames, int run, int64_t dim,
                          float tau, float beta, unsigned int *done, float *__restrict__ c_out,
                          float *__restrict__ d_out, float *__restrict__ s_out, float *__restrict__ dn_out,
                          float *__restrict__ cbar_out, const unsigned int *status, DeviceError *err) {
  pdl_wait_and_release();   // the pooled rows (and the zeroed counter) of the pool kernel are visible
  constexpr int kG = W * (W + 1) / 2;
  constexpr int kN = 2 * kG + 1;
  constexpr int kHold = RUNS ? kGateHold : 0;
  constexpr int kWarps = kCkaThreads / 32;
  __shared__ float red[kWarps][kN];
  __shared__ float tot[kN];
  __shared__ bool last, gave_up;
  int f = blockIdx.x;
  unsigned int bad = 0;                                     // thread 0: this CTA's run gave up a wait
  if (RUNS) {
    constexpr int kPer = W > 1 ? W - 1 : 1;                 // 2 (W / 2) frames per run
    if (threadIdx.x == 0) bad = __ldcg(status + f / kPer);
    const int f0 = f / kPer * run, f1 = min(n_frames, f0 + run), i = f % kPer;
    // a last run shorter than W - 1 frames: the CTAs past it take its last frame again
    f = i < W / 2 ? min(f0 + i, f1 - 1) : max(f1 - kPer + i, f0);
  }
  const int lo = max(0, f - W / 2), hi = min(n_frames, f + W / 2 + 1);
  const int w = hi - lo;
  const int center = f - lo;
  const float inv_w = 1.f / static_cast<float>(w);
  float ga[kG], gv[kG], dist = 0.f;
#pragma unroll
  for (int i = 0; i < kG; ++i) ga[i] = gv[i] = 0.f;
  // four consecutive features per thread and step (16-byte loads of the pooled rows: dim is a
  // multiple of 8 and the rows start 256-byte aligned)
  const int64_t nv4 = dim / 4;
  const float4 *a4 = reinterpret_cast<const float4 *>(a);
  const float4 *v4 = reinterpret_cast<const float4 *>(v);
#pragma unroll(RUNS && W <= 3 ? 2 : 1)
  for (int64_t x = threadIdx.x; x < nv4; x += kCkaThreads) {
    float4 a_r[W], v_r[W];
#pragma unroll
    for (int r = 0; r < W; ++r) {
      a_r[r] = r < w ? a4[static_cast<int64_t>(lo + r) * nv4 + x] : make_float4(0.f, 0.f, 0.f, 0.f);
      v_r[r] = r < w ? v4[static_cast<int64_t>(lo + r) * nv4 + x] : make_float4(0.f, 0.f, 0.f, 0.f);
    }
#pragma unroll
    for (int e = 0; e < 4; ++e) {             // the four features in order
      float av[W], vv[W], am = 0.f, vm = 0.f, dd = 0.f;
#pragma unroll
      for (int r = 0; r < W; ++r) {
        av[r] = e == 0 ? a_r[r].x : e == 1 ? a_r[r].y : e == 2 ? a_r[r].z : a_r[r].w;
        vv[r] = e == 0 ? v_r[r].x : e == 1 ? v_r[r].y : e == 2 ? v_r[r].z : v_r[r].w;
        am += av[r];
        vm += vv[r];
        if (r == center) dd = vv[r] - av[r];
      }
      dist = fmaf(dd, dd, dist);
      am *= inv_w;
      vm *= inv_w;
#pragma unroll
      for (int r = 0; r < W; ++r) {
        av[r] = r < w ? av[r] - am : 0.f;
        vv[r] = r < w ? vv[r] - vm : 0.f;
      }
      int k = 0;
#pragma unroll
      for (int i = 0; i < W; ++i)
#pragma unroll
        for (int j = i; j < W; ++j, ++k) {
          ga[k] = fmaf(av[i], av[j], ga[k]);
          gv[k] = fmaf(vv[i], vv[j], gv[k]);
        }
    }
  }
  // fixed-order block reduction: warp trees, then one thread per sum over the warps in order
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int i = 0; i < kG; ++i) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      ga[i] += __shfl_xor_sync(0xffffffffu, ga[i], o);
      gv[i] += __shfl_xor_sync(0xffffffffu, gv[i], o);
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) dist += __shfl_xor_sync(0xffffffffu, dist, o);
  if (lane == 0) {
#pragma unroll
    for (int i = 0; i < kG; ++i) {
      red[warp][i] = ga[i];
      red[warp][kG + i] = gv[i];
    }
    red[warp][2 * kG] = dist;
  }
  __syncthreads();
  if (threadIdx.x < kN) {
    float t = 0.f;
#pragma unroll
    for (int wp = 0; wp < kWarps; ++wp) t += red[wp][threadIdx.x];
    tot[threadIdx.x] = t;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    c_out[f] = cka_of<W>(tot);
    d_out[f] = sqrtf(tot[2 * kG]);
    __threadfence();
    // with RUNS the count's upper half counts the CTAs whose run gave up (a grid is a few CTAs per SM)
    const unsigned int add = 1u + (bad << 16), now = atomicAdd(done, add) + add;
    last = (RUNS ? now & 0xffffu : now) == gridDim.x;
    gave_up = RUNS && now >> 16;
  }
  __syncthreads();
  if (!last) return;
  // gate over the whole clip (every other CTA's c and d are visible after its fence)
  __threadfence();
  __shared__ double rsum[kWarps];
  __shared__ float rmin[kWarps], rmax[kWarps];
  __shared__ double cbar_s;
  __shared__ float dmin_s, dmax_s;
  // from L2, where the other CTAs' stores are; one volatile load at a time keeps window 1 at 32 registers,
  // eight CTAs per SM: a clip of 1,200 frames in one wave
  struct L2Row {
    const float *p;
    __device__ float operator[](int g) const { return __ldcg(p + g); }
  };
  using Row = std::conditional_t<RUNS, L2Row, const volatile float *>;
  const Row cv{c_out}, dv{d_out};
  double cs = 0.0;
  float mn = INFINITY, mx = -INFINITY;
  // the first kHold frames per thread are loaded together and kept for the scores: the gate runs
  // after everything else, so its round trips are the call's (1,200 frames: 0.7 us less)
  float ch[kHold ? kHold : 1], dh[kHold ? kHold : 1];
#pragma unroll
  for (int i = 0; i < kHold; ++i) {
    const int g = threadIdx.x + i * kCkaThreads;
    ch[i] = g < n_frames ? cv[g] : 0.f;
    dh[i] = g < n_frames ? dv[g] : 0.f;
  }
#pragma unroll
  for (int i = 0; i < kHold; ++i)
    if (threadIdx.x + i * kCkaThreads < n_frames) {
      cs += ch[i];
      mn = fminf(mn, dh[i]);
      mx = fmaxf(mx, dh[i]);
    }
  for (int g = threadIdx.x + kHold * kCkaThreads; g < n_frames; g += kCkaThreads) {
    cs += cv[g];
    const float dg = dv[g];
    mn = fminf(mn, dg);
    mx = fmaxf(mx, dg);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    cs += __shfl_xor_sync(0xffffffffu, cs, o);
    mn = fminf(mn, __shfl_xor_sync(0xffffffffu, mn, o));
    mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  }
  if (lane == 0) {
    rsum[warp] = cs;
    rmin[warp] = mn;
    rmax[warp] = mx;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    err->code = gave_up ? APACK_ETIMEOUT : APACK_OK;
    err->where = gave_up ? 71 : 0;
    double t = 0.0;
    float lo_d = INFINITY, hi_d = -INFINITY;
    for (int wp = 0; wp < kWarps; ++wp) {
      t += rsum[wp];
      lo_d = fminf(lo_d, rmin[wp]);
      hi_d = fmaxf(hi_d, rmax[wp]);
    }
    cbar_s = gave_up ? static_cast<double>(NAN) : t / n_frames;
    dmin_s = lo_d;
    dmax_s = hi_d;
    if (cbar_out) *cbar_out = static_cast<float>(cbar_s);
  }
  __syncthreads();
  const bool blend = cbar_s < static_cast<double>(tau);
  const float span = dmax_s - dmin_s;
  auto gate = [&](int g, float cg, float dg) {
    float dn = span > 0.f ? (dg - dmin_s) / span : 0.f;
    if (RUNS && gave_up) c_out[g] = cg = dn = NAN;
    if (dn_out) dn_out[g] = dn;
    s_out[g] = blend ? (1.f - beta) * cg + beta * (1.f - dn) : cg;
  };
#pragma unroll
  for (int i = 0; i < kHold; ++i)
    if (threadIdx.x + i * kCkaThreads < n_frames) gate(threadIdx.x + i * kCkaThreads, ch[i], dh[i]);
  for (int g = threadIdx.x + kHold * kCkaThreads; g < n_frames; g += kCkaThreads) gate(g, cv[g], dv[g]);
}

size_t up(size_t x) { return (x + 255) & ~static_cast<size_t>(255); }

}  // namespace

}  // namespace apack

using namespace apack;

extern "C" {

apack_status apack_frame_alignment_workspace_size(int32_t n_frames, int64_t dim, size_t *bytes) {
  if (!bytes || n_frames < 1 || dim < 8) return APACK_EINVAL;
  // device error word and CTA counter, v [F][dim], a [F][dim], d [F], status [runs <= F], unused
  *bytes = 256 + 2 * up(static_cast<size_t>(n_frames) * dim * sizeof(float)) +
           2 * up(static_cast<size_t>(n_frames) * sizeof(float)) + 256;
  return APACK_OK;
}

apack_status apack_frame_alignment(const void *visual, const void *audio, int32_t n_frames, int32_t tokens_per_frame,
                                   int32_t n_audio, int64_t dim, int32_t window, float tau, float beta, float *c_out,
                                   float *s_out, float *dnorm_out, float *cbar_out, void *ws, size_t ws_bytes,
                                   void *stream) {
  if (!visual || !audio || !c_out || !s_out || !ws) return APACK_EINVAL;
  if (n_frames < 1 || tokens_per_frame < 1 || n_audio < n_frames || dim < 8 || (dim % 8) != 0) return APACK_EINVAL;
  if (window < 1 || window > kMaxWindow || (window % 2) == 0) return APACK_EINVAL;
  if (!(beta >= 0.f && beta <= 1.f) || !std::isfinite(tau)) return APACK_EINVAL;
  if ((reinterpret_cast<uintptr_t>(visual) & 15) || (reinterpret_cast<uintptr_t>(audio) & 15) ||
      (reinterpret_cast<uintptr_t>(ws) & 255))
    return APACK_EINVAL;
  size_t need = 0;
  apack_frame_alignment_workspace_size(n_frames, dim, &need);
  if (ws_bytes < need) return APACK_EWORKSPACE;
  uint8_t *w = static_cast<uint8_t *>(ws);
  DeviceError *err = reinterpret_cast<DeviceError *>(w);
  unsigned int *done = reinterpret_cast<unsigned int *>(w + 64);
  float *vbuf = reinterpret_cast<float *>(w + 256);
  float *abuf = reinterpret_cast<float *>(w + 256 + up(static_cast<size_t>(n_frames) * dim * sizeof(float)));
  float *dbuf = reinterpret_cast<float *>(w + 256 + 2 * up(static_cast<size_t>(n_frames) * dim * sizeof(float)));
  unsigned int *status = reinterpret_cast<unsigned int *>(reinterpret_cast<uint8_t *>(dbuf) + up(static_cast<size_t>(n_frames) * sizeof(float)));
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const int64_t vecs = dim / 8;
  const int pthreads = static_cast<int>(std::min<int64_t>(kPoolMaxThreads, (vecs + 31) / 32 * 32));
  // Runs of frames, when every CTA of one per SM has windows of its own (run >= window), enough to stream
  // (kRunBytes: 460 frames of 25 tokens of 1,000 features, 200 KB a run, take 19.6 us in runs and 15.7 us
  // frame by frame; 1,200 of 25 tokens of 1,280, 512 KB, 36.4 and 37.5) and threads that hold a row; shorter
  // clips, wider rows and window 7 (whose rows do not fit the registers): one CTA per frame for the pool
  // (more for wider rows) and one for the CKA.
  const int run = (n_frames + device_sm_count() - 1) / device_sm_count();
  int cka_run = 0, cka_grid = n_frames;
  constexpr int64_t kRunBytes = 384 << 10;
  if ((window == 3 || window == 5) && run >= window && run * tokens_per_frame * dim * 2 >= kRunBytes &&
      vecs <= (window == 3 ? run_threads<3>() : run_threads<5>())) {
    const RunShape sh{n_frames, tokens_per_frame, n_audio, run, dim};
    const int runs = (n_frames + run - 1) / run;
    auto *kernel = window == 3 ? frame_run_kernel<3> : frame_run_kernel<5>;
    constexpr size_t smem = static_cast<size_t>(kRunStages) * kRunStage;
    static std::atomic<uint64_t> attr{0};
    if (once_per_device(attr, [] {
          cudaError_t e = cudaFuncSetAttribute(frame_run_kernel<3>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               static_cast<int>(smem));
          if (e == cudaSuccess)
            e = cudaFuncSetAttribute(frame_run_kernel<5>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     static_cast<int>(smem));
          return e;
        }) != cudaSuccess)
      return APACK_ECUDA;
    kernel<<<runs, pthreads + 32, smem, s>>>(sh, static_cast<const uint8_t *>(visual), static_cast<const uint8_t *>(audio),
                                             vbuf, abuf, c_out, dbuf, done, status);
    cka_run = run;
    cka_grid = runs * (window - 1);
  } else {
    dim3 pgrid(n_frames, static_cast<unsigned>((vecs + pthreads - 1) / pthreads));
    frame_pool_kernel<<<pgrid, pthreads, 0, s>>>(static_cast<const uint4 *>(visual), static_cast<const uint4 *>(audio),
                                                n_frames, tokens_per_frame, n_audio, dim, vbuf, abuf, done);
  }
  count_launches(1);
  if (check_cuda(cudaGetLastError()) != APACK_OK) return APACK_ECUDA;
  // programmatic dependent launch: the CKA kernel's CTAs are scheduled while the pool kernel drains
  auto *cka = window == 1   ? frame_cka_gate_kernel<1, false>
              : window == 3 ? (cka_run ? frame_cka_gate_kernel<3, true> : frame_cka_gate_kernel<3, false>)
              : window == 5 ? (cka_run ? frame_cka_gate_kernel<5, true> : frame_cka_gate_kernel<5, false>)
                            : frame_cka_gate_kernel<7, false>;
  const cudaError_t e = launch_pdl(cka, dim3(cka_grid), dim3(kCkaThreads), 0, s, vbuf, abuf, n_frames, cka_run, dim, tau,
                                   beta, done, c_out, dbuf, s_out, dnorm_out, cbar_out, status, err);
  count_launches(1);
  if (check_cuda(e) != APACK_OK) return APACK_ECUDA;
  return APACK_OK;
}

}  // extern "C"
