// narrow_plan.cuh -- launch plan of the narrow scoring path, shared by its CUDA-core and
// tensor-core logits kernels and by the merge and final kernels.
#pragma once
#include <cstdint>

#include "internal.cuh"

namespace apack {

struct NSeq {
  int32_t t0, len;
  int32_t q_off, n_q;
  int32_t unit_begin;                  // first 256-key CTA of this sequence (general logits kernel)
  int32_t unit8_begin;                 // first CTA of this sequence (tensor-core logits kernel)
  int32_t chunk;                       // tensor-core kernel: stages (KV head of a 128-key tile) per CTA
  int32_t stages;                      // and in all
  int32_t final_begin;                 // first CTA of this sequence (final kernel)
  int32_t nparts;                      // CTA partials of the logits kernel in use
  int32_t rows;                        // logit rows R = Hq * n_q
  int32_t q_pos;                       // causal rows: position of query row 0 within the sequence
  int64_t lstride;                     // logit row stride: len rounded up to kLogitPad
  int64_t logit_base;                  // float offset of this sequence's logits [R][lstride]
  int64_t part_base;                   // float2 offset of its CTA partials [R][nparts]
  int64_t lse_base;                    // float offset of its lse2 [R]
};

struct NarrowPlan {
  int32_t nseq;
  int32_t hq, hkv, group;
  int32_t stream_keys;                 // tensor-core kernel: keys are the first to leave L2
  int32_t causal;                      // APACK_SOFTMAX_CAUSAL_ROW: row r of n_q sees keys <= q_pos + r
  float scale2;
  NSeq seq[kSeqsPerLaunch];
};

__device__ __forceinline__ int find_unit_seq(const NarrowPlan &p, int u) {
  int s = 0;
  while (s + 1 < p.nseq && p.seq[s + 1].unit_begin <= u) ++s;
  return s;
}

__device__ __forceinline__ int find_final_seq(const NarrowPlan &p, int u) {
  int s = 0;
  while (s + 1 < p.nseq && p.seq[s + 1].final_begin <= u) ++s;
  return s;
}

__device__ __forceinline__ int find_unit8_seq(const NarrowPlan &p, int u) {
  int s = 0;
  while (s + 1 < p.nseq && p.seq[s + 1].unit8_begin <= u) ++s;
  return s;
}

// Tensor-core logits kernel of the narrow path (score_narrow_tc.cu): Hkv = 1, 2, 4 or 8, at most
// max_rg <= 32 query rows per KV head group; `grid` CTAs, placed by unit8_begin and chunk.
cudaError_t launch_narrow_tc(int max_rg, int grid, cudaStream_t stream, const CUtensorMap &kmap, const NarrowPlan &P,
                             const uint16_t *q, const uint8_t *modality, float *logits, float2 *part,
                             DeviceError *err);

}  // namespace apack
