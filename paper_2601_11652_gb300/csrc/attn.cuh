// attn.cuh -- parameters of the attention kernels.
#pragma once

#include "plan.cuh"

namespace wisp {

struct AttnParams {
  int B, Hq, Hkv, D, max_blocks_per_seq, num_blocks;
  const int64_t *request_ids;
  const int32_t *block_tables;
  const void *q, *k_cache, *v_cache;
  void *out;
  DeviceStatus *status;
  const int32_t *req_chunks;
  const PlanHeader *header;
  PlanHeader *header_mut;  // same object: the work counter
  const WorkItem *items;  // in dispatch order
  float *partials;
  int row_groups;      // row groups per (request, head) at most
  int32_t *pair_done;  // [B * Hkv * row_groups] finished chunks of each split (request, head, row group), zeroed
                       // by the planner
};

// Host launchers (defined next to their kernels): programmatic dependents of the planner, which they wait for
// before they read the plan.
// CUDA-core kernel for fp32 KV, D in {64, 128}; `grid` persistent CTAs
cudaError_t attn_f32_setup();  // once per device: shared-memory attributes
cudaError_t attn_f32_launch(const AttnParams &p, int grid, cudaStream_t s);
// tcgen05 / TMA kernel for bf16 KV, D in {64, 128}; `grid` persistent CTAs
cudaError_t attn_tc_setup();
cudaError_t attn_tc_launch(const AttnParams &p, int grid, cudaStream_t s);

}  // namespace wisp
