// What score.cu hands to score_cluster.cu.
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "smartgen.h"

namespace sg {
struct ScoreLaunch {
  float* importance;
  int32_t* dev_status;
  int32_t withhold_unit;   // testing only
  uint32_t wait_ns;
  cudaStream_t stream;
};
// Selection and packing behind the scores (arguments of sg_select_pack_kv).
struct PackLaunch {
  const int32_t* cu_k;
  int32_t total_sel;
  const void* k_cache;
  const void* v_cache;
  int32_t* sel_idx;
  void* packed_k;
  void* packed_v;
};
// CTAs per part where score_cluster.cu's kernel takes calls of this shape (one that score.cu supports), else 0.  packs: with selection
// and packing.
int score_cluster_size(const sg_shape* shape, bool packs);
// The tensor maps are score.cu's.  pack = null: scores only.
sg_status score_cluster_launch(const sg_shape* shape, const CUtensorMap& q, const CUtensorMap& k, const ScoreLaunch& args, const PackLaunch* pack);
}  // namespace sg
