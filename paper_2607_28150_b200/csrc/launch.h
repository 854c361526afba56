// Host-side helpers shared between translation units of the library (not part of the public ABI).
#pragma once
#include <stddef.h>
#include <stdint.h>

#include "smartgen.h"

namespace sg {
size_t score_workspace_bytes(const sg_shape* shape);
size_t decode_workspace_bytes(const sg_shape* shape, int32_t total_sel, int32_t total_loc);
// Cluster size (CTAs per sequence and KV head) the decode kernel uses for a call of this size.
void decode_plan(const sg_shape* shape, int32_t total_sel, int32_t total_loc, bool two_lane, int* csize, int* warps, int* slots);
// Threshold selection in one kernel, for rows that the register-resident selection holds.
bool select_threshold_fits(const sg_shape* shape);
sg_status select_threshold_launch(const sg_shape* shape, const float* scores, float alpha, const int32_t* cu_cap, int32_t total_cap,
                                  int32_t* sel_idx, int32_t* sel_count, int32_t* dev_status, void* stream);
}  // namespace sg
