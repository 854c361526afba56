// What the library exports for csrc/native.cpp alone (not part of the public ABI).
#pragma once
#include "smartgen.h"

// sg_score, then sg_select_pack_kv, where one kernel does both; SG_ERR_UNSUPPORTED, with nothing launched, for everything else, bad
// arguments included (the two calls then say what is wrong).
extern "C" sg_status sg_internal_score_select_pack(const sg_shape* shape, const void* q_win, const void* k_cache, const void* v_cache,
                                                   float* importance, void* workspace, size_t workspace_bytes, const int32_t* cu_k,
                                                   int32_t total_sel, int32_t* sel_idx, void* packed_k, void* packed_v,
                                                   int32_t* dev_status, void* stream);
