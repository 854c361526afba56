// sg_split_index: Algorithm 1 (KV index splitting and reordering) on the device.
//
// One CTA owns one row of the KV index (one sequence, one KV head).  It looks up the int8 class of every
// selected token in the KV mask (2 = remote, 1 = local, 0 = padding) and forms a stable three-way partition of
// the row by class -- remote first, then local, then padding -- with ballots and prefix counts: no atomics, so
// the output order is a pure function of the input.  The partitioned row (when asked for) and the local and
// remote index lists with their counts are written.  Integer work only, bound by latency (a row is a few KB): two
// dependent loads per entry, index then mask.  So every thread has several entries in flight, and a row that they cover is
// looked up once and stays in registers between the counting and the placing.
#include "common.cuh"

namespace sg {
namespace {

struct SplitParams {
  const int32_t* kv_index;
  const int8_t* kv_mask;
  const int32_t* cu;
  const int32_t* cu_k;
  int32_t* reordered;
  int32_t* local_index;
  int32_t* remote_index;
  int32_t* n_local;
  int32_t* n_remote;
  int32_t* dev_status;
  int32_t K_tot, B, Hkv, reorder;
};

// kFlight: entries in flight per thread.
template <int kSplitThreads, int kFlight>
__global__ void __launch_bounds__(kSplitThreads) split_index_kernel(const SplitParams p) {
  constexpr int kSplitWarps = kSplitThreads / 32;
  __shared__ uint32_t w_cnt[3][kSplitWarps];     // per-warp counts of classes remote / local / padding
  __shared__ uint32_t w_base[3][kSplitWarps];
  __shared__ uint32_t tot[3];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int b = blockIdx.x / p.Hkv, g = blockIdx.x - b * p.Hkv;
  pdl_wait();
  const int c0 = p.cu[b], N = p.cu[b + 1] - c0;
  const int ck = p.cu_k[b], kb = p.cu_k[b + 1] - ck;
  const int64_t base = (int64_t)g * p.K_tot + ck;
  // warp w owns positions [w*C, (w+1)*C) of the row, C a multiple of 32; lane i its positions beg + i, + 32, ...
  const int C = (((kb + kSplitWarps - 1) / kSplitWarps) + 31) & ~31;
  const int beg = warp * C, end = min(kb, beg + C);
  int t[kFlight], cls[kFlight];                      // class: 0 remote, 1 local, 2 padding (or invalid), 3 nothing
  auto look_up = [&](int j0) {
#pragma unroll
    for (int i = 0; i < kFlight; ++i) {
      const int j = j0 + 32 * i + lane;
      t[i] = j < end ? p.kv_index[base + j] : -1;
    }
#pragma unroll
    for (int i = 0; i < kFlight; ++i) {
      const bool in = t[i] >= 0 && t[i] < N;
      const int m = in ? p.kv_mask[c0 + t[i]] : 0;
      cls[i] = j0 + 32 * i + lane >= end ? 3 : (m == 2 ? 0 : (m == 1 ? 1 : 2));
      if (cls[i] != 3 && !in) raise(p.dev_status, SG_ERR_INDEX);
    }
  };
  uint32_t cnt[3] = {0, 0, 0};
  for (int j0 = beg; j0 < end; j0 += 32 * kFlight) {
    look_up(j0);
#pragma unroll
    for (int i = 0; i < kFlight; ++i)
#pragma unroll
      for (int c = 0; c < 3; ++c) cnt[c] += __popc(__ballot_sync(0xffffffffu, cls[i] == c));
  }
  if (lane == 0) { w_cnt[0][warp] = cnt[0]; w_cnt[1][warp] = cnt[1]; w_cnt[2][warp] = cnt[2]; }
  __syncthreads();
  if (warp < 3) {
    const uint32_t v = lane < kSplitWarps ? w_cnt[warp][lane] : 0u;
    uint32_t inc = v;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const uint32_t u = __shfl_up_sync(0xffffffffu, inc, off);
      if (lane >= off) inc += u;
    }
    if (lane < kSplitWarps) w_base[warp][lane] = inc - v;
    if (lane == 31) tot[warp] = inc;
  }
  __syncthreads();
  const uint32_t n_rem = tot[0], n_loc = tot[1];
  if (tid == 0) { p.n_remote[b * p.Hkv + g] = (int32_t)n_rem; p.n_local[b * p.Hkv + g] = (int32_t)n_loc; }
  uint32_t run[3] = {w_base[0][warp], w_base[1][warp], w_base[2][warp]};
  const uint32_t lt = (1u << lane) - 1u;
  for (int j0 = beg; j0 < end; j0 += 32 * kFlight) {
    if (C > 32 * kFlight) look_up(j0);               // shorter pieces are still in registers
#pragma unroll
    for (int i = 0; i < kFlight; ++i) {
      uint32_t bal[3];
#pragma unroll
      for (int c = 0; c < 3; ++c) bal[c] = __ballot_sync(0xffffffffu, cls[i] == c);
      if (cls[i] < 3) {
        const uint32_t rank = (cls[i] == 0 ? run[0] : cls[i] == 1 ? run[1] : run[2]) + __popc((cls[i] == 0 ? bal[0] : cls[i] == 1 ? bal[1] : bal[2]) & lt);
        if (cls[i] == 0) p.remote_index[base + rank] = t[i];
        if (cls[i] == 1) p.local_index[base + rank] = t[i];
        if (p.reordered) {
          const uint32_t dst = p.reorder ? (cls[i] == 0 ? rank : (cls[i] == 1 ? n_rem + rank : n_rem + n_loc + rank)) : (uint32_t)(j0 + 32 * i + lane);
          p.reordered[base + dst] = t[i];
        }
      }
#pragma unroll
      for (int c = 0; c < 3; ++c) run[c] += __popc(bal[c]);
    }
  }
}

}  // namespace
}  // namespace sg

extern "C" sg_status sg_split_index(const sg_shape* shape, const int32_t* kv_index, const int32_t* cu_k,
                                    int32_t total_sel, const int8_t* kv_mask, int32_t reorder, int32_t* reordered,
                                    int32_t* local_index, int32_t* remote_index, int32_t* n_local, int32_t* n_remote,
                                    int32_t* dev_status, void* stream) {
  using namespace sg;
  sg_status st = check_shape(shape, false);
  if (st != SG_OK) return st;
  if (shape->num_layers != 1 || total_sel < 0) return SG_ERR_INVALID;
  if (!cu_k || !n_local || !n_remote) return SG_ERR_INVALID;
  if (total_sel > 0 && (!kv_index || !kv_mask || !local_index || !remote_index)) return SG_ERR_INVALID;
  if (!aligned16(kv_index) || !aligned16(cu_k) || !aligned16(local_index) || !aligned16(remote_index) ||
      !aligned16(reordered) || (reinterpret_cast<uintptr_t>(n_local) & 3u) || (reinterpret_cast<uintptr_t>(n_remote) & 3u))
    return SG_ERR_INVALID;
  const int64_t rows = (int64_t)shape->batch * shape->num_kv_heads;
  if (rows > 0x7fffffffLL) return SG_ERR_UNSUPPORTED;
  SplitParams p;
  p.kv_index = kv_index;
  p.kv_mask = kv_mask;
  p.cu = shape->cu_seqlens;
  p.cu_k = cu_k;
  p.reordered = reordered;
  p.local_index = local_index;
  p.remote_index = remote_index;
  p.n_local = n_local;
  p.n_remote = n_remote;
  p.dev_status = dev_status;
  p.K_tot = total_sel;
  p.B = shape->batch;
  p.Hkv = shape->num_kv_heads;
  p.reorder = reorder ? 1 : 0;
  // The CTA size is chosen for a row of the longest sequence, if the budgets are shares of the lengths (any row is split
  // correctly): four entries per thread hold the row in registers, two for the shortest rows, eight up to 8192 entries; longer
  // rows are looked up twice in flights of four.  More threads or entries than the row needs are idle steps in every ballot
  // loop, and fewer CTAs are resident.  Microseconds (1024 threads with eight entries each for every row -> these rules; 256
  // threads, one entry at a time): 320 rows of 128 entries 7.8 -> 2.2 (3.0), 320 of 820 12.4 -> 3.7 (5.6), 64 of 2000 5.2 -> 3.3
  // (7.7), 64 of 3277 5.3 -> 4.1 (11.2), 64 of 6000 6.3 (20.7; four entries per thread 7.5), 64 of 16000 14.8 -> 14.3 (51.7).
  const int64_t average = total_sel / shape->batch;
  const int64_t scaled = shape->total_tokens > 0 ? (int64_t)total_sel * shape->max_seqlen / shape->total_tokens : 0;
  const int64_t longest = scaled > average ? scaled : average;
  const dim3 grid((unsigned)rows);
  if (longest <= 256) return launch_chained(split_index_kernel<128, 2>, grid, 128, p, stream);
  if (longest <= 1024) return launch_chained(split_index_kernel<256, 4>, grid, 256, p, stream);
  if (longest <= 2048) return launch_chained(split_index_kernel<512, 4>, grid, 512, p, stream);
  if (longest > 4096 && longest <= 8192) return launch_chained(split_index_kernel<1024, 8>, grid, 1024, p, stream);
  return launch_chained(split_index_kernel<1024, 4>, grid, 1024, p, stream);
}
