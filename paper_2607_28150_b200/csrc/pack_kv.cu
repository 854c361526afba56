// sg_pack_kv: index-driven gather of selected K/V rows into a contiguous buffer.
//
// Pure byte movement, bound by HBM: every selected row (2*d bytes of K, 2*d bytes of V) is read
// once and written once.  A CTA takes 64 (d = 128) or 128 (d = 64) neighbouring entries of one (layer, KV head) of the
// KV index.  First one thread per entry reads the index and works out where the row comes from and goes to; then
// groups of d/8 threads move the rows with 16-byte vectors, so a warp's accesses cover whole 128-byte lines on both
// sides, four rows (eight loads) per group in flight before the first store.  With every thread of a group working
// out its own row (two 64-bit divisions, a search and four dependent loads per row), the address chain and not the bytes
// set the pace of short and of counted calls.
#include "common.cuh"

namespace sg {
namespace {

constexpr int kPackThreads = 256;
constexpr int kUnroll = 4;

struct PackParams {
  const uint16_t* k_cache;
  const uint16_t* v_cache;
  const int32_t* sel_idx;
  const int32_t* cu;
  const int32_t* cu_k;
  const int32_t* sel_count;   // [L][B][Hkv] entries selected per row, or null: every entry of the row
  uint16_t* packed_k;
  uint16_t* packed_v;
  int32_t* dev_status;
  int64_t ls, ts, hs;
  int32_t K_tot, B, Hkv;
  int32_t chunks;          // CTAs per (layer, KV head)
};

// kCounted: rows beyond a head's count (PackParams::sel_count) are skipped; the plain instantiation carries none of it.
template <int D, bool kCounted>
__global__ void __launch_bounds__(kPackThreads) pack_kv_kernel(const PackParams p) {
  constexpr int kTPR = D / 8;                       // threads per row, 16 bytes each
  constexpr int kGroups = kPackThreads / kTPR, kRows = kGroups * kUnroll;
  __shared__ int64_t s_src[kRows], s_dst[kRows];    // element offsets; source -1: zeros, destination -1: nothing to do
  pdl_wait();
  const int lg = blockIdx.x / p.chunks, e0 = (blockIdx.x - lg * p.chunks) * kRows;
  const int l = lg / p.Hkv, g = lg - l * p.Hkv;
  if (threadIdx.x < kRows) {
    const int e = e0 + threadIdx.x, lane = threadIdx.x & 31;
    int64_t src = -1, dst = -1;
    // the sequence that holds the warp's first entry, then on from there
    int b = 0;
    if (p.B > 32) {
      b = upper_segment(p.cu_k, p.B, e - lane);
    } else if (p.B > 1) {
      const int end = lane < p.B ? p.cu_k[lane + 1] : 0x7fffffff;
      b = min(__popc(__ballot_sync(0xffffffffu, end <= e - lane)), p.B - 1);
    }
    if (e < p.K_tot) {
      int ck = p.cu_k[b], ce = p.cu_k[b + 1];
      while (e >= ce && b + 1 < p.B) { ++b; ck = ce; ce = p.cu_k[b + 1]; }
      const int kb = ce - ck, j = e - ck;
      if (j >= kb) {
        raise(p.dev_status, SG_ERR_INVALID);          // the host's total is larger than cu_k[B]: no row owns the entry
      } else if (!kCounted || j < p.sel_count[((int64_t)l * p.B + b) * p.Hkv + g]) {
        dst = ((int64_t)l * p.K_tot * p.Hkv + (int64_t)ck * p.Hkv + (int64_t)g * kb + j) * D;
        const int t = p.sel_idx[(int64_t)lg * p.K_tot + e];
        const int c0 = p.cu[b];
        if (t >= 0 && t < p.cu[b + 1] - c0) src = l * p.ls + ((int64_t)c0 + t) * p.ts + (int64_t)g * p.hs;
        else raise(p.dev_status, SG_ERR_INDEX);
      }
    }
    s_src[threadIdx.x] = src;
    s_dst[threadIdx.x] = dst;
  }
  __syncthreads();
  const int x = (threadIdx.x % kTPR) * 8, group = threadIdx.x / kTPR;
  int4 kv[kUnroll][2];
#pragma unroll
  for (int u = 0; u < kUnroll; ++u) {
    const int64_t src = s_src[group + u * kGroups];
    kv[u][0] = make_int4(0, 0, 0, 0);
    kv[u][1] = make_int4(0, 0, 0, 0);
    if (src >= 0) {
      kv[u][0] = __ldcs(reinterpret_cast<const int4*>(p.k_cache + src + x));
      kv[u][1] = __ldcs(reinterpret_cast<const int4*>(p.v_cache + src + x));
    }
  }
#pragma unroll
  for (int u = 0; u < kUnroll; ++u) {
    const int64_t dst = s_dst[group + u * kGroups];
    if (dst >= 0) {
      __stcs(reinterpret_cast<int4*>(p.packed_k + dst + x), kv[u][0]);
      __stcs(reinterpret_cast<int4*>(p.packed_v + dst + x), kv[u][1]);
    }
  }
}

}  // namespace
}  // namespace sg

namespace sg {
namespace {
sg_status pack_kv_launch(const sg_shape* shape, const void* k_cache, const void* v_cache, const int32_t* sel_idx,
                         const int32_t* cu_k, int32_t total_sel, const int32_t* sel_count, void* packed_k, void* packed_v,
                         int32_t* dev_status, void* stream);
}
}  // namespace sg

extern "C" sg_status sg_pack_kv(const sg_shape* shape, const void* k_cache, const void* v_cache,
                                const int32_t* sel_idx, const int32_t* cu_k, int32_t total_sel,
                                void* packed_k, void* packed_v, int32_t* dev_status, void* stream) {
  return sg::pack_kv_launch(shape, k_cache, v_cache, sel_idx, cu_k, total_sel, nullptr, packed_k, packed_v, dev_status, stream);
}

extern "C" sg_status sg_pack_kv_counted(const sg_shape* shape, const void* k_cache, const void* v_cache,
                                        const int32_t* sel_idx, const int32_t* cu_cap, int32_t total_cap,
                                        const int32_t* sel_count, void* packed_k, void* packed_v, int32_t* dev_status,
                                        void* stream) {
  if (!sel_count || !sg::aligned16(sel_count)) return SG_ERR_INVALID;
  return sg::pack_kv_launch(shape, k_cache, v_cache, sel_idx, cu_cap, total_cap, sel_count, packed_k, packed_v, dev_status, stream);
}

namespace sg {
namespace {
sg_status pack_kv_launch(const sg_shape* shape, const void* k_cache, const void* v_cache, const int32_t* sel_idx,
                         const int32_t* cu_k, int32_t total_sel, const int32_t* sel_count, void* packed_k, void* packed_v,
                         int32_t* dev_status, void* stream) {
  using namespace sg;
  sg_status st = check_shape(shape, false);
  if (st != SG_OK) return st;
  if (total_sel < 0) return SG_ERR_INVALID;
  if (total_sel == 0) return SG_OK;
  if (!k_cache || !v_cache || !sel_idx || !cu_k || !packed_k || !packed_v) return SG_ERR_INVALID;
  if (!aligned16(k_cache) || !aligned16(v_cache) || !aligned16(sel_idx) || !aligned16(cu_k) ||
      !aligned16(packed_k) || !aligned16(packed_v))
    return SG_ERR_INVALID;
  PackParams p;
  p.k_cache = static_cast<const uint16_t*>(k_cache);
  p.v_cache = static_cast<const uint16_t*>(v_cache);
  p.sel_idx = sel_idx;
  p.cu = shape->cu_seqlens;
  p.cu_k = cu_k;
  p.sel_count = sel_count;
  p.packed_k = static_cast<uint16_t*>(packed_k);
  p.packed_v = static_cast<uint16_t*>(packed_v);
  p.dev_status = dev_status;
  p.ls = shape->cache_layer_stride;
  p.ts = shape->cache_token_stride;
  p.hs = shape->cache_head_stride;
  p.K_tot = total_sel;
  p.B = shape->batch;
  p.Hkv = shape->num_kv_heads;
  const int rows = kPackThreads / (shape->head_dim / 8) * kUnroll;
  p.chunks = total_sel / rows + (total_sel % rows != 0);
  const int64_t grid = (int64_t)p.chunks * shape->num_layers * shape->num_kv_heads;
  if (grid > 0x7fffffffLL) return SG_ERR_UNSUPPORTED;
  if (shape->head_dim == 128)
    return launch_chained(sel_count ? pack_kv_kernel<128, true> : pack_kv_kernel<128, false>, dim3((unsigned)grid), kPackThreads, p, stream);
  return launch_chained(sel_count ? pack_kv_kernel<64, true> : pack_kv_kernel<64, false>, dim3((unsigned)grid), kPackThreads, p, stream);
}
}  // namespace
}  // namespace sg
