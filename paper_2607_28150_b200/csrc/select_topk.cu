// sg_select_topk: per-(layer, sequence, KV head) top-k by exact selection of the k-th largest key.
//
// One CTA owns one importance row.  The row's fp32 values are mapped to order-preserving uint32 keys.
// Rows of up to 32768 tokens keep their keys in registers (second kernel below: histograms over a shrinking
// key interval, direct ranking of the last few keys, output from bit masks; optionally fused with the gather
// of the selected K/V rows).  Longer rows keep the keys in shared memory (up to ~55K tokens) or re-read them
// from L2 (first kernel): four 8-bit MSB-first histogram passes find the k-th largest key exactly and a final
// ordered compaction (ballot + prefix counts, no atomics) emits the selected positions in ascending order.
// Both take equal-to-threshold entries from the lowest positions first.  The result is therefore a pure
// function of the input row: identical on every run and identical to a full sort.
#include <type_traits>

#include "common.cuh"
#include "select_key.cuh"

namespace sg {
namespace {

constexpr int kSelThreads = 1024;
constexpr int kSelWarps = kSelThreads / 32;
constexpr int kHistCopies = 8;
constexpr int kMaxSmemBytes = 227 * 1024;
constexpr int kSelFixedSmem = (kHistCopies * 256 + 256 + 4 * kSelWarps + 8) * 4;
constexpr int kSelKeyCap = (kMaxSmemBytes - kSelFixedSmem) / 4;

struct SelParams {
  const float* importance;
  const int32_t* cu;
  const int32_t* cu_k;
  int32_t* sel_idx;
  int32_t* dev_status;
  int64_t T;
  int32_t K_tot, B, Hkv;
  int32_t capacity;        // longest row the launched kernel variant can hold (from shape->max_seqlen); 0 = any length
  // fused packing (select_topk_reg_kernel with PD > 0): the CTA that selected a row also gathers its K/V rows
  const uint16_t* k_cache;
  const uint16_t* v_cache;
  uint16_t* packed_k;
  uint16_t* packed_v;
  int64_t ls, ts, hs;
  // threshold selection (select_topk_reg_kernel with kThr): keep only what exceeds the row maximum minus alpha
  int32_t* sel_count;      // [L][B][Hkv]
  float alpha;
};

// The selection kernels are launched with programmatic stream serialization: when the kernel before them in the
// stream (normally the scoring kernel) lets its dependents go early, their CTAs are placed while it drains, and
// the launch latency disappears behind it.  They do not let their own dependents go early: with the gather of 64 ragged rows
// placed beside its selection (84 SMs free) a call of scoring, selection and packing, replayed from a graph, took 139.0 us, 136.1 without.

template <bool kInSmem>
__global__ void __launch_bounds__(kSelThreads, 1) select_topk_kernel(const SelParams p) {
  pdl_wait();
  extern __shared__ __align__(16) uint32_t smem[];
  uint32_t* hist = smem;                              // [kHistCopies][256]
  uint32_t* total = hist + kHistCopies * 256;         // [256]
  uint32_t* wgt = total + 256;                        // [kSelWarps] per-warp counts / bases
  uint32_t* weq = wgt + kSelWarps;
  uint32_t* wgt_base = weq + kSelWarps;
  uint32_t* weq_base = wgt_base + kSelWarps;
  uint32_t* sh = weq_base + kSelWarps;                // [0] chosen bin, [1] remaining need
  uint32_t* keys = sh + 8;                            // [N] when kInSmem

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int row = blockIdx.x;
  const int l = row / (p.B * p.Hkv);
  const int rem = row - l * (p.B * p.Hkv);
  const int b = rem / p.Hkv;
  const int g = rem - b * p.Hkv;
  const int c0 = p.cu[b];
  const int N = p.cu[b + 1] - c0;
  const int ck = p.cu_k[b];
  const int kb = p.cu_k[b + 1] - ck;
  if (kb <= 0) return;
  int32_t* out = p.sel_idx + ((int64_t)l * p.Hkv + g) * p.K_tot + ck;
  if (p.capacity > 0 && N > p.capacity) {
    // The row is longer than the shape's max_seqlen promised (the key array was sized from it): flag it and
    // emit an empty row instead of touching memory the launch did not provide.
    if (tid == 0) raise(p.dev_status, SG_ERR_INVALID);
    for (int j = tid; j < kb; j += kSelThreads) out[j] = -1;
    return;
  }
  if (kb >= N) {                                      // whole prompt (or an over-sized budget)
    if (kb > N && tid == 0) raise(p.dev_status, SG_ERR_INVALID);
    for (int j = tid; j < kb; j += kSelThreads) out[j] = j < N ? j : -1;
    return;
  }
  const uint32_t* x = reinterpret_cast<const uint32_t*>(p.importance) + ((int64_t)l * p.Hkv + g) * p.T + c0;

  if (kInSmem) {
    for (int t = tid; t < N; t += kSelThreads) keys[t] = order_key(x[t]);
  }
  auto key_at = [&](int t) -> uint32_t { return kInSmem ? keys[t] : order_key(x[t]); };

  // ---- radix select: find the kb-th largest key ----
  uint32_t prefix = 0, decided = 0, need = (uint32_t)kb;
#pragma unroll 1
  for (int pass = 0; pass < 4; ++pass) {
    const int shift = 24 - 8 * pass;
    for (int i = tid; i < kHistCopies * 256; i += kSelThreads) hist[i] = 0;
    __syncthreads();
    uint32_t* my_hist = hist + (warp % kHistCopies) * 256;
    for (int t = tid; t < N; t += kSelThreads) {
      const uint32_t k = key_at(t);
      if ((k & decided) == prefix) atomicAdd(&my_hist[(k >> shift) & 255u], 1u);
    }
    __syncthreads();
    if (tid < 256) {
      uint32_t s = 0;
#pragma unroll
      for (int c = 0; c < kHistCopies; ++c) s += hist[c * 256 + tid];
      total[tid] = s;
    }
    __syncthreads();
    if (warp == 0) {
      uint32_t c[8], s = 0;
#pragma unroll
      for (int i = 0; i < 8; ++i) { c[i] = total[255 - (lane * 8 + i)]; s += c[i]; }
      uint32_t inc = s;
#pragma unroll
      for (int off = 1; off < 32; off <<= 1) {
        const uint32_t v = __shfl_up_sync(0xffffffffu, inc, off);
        if (lane >= off) inc += v;
      }
      const uint32_t exc = inc - s;                   // candidates in bins above this lane's bins
      if (exc < need && need <= inc) {
        uint32_t run = exc;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          if (run < need && need <= run + c[i]) { sh[0] = 255u - (uint32_t)(lane * 8 + i); sh[1] = need - run; }
          run += c[i];
        }
      }
    }
    __syncthreads();
    prefix |= sh[0] << shift;
    decided |= 255u << shift;
    need = sh[1];
    __syncthreads();
  }
  const uint32_t tau = prefix;                        // the kb-th largest key
  const uint32_t need_eq = need;                      // entries equal to tau to keep, lowest positions first

  // ---- ordered compaction: warp w owns positions [w*C, (w+1)*C) ----
  const int C = (((N + kSelWarps - 1) / kSelWarps) + 31) & ~31;
  const int beg = warp * C;
  const int end = min(N, beg + C);
  uint32_t ngt = 0, neq = 0;
  for (int t0 = beg; t0 < end; t0 += 32) {
    const int t = t0 + lane;
    const uint32_t k = t < end ? key_at(t) : 0u;
    ngt += __popc(__ballot_sync(0xffffffffu, t < end && k > tau));
    neq += __popc(__ballot_sync(0xffffffffu, t < end && k == tau));
  }
  if (lane == 0) { wgt[warp] = ngt; weq[warp] = neq; }
  __syncthreads();
  if (warp == 0) {
    uint32_t a = wgt[lane], e = weq[lane], ia = a, ie = e;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const uint32_t va = __shfl_up_sync(0xffffffffu, ia, off);
      const uint32_t ve = __shfl_up_sync(0xffffffffu, ie, off);
      if (lane >= off) { ia += va; ie += ve; }
    }
    wgt_base[lane] = ia - a;
    weq_base[lane] = ie - e;
  }
  __syncthreads();
  uint32_t gt_run = wgt_base[warp], eq_run = weq_base[warp];
  const uint32_t lt_mask = (1u << lane) - 1u;
  for (int t0 = beg; t0 < end; t0 += 32) {
    const int t = t0 + lane;
    const uint32_t k = t < end ? key_at(t) : 0u;
    const bool is_gt = t < end && k > tau;
    const bool is_eq = t < end && k == tau;
    const uint32_t bg = __ballot_sync(0xffffffffu, is_gt);
    const uint32_t be = __ballot_sync(0xffffffffu, is_eq);
    const uint32_t gt_before = gt_run + __popc(bg & lt_mask);
    const uint32_t eq_before = eq_run + __popc(be & lt_mask);
    if (is_gt || (is_eq && eq_before < need_eq)) out[gt_before + min(eq_before, need_eq)] = t;
    gt_run += __popc(bg);
    eq_run += __popc(be);
  }
}


// ------------------------------------------------------------------------------------------------
// Register-resident variant for rows of up to 32768 tokens: thread t owns E consecutive positions
// [t*E, (t+1)*E) and keeps their keys in registers (16-byte loads from the boundary at or before the
// row's start).  Histogram passes over a shrinking key interval find the k-th largest key exactly, at most three of 2048 bins
// (512 threads and more; four of 1024 or 512 with 256 or 128); after the first pass only the few
// keys inside the threshold bin take part.  Because ownership is contiguous, one block-wide prefix sum over
// per-thread (greater, equal) counts gives every thread the output offset of its first selected position, and
// it writes its positions in ascending order from two bit masks.
//
// PD > 0 (head dimension 64 or 128) fuses the packing: the positions also go to shared memory and the same CTA
// copies the row's kb selected K and V rows (16 bytes per thread, kPackUnroll rows in flight per thread group)
// into the packed buffers.  Rows are independent, so while one CTA of an SM is in its latency-bound
// selection another streams rows: the two phases overlap across CTAs without any inter-CTA wait.
//
// kThr is the threshold selection (sg_select_threshold): keys above row maximum - alpha, at most kb of them.  The threshold
// is known from the row maximum alone, so the keys above it are counted first; only a row that has more than kb of them goes
// through the narrowing (8B shape, 256 rows, cap 20 %: exact top-cap and a trimming kernel behind it took 13.7 + 7.6 us,
// this 9.0 us when no row reaches its cap).  NaNs do not take part.
constexpr int kPackUnroll = 4;
// Interval populations up to kFinishMax are finished by direct ranking.  Rows of 8192 (one CTA each, 256 of them), the selection
// alone: 64 takes 13.8 us (most rows need another histogram pass), 128 takes 10.1, 256 takes 12.8; with the gather fused in, 43 us
// in each case.  Up to kAtomicGather of them are gathered
// with one shared atomic per thread that has any, more of them through a block-wide prefix sum: the atomics of 100 threads
// took 9 k clocks in a row of 32768, the prefix sum costs rows of 8192 and less 0.1 us when there are few.
constexpr int kFinishMax = 128;
constexpr uint32_t kAtomicGather = 64;
constexpr int64_t kFuseMinRows = kNumSMs;               // fewer rows than SMs cannot fill the machine with their gathers
// Bins of a histogram: four per thread, 2048 at most (eight per thread for 128 and 256 threads: 0.5 to 1 us slower).
template <int T>
constexpr int kRegBinBits = T >= 512 ? 11 : T >= 256 ? 10 : 9;
constexpr int kRegCopies = 2;

// Block-wide exclusive prefix sum of one value per thread (T threads); `wsum` holds T/32 words.  One barrier: every
// warp adds up the totals of the warps before it by itself.  The caller keeps a barrier between two calls.
template <int T>
__device__ __forceinline__ uint32_t block_exclusive_scan(uint32_t v, uint32_t* wsum, int lane, int warp) {
  uint32_t inc = v;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const uint32_t u = __shfl_up_sync(0xffffffffu, inc, off);
    if (lane >= off) inc += u;
  }
  if (lane == 31) wsum[warp] = inc;
  __syncthreads();
  const uint32_t before = __reduce_add_sync(0xffffffffu, (lane < T / 32 && lane < warp) ? wsum[lane] : 0u);
  return before + inc - v;
}

template <int E, int T, int PD, bool kThr>
__global__ void __launch_bounds__(T) select_topk_reg_kernel(const SelParams p) {
  pdl_wait();
  constexpr int kBinBits = kRegBinBits<T>, kRegBins = 1 << kBinBits;
  extern __shared__ __align__(16) uint32_t smem[];
  uint32_t* wsum = smem;                               // [2][T/32]
  uint32_t* sh = wsum + 2 * (T / 32);                  // [0] chosen bin, [1] remaining need ... [6], [7] barrier
  uint32_t* cand = sh + 8;                             // [kFinishMax + 4] keys that are ranked directly
  uint32_t* hist = cand + kFinishMax + 4;              // [kRegCopies][kRegBins]
  uint32_t* stage = hist + kRegCopies * kRegBins;      // E > 16: [T * E] values of the row
  // [T * E] selected positions (PD > 0), over what has been used; in 16 bits where they would not fit in 32 (whose gather starts 0.2 us sooner)
  using Pos = typename std::conditional<E <= 8, uint32_t, uint16_t>::type;
  Pos* list = reinterpret_cast<Pos*>(E > 16 ? stage : hist);

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int row = blockIdx.x;
  const int l = row / (p.B * p.Hkv);
  const int rem = row - l * (p.B * p.Hkv);
  const int b = rem / p.Hkv;
  const int g = rem - b * p.Hkv;
  const int c0 = p.cu[b];
  const int N = p.cu[b + 1] - c0;
  const int ck = p.cu_k[b];
  const int kb = p.cu_k[b + 1] - ck;
  // the host's total is larger than cu_k[B]: as sg_pack_kv, entries that no row owns are not written
  if (PD > 0 && row == (int)gridDim.x - 1 && tid == 0 && ck + kb < p.K_tot) raise(p.dev_status, SG_ERR_INVALID);
  auto write_count = [&](int n) { if (kThr && tid == 0) p.sel_count[((int64_t)l * p.B + b) * p.Hkv + g] = n; };
  if (kb <= 0) { write_count(0); return; }
  int32_t* out = p.sel_idx + ((int64_t)l * p.Hkv + g) * p.K_tot + ck;
  // fused packing: thread group `grp` (D/8 threads, 16 bytes each) copies selected row j of this (layer, sequence, head)
  auto pack_rows = [&](auto pos_of) {
    if constexpr (PD > 0) {
      constexpr int kTPR = PD / 8, kGroups = T / kTPR;
      const int lane_in_row = tid % kTPR, grp = tid / kTPR;
      const int64_t src0 = (int64_t)l * p.ls + (int64_t)c0 * p.ts + (int64_t)g * p.hs + lane_in_row * 8;
      const int64_t dst0 = (((int64_t)l * p.K_tot + ck) * p.Hkv + (int64_t)g * kb) * PD + lane_in_row * 8;
      // rotating pipeline: kPackUnroll rows per thread group stay in flight; a row's registers are refilled right
      // after its store is issued, so loads never drain while stores go out
      auto load_row = [&](int j, int4& a, int4& b) {
        a = make_int4(0, 0, 0, 0);
        b = make_int4(0, 0, 0, 0);
        if (j < kb) {
          const int t = pos_of(j);
          if (t >= 0) {                                // -1 only behind the end of an over-sized budget: zero rows
            const int64_t src = src0 + (int64_t)t * p.ts;
            a = __ldcs(reinterpret_cast<const int4*>(p.k_cache + src));
            b = __ldcs(reinterpret_cast<const int4*>(p.v_cache + src));
          }
        }
      };
      int4 kv[kPackUnroll][2];
#pragma unroll
      for (int u = 0; u < kPackUnroll; ++u) load_row(grp + u * kGroups, kv[u][0], kv[u][1]);
      for (int j0 = grp; j0 < kb; j0 += kGroups * kPackUnroll) {
#pragma unroll
        for (int u = 0; u < kPackUnroll; ++u) {
          const int j = j0 + u * kGroups;
          if (j < kb) {
            const int64_t dst = dst0 + (int64_t)j * PD;
            __stcs(reinterpret_cast<int4*>(p.packed_k + dst), kv[u][0]);
            __stcs(reinterpret_cast<int4*>(p.packed_v + dst), kv[u][1]);
          }
          load_row(j + kGroups * kPackUnroll, kv[u][0], kv[u][1]);
        }
      }
    }
  };
  if (N > p.capacity) {
    // Longer than the E*T positions this variant holds (it was chosen from shape->max_seqlen, which the row
    // exceeds): flag it, emit an empty row (and zero rows in the fused gather) and leave.
    if (tid == 0) {
      raise(p.dev_status, SG_ERR_INVALID);
      if (PD > 0) raise(p.dev_status, SG_ERR_INDEX);
    }
    for (int j = tid; j < kb; j += T) out[j] = -1;
    pack_rows([&](int) { return -1; });
    write_count(0);
    return;
  }
  if (kThr && kb > N && tid == 0) raise(p.dev_status, SG_ERR_INVALID);
  if (!kThr && kb >= N) {                             // whole prompt (or an over-sized budget)
    if (kb > N && tid == 0) {
      raise(p.dev_status, SG_ERR_INVALID);
      if (PD > 0) raise(p.dev_status, SG_ERR_INDEX);   // what the packing kernel reports for the -1 entries
    }
    for (int j = tid; j < kb; j += T) out[j] = j < N ? j : -1;
    pack_rows([&](int j) { return j < N ? j : -1; });
    return;
  }
  const uint32_t* x = reinterpret_cast<const uint32_t*>(p.importance) + ((int64_t)l * p.Hkv + g) * p.T + c0;
  // Thread t owns E consecutive values, from the 16-byte boundary at or before the row's start (`off` values early): its positions are
  // those from t*E - off.  Up to 16 values it reads itself, 16 bytes at a time (the lines of a warp's first load serve its later ones
  // from L1).  For E = 32 the row comes to shared memory with one bulk copy, the up to three values behind the last boundary with
  // plain loads; a thread reads its values 16 bytes at a time, starting at another quad of its segment than its neighbours (no bank
  // conflicts), so its registers hold the segment turned by `turn` quads, and bit masks over them are turned back before use.
  // A row of 32768: 5.7 k clocks; by the threads themselves 10.7 k (the row is larger than the L1 that shared memory leaves:
  // every line comes from L2 several times).  With 16 values or fewer the bulk copy loses: 3.8 against 2.9 k clocks for a row of
  // 8192, 2.8 against 2.3 k for 1024.
  constexpr bool kBulk = E > 16;
  constexpr uint32_t kAll = E >= 32 ? 0xffffffffu : ((1u << (E & 31)) - 1u);
  constexpr int kQuads = E / 4;
  const int turn = kBulk ? (lane / (8 / (kQuads < 8 ? kQuads : 8))) % kQuads : 0;
  auto turned = [&](uint32_t m, int by) -> uint32_t {  // rotate the E-bit mask left by `by` quads
    if constexpr (!kBulk) return m;
    const int sft = 4 * by;
    return sft == 0 ? m : ((m << sft) | (m >> (E - sft))) & kAll;
  };
  int off = (int)((reinterpret_cast<uintptr_t>(x) & 15u) >> 2);
  const bool wide = N + off <= E * T;                  // else the values in front of the row would push its end out of the registers
  const bool bulk = kBulk && wide;
  if (!wide) off = 0;
  const int span = N + off, whole = bulk ? span & ~3 : 0;                // values from the boundary on; of the bulk copy
  const uint32_t bar = smem_u32(sh + 6);               // 8 bytes, 8-byte aligned
  if (bulk && tid == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(whole * 4) : "memory");
    if (whole > 0)
      asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(smem_u32(stage)), "l"(x - off),
                   "r"(whole * 4), "r"(bar) : "memory");
  }
  for (int i = tid; i < kRegCopies * kRegBins; i += T) hist[i] = 0;
  const int first = tid * E - off;                     // position of the thread's first value (negative: before the row)
  const int nvalid = min(max(N - first, 0), E);
  uint32_t vmask = nvalid >= 32 ? 0xffffffffu : ((1u << nvalid) - 1u);
  if (first < 0) vmask &= ~((1u << -first) - 1u);      // the boundary's values in front of the row
  vmask = turned(vmask, (kQuads - turn) % kQuads);     // as the registers hold the segment
  uint32_t key[E];
  if constexpr (kBulk) {
    for (int i = whole + tid; i < span; i += T) stage[i] = x[i - off];
    __syncthreads();                                   // barrier set up, histogram cleared, plainly loaded values there
    uint32_t done = bulk ? 0u : 1u;
    for (uint32_t tries = 0; tries < (1u << 22) && !done; ++tries)
      asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], 0;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(done) : "r"(bar) : "memory");
    if (!__syncthreads_and((int)done)) {               // does not happen: the copy has a valid source and size
      if (tid == 0) raise(p.dev_status, SG_ERR_TIMEOUT);
      for (int j = tid; j < kb; j += T) out[j] = -1;
      pack_rows([&](int) { return -1; });
      write_count(0);
      return;
    }
#pragma unroll
    for (int q = 0; q < kQuads; ++q) {
      const uint4 v = *reinterpret_cast<const uint4*>(stage + tid * E + 4 * ((q + turn) % kQuads));
      key[4 * q] = order_key(v.x); key[4 * q + 1] = order_key(v.y);
      key[4 * q + 2] = order_key(v.z); key[4 * q + 3] = order_key(v.w);
    }
  } else {
    uint4 v[kQuads];
#pragma unroll
    for (int q = 0; q < kQuads; ++q) {
      const int i = first + 4 * q;
      v[q] = make_uint4(0u, 0u, 0u, 0u);
      if (wide && i + 3 < N) {
        v[q] = *reinterpret_cast<const uint4*>(x + i);
      } else if (i < N) {                              // the row's ends: what the mask leaves out may be any value of the row
        v[q] = make_uint4(x[max(i, 0)], x[min(max(i + 1, 0), N - 1)], x[min(max(i + 2, 0), N - 1)], x[min(max(i + 3, 0), N - 1)]);
      }
    }
#pragma unroll
    for (int q = 0; q < kQuads; ++q) {
      key[4 * q] = order_key(v[q].x); key[4 * q + 1] = order_key(v[q].y);
      key[4 * q + 2] = order_key(v[q].z); key[4 * q + 3] = order_key(v[q].w);
    }
    __syncthreads();                                   // histogram cleared
  }

  // ---- exact k-th largest key by narrowing a key interval [lo, hi] that holds it, kBinBits bits of the interval per pass.
  // The digit of a pass is (key - lo) >> shift with shift chosen so that the interval spans at most kRegBins bins:
  // unlike the fixed top bits of a float, it spreads whatever range the row really has over all bins, so the
  // threshold bin of the first pass keeps tens of keys, not a quarter of the row, and the later passes touch few.
  if constexpr (kThr) {                                // the keys of -inf .. +inf: everything outside is a NaN
#pragma unroll
    for (int e = 0; e < E; ++e)
      if (key[e] < kKeyNegInf || key[e] > kKeyPosInf) vmask &= ~(1u << e);
  }
  uint32_t kmin = 0xffffffffu, kmax = 0u;
#pragma unroll
  for (int e = 0; e < E; ++e)
    if ((vmask >> e) & 1u) { kmin = min(kmin, key[e]); kmax = max(kmax, key[e]); }
  kmin = __reduce_min_sync(0xffffffffu, kmin);
  kmax = __reduce_max_sync(0xffffffffu, kmax);
  if (lane == 0) { wsum[warp] = kmin; wsum[T / 32 + warp] = kmax; }
  __syncthreads();
  kmin = __reduce_min_sync(0xffffffffu, lane < T / 32 ? wsum[lane] : 0xffffffffu);
  kmax = __reduce_max_sync(0xffffffffu, lane < T / 32 ? wsum[T / 32 + lane] : 0u);
  __syncthreads();                                     // wsum is reused by the scans below
  uint32_t lo = kmin, hi = kmax, need = (uint32_t)kb;
  int above_thr = kb;                                  // kThr: number selected
  if constexpr (kThr) {
    float thr;                                         // IEEE subtraction without flush-to-zero, whatever the compile flags
    asm("sub.rn.f32 %0, %1, %2;" : "=f"(thr) : "f"(__uint_as_float(key_to_bits(kmax))), "f"(p.alpha));
    uint32_t thr_bits = __float_as_uint(thr);
    if ((thr_bits & 0x7fffffffu) == 0u) thr_bits = 0u;  // -0 and +0 compare equal as floats: use +0's key
    const uint32_t kthr = order_key(thr_bits);
    uint32_t n = 0;
#pragma unroll
    for (int e = 0; e < E; ++e) n += ((vmask >> e) & 1u) && key[e] > kthr ? 1u : 0u;
    n = __reduce_add_sync(0xffffffffu, n);
    if (lane == 0) wsum[warp] = n;
    __syncthreads();
    above_thr = kmax == 0u ? 0 : (int)__reduce_add_sync(0xffffffffu, lane < T / 32 ? wsum[lane] : 0u);
    __syncthreads();                                   // wsum is reused by the scans below
    if (above_thr <= kb) { lo = hi = kmax == 0u ? 0xffffffffu : kthr; need = 0; }      // everything above, nothing equal
    else above_thr = kb;
  }
#pragma unroll 1
  for (int pass = 0; lo != hi; ++pass) {
    const uint32_t width = hi - lo;
    const int shift = max(0, 32 - __clz(width) - kBinBits);
    const int copies = pass == 0 ? kRegCopies : 1;     // later passes see few candidates: one copy is enough
    uint32_t* my_hist = hist + (warp % copies) * kRegBins;
#pragma unroll
    for (int e = 0; e < E; ++e) {
      const uint32_t rel = key[e] - lo;
      if (((vmask >> e) & 1u) && rel <= width) atomicAdd(&my_hist[rel >> shift], 1u);
    }
    __syncthreads();
    // suffix search: thread t looks at bins kRegBins-1-t*kBpt ... (descending) for the bin holding the need-th largest
    constexpr int kBpt = kRegBins / T;
    uint32_t c[kBpt];
    const int bin0 = kRegBins - 1 - tid * kBpt;        // this thread's highest bin; it owns bin0, bin0-1, ...
    uint32_t ssum = 0;
#pragma unroll
    for (int i = 0; i < kBpt; ++i) {
      c[i] = hist[bin0 - i];
      if (copies > 1) c[i] += hist[kRegBins + bin0 - i];
    }
#pragma unroll
    for (int i = 0; i < kBpt; ++i) {                   // cleared for the next pass
      hist[bin0 - i] = 0;
      if (copies > 1) hist[kRegBins + bin0 - i] = 0;
      ssum += c[i];
    }
    const uint32_t exc = block_exclusive_scan<T>(ssum, wsum, lane, warp);   // candidates in bins above this thread's
    if (exc < need && need <= exc + ssum) {
      uint32_t run = exc;
#pragma unroll
      for (int i = 0; i < kBpt; ++i) {
        if (run < need && need <= run + c[i]) { sh[0] = (uint32_t)(bin0 - i); sh[1] = need - run; sh[2] = c[i]; sh[3] = 0; }
        run += c[i];
      }
    }
    __syncthreads();
    lo += sh[0] << shift;
    hi = lo + min(hi - lo, (1u << shift) - 1u);
    need = sh[1];
    const uint32_t ncand = sh[2];
    if (lo != hi && ncand <= (uint32_t)kFinishMax) {
      // Few keys left in the interval: instead of more block-wide passes, gather them and count for each the keys above it
      // and equal to it; the key whose rank range covers `need` is the threshold.
      const uint32_t w = hi - lo;
      uint32_t mine = 0;
#pragma unroll
      for (int e = 0; e < E; ++e) mine |= (key[e] - lo <= w ? 1u : 0u) << e;
      mine &= vmask;
      uint32_t at = 0;
      if (ncand > kAtomicGather)
        at = block_exclusive_scan<T>((uint32_t)__popc(mine), wsum, lane, warp);
      else if (mine)
        at = atomicAdd(&sh[3], (uint32_t)__popc(mine));
      if (mine) {
#pragma unroll
        for (int e = 0; e < E; ++e)
          if ((mine >> e) & 1u) cand[at++] = key[e];
      }
      __syncthreads();
      // four lanes per key, a quarter of the list each
      for (int i0 = 0; i0 < (int)ncand; i0 += T / 4) {
        const int i = i0 + (tid >> 2), part = tid & 3;
        if (i0 + (warp << 3) >= (int)ncand) break;     // nothing for this warp
        const uint32_t k = i < (int)ncand ? cand[i] : 0u;
        uint32_t above = 0, same = 0;
        for (int j = 4 * part; j < (int)ncand; j += 16) {
          const uint4 o = *reinterpret_cast<const uint4*>(cand + j);     // values behind the list's end do not count
          const int left = (int)ncand - j;
          above += (o.x > k ? 1u : 0u) + (left > 1 && o.y > k ? 1u : 0u) + (left > 2 && o.z > k ? 1u : 0u) + (left > 3 && o.w > k ? 1u : 0u);
          same += (o.x == k ? 1u : 0u) + (left > 1 && o.y == k ? 1u : 0u) + (left > 2 && o.z == k ? 1u : 0u) + (left > 3 && o.w == k ? 1u : 0u);
        }
#pragma unroll
        for (int o = 1; o < 4; o <<= 1) {
          above += __shfl_xor_sync(0xffffffffu, above, o);
          same += __shfl_xor_sync(0xffffffffu, same, o);
        }
        if (part == 0 && i < (int)ncand && above < need && need <= above + same) { sh[4] = k; sh[5] = need - above; }   // equal keys write equal values
      }
      __syncthreads();
      lo = hi = sh[4];
      need = sh[5];
    }
  }
  const uint32_t tau = lo, need_eq = need;

  // per-thread bit masks of the positions above / equal to the threshold; their counts, packed (greater in the low half,
  // equal in the high half), go through one block-wide exclusive prefix sum
  uint32_t mgt = 0, meq = 0;
#pragma unroll
  for (int e = 0; e < E; ++e) {
    mgt |= (key[e] > tau ? 1u : 0u) << e;
    meq |= (key[e] == tau ? 1u : 0u) << e;
  }
  mgt = turned(mgt & vmask, turn);
  meq = turned(meq & vmask, turn);
  const uint32_t cnt = (uint32_t)__popc(mgt) | ((uint32_t)__popc(meq) << 16);
  const uint32_t before = block_exclusive_scan<T>(cnt, wsum, lane, warp);
  const uint32_t gt_before = before & 0xffffu, eq_before = before >> 16;
  // of this thread's equal entries only the first (need_eq - eq_before) are kept: drop the highest ones beyond that
  int extra = __popc(meq) - (int)(need_eq > eq_before ? min(need_eq - eq_before, (uint32_t)E) : 0u);
  while (extra > 0) { meq &= ~(0x80000000u >> __clz(meq)); --extra; }
  uint32_t m = mgt | meq;
  uint32_t slot = gt_before + min(eq_before, need_eq);
  while (m) {                                          // ascending positions
    const int e = __ffs(m) - 1;
    m &= m - 1;
    out[slot] = first + e;
    if constexpr (PD > 0) list[slot] = (Pos)(first + e);
    ++slot;
  }
  if constexpr (kThr) {
    for (int j = above_thr + tid; j < kb; j += T) out[j] = -1;
    write_count(above_thr);
  }
  if constexpr (PD > 0) {
    __syncthreads();
    pack_rows([&](int j) { return (int)list[j]; });
  }
}

// What the selection needs of shared memory is what the gather lacks of L1, which holds the lines that are on their way: 256 rows of
// 8192 with 57 KB per CTA (rows staged, positions in 32 bits beside the histograms) took 43.6 us, 43.2 with 17 KB; 51 with the whole L1
// asked for as shared memory.
template <int E, int T>
constexpr int select_reg_smem_bytes(bool lists) {
  const int hist = kRegCopies * (4 << kRegBinBits<T>), list = lists && E <= 16 ? E * T * (E <= 8 ? 4 : 2) : 0;
  return (2 * (T / 32) + 8 + kFinishMax + 4) * 4 + (hist > list ? hist : list) + (E > 16 ? E * T * 4 : 0);
}

}  // namespace
}  // namespace sg

namespace sg {
namespace {
// Launches the selection.  kPack and kThreshold are done by the register-resident kernels only (the caller has checked that
// the rows fit them).
enum SelectKind { kSelect, kPack, kThreshold };
sg_status select_launch(const sg_shape* shape, SelParams& p, SelectKind kind, void* stream) {
  const int64_t rows = (int64_t)shape->num_layers * shape->batch * shape->num_kv_heads;
  if (rows > 0x7fffffffLL) return SG_ERR_UNSUPPORTED;
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.stream = static_cast<cudaStream_t>(stream);
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  cfg.gridDim = dim3((unsigned)rows);
  const int pd = kind == kPack ? shape->head_dim : 0;
#define SG_LAUNCH_SELECT_REG_PD(E, T, PD, THR)                                                     \
  do {                                                                                          \
    p.capacity = (E) * (T);                                                                     \
    SG_ENSURE_SMEM((select_topk_reg_kernel<E, T, PD, THR>), (select_reg_smem_bytes<E, T>(PD > 0)));         \
    cfg.blockDim = dim3(T);                                                                     \
    cfg.dynamicSmemBytes = select_reg_smem_bytes<E, T>(PD > 0);                                       \
    SG_CUDA_TRY(cudaLaunchKernelEx(&cfg, select_topk_reg_kernel<E, T, PD, THR>, p));                  \
  } while (0)
#define SG_LAUNCH_SELECT_REG(E, T)                                              \
  do {                                                                          \
    if (kind == kThreshold) SG_LAUNCH_SELECT_REG_PD(E, T, 0, true);             \
    else if (pd == 128) SG_LAUNCH_SELECT_REG_PD(E, T, 128, false);              \
    else if (pd == 64) SG_LAUNCH_SELECT_REG_PD(E, T, 64, false);                \
    else SG_LAUNCH_SELECT_REG_PD(E, T, 0, false);                               \
  } while (0)
  // Short rows take as many threads as have keys: with 512 for every row a wave held two rows per SM.  Microseconds with 512 threads -> with
  // 128 (rows of up to 1024) or 256 (2048): the selection alone, 8 rows of 1000 4.3 -> 3.7, 256 of 1024 5.5 -> 4.0, 832 of 640 14.3 -> 5.1,
  // 1280 of 100 20.9 -> 6.4, 256 of 2000 5.7 -> 4.7; by a threshold, 832 of 640 16.3 -> 10.1, 256 of 2000 7.6 -> 6.3, but 128 of 900 5.1 ->
  // 6.0.  A gather needs threads for its rows on the way: 832 rows of 640 19.5 -> 9.2, but 256 of 1000, a fifth kept, 13.5 -> 15.9.
  const int64_t fewest[] = {1, 4 * kNumSMs, kNumSMs};   // rows from which on, by kind
  if (rows < kNumSMs && kind != kPack && shape->max_seqlen <= 8192 && shape->max_seqlen > 4096) {
    // fewer rows than SMs: one CTA per SM anyway, so twice the threads per row (half the keys each) shorten the chains
    if (kind == kThreshold) SG_LAUNCH_SELECT_REG_PD(8, 1024, 0, true);
    else SG_LAUNCH_SELECT_REG_PD(8, 1024, 0, false);
  } else if (shape->max_seqlen <= 1024 && rows >= fewest[kind]) {
    SG_LAUNCH_SELECT_REG(8, 128);
  } else if (shape->max_seqlen <= 2048 && (kind != kPack || rows >= fewest[kind])) {
    SG_LAUNCH_SELECT_REG(8, 256);
  } else if (shape->max_seqlen <= 4096) {
    SG_LAUNCH_SELECT_REG(8, 512);
  } else if (shape->max_seqlen <= 8192) {
    SG_LAUNCH_SELECT_REG(16, 512);
  } else if (shape->max_seqlen <= 16384) {
    SG_LAUNCH_SELECT_REG(16, 1024);
  } else if (shape->max_seqlen <= 32768) {
    SG_LAUNCH_SELECT_REG(32, 1024);
  } else if (kind != kSelect) {
    return SG_ERR_UNSUPPORTED;
  } else if (shape->max_seqlen <= kSelKeyCap) {
    const int smem = kSelFixedSmem + shape->max_seqlen * 4;
    p.capacity = shape->max_seqlen;
    SG_ENSURE_SMEM(select_topk_kernel<true>, smem);
    cfg.blockDim = dim3(kSelThreads);
    cfg.dynamicSmemBytes = smem;
    SG_CUDA_TRY(cudaLaunchKernelEx(&cfg, select_topk_kernel<true>, p));
  } else {
    p.capacity = 0;                                    // keys are re-read from global memory: any length
    cfg.blockDim = dim3(kSelThreads);
    cfg.dynamicSmemBytes = kSelFixedSmem;
    SG_CUDA_TRY(cudaLaunchKernelEx(&cfg, select_topk_kernel<false>, p));
  }
#undef SG_LAUNCH_SELECT_REG
#undef SG_LAUNCH_SELECT_REG_PD
  SG_CUDA_TRY(cudaGetLastError());
  return SG_OK;
}
}  // namespace
}  // namespace sg

namespace sg {
bool select_threshold_fits(const sg_shape* shape) { return shape->max_seqlen <= 32768; }
sg_status select_threshold_launch(const sg_shape* shape, const float* scores, float alpha, const int32_t* cu_cap, int32_t total_cap,
                                  int32_t* sel_idx, int32_t* sel_count, int32_t* dev_status, void* stream) {
  SelParams p = {};
  p.importance = scores;
  p.cu = shape->cu_seqlens;
  p.cu_k = cu_cap;
  p.sel_idx = sel_idx;
  p.dev_status = dev_status;
  p.T = shape->total_tokens;
  p.K_tot = total_cap;
  p.B = shape->batch;
  p.Hkv = shape->num_kv_heads;
  p.sel_count = sel_count;
  p.alpha = alpha;
  return select_launch(shape, p, kThreshold, stream);
}
}  // namespace sg

extern "C" sg_status sg_select_topk(const sg_shape* shape, const float* importance, const int32_t* cu_k,
                                    int32_t total_sel, int32_t* sel_idx, void* workspace,
                                    size_t workspace_bytes, int32_t* dev_status, void* stream) {
  using namespace sg;
  (void)workspace;
  (void)workspace_bytes;
  sg_status st = check_shape(shape, false);
  if (st != SG_OK) return st;
  if (total_sel < 0) return SG_ERR_INVALID;
  if (total_sel == 0) return SG_OK;
  if (!importance || !cu_k || !sel_idx) return SG_ERR_INVALID;
  if (!aligned16(importance) || !aligned16(cu_k) || !aligned16(sel_idx)) return SG_ERR_INVALID;
  SelParams p = {};
  p.importance = importance;
  p.cu = shape->cu_seqlens;
  p.cu_k = cu_k;
  p.sel_idx = sel_idx;
  p.dev_status = dev_status;
  p.T = shape->total_tokens;
  p.K_tot = total_sel;
  p.B = shape->batch;
  p.Hkv = shape->num_kv_heads;
  return select_launch(shape, p, kSelect, stream);
}

extern "C" sg_status sg_select_pack_kv(const sg_shape* shape, const float* importance, const int32_t* cu_k,
                                       int32_t total_sel, const void* k_cache, const void* v_cache, int32_t* sel_idx,
                                       void* packed_k, void* packed_v, int32_t* dev_status, void* stream) {
  using namespace sg;
  sg_status st = check_shape(shape, false);
  if (st != SG_OK) return st;
  if (total_sel < 0) return SG_ERR_INVALID;
  if (total_sel == 0) return SG_OK;
  if (!importance || !cu_k || !sel_idx || !k_cache || !v_cache || !packed_k || !packed_v) return SG_ERR_INVALID;
  if (!aligned16(importance) || !aligned16(cu_k) || !aligned16(sel_idx) || !aligned16(k_cache) || !aligned16(v_cache) ||
      !aligned16(packed_k) || !aligned16(packed_v))
    return SG_ERR_INVALID;
  // One fused launch pays when the rows fit the register-resident kernels and there are enough of them to keep every SM
  // streaming while others select; otherwise the two kernels run back to back.
  const int64_t rows = (int64_t)shape->num_layers * shape->batch * shape->num_kv_heads;
  const bool fuse = shape->max_seqlen <= 32768 && rows >= kFuseMinRows;
  if (!fuse) {
    st = sg_select_topk(shape, importance, cu_k, total_sel, sel_idx, nullptr, 0, dev_status, stream);
    if (st != SG_OK) return st;
    return sg_pack_kv(shape, k_cache, v_cache, sel_idx, cu_k, total_sel, packed_k, packed_v, dev_status, stream);
  }
  SelParams p = {};
  p.importance = importance;
  p.cu = shape->cu_seqlens;
  p.cu_k = cu_k;
  p.sel_idx = sel_idx;
  p.dev_status = dev_status;
  p.T = shape->total_tokens;
  p.K_tot = total_sel;
  p.B = shape->batch;
  p.Hkv = shape->num_kv_heads;
  p.k_cache = static_cast<const uint16_t*>(k_cache);
  p.v_cache = static_cast<const uint16_t*>(v_cache);
  p.packed_k = static_cast<uint16_t*>(packed_k);
  p.packed_v = static_cast<uint16_t*>(packed_v);
  p.ls = shape->cache_layer_stride;
  p.ts = shape->cache_token_stride;
  p.hs = shape->cache_head_stride;
  return select_launch(shape, p, kPack, stream);
}
