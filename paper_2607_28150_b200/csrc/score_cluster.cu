// Scoring of calls that fit the chip at once, one kernel: a thread-block cluster per part (layer, sequence, KV head), and, for a
// prefill, selection and packing in the same kernel.
//
// A call of few and short parts (one layer of one prompt, a small model) is bound by latency: score.cu's two passes, the
// selection and the gather are four launches in a row, each with its set-up, first loads and completion, around a few
// microseconds of work.  Here the key tiles of a part are dealt out over the CTAs of one cluster and stay in shared memory:
//
//   1. row statistics  D[row][key] = Q x K_tile^T, as pass 1 of score.cu; every CTA sends its rows' (reference, sum of exp2)
//      to all CTAs of the cluster through distributed shared memory;
//   2. column sums     D[key][row] = K_tile x Q^T on the same tiles, as pass 2; the MMAs run while the statistics travel;
//   3. selection       every CTA sends its importances to all CTAs, and every CTA finds the row's k-th largest by itself, on all
//      keys.  (Sharing the work out instead, 1024 bins of every CTA to every CTA and then the keys of one bin, took 1.4 us more at
//      1024 keys and 1.7 at 2048: what counts is the number of steps, not the keys per step.)
//   4. packing         every CTA knows which of its own keys are selected and where they go; their K rows are in its shared
//      memory, only the V rows are read.
//
// So K comes from HBM once, and the two exchanges (a third of a microsecond each) are all that CTAs wait for one another.  A call is
// bound by its chain of steps (1024 keys, 17 k clocks: set-up and first tile 5.1 k, statistics and their exchange 2.5 k, sums 1.3 k,
// second exchange 1.8 k, selection 4.5 k, packing 1.1 k), with several tiles per CTA by the epilogue, about 1250 clocks per
// block and pass.
//
// All sixteen worker warps share every block: a block is 128 x 128 scores in one TMEM stage, warp w takes the lanes of quarter
// w mod 4 and the columns of quarter w / 4, so that one tile per CTA keeps all schedulers busy.
//
// Every wait on an mbarrier is bounded, as in score.cu: on expiry the CTA raises SG_ERR_TIMEOUT, tells the other CTAs of its cluster, waits
// (bounded) for its own TMA copies and MMAs and for what is on its way to it, frees its TMEM and returns.  The cluster barriers have no
// limit of their own: every warp of every CTA arrives at each of them on every path.
#include <cuda.h>

#include "common.cuh"
#include "launch.h"
#include "score_launch.h"
#include "score_math.cuh"
#include "select_key.cuh"
#include "tcgen05.cuh"

namespace sg {
namespace {

constexpr int kWorkWarps = 16, kWork = 32 * kWorkWarps;      // workers
constexpr int kLoadWarp = kWorkWarps, kIssueWarp = kLoadWarp + 1;
constexpr int kThreads = 32 * (kIssueWarp + 1);
constexpr int kTileKeys = 128;
constexpr int kStages = 4;               // TMEM stages of 128 columns
// Most key tiles of a CTA, with selection and packing and without (cluster_pays says when).
constexpr int kMaxOwn = 8, kMaxOwnScore = 4;
constexpr int kBins = 2048;
constexpr int kRankMax = 128;            // keys that are ranked directly
constexpr int kSweeps = (kMaxOwn * kTileKeys + kWork - 1) / kWork;
constexpr int kCandAt = (24 + kSweeps * kWorkWarps + 3) & ~3;
constexpr int kFailedAt = kCandAt + kRankMax + 4, kMiscWords = kFailedAt + 4;
constexpr int kBars = 2 * kMaxOwn + 16;

struct ClusterParams {
  const int32_t* cu;
  const int32_t* cu_k;
  float* importance;
  int32_t* sel_idx;
  const uint16_t* k_cache;
  const uint16_t* v_cache;
  uint16_t* packed_k;
  uint16_t* packed_v;
  int32_t* dev_status;
  int64_t T, ls, ts, hs;
  int32_t K_tot, B, Hkv, G, W, R, Ralloc;
  int32_t csize, own, cap;               // CTAs per part; most tiles of a CTA; key tiles that it holds at a time
  int32_t withhold_unit;                 // testing only: the first CTA never sends the statistics of this unit (-1 = none)
  uint32_t wait_ns;
  float scale_log2;
};

// Byte offsets into the (1024-byte aligned) dynamic shared memory; the other CTAs write to rec, vals and minmax.
struct Carve {
  int k, rec, vals, minmax, slots, neg_lse, hist, misc, bars, total;
};
__host__ __device__ __forceinline__ Carve carve(int D, int Ralloc, int csize, int own, int cap) {
  Carve c;
  c.k = Ralloc * D * 2;
  c.rec = c.k + cap * kTileKeys * D * 2;
  c.vals = c.rec + csize * Ralloc * 8;
  c.minmax = c.vals + csize * own * kTileKeys * 4;
  c.slots = (c.minmax + csize * own * 8 + 15) & ~15;
  const int slots = 4 * Ralloc * 8, cols = 4 * own * kTileKeys * 4;      // row statistics, later column sums, later positions
  c.neg_lse = c.slots + (slots > cols ? slots : cols);
  c.hist = c.neg_lse + Ralloc * 4;
  c.misc = c.hist + kBins * 4;
  c.bars = c.misc + kMiscWords * 4;
  c.total = c.bars + kBars * 8;
  return c;
}

// Relaxed: what the CTAs tell each other is ordered by mbarriers; a releasing arrival took 0.4 us.
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_arrive_release() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ uint32_t at_rank(uint32_t addr, int rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void push2(uint32_t addr, uint32_t bar, uint32_t a, uint32_t b) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v2.b32 [%0], {%1, %2}, [%3];" ::"r"(addr), "r"(a), "r"(b), "r"(bar) : "memory");
}
// A barrier of the workers that also agrees on whether all of them are well.
__device__ __forceinline__ bool work_sync(bool ok) {
  uint32_t r;
  __syncwarp();
  asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.u32 p, %1, 0;\n\tbar.red.and.pred q, 1, %2, p;\n\tselp.u32 %0, 1, 0, q;\n\t}"
               : "=r"(r) : "r"((uint32_t)ok), "n"(kWork) : "memory");
  return r != 0;
}
// Phase 0 of a barrier whose bytes come from other CTAs of the cluster.
__device__ __forceinline__ bool mbar_test_cluster(uint32_t bar) {
  uint32_t ok;
  asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], 0;\n\tselp.u32 %0, 1, 0, p;\n\t}"
               : "=r"(ok) : "r"(bar) : "memory");
  return ok != 0;
}
static __device__ __noinline__ bool mbar_wait_cluster(uint32_t bar, volatile int* abort_flag, uint32_t limit_ns) {
  uint64_t t0 = 0;
  for (uint32_t it = 0;; ++it) {
    if (mbar_test_cluster(bar)) return true;
    if ((it & 63u) == 63u) {
      if (*abort_flag) return false;
      const uint64_t now = global_timer_ns();
      if (t0 == 0) t0 = now;
      else if (now - t0 > (uint64_t)limit_ns) { *abort_flag = 1; return false; }
    }
  }
}
// Entries from `from` on of a part's kb that name no position: -1 and zero rows, by the workers of all CTAs of the part.
template <int D>
__device__ __forceinline__ void clear_entries(int32_t* out, uint16_t* rows_k, uint16_t* rows_v, int from, int kb, int worker, int rank, int csize) {
  constexpr int kTPR = D / 8, kRowGroups = kWork / kTPR;
  const int x = worker % kTPR, grp = worker / kTPR;
  for (int j = from + rank * kRowGroups + grp; j < kb; j += csize * kRowGroups) {
    if (x == 0) out[j] = -1;
    *reinterpret_cast<int4*>(rows_k + (int64_t)j * D + x * 8) = make_int4(0, 0, 0, 0);
    *reinterpret_cast<int4*>(rows_v + (int64_t)j * D + x * 8) = make_int4(0, 0, 0, 0);
  }
}
// A CTA gives up (the workers' first warp): every CTA of the cluster knows it behind the cluster barrier that this warp arrives at.
__device__ __noinline__ void tell_failed(uint32_t failed, int csize) {
  const int lane = threadIdx.x & 31;
  if (lane < csize) asm volatile("st.shared::cluster.u32 [%0], 1;" ::"r"(at_rank(failed, lane)) : "memory");
  __syncwarp();
  cluster_arrive_release();
}
// All CTAs of a cluster of which one has given up.  It does not know its entries, so none of the part's rows may pass for selected ones.
// (Out of line, as tell_failed: inside the kernel they cost every call 0.5 us.)
template <int D, bool kPack>
__device__ __noinline__ void give_up(uint32_t bar_rec, uint32_t bar_val, uint32_t wait_ns, const int32_t* cu_k, int32_t* sel_idx, uint16_t* packed_k,
                                     uint16_t* packed_v, int K_tot, int Hkv, int csize) {
  // What the CTAs had sent one another may still be on its way, and nobody may have waited for it: no CTA leaves before it has landed
  // everywhere.  What was never sent ends the wait at its limit, long behind the landing of what was.
  const uint64_t t0 = global_timer_ns();
  while (!(mbar_test_cluster(bar_rec) && (!kPack || mbar_test_cluster(bar_val))) && global_timer_ns() - t0 <= wait_ns) {}
  __syncwarp();
  cluster_arrive_release();                            // (behind what the other CTAs have packed, too)
  cluster_wait();
  if (!kPack || threadIdx.x >= kWork) return;
  const int l = blockIdx.z, b = blockIdx.y / Hkv, g = blockIdx.y - b * Hkv, ck = cu_k[b], kb = cu_k[b + 1] - ck;
  const int64_t row0 = (((int64_t)l * K_tot + ck) * Hkv + (int64_t)g * kb) * D;
  clear_entries<D>(sel_idx + ((int64_t)l * Hkv + g) * K_tot + ck, packed_k + row0, packed_v + row0, 0, kb, threadIdx.x, blockIdx.x, csize);
}
// kTwice: up to 64 query rows stand twice, as in pass 1 of score.cu; else half of the warps, those of two of the four schedulers, would have
// padding (one layer of 8192 tokens, 8 heads of 64, 21.0 -> 19.3 us, 3000 tokens 13.4 -> 12.8; a kernel of its
// own, because as a branch it cost 128 rows of 2048 tokens 0.3 us).
template <int D, bool kPack, bool kTwice>
__global__ void __launch_bounds__(kThreads, 1)
score_cluster_kernel(const __grid_constant__ CUtensorMap tmap_q, const __grid_constant__ CUtensorMap tmap_k, const ClusterParams p) {
  constexpr int kSub = D / 64;
  constexpr int kKSubBytes = kTileKeys * 128, kKStageBytes = kSub * kKSubBytes;
  extern __shared__ uint8_t smem_dyn[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_dyn) + 1023) & ~uintptr_t(1023));
  const Carve cv = carve(D, p.Ralloc, p.csize, p.own, p.cap);
  uint8_t* const q_smem = smem;
  uint8_t* const k_smem = smem + cv.k;
  float2* const rec = reinterpret_cast<float2*>(smem + cv.rec);            // [csize][Ralloc] statistics of every CTA
  uint32_t* const vals = reinterpret_cast<uint32_t*>(smem + cv.vals);      // [csize * own * 128] importances, as ordered keys
  uint2* const minmax = reinterpret_cast<uint2*>(smem + cv.minmax);        // [csize * own] of a tile's keys
  float* const slot_m = reinterpret_cast<float*>(smem + cv.slots);         // [4][Ralloc] statistics by quarter of the columns
  float* const slot_l = slot_m + 4 * p.Ralloc;
  float* const cols = slot_m;                                              // [4][own * 128] column sums by quarter of the rows
  int* const list = reinterpret_cast<int*>(slot_m);                        // [own * 128] selected positions of this CTA
  float* const neg_lse = reinterpret_cast<float*>(smem + cv.neg_lse);      // [Ralloc]
  uint32_t* const misc = reinterpret_cast<uint32_t*>(smem + cv.misc);
  uint32_t* const hist = reinterpret_cast<uint32_t*>(smem + cv.hist);      // [kBins]
  const uint32_t bar0 = smem_u32(smem + cv.bars);
  const uint32_t bar_q = bar0, bar_drain = bar0 + 8u, bar_rec = bar0 + 16u, bar_val = bar0 + 24u;
  auto bar_afull = [&](uint32_t s) { return bar0 + 8u * (8 + s); };
  auto bar_aempty = [&](uint32_t s) { return bar0 + 8u * (12 + s); };
  auto bar_kfull = [&](uint32_t s) { return bar0 + 8u * (16 + s); };
  auto bar_kempty = [&](uint32_t s) { return bar0 + 8u * (16 + kMaxOwn + s); };
  uint32_t* const tmem_slot = misc;
  volatile int* const abort_flag = reinterpret_cast<volatile int*>(misc + 1);
  uint32_t* const sh = misc + 2;                       // [0] chosen bin, [1] remaining need, [2] keys in it, [3] gathered, [4] threshold, [5] need
  uint32_t* const wsum = misc + 8;                     // [16]
  uint32_t* const wsum2 = misc + 24;                   // [kSweeps][16] selected keys by warp
  uint32_t* const cand = misc + kCandAt;               // [kRankMax + 4]
  volatile uint32_t* const failed = misc + kFailedAt;  // a CTA of this cluster has given up (it writes the word of every CTA)

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  // (an integer division takes a hundred clocks: none where there is one sequence, or where all tiles fit)
  const int rank = blockIdx.x, l = blockIdx.z, b = p.B == 1 ? 0 : blockIdx.y / p.Hkv, g = blockIdx.y - b * p.Hkv, u = l * p.Hkv + g;
  const int nblk = p.Ralloc >> 7;

  // ---- set-up: nothing ahead of pdl_wait() touches what an earlier kernel may be writing
  if (tid == 0) {
    mbar_init(bar_drain, 1); mbar_init(bar_rec, 1); mbar_init(bar_val, 1);
    for (int s = 0; s < kStages; ++s) { mbar_init(bar_afull(s), 1); mbar_init(bar_aempty(s), kWorkWarps); }
    *abort_flag = 0;
    fence_barrier_init();
    mbar_arrive_expect_tx(bar_rec, (uint32_t)(p.csize * (kTwice ? 64 : p.Ralloc) * 8));
  }
  if (warp == kIssueWarp) {
    tmem_alloc(smem_u32(tmem_slot), 512);
    tmem_relinquish();
  }
  if (warp == kLoadWarp && lane == 1) *failed = 0;
  if (warp == kLoadWarp && lane == 0) {
    tma_prefetch_map(&tmap_q);
    tma_prefetch_map(&tmap_k);
    mbar_init(bar_q, 1);
    for (int s = 0; s < p.cap; ++s) { mbar_init(bar_kfull(s), 1); mbar_init(bar_kempty(s), 1); }
    fence_barrier_init();
    fence_proxy_async();
  }
  if (warp < kWorkWarps) {
    if (kPack) reinterpret_cast<uint4*>(hist)[tid] = make_uint4(0, 0, 0, 0);
    if (p.R < p.Ralloc) {
      // rows R.. of Q are never written by TMA: zero, so that padded MMA columns are finite
      const int span = kTwice ? 64 : p.Ralloc, words = (span - p.R) * 32;
      for (int dc = 0; dc < kSub; ++dc)
        for (int row = p.R; row < p.Ralloc; row += span) {
          uint32_t* z = reinterpret_cast<uint32_t*>(q_smem + dc * p.Ralloc * 128 + row * 128);
          for (int i = tid; i < words; i += kWork) z[i] = 0u;
        }
      fence_proxy_async();
    }
  }
  pdl_wait();
  const int c0 = p.B == 1 ? 0 : p.cu[b], N = p.B == 1 ? (int)p.T : p.cu[b + 1] - c0;
  const int ntiles = (N + kTileKeys - 1) / kTileKeys;
  const int t0 = rank * ntiles / p.csize, n_my = (rank + 1) * ntiles / p.csize - t0;     // this CTA's tiles
  const bool fits = ntiles <= p.csize * p.own;         // else max_seqlen was no upper bound: the row's keys do not fit `vals`
  volatile int never = 0;
  // Tile i of the CTA lives in stage i mod cap.  The row statistics take the tiles upwards, the column sums downwards: the last
  // `cap` tiles are still there, the others are loaded again (from L2), and in the end the first `cap` are there.  A stage's
  // loads are counted: tile i is load i / cap for the statistics and, downwards again, load phase2(i) for the column sums.
  auto stage_of = [&](int i) { return i < p.cap ? i : i % p.cap; };
  auto phase2 = [&](int i) { return n_my <= p.cap ? 0 : 2 * ((n_my - 1 - i % p.cap) / p.cap) - i / p.cap; };
  // The first tiles are requested as soon as there are barriers for them, beside the rest of the set-up.
  bool load_ok = true;
  uint32_t used = 0, odd = 0;                          // stages that were loaded; parity of their last load
  auto load = [&](int i, int phase) {                  // tile i of this CTA; its stage's earlier tile has been used
    const int s = stage_of(i);
    if (phase > 0) load_ok = mbar_wait<true>(bar_kempty(s), (uint32_t)((phase - 1) & 1), abort_flag, p.wait_ns, 100u);
    if (!load_ok) return;
    mbar_arrive_expect_tx(bar_kfull(s), (uint32_t)kKStageBytes);
#pragma unroll
    for (int dc = 0; dc < kSub; ++dc)
      tma_load_4d(smem_u32(k_smem + s * kKStageBytes + dc * kKSubBytes), &tmap_k, bar_kfull(s), dc * 64, g, c0 + (t0 + i) * kTileKeys, l);
    if (phase & 1) odd |= 1u << s; else odd &= ~(1u << s);
    used |= 1u << s;
  };
  if (warp == kLoadWarp && lane == 0 && n_my > 0) {
    mbar_arrive_expect_tx(bar_q, (uint32_t)((kTwice ? 2 : 1) * kSub * p.G * p.W * 128));
#pragma unroll
    for (int dc = 0; dc < kSub; ++dc)
      for (int at = 0; at <= (kTwice ? 64 : 0); at += 64)
        tma_load_4d(smem_u32(q_smem + dc * p.Ralloc * 128 + at * 128), &tmap_q, bar_q, dc * 64, g * p.G, 0, l * p.B + b);
    for (int i = 0; i < min(n_my, p.cap); ++i) load(i, 0);
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  // "this CTA runs and its barriers are set up": awaited before the first push.  (The warp that wrote `failed` arrives below, releasing it.)
  if (warp != kLoadWarp) cluster_arrive();
  const uint32_t tmem_base = *tmem_slot;
  auto wait = [&](uint32_t bar, uint32_t parity) {
    if (__all_sync(0xffffffffu, mbar_test(bar, parity))) return true;
    return __all_sync(0xffffffffu, mbar_wait_slow<true>(bar, parity, abort_flag, p.wait_ns)) != 0;
  };
  auto wait_cluster = [&](uint32_t bar) {
    if (__all_sync(0xffffffffu, mbar_test_cluster(bar))) return true;
    return __all_sync(0xffffffffu, mbar_wait_cluster(bar, abort_flag, p.wait_ns)) != 0;
  };

  if (warp == kLoadWarp) {
    // ------------------------------------------------------------ TMA producer (one thread)
    cluster_arrive_release();
    if (lane == 0 && n_my > 0) {
      for (int i = p.cap; i < n_my && load_ok; ++i) load(i, i / p.cap);
      for (int i = n_my - p.cap - 1; i >= 0 && load_ok; --i) load(i, phase2(i));
      // every copy has landed before the CTA can end, also when its waits run out
      for (int s = 0; s < p.cap; ++s)
        if ((used >> s) & 1u) mbar_wait<true>(bar_kfull(s), (odd >> s) & 1u, &never, p.wait_ns, 100u);
      mbar_wait<true>(bar_q, 0u, &never, p.wait_ns, 100u);
    }
    // the host's total is larger than cu_k[B]: flagged, as by sg_pack_kv, and entries that no row owns are not written (here, because the
    // workers' chain of steps is what the call takes)
    if (kPack && lane == 1 && (blockIdx.x | blockIdx.y | blockIdx.z) == 0 && p.cu_k[p.B] < p.K_tot) raise(p.dev_status, SG_ERR_INVALID);
    __syncwarp();
    cluster_wait();
    cluster_arrive();
  } else if (warp == kIssueWarp) {
    // ------------------------------------------------------------ MMA issuer (converged warp, one elected lane issues)
    const bool leader = elect_one();
    const uint32_t q_lo0 = smem_desc_lo(smem_u32(q_smem)), k_lo0 = smem_desc_lo(smem_u32(k_smem));
    const uint32_t q_sub_lo = (uint32_t)(p.Ralloc * 128) >> 4;
    constexpr uint32_t k_stage_lo = (uint32_t)kKStageBytes >> 4, k_sub_lo = (uint32_t)kKSubBytes >> 4, q_blk_lo = (128u * 128u) >> 4;
    const uint32_t idesc = make_idesc(128, 128);
    bool ok = n_my == 0 || wait(bar_q, 0u);
    uint32_t n = 0;
    for (int i = 0; i < 2 * n_my && ok; ++i) {
      const bool first = i < n_my;
      const int tile = first ? i : 2 * n_my - 1 - i, ks = stage_of(tile);
      const bool reload = first ? tile < n_my - p.cap : tile >= p.cap;       // the stage's next load waits for this use
      ok = wait(bar_kfull(ks), (uint32_t)((!first ? phase2(tile) : tile < p.cap ? 0 : tile / p.cap) & 1));
      const uint32_t k_lo = k_lo0 + ks * k_stage_lo;
      uint32_t q_lo = q_lo0;
      for (int blk = 0; blk < nblk && ok; ++blk, q_lo += q_blk_lo, ++n) {
        const uint32_t st = n & (kStages - 1);
        ok = wait(bar_aempty(st), ((n / kStages) & 1u) ^ 1u);
        if (!ok) break;
        tc_fence_after();
        if (leader) {
          if (first) umma_block<4 * kSub>(tmem_base + st * 128u, q_lo, k_lo, q_sub_lo, k_sub_lo, idesc);
          else umma_block<4 * kSub>(tmem_base + st * 128u, k_lo, q_lo, k_sub_lo, q_sub_lo, idesc);
          umma_commit(bar_afull(st));
          if (reload && blk == nblk - 1) umma_commit(bar_kempty(ks));
        }
        __syncwarp();
      }
    }
    if (leader) {
      umma_commit(bar_drain);                          // every MMA has completed before the CTA frees its tensor memory
      mbar_wait<true>(bar_drain, 0u, &never, p.wait_ns, 0u);
    }
    __syncwarp();
    cluster_wait();
    cluster_arrive();
  } else {
    // ------------------------------------------------------------ workers
    const int part_c = warp >> 2, quarter = warp & 3;  // quarter of a block's columns, of its lanes
    const int lane_row = quarter * 32 + lane;
    const uint32_t t_lane = tmem_base + ((uint32_t)(quarter * 32) << 16);
    const uint64_t scale2 = pack2(p.scale_log2, p.scale_log2);
    const int Weff = min(p.W, N), first_win = N - Weff, vis_end = (first_win + 1) / kTileKeys;
    bool ok = true;
    uint32_t n = 0;
    auto release = [&](uint32_t st) {
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(bar_aempty(st));
    };
    int ck = 0, kb = 0;
    if (kPack) { ck = p.cu_k[b]; kb = p.cu_k[b + 1] - ck; }
    const bool selects = kPack && fits && kb > 0 && kb < N;
    // "this CTA has received everything, and sends nothing more"; or it has given up (`ok` is that of all workers)
    auto last_arrive = [&] {
      __syncwarp();
      if (__builtin_expect(!ok && warp == 0, 0)) tell_failed(smem_u32(const_cast<uint32_t*>(failed)), p.csize);
      else cluster_arrive();
    };
    if (selects && tid == 0) mbar_arrive_expect_tx(bar_val, (uint32_t)((ntiles - n_my) * kTileKeys * 4 + ntiles * 8));

    // ---- 1. row statistics: a running (maximum, sum of exp2) of the thread's row over its quarter of the columns
    for (int blk = 0; blk < nblk; ++blk) {
      slot_m[part_c * p.Ralloc + blk * 128 + lane_row] = -INFINITY;
      slot_l[part_c * p.Ralloc + blk * 128 + lane_row] = 0.f;
    }
    for (int i = 0; i < n_my && ok; ++i) {
      const int tile = t0 + i;
      const bool hidden = tile >= vis_end || Weff != p.W;
      for (int blk = 0; blk < nblk; ++blk, ++n) {
        const uint32_t st = n & (kStages - 1);
        ok = wait(bar_afull(st), (n / kStages) & 1u);
        if (!ok) break;
        tc_fence_after();
        auto rows_of = [&](auto& a, int r, int col0) {  // row r, columns from col0 on
          constexpr int kCols = sizeof(a) / 4;
          if (hidden) {
            const int cmax = (r < p.R && r / p.G < Weff ? first_win + r / p.G - tile * kTileKeys : -1) - col0;     // last visible column
#pragma unroll
            for (int c = 0; c < kCols; ++c) a[c] = c <= cmax ? a[c] : 0xff800000u;
          }
          float x = fmaxf(__uint_as_float(a[0]), __uint_as_float(a[1]));
#pragma unroll
          for (int c = 2; c < kCols; c += 2) x = max3(x, __uint_as_float(a[c]), __uint_as_float(a[c + 1]));
          const int at = part_c * p.Ralloc + blk * 128 + lane_row;
          const float m = slot_m[at], mn = fmaxf(m, x * p.scale_log2);
          const float ref = mn == -INFINITY ? 0.f : mn;  // nothing visible yet: all terms are 0 (or NaN)
          uint64_t s0 = 0ull, s1 = 0ull;
          chunk_rows(a, scale2, pack2(-ref, -ref), s0, s1);
          float lo, hi;
          unpack2(add2(s0, s1), lo, hi);
          slot_l[at] = slot_l[at] * exp2f(m - ref) + (lo + hi);
          slot_m[at] = mn;
        };
        if constexpr (kTwice) {
          const int col0 = part_c * 32 + (quarter >> 1) * 16;
          uint32_t a[16];
          tmem_ld16_issue(a, t_lane + st * 128u + col0);
          tmem_ld_wait(a);
          release(st);
          if ((quarter & 1) * 32 < p.R) rows_of(a, lane_row & 63, col0);
        } else {
          if (blk * 128 + quarter * 32 >= p.R) { release(st); continue; }
          uint32_t a[32];
          tmem_ld32_issue(a, t_lane + st * 128u + part_c * 32u);
          tmem_ld_wait(a);
          release(st);
          rows_of(a, blk * 128 + lane_row, part_c * 32);
        }
      }
    }
    ok = work_sync(ok);
    // ---- exchange: every CTA gets every CTA's statistics
    cluster_wait();                                    // all CTAs of the cluster run
    if (ok && (u != p.withhold_unit || rank != 0)) {
      for (int r = tid & 127; r < (kTwice ? 64 : p.Ralloc); r += 128) {
        float m[8], M = -INFINITY, L = 0.f;
#pragma unroll
        for (int w = 0; w < 8; ++w) {                  // (the second half only where the rows stand twice)
          m[w] = w < 4 || kTwice ? slot_m[(w & 3) * p.Ralloc + r + (w >> 2) * 64] : -INFINITY;
          M = fmaxf(M, m[w]);
        }
        const float Mu = M == -INFINITY ? 0.f : M;
#pragma unroll
        for (int w = 0; w < 8; ++w)
          if (w < 4 || kTwice) L += slot_l[(w & 3) * p.Ralloc + r + (w >> 2) * 64] * exp2f(m[w] - Mu);
        const uint32_t own_rec = smem_u32(rec + rank * p.Ralloc + r);
        for (int to = tid >> 7; to < p.csize; to += 4) push2(at_rank(own_rec, to), at_rank(bar_rec, to), __float_as_uint(M), __float_as_uint(L));
      }
    }
    __syncwarp();
    if (ok) ok = wait_cluster(bar_rec);
    if (ok) {
      // One thread per row: what four warps per scheduler take for their instructions is more than what the loads in a row take.
      for (int r = tid; r < p.Ralloc; r += kWork) {
        float M = -INFINITY, L = 0.f;
        for (int q0 = 0; q0 < p.csize; q0 += 8) {
          float2 v[8];
          float m = M;
#pragma unroll
          for (int c = 0; c < 8; ++c) {
            v[c] = q0 + c < p.csize ? rec[(q0 + c) * p.Ralloc + r] : make_float2(-INFINITY, 0.f);
            m = fmaxf(m, v[c].x);
          }
          const float Mu = m == -INFINITY ? 0.f : m;
          L *= exp2f(M - Mu);
#pragma unroll
          for (int c = 0; c < 8; ++c) L += v[c].y * exp2f(v[c].x - Mu);
          M = m;
        }
        neg_lse[r] = r < p.R && r < Weff * p.G ? -(M + log2f(L)) : -INFINITY;
      }
    }
    ok = work_sync(ok);

    // ---- 2. column sums of the thread's key over its quarter of the rows
    for (int i1 = n_my; i1 > 0 && ok; i1 -= p.own) {   // (one trip, unless max_seqlen was no upper bound)
      const int i0 = max(0, i1 - p.own);
      for (int i = i1 - 1; i >= i0 && ok; --i) {
        const int tile = t0 + i, rmin = (tile * kTileKeys + lane_row - first_win) * p.G;        // rows below rmin cannot see the key
        uint64_t s0 = 0ull, s1 = 0ull;
        for (int blk = 0; blk < nblk; ++blk, ++n) {
          const uint32_t st = n & (kStages - 1);
          ok = wait(bar_afull(st), (n / kStages) & 1u);
          if (!ok) break;
          tc_fence_after();
          const int rows = min(128, p.R - blk * 128);
          auto columns = [&](auto& a, int r0) {
            constexpr int kCols = sizeof(a) / 4;
            if (tile >= vis_end) {
              const int c_lo = rmin - blk * 128 - r0;
#pragma unroll
              for (int c = 0; c < kCols; ++c) a[c] = c >= c_lo ? a[c] : 0xff800000u;
            }
            chunk_cols(a, scale2, neg_lse + blk * 128 + r0, s0, s1);
          };
          if (rows > 64) {
            const int r0 = part_c * 32;
            if (r0 >= rows) { release(st); continue; }
            uint32_t a[32];
            tmem_ld32_issue(a, t_lane + st * 128u + r0);
            tmem_ld_wait(a);
            release(st);
            columns(a, r0);
          } else {
            const int r0 = part_c * 16;
            if (r0 >= rows) { release(st); continue; }
            uint32_t a[16];
            tmem_ld16_issue(a, t_lane + st * 128u + r0);
            tmem_ld_wait(a);
            release(st);
            columns(a, r0);
          }
        }
        float lo, hi;
        unpack2(add2(s0, s1), lo, hi);
        cols[part_c * (p.own * kTileKeys) + (i - i0) * kTileKeys + lane_row] = lo + hi;
      }
      ok = work_sync(ok);
      if (!ok) break;
      for (int ti = warp; ti < i1 - i0; ti += kWorkWarps) {
        const int at = ti * kTileKeys + lane * 4, tile = t0 + i0 + ti, t = tile * kTileKeys + lane * 4;
        float4 s = *reinterpret_cast<const float4*>(cols + at);
#pragma unroll
        for (int w = 1; w < 4; ++w) {
          const float4 v = *reinterpret_cast<const float4*>(cols + w * (p.own * kTileKeys) + at);
          s.x += v.x; s.y += v.y; s.z += v.z; s.w += v.w;
        }
        if (selects) {
          const uint4 k = make_uint4(order_key(__float_as_uint(s.x)), order_key(__float_as_uint(s.y)), order_key(__float_as_uint(s.z)), order_key(__float_as_uint(s.w)));
          *reinterpret_cast<uint4*>(vals + t) = k;
          uint32_t kmin = 0xffffffffu, kmax = 0u;
          if (t < N) { kmin = min(kmin, k.x); kmax = max(kmax, k.x); }
          if (t + 1 < N) { kmin = min(kmin, k.y); kmax = max(kmax, k.y); }
          if (t + 2 < N) { kmin = min(kmin, k.z); kmax = max(kmax, k.z); }
          if (t + 3 < N) { kmin = min(kmin, k.w); kmax = max(kmax, k.w); }
          kmin = __reduce_min_sync(0xffffffffu, kmin);
          kmax = __reduce_max_sync(0xffffffffu, kmax);
          if (lane < p.csize) push2(at_rank(smem_u32(minmax + tile), lane), at_rank(bar_val, lane), kmin, kmax);
        }
        float* o = p.importance + (int64_t)u * p.T + c0 + t;
        if (t + 3 < N && (reinterpret_cast<uintptr_t>(o) & 15u) == 0) {
          *reinterpret_cast<float4*>(o) = s;
        } else {
          if (t < N) o[0] = s.x;
          if (t + 1 < N) o[1] = s.y;
          if (t + 2 < N) o[2] = s.z;
          if (t + 3 < N) o[3] = s.w;
        }
      }
      if (i0 > 0) ok = work_sync(ok);                  // `cols` is written again
    }
    if (selects) {
      // This CTA's keys to all others, a bulk copy each.  (16-byte remote stores: 28 warps' worth for seven tiles and ten CTAs took
      // 5.0 k clocks.)
      fence_proxy_async();
      ok = work_sync(ok);
      if (ok && warp == 0 && lane < p.csize && lane != rank && n_my > 0) {
        const uint32_t from = smem_u32(vals + t0 * kTileKeys);
        asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                     ::"r"(at_rank(from, lane)), "r"(from), "r"(n_my * kTileKeys * 4), "r"(at_rank(bar_val, lane)) : "memory");
      }
      __syncwarp();
    }
    if constexpr (kPack) {
      const int64_t row0 = ((int64_t)l * p.K_tot + ck) * p.Hkv + (int64_t)g * kb;          // packed row of entry 0
      int32_t* const out = p.sel_idx + ((int64_t)l * p.Hkv + g) * p.K_tot + ck;
      constexpr int kTPR = D / 8, kRowGroups = kWork / kTPR;
      const int x = tid % kTPR, grp = tid / kTPR;      // 16-byte piece of a row
      const int p0 = t0 * kTileKeys, own = min(N, (t0 + n_my) * kTileKeys) - p0;           // this CTA's keys (none: not positive)
      // entry j is position t, one of this CTA's keys: K from its tile where that is still there, V from the cache
      const int64_t src = (int64_t)l * p.ls + (int64_t)c0 * p.ts + (int64_t)g * p.hs + x * 8;
      auto pack_own = [&](int count, int first, auto pos_of) {
        constexpr int kFlight = 4;
        for (int j0 = grp; j0 < count; j0 += kFlight * kRowGroups) {
          int4 k[kFlight], v[kFlight];
          int t[kFlight];
#pragma unroll
          for (int f = 0; f < kFlight; ++f) {
            const int j = j0 + f * kRowGroups;
            t[f] = j < count ? pos_of(j) : -1;
            if (t[f] < 0) continue;
            v[f] = __ldcs(reinterpret_cast<const int4*>(p.v_cache + src + (int64_t)t[f] * p.ts));
            const int ti = (t[f] >> 7) - t0, r = t[f] & (kTileKeys - 1);
            if (ti < p.cap) k[f] = *reinterpret_cast<const int4*>(k_smem + ti * kKStageBytes + (x >> 3) * kKSubBytes + r * 128 + (((x & 7) ^ (r & 7)) << 4));
            else k[f] = __ldcs(reinterpret_cast<const int4*>(p.k_cache + src + (int64_t)t[f] * p.ts));
          }
#pragma unroll
          for (int f = 0; f < kFlight; ++f) {
            if (t[f] < 0) continue;
            const int64_t dst = (row0 + first + j0 + f * kRowGroups) * D + x * 8;
            __stcs(reinterpret_cast<int4*>(p.packed_k + dst), k[f]);
            __stcs(reinterpret_cast<int4*>(p.packed_v + dst), v[f]);
          }
        }
      };
      auto zero_rows = [&](int from) { clear_entries<D>(out, p.packed_k + row0 * D, p.packed_v + row0 * D, from, kb, tid, rank, p.csize); };
      for (int i = 0; i < min(n_my, p.cap) && ok; ++i)  // the tiles' bytes are seen by this thread (the MMAs have used them long ago)
        ok = wait(bar_kfull(i), (uint32_t)(phase2(i) & 1));
      if (selects) {
        // ---- 3. selection, by every CTA on all keys of the row: an interval [lo, hi] of keys that holds the kb-th largest is narrowed by
        // histograms of 2048 bins until few enough are left to be ranked (as select_topk.cu)
        __syncwarp();
        if (ok) ok = wait_cluster(bar_val);
        ok = work_sync(ok);
        last_arrive();
        if (ok) {
          uint32_t lo = 0xffffffffu, hi = 0u, need = (uint32_t)kb;
          for (int i = lane; i < ntiles; i += 32) { const uint2 v = minmax[i]; lo = min(lo, v.x); hi = max(hi, v.y); }
          lo = __reduce_min_sync(0xffffffffu, lo);
          hi = __reduce_max_sync(0xffffffffu, hi);
          const uint4* const vals4 = reinterpret_cast<const uint4*>(vals);
          const int quads = (N + 3) >> 2;
          auto in_row = [&](int q, int e) { return 4 * q + e < N; };     // the last quad may hold keys behind the row's end
#pragma unroll 1
          while (lo != hi) {
            const uint32_t width = hi - lo;
            const int shift = max(0, 32 - __clz(width) - 11);
#pragma unroll 1
            for (int q = tid; q < quads; q += kWork) {
              const uint4 k = vals4[q];
              if (k.x - lo <= width) atomicAdd(&hist[(k.x - lo) >> shift], 1u);
              if (k.y - lo <= width && in_row(q, 1)) atomicAdd(&hist[(k.y - lo) >> shift], 1u);
              if (k.z - lo <= width && in_row(q, 2)) atomicAdd(&hist[(k.z - lo) >> shift], 1u);
              if (k.w - lo <= width && in_row(q, 3)) atomicAdd(&hist[(k.w - lo) >> shift], 1u);
            }
            work_sync(true);
            // thread t looks at the bins from 2047 - 4t down
            uint4* const h = reinterpret_cast<uint4*>(hist) + (kBins / 4 - 1 - tid);
            const uint4 c = *h;
            *h = make_uint4(0, 0, 0, 0);
            const uint32_t mine = c.x + c.y + c.z + c.w;
            uint32_t inc = mine;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
              const uint32_t v = __shfl_up_sync(0xffffffffu, inc, off);
              if (lane >= off) inc += v;
            }
            if (lane == 31) wsum[warp] = inc;
            work_sync(true);
            const uint32_t above = __reduce_add_sync(0xffffffffu, lane < warp ? wsum[lane & 15] : 0u) + inc - mine;
            if (above < need && need <= above + mine) {
              uint32_t run = above, which = 0, cnt = c.w;
              if (need > run + cnt) { run += cnt; which = 1; cnt = c.z; }
              if (need > run + cnt) { run += cnt; which = 2; cnt = c.y; }
              if (need > run + cnt) { run += cnt; which = 3; cnt = c.x; }
              sh[0] = (uint32_t)(kBins - 1 - 4 * tid) - which; sh[1] = need - run; sh[2] = cnt; sh[3] = 0;
            }
            work_sync(true);
            lo += sh[0] << shift;
            hi = lo + min(hi - lo, (1u << shift) - 1u);
            need = sh[1];
            const int ncand = (int)sh[2];
            if (lo != hi && ncand <= kRankMax) {
              const uint32_t w = hi - lo;
#pragma unroll 1
              for (int q0 = warp * 32; q0 < quads; q0 += kWork) {
                const int q = q0 + lane;
                const uint4 k = q < quads ? vals4[q] : make_uint4(0, 0, 0, 0);
                const uint32_t kk[4] = {k.x, k.y, k.z, k.w};
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                  const bool in = q < quads && in_row(q, e) && kk[e] - lo <= w;
                  const uint32_t m = __ballot_sync(0xffffffffu, in);
                  if (m == 0) continue;
                  uint32_t base = 0;
                  if (lane == 0) base = atomicAdd(&sh[3], (uint32_t)__popc(m));
                  base = __shfl_sync(0xffffffffu, base, 0);
                  if (in) cand[base + __popc(m & ((1u << lane) - 1u))] = kk[e];
                }
              }
              work_sync(true);
              // four lanes per key, a quarter of the list each; values behind the list's end do not count
              const int i = tid >> 2, sub = tid & 3;
              if (warp * 8 < ncand) {
                const uint32_t k = i < ncand ? cand[i] : 0u;
                uint32_t greater = 0, same = 0;
                for (int j = 4 * sub; j < ncand; j += 16) {
                  const uint4 o = *reinterpret_cast<const uint4*>(cand + j);
                  const int left = ncand - j;
                  greater += (o.x > k ? 1u : 0u) + (left > 1 && o.y > k ? 1u : 0u) + (left > 2 && o.z > k ? 1u : 0u) + (left > 3 && o.w > k ? 1u : 0u);
                  same += (o.x == k ? 1u : 0u) + (left > 1 && o.y == k ? 1u : 0u) + (left > 2 && o.z == k ? 1u : 0u) + (left > 3 && o.w == k ? 1u : 0u);
                }
#pragma unroll
                for (int o = 1; o < 4; o <<= 1) {
                  greater += __shfl_xor_sync(0xffffffffu, greater, o);
                  same += __shfl_xor_sync(0xffffffffu, same, o);
                }
                if (sub == 0 && i < ncand && greater < need && need <= greater + same) { sh[4] = k; sh[5] = need - greater; }    // equal keys write equal values
              }
              work_sync(true);
              lo = hi = sh[4];
              need = sh[5];
            }
          }
          const uint32_t tau = lo, need_eq = need;     // keep all above tau and the first need_eq of those equal to it

          // this CTA's entries: keys in front of its range are counted, its own ranked (greater in the low half of a word, equal in
          // the high half: a row has at most 32768 keys)
          uint32_t before = 0;
#pragma unroll 1
          for (int q = tid; q < p0 / 4; q += kWork) {
            const uint4 k = vals4[q];
            before += (k.x > tau ? 1u : 0u) + (k.y > tau ? 1u : 0u) + (k.z > tau ? 1u : 0u) + (k.w > tau ? 1u : 0u);
            before += (k.x == tau ? 0x10000u : 0u) + (k.y == tau ? 0x10000u : 0u) + (k.z == tau ? 0x10000u : 0u) + (k.w == tau ? 0x10000u : 0u);
          }
          before = __reduce_add_sync(0xffffffffu, before);
          if (lane == 0) wsum[warp] = before;
          uint32_t bgt[kSweeps], beq[kSweeps];
#pragma unroll
          for (int i = 0; i < kSweeps; ++i) {
            bgt[i] = beq[i] = 0u;
            if (i * kWork >= own) continue;
            const int j = i * kWork + tid;
            const uint32_t k = j < own ? vals[p0 + j] : 0u;
            bgt[i] = __ballot_sync(0xffffffffu, j < own && k > tau);
            beq[i] = __ballot_sync(0xffffffffu, j < own && k == tau);
            if (lane == 0) wsum2[i * kWorkWarps + warp] = (uint32_t)__popc(bgt[i]) | ((uint32_t)__popc(beq[i]) << 16);
          }
          work_sync(true);
          const uint32_t base = __reduce_add_sync(0xffffffffu, lane < kWorkWarps ? wsum[lane] : 0u);    // in front of the range
          const uint32_t first = (base & 0xffffu) + min(base >> 16, need_eq);
          uint32_t total = base;
#pragma unroll
          for (int i = 0; i < kSweeps; ++i) {
            if (i * kWork >= own) continue;
            const uint32_t v = lane < kWorkWarps ? wsum2[i * kWorkWarps + lane] : 0u;
            const uint32_t at = total + __reduce_add_sync(0xffffffffu, lane < warp ? v : 0u);
            total += __reduce_add_sync(0xffffffffu, v);
            const uint32_t lt = (1u << lane) - 1u;
            const uint32_t eq = (at >> 16) + __popc(beq[i] & lt), slot = (at & 0xffffu) + __popc(bgt[i] & lt) + min(eq, need_eq);
            const bool is_gt = (bgt[i] >> lane) & 1u, is_eq = (beq[i] >> lane) & 1u;
            if (is_gt || (is_eq && eq < need_eq)) {
              const int t = p0 + i * kWork + tid;
              out[slot] = t;
              list[slot - first] = t;
            }
          }
          const int count = (int)((total & 0xffffu) + min(total >> 16, need_eq) - first);
          work_sync(true);
          // ---- 4. packing
          pack_own(count, (int)first, [&](int j) { return list[j]; });
        }
      } else {
        ok = work_sync(ok);
        last_arrive();
      }
      if (kb > 0 && !fits) {
        // longer than max_seqlen promised: as sg_select_pack_kv
        if (rank == 0 && tid == 0) { raise(p.dev_status, SG_ERR_INVALID); raise(p.dev_status, SG_ERR_INDEX); }
        zero_rows(0);
      } else if (kb > 0 && !selects) {
        // the whole prompt (or an over-sized budget)
        if (kb > N && rank == 0 && tid == 0) { raise(p.dev_status, SG_ERR_INVALID); raise(p.dev_status, SG_ERR_INDEX); }
        if (ok) {
          for (int j = tid; j < own; j += kWork) out[p0 + j] = p0 + j;
          pack_own(own, p0, [&](int j) { return p0 + j; });
        }
        zero_rows(N);
      }
    } else {
      last_arrive();
    }
  }
  // ---------------------------------------------------------------- teardown
  if (!kPack) pdl_launch_dependents();                 // (the packed rows of a prefill may be inputs that the next kernel reads at once)
  __syncwarp();
  cluster_wait();                                      // nobody sends to this CTA or reads from it any more
  if (__builtin_expect(*failed, 0)) give_up<D, kPack>(bar_rec, bar_val, p.wait_ns, p.cu_k, p.sel_idx, p.packed_k, p.packed_v, p.K_tot, p.Hkv, p.csize);
  tc_fence_before();
  __syncthreads();
  if (warp == kIssueWarp) {
    tc_fence_after();
    tmem_dealloc(tmem_base, 512);
  }
  if (tid == 0 && *abort_flag) raise(p.dev_status, SG_ERR_TIMEOUT);
}

// ---------------------------------------------------------------- host side
constexpr int kSmemLimit = 232448, kMaxCluster = 16;

template <int D, bool kPack, bool kTwice>
cudaError_t prepare_kernel() {
  // once per device: the clusters' size may exceed the portable eight, the shared memory the default
  static std::atomic<int> done[64];
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev >= 0 && dev < 64 && done[dev].load(std::memory_order_relaxed)) return cudaSuccess;
  e = cudaFuncSetAttribute(score_cluster_kernel<D, kPack, kTwice>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemLimit);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(score_cluster_kernel<D, kPack, kTwice>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e == cudaSuccess && dev >= 0 && dev < 64) done[dev].store(1, std::memory_order_relaxed);
  return e;
}

// How many clusters of `csize` CTAs (one per SM) the current device holds at once; asked once per device and size.
int clusters_at_once(int csize) {
  static std::atomic<int> known[64][kMaxCluster + 1];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
  int n = known[dev][csize].load(std::memory_order_relaxed);
  if (n == 0) {
    if (prepare_kernel<128, true, false>() != cudaSuccess) return 0;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim = {(unsigned)csize, 1, 1};
    cfg.gridDim = dim3((unsigned)csize);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = kSmemLimit;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    int got = 0;
    if (cudaOccupancyMaxActiveClusters(&got, score_cluster_kernel<128, true, false>, &cfg) != cudaSuccess) {
      (void)cudaGetLastError();
      got = 0;
    }
    n = got + 1;                                       // 0 stands for "not asked yet"
    known[dev][csize].store(n, std::memory_order_relaxed);
  }
  return n - 1;
}

struct ClusterPlan {
  int csize, own, cap, smem;
  bool ok;
};
// Whether one kernel takes less than the launches one by one.  Its time is that of the CTA with the most blocks (key tiles x 128 query
// rows): 9.5 us and, per tile, 0.65 + 1.4 us per row block.  score.cu deals the tiles of all parts out evenly, so that its time goes with
// the tiles per SM: with one row block about 18 us with one, 24 with three, 26 with four, 30 with five; with two 22, 33, 37; with four 26
// with one.  Up to eight tiles of single prompts and of batches of equal lengths that is the one kernel's, but a batch with one long
// prompt among short ones leaves most of its CTAs idle.  Measured on 400 shapes, calls in a row and on keys not in L2, microseconds one by
// one -> one kernel; taken, 32 query and 8 KV heads of 128, 128 rows: 512 tokens 16.8 -> 10.2, 2048 19.9 -> 12.6, 4096 (four tiles)
// 22.6 -> 17.0, 8192 (seven) 25.8 -> 25.0 (keys not in L2 28.8 -> 26.5), 10000 (eight) 30.1 -> 28.3, seven of 100 and one of 1790 (seven)
// 23.5 -> 23.2, 2040 and 100 in turn, four each (eight) 29.3 -> 25.6; 256 rows: 7500 (six) 35.2 -> 32.8, four of 1270 and of 100 (five)
// 36.9 -> 27.5; 64 rows, heads of 64, 6000 and 100 (eight) 23.9 -> 20.8.
// Not taken, 128 rows: seven of 100 and one of 2048 (eight) 23.3 -> 25.0, 3000 and 6000 (eight) 26.0 -> 26.8; 256 rows: seven of 100 and one of
// 1270 (five) 24.3 -> 27.0, of 2040 28.7 -> 36.5; 512 rows, 2 heads: 20 of 100 and one of 2900 26.6 -> 58.2.
// Scores alone, taken: 128 rows, 4096 tokens (four) 13.3 -> 11.9; 256 rows, 3000 (three) 0.86 of the time; 512 rows, 8 layers of 2000, 2 heads
// (three) 0.90.  Not taken: 6500 (six) 14.4 -> 14.9; 256 rows, seven of 100 and one of 1000 (four) 1.18, 512 rows, 20 of 100 and one of 1000 (three) 1.30.
bool cluster_pays(const sg_shape* s, int own, int Ralloc, bool packs) {
  const int R = s->num_q_heads / s->num_kv_heads * s->window, blocks = own * (Ralloc / 128);
  const double parts = (double)s->num_layers * s->batch * s->num_kv_heads;
  const double even = (s->total_tokens / 64.0 + s->batch) * s->num_layers * s->num_kv_heads / (2 * kNumSMs);     // expected tiles per SM
  if (!packs) return own <= kMaxOwnScore && (own == 1 || blocks <= 4 || (even >= 1 && blocks <= 4 + 5 * even));
  if (own == kMaxOwn && !(even >= 4 || (even >= 3 && parts >= 32) || (R <= 64 && (s->head_dim == 64 || even >= 2)))) return false;
  return own <= kMaxOwn && blocks <= 7 + 1.4 * (Ralloc / 128) * even;
}
// The largest cluster with which all parts are resident at once (on B200 15 clusters of 9, 11 of 10, 7 of 16), no larger than the longest
// sequence has tiles.
ClusterPlan plan_cluster(const sg_shape* s, int Ralloc, bool packs) {
  ClusterPlan pl{};
  const int64_t parts = (int64_t)s->num_layers * s->batch * s->num_kv_heads;
  if (parts > kNumSMs) return pl;
  if (packs && s->batch == 1 && s->max_seqlen < s->total_tokens) return pl;      // broken promise: the selection says so
  const int longest = s->batch == 1 ? s->total_tokens : s->max_seqlen, tiles = longest / kTileKeys + (longest % kTileKeys != 0);
  int cs = kMaxCluster;
  while (cs > 1 && (cs > tiles || parts * cs > kNumSMs || parts > clusters_at_once(cs))) --cs;
  if (parts > clusters_at_once(cs)) return pl;
  pl.csize = cs;
  pl.own = tiles > cs ? (tiles + cs - 1) / cs : 1;
  if (!cluster_pays(s, pl.own, Ralloc, packs)) return pl;
  pl.cap = pl.own;
  while (pl.cap > 0 && carve(s->head_dim, Ralloc, cs, pl.own, pl.cap).total + 1024 > kSmemLimit) --pl.cap;
  if (pl.cap < pl.own && pl.cap < 2) return pl;        // tiles that are loaded twice need a second stage
  pl.smem = carve(s->head_dim, Ralloc, cs, pl.own, pl.cap).total + 1024;
  if (pl.smem < 120 * 1024) pl.smem = 120 * 1024;      // one CTA per SM: each takes the whole TMEM
  pl.ok = true;
  return pl;
}

template <int D, bool kPack, bool kTwice>
sg_status launch_kernel(const CUtensorMap& q, const CUtensorMap& k, const ClusterParams& p, const ClusterPlan& pl, const sg_shape* shape, cudaStream_t s) {
  SG_CUDA_TRY((prepare_kernel<D, kPack, kTwice>()));
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim = {(unsigned)pl.csize, 1, 1};
  cfg.gridDim = dim3((unsigned)pl.csize, (unsigned)(shape->batch * shape->num_kv_heads), (unsigned)shape->num_layers);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = (size_t)pl.smem;
  cfg.stream = s;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  SG_CUDA_TRY(cudaLaunchKernelEx(&cfg, score_cluster_kernel<D, kPack, kTwice>, q, k, p));
  return SG_OK;
}
template <int D, bool kPack>
sg_status launch(const CUtensorMap& q, const CUtensorMap& k, const ClusterParams& p, const ClusterPlan& pl, const sg_shape* shape, cudaStream_t s) {
  return p.R <= 64 ? launch_kernel<D, kPack, true>(q, k, p, pl, shape, s) : launch_kernel<D, kPack, false>(q, k, p, pl, shape, s);
}

}  // namespace

int score_cluster_size(const sg_shape* s, bool packs) {
  const int R = s->num_q_heads / s->num_kv_heads * s->window;
  const ClusterPlan pl = plan_cluster(s, (R + 127) & ~127, packs);
  return pl.ok ? pl.csize : 0;
}

sg_status score_cluster_launch(const sg_shape* s, const CUtensorMap& q, const CUtensorMap& k, const ScoreLaunch& a, const PackLaunch* pack) {
  ClusterParams p = {};
  p.cu = s->cu_seqlens;
  p.importance = a.importance;
  p.dev_status = a.dev_status;
  p.T = s->total_tokens;
  p.B = s->batch;
  p.Hkv = s->num_kv_heads;
  p.G = s->num_q_heads / s->num_kv_heads;
  p.W = s->window;
  p.R = p.G * p.W;
  p.Ralloc = (p.R + 127) & ~127;
  const ClusterPlan pl = plan_cluster(s, p.Ralloc, pack != nullptr);
  if (!pl.ok) return SG_ERR_UNSUPPORTED;
  p.csize = pl.csize;
  p.own = pl.own;
  p.cap = pl.cap;
  p.withhold_unit = a.withhold_unit;
  p.wait_ns = a.wait_ns;
  p.scale_log2 = kLog2e / sqrtf((float)s->head_dim);
  if (!pack) return s->head_dim == 128 ? launch<128, false>(q, k, p, pl, s, a.stream) : launch<64, false>(q, k, p, pl, s, a.stream);
  p.cu_k = pack->cu_k;
  p.K_tot = pack->total_sel;
  p.sel_idx = pack->sel_idx;
  p.k_cache = static_cast<const uint16_t*>(pack->k_cache);
  p.v_cache = static_cast<const uint16_t*>(pack->v_cache);
  p.packed_k = static_cast<uint16_t*>(pack->packed_k);
  p.packed_v = static_cast<uint16_t*>(pack->packed_v);
  p.ls = s->cache_layer_stride;
  p.ts = s->cache_token_stride;
  p.hs = s->cache_head_stride;
  return s->head_dim == 128 ? launch<128, true>(q, k, p, pl, s, a.stream) : launch<64, true>(q, k, p, pl, s, a.stream);
}

}  // namespace sg
