// sg_score: window-query x key-cache scoring with a fused softmax and row-reduce (sm_100a).
//
// For one (layer, sequence, KV head) -- a "part" -- the R = G*W window queries are scored against all N keys: a dense
// R x N x d contraction, so it runs on the 5th-generation tensor cores.  importance[t] = sum_r softmax_row_r(s)[t] needs
// every row's normaliser before any probability can be summed down a column, so the work is two passes over the keys,
// each a kernel of its own:
//
//   pass 1 (row statistics)  D[row r][key t]  = Q_blk (A, 128 rows) x K_tile^T (B, 128 keys):
//          each epilogue thread owns one query row (one TMEM lane) and keeps a running
//          (reference, sum of exp2) over the key columns -- no cross-thread reduction.
//   pass 2 (column sums)     D[key t][row r]  = K_tile (A, 128 keys) x Q_blk^T (B, 128 rows):
//          each epilogue thread owns one key (one TMEM lane) and adds exp2(s*c - lse_r) over the
//          query-row columns; lse_r is a per-column constant read from shared memory.
//
// The score matrix never leaves the SM.  The key tiles of all parts of a launch, in order, are cut into one contiguous
// range per CTA, so every CTA has the same work to within a tile; a CTA's piece of a part is a "segment".  Pass 1 leaves one
// record per segment ((reference, sum) of every row), pass 2 merges a part's records into its rows' log-sum-exps.  The
// kernel boundary is the only synchronisation between CTAs: measured against one persistent kernel that ran both passes
// behind per-part counters in global memory, no CTA waits for another CTA's statistics in mid-kernel (a third of the time
// of a one-layer call), and each kernel holds one hot loop.  The launches follow one another by programmatic dependent
// launch: a kernel sets itself up (pass 2 also requests its first tiles) while the one before it drains; so does pass 1 behind
// whatever precedes the call (a whole call for one layer of 8192 tokens: 35.0 -> 30.8 us).
//
// Roles of a CTA (one per SM): twelve epilogue warps (three warpgroups, each taking every third block, a block being a
// key tile x row block), one warp feeding Q and 128-key K tiles with TMA into 128-byte-swizzled shared memory, one issuing
// tcgen05.mma into four 128-column TMEM stages, two helper warps (merging statistics and, for several row blocks per
// tile, adding up the warpgroups' column sums) off the epilogue's path.
//
// Every wait is bounded: on expiry the CTA raises SG_ERR_TIMEOUT in the status word, stops issuing work, waits
// (bounded) for its own TMA copies and MMAs, frees its TMEM and returns.
#include <cuda.h>

#include "common.cuh"
#include "internal.h"
#include "launch.h"
#include "score_launch.h"
#include "score_math.cuh"
#include "tcgen05.cuh"

namespace sg {
namespace {

constexpr int kGroups = 3;                // epilogue warpgroups (four warps each, one per TMEM lane quarter)
constexpr int kEpiWarps = 4 * kGroups;
constexpr int kTmaWarp = kEpiWarps, kMmaWarp = kTmaWarp + 1, kHelperWarp = kMmaWarp + 1 /* two */;
constexpr int kThreads = 32 * (kHelperWarp + 2);
constexpr int kTileKeys = 128;
constexpr int kStages = 4;                // 4 x 128 fp32 columns = the whole 512-column TMEM
constexpr int kColSlots = 4;              // pass 2, several row blocks per tile: partial column sums of four tiles in flight
constexpr int kMaxKStages = 4;
constexpr int kSmemLimit = 232448;        // 227 KB opt-in dynamic shared memory per CTA

// Debug build (-DSG_CHECKS): device-side checks of the shared-memory carve-up and of every TMA coordinate (tile inside
// the tensor or hanging over its end only where the fill value is wanted).  A failed check never traps: it sets the
// SG_ERR_INVALID bit of the status word and the access is still made only if it is known to be harmless (TMA loads
// past the end are zero-filled by the hardware), so a debug run ends like any other and reports the bit.
#ifdef SG_CHECKS
#define SG_CHECK(cond) do { if (!(cond)) raise(p.dev_status, SG_ERR_INVALID); } while (0)
#else
#define SG_CHECK(cond) do { } while (0)
#endif

// Profiling build (-DSG_SCORE_PROFILE): the MMA warp and one warp per warpgroup add up the clocks they spend waiting; the
// sums go behind the CTA's four clock words of the testing clock buffer (32 words per CTA).
#ifdef SG_SCORE_PROFILE
constexpr int kClockWords = 32;
#define SG_PROF_WAIT(acc, expr) do { const long long _t = clock64(); expr; acc += clock64() - _t; } while (0)
#define SG_PROF_STORE(slot, v) do { if (p.clock_out && lane == 0) p.clock_out[32 * (size_t)blockIdx.x + (slot)] = (unsigned long long)(v); } while (0)
#else
constexpr int kClockWords = 4;
#define SG_PROF_WAIT(acc, expr) do { expr; } while (0)
#define SG_PROF_STORE(slot, v) do { (void)(v); } while (0)
#endif

struct ScoreParams {
  const int32_t* cu;
  float* importance;
  float2* records;         // [parts + CTAs][Ralloc] row statistics (log2-domain reference, sum of exp2) of a segment
  int32_t* dev_status;
  int64_t T;
  int32_t B, Hkv, G, W, R, Ralloc;
  int32_t units;           // (layer, KV head) units of the call
  int32_t k_stages, q_bufs;
  int32_t smem_bytes;      // dynamic shared memory of the launch (debug checks)
  int32_t withhold_unit;   // testing only: the statistics of this unit's segments are never handed to the helpers (-1 = none)
  uint32_t wait_ns;        // limit of every bounded wait, nanoseconds
  unsigned long long* clock_out;   // testing only: per CTA {clock64 start, end, globaltimer start, end}, or null
  float scale_log2;
};

// ---------------------------------------------------------------- schedule
// CTAs that get tiles (the host sizes the grid by an upper bound of the tile count).
__device__ __forceinline__ int busy_ctas(long long tt) { return tt < (long long)gridDim.x ? (int)tt : (int)gridDim.x; }
// The CTA whose range holds tile `pos` of the launch's `tt`.
__device__ __forceinline__ int cta_of(long long pos, long long tt, int busy) { return (int)(((pos + 1) * busy - 1) / tt); }
// A CTA's segments: its range of the launch's key tiles [c * tt / busy, (c + 1) * tt / busy), cut at part boundaries.  Pass 2
// walks the range backwards, segments and tiles: what pass 1 read last is still in L2.
struct Segment {
  int u, b;                // unit and sequence
  int c0, N;               // first token and length of sequence b
  int tile_beg, tile_end;  // tiles of the part
  int part;
};
template <int PASS>
struct SegmentWalk {
  int C, B, pos, end;
  const int *cu, *prefix;  // prefix[b] = tiles of the sequences before b (prefix[B] = C)
  __device__ __forceinline__ SegmentWalk(int C_, int units, int B_, const int* cu_, const int* prefix_) : C(C_), B(B_), cu(cu_), prefix(prefix_) {
    const long long tt = (long long)units * C;
    const int g = busy_ctas(tt);
    pos = (int)blockIdx.x < g ? (int)(tt * blockIdx.x / g) : 0;
    end = (int)blockIdx.x < g ? (int)(tt * (blockIdx.x + 1) / g) : 0;
  }
  __device__ __forceinline__ bool next(Segment& s) {
    if (pos >= end) return false;
    const int at = PASS == 1 ? pos : end - 1;         // a tile of the segment
    const int u = at / C, j = at - u * C;
    int lo = 0, hi = B;
    while (hi - lo > 1) {
      const int mid = (lo + hi) >> 1;
      if (prefix[mid] <= j) lo = mid; else hi = mid;
    }
    s.u = u;
    s.b = lo;
    s.c0 = cu[lo];
    s.N = cu[lo + 1] - s.c0;
    const int tile = j - prefix[lo];
    s.tile_beg = PASS == 1 ? tile : max(0, tile - (at - pos));
    s.tile_end = PASS == 1 ? min(prefix[lo + 1] - prefix[lo], tile + (end - pos)) : tile + 1;
    s.part = u * B + lo;
    if (PASS == 1) pos += s.tile_end - s.tile_beg; else end -= s.tile_end - s.tile_beg;
    return true;
  }
};
// The i-th tile of a segment in the order of the pass.
template <int PASS>
__device__ __forceinline__ int tile_at(const Segment& s, int i) { return PASS == 1 ? s.tile_beg + i : s.tile_end - 1 - i; }

// Log-sum-exps of a part's rows from its segments' records: rows r0, r0 + step, ..., kFlight records in flight, of up to kRows rows.  Negated, as
// the epilogue of pass 2 adds them; rows outside the window get -inf: exp2(x - inf) = 0.
template <int kFlight, int kRows>
__device__ __forceinline__ void merge_records(const ScoreParams& p, const Segment& sg, const int* prefix, int C, float* neg_lse, int r0, int step) {
  const long long tt = (long long)p.units * C, first = (long long)sg.u * C + prefix[sg.b];
  const int busy = busy_ctas(tt), Weff = min(p.W, sg.N);
  const int c_lo = cta_of(first, tt, busy), nrec = cta_of(first + (prefix[sg.b + 1] - prefix[sg.b]) - 1, tt, busy) - c_lo + 1;
  constexpr int kRecs = 4;
  if (kRows > 1 && nrec <= kRecs) {
    // Short parts: a warp has many rows of one or two records each and a segment of the next part every few microseconds, so
    // several rows' records are in flight together (640 parts of 486 to 827 keys, 152 query rows, whole call: 136.9 us with
    // one row at a time, which made the helper the slowest warp; 116.5 with four; one layer of 8192 keys 30.8 -> 28.9).
    for (int rb = r0; rb < p.Ralloc; rb += kRows * step) {
      float2 v[kRows][kRecs];
#pragma unroll
      for (int k = 0; k < kRows; ++k) {
        const int r = rb + k * step;
#pragma unroll
        for (int i = 0; i < kRecs; ++i)
          v[k][i] = i < nrec && r < p.R ? __ldcg(p.records + (size_t)(sg.part + c_lo + i) * p.Ralloc + r) : make_float2(-INFINITY, 0.f);
      }
#pragma unroll
      for (int k = 0; k < kRows; ++k) {
        const int r = rb + k * step;
        float M = v[k][0].x, L = 0.f;
#pragma unroll
        for (int i = 1; i < kRecs; ++i) M = fmaxf(M, v[k][i].x);
        if (M != -INFINITY) {
#pragma unroll
          for (int i = 0; i < kRecs; ++i) L += v[k][i].y * exp2f(v[k][i].x - M);
        }
        if (r < p.Ralloc) neg_lse[r] = (r < p.R && r / p.G < Weff) ? -(M + log2f(L)) : -INFINITY;
      }
    }
    return;
  }
  for (int r = r0; r < p.Ralloc; r += step) {
    const float2* rec = p.records + (size_t)(sg.part + c_lo) * p.Ralloc + r;
    float M = -INFINITY, L = 0.f;
    for (int i0 = 0; i0 < nrec; i0 += kFlight) {
      float2 v[kFlight];
#pragma unroll
      for (int i = 0; i < kFlight; ++i) v[i] = i0 + i < nrec ? __ldcg(rec + (size_t)(i0 + i) * p.Ralloc) : make_float2(-INFINITY, 0.f);
      float m = v[0].x;
#pragma unroll
      for (int i = 1; i < kFlight; ++i) m = fmaxf(m, v[i].x);
      if (m != -INFINITY) {                            // else nothing of row r is visible in these segments
        const float Mn = fmaxf(M, m);
        float acc = L * exp2f(M - Mn);
#pragma unroll
        for (int i = 0; i < kFlight; ++i) acc += v[i].y * exp2f(v[i].x - Mn);    // a (-inf, 0) pair adds 0
        M = Mn; L = acc;
      }
    }
    neg_lse[r] = (r < p.R && r / p.G < Weff) ? -(M + log2f(L)) : -INFINITY;
  }
}

// Pass 2, several row blocks per tile: a helper warp merges a later segment's records one segment ahead, hidden behind the
// segment before it if that is long enough.  Round trips to L2 per lane that takes, each about as long as a block of the epilogue:
__host__ __device__ __forceinline__ int helper_trips(int Ralloc, int nrec) {
  return nrec <= 4 ? Ralloc >> 7 : (Ralloc >> 5) * ((nrec + 23) / 24);
}
// A part over many CTAs behind a short segment is not hidden (two layers of one KV head, 1024 query rows, sequences of 30000, 10
// and 200 keys: 74 records of 1024 rows merged by one warp while a CTA's epilogue stood, 158 us; 82 with this rule, 107
// before the helpers merged at all): then the epilogue warps merge the records themselves.  `per16` = sixteenths of a key tile per
// CTA.
__device__ __forceinline__ bool epilogue_merges(const ScoreParams& p, int part_tiles, int per16, int blocks_before) {
  const int nrec = part_tiles * 16 / per16 + 1;
  return helper_trips(p.Ralloc, nrec) > blocks_before + 2 + (p.Ralloc + 32 * kEpiWarps - 1) / (32 * kEpiWarps) * ((nrec + 11) / 12);
}

// kVariant, pass 1: kTwice, for up to 64 query rows (below); pass 2: kOwn, the epilogue warps may merge later segments, too (plan_score
// says when).  Kernels of their own: the branches cost the hot loops of the others 0.5 to 3 %.
template <int D, int PASS, bool kVariant>
__global__ void __launch_bounds__(kThreads, 1)
score_kernel(const __grid_constant__ CUtensorMap tmap_q, const __grid_constant__ CUtensorMap tmap_k, const ScoreParams p) {
  constexpr bool kOwn = PASS == 2 && kVariant;
  // Up to 64 query rows leave half of the lanes of pass 1 with padding.  So the queries stand in rows 64 on once more, and the lanes of
  // either half take half of the columns: the same MMAs, half of the exponentials.  Scores of 64 rows against heads of 64, in a row: 32 layers
  // of 8192 tokens 138.8 -> 130.0 us, of 8 x 1500 63.8 -> 55.8, 13 of 8 x 640 52.3 -> 46.3, one of 32768 26.5 -> 24.7.
  constexpr bool kTwice = PASS == 1 && kVariant;
  constexpr int kSub = D / 64;                        // 64-element (128-byte) sub-tiles along d
  constexpr int kKSubBytes = kTileKeys * 128;         // one sub-tile of a K stage
  constexpr int kKStageBytes = kSub * kKSubBytes;
  extern __shared__ uint8_t smem_dyn[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_dyn) + 1023) & ~uintptr_t(1023));
  const int q_sub_bytes = p.Ralloc * 128;
  const int q_buf_bytes = kSub * q_sub_bytes;
  uint8_t* q_smem = smem;                                            // [q_bufs] Q operands
  uint8_t* k_smem = q_smem + p.q_bufs * q_buf_bytes;                  // [k_stages] K tiles
  uint64_t* bars = reinterpret_cast<uint64_t*>(k_smem + p.k_stages * kKStageBytes);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 38);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  int* const s_per16 = reinterpret_cast<int*>(bars + 39);            // sixteenths of a key tile per CTA (kOwn)
  float* table = reinterpret_cast<float*>(bars + 40);
  // pass 1: [2 buffers][kGroups]{m[Ralloc], l[Ralloc]} running statistics of a segment
  // pass 2: [2 buffers][Ralloc] negated log-sum-exps, [kColSlots][kGroups][128] partial column sums
  float* const stat = table;
  float* const neg_lse = table;
  float* const cols = table + 2 * p.Ralloc;
  int* s_cu = reinterpret_cast<int*>(table + (PASS == 1 ? 4 * kGroups * p.Ralloc : 2 * p.Ralloc + kColSlots * kGroups * 128));
  int* s_prefix = s_cu + p.B + 1;

  const uint32_t bar0 = smem_u32(bars);
  auto bar_qfull = [&](uint32_t s) { return bar0 + 8u * s; };
  auto bar_qempty = [&](uint32_t s) { return bar0 + 8u * (2 + s); };
  auto bar_kfull = [&](uint32_t s) { return bar0 + 8u * (4 + s); };
  auto bar_kempty = [&](uint32_t s) { return bar0 + 8u * (8 + s); };
  auto bar_afull = [&](uint32_t s) { return bar0 + 8u * (12 + s); };
  auto bar_aempty = [&](uint32_t s) { return bar0 + 8u * (16 + s); };
  // pass 1: statistics complete (epilogue -> helpers) / published; pass 2: log-sum-exps there (helper -> epilogue) / used
  auto bar_tab_full = [&](uint32_t s) { return bar0 + 8u * (20 + s); };
  auto bar_tab_free = [&](uint32_t s) { return bar0 + 8u * (22 + s); };
  auto bar_cols_full = [&](uint32_t s) { return bar0 + 8u * (24 + s); };   // epilogue -> helper: partial column sums of a tile complete
  auto bar_cols_free = [&](uint32_t s) { return bar0 + 8u * (28 + s); };
  const uint32_t bar_drain = bar0 + 8u * 32u;
  const uint32_t bar_own = bar0 + 8u * 33u;            // pass 2: the epilogue warps' own merge of a segment's log-sum-exps

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  unsigned long long clk0 = 0, gt0 = 0;
  if (p.clock_out && tid == 0) { clk0 = (unsigned long long)clock64(); gt0 = global_timer_ns(); }
  const int nblk = p.Ralloc >> 7;                      // row blocks
  if (warp == kTmaWarp && lane == 0) { tma_prefetch_map(&tmap_q); tma_prefetch_map(&tmap_k); }
  if (tid == 0) {
    SG_CHECK(reinterpret_cast<uint8_t*>(s_prefix + p.B + 1) <= smem_dyn + p.smem_bytes);     // carve-up fits the launch's shared memory
    SG_CHECK((smem_u32(q_smem) & 1023u) == 0 && (smem_u32(k_smem) & 1023u) == 0);            // swizzled operands on 1024-byte boundaries
    for (int s = 0; s < 2; ++s) {
      mbar_init(bar_qfull(s), 1); mbar_init(bar_qempty(s), 1);
      mbar_init(bar_tab_full(s), PASS == 1 ? kEpiWarps : nblk == 1 ? 2 : 1); mbar_init(bar_tab_free(s), PASS == 1 ? 2 : kEpiWarps);
    }
    for (int s = 0; s < kMaxKStages; ++s) { mbar_init(bar_kfull(s), 1); mbar_init(bar_kempty(s), 1); }
    for (int s = 0; s < kStages; ++s) { mbar_init(bar_afull(s), 1); mbar_init(bar_aempty(s), 4); }
    for (int s = 0; s < kColSlots; ++s) { mbar_init(bar_cols_full(s), 4 * min(nblk, kGroups)); mbar_init(bar_cols_free(s), 1); }
    mbar_init(bar_drain, 1);
    mbar_init(bar_own, kEpiWarps);
    *abort_flag = 0;
    fence_barrier_init();
    fence_proxy_async();
  }
  if (warp == kMmaWarp) {
    tmem_alloc(smem_u32(tmem_slot), 512);
    tmem_relinquish();
  }
  if (warp == 0) {
    if (PASS == 1 && p.B > 1) pdl_wait();              // (pass 2 is let go by pass 1 only behind its wait, below)
    // sequence offsets and the per-sequence tile prefix, once per CTA (one sequence: {0, T}, no load)
    int acc = 0;
    for (int b0 = 0; b0 <= p.B; b0 += 32) {
      const int b = b0 + lane;
      int nt = 0;
      if (p.B == 1) {
        if (b <= 1) s_cu[b] = b * (int)p.T;
        if (b == 0) nt = ((int)p.T + kTileKeys - 1) / kTileKeys;
      } else {
        if (b <= p.B) s_cu[b] = p.cu[b];
        if (b < p.B) nt = (p.cu[b + 1] - p.cu[b] + kTileKeys - 1) / kTileKeys;
      }
      int inc = nt;
#pragma unroll
      for (int off = 1; off < 32; off <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, inc, off);
        if (lane >= off) inc += v;
      }
      if (b < p.B) s_prefix[b + 1] = acc + inc;
      acc += __shfl_sync(0xffffffffu, inc, 31);
    }
    if (lane == 0) s_prefix[0] = 0;
    if (kOwn && lane == 0) *s_per16 = max(16, (int)((long long)p.units * acc * 16 / gridDim.x));
  }
  if (p.R < p.Ralloc) {
    // Rows R..Ralloc-1 of the Q operands are never written by TMA: zero them once so that padded MMA
    // rows/columns are finite.  (The 128-byte swizzle only permutes 16-byte chunks inside a row's own 128 bytes.)
    const int span = kTwice ? 64 : p.Ralloc, words = (span - p.R) * 32;
    for (int qb = 0; qb < p.q_bufs; ++qb)
      for (int dc = 0; dc < kSub; ++dc)
        for (int row = p.R; row < p.Ralloc; row += span) {
          uint32_t* z = reinterpret_cast<uint32_t*>(q_smem + qb * q_buf_bytes + dc * q_sub_bytes + row * 128);
          for (int i = tid; i < words; i += kThreads) z[i] = 0u;
        }
    fence_proxy_async();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  const int C = s_prefix[p.B];
  volatile int never = 0;
  // Pass 1 waits for whatever precedes the call (it may have written the queries, the keys, the sequence offsets) before it
  // lets pass 2 be set up: pass 2 loads queries, keys and offsets without a wait of its own, so everything ahead of the call
  // has to be complete and visible by then, also behind a kernel that starts its dependents early.  (Pass 2 does wait
  // for all of pass 1 before it reads or overwrites anything that a launch wrote.)
  if (PASS == 1) {
    pdl_wait();
    pdl_launch_dependents();
  }
  SegmentWalk<PASS> walk(C, p.units, p.B, s_cu, s_prefix);
  Segment sg;
  // In pass 2 loads and MMAs run ahead while the epilogue waits for pass 1: what their limits count starts behind pass 1.
  constexpr bool kBehind = PASS == 1;
  // A warp's wait: every lane sees the phase complete, or none goes on.
  auto wait = [&](uint32_t bar, uint32_t parity) {
    if (__all_sync(0xffffffffu, mbar_test(bar, parity))) return true;
    return __all_sync(0xffffffffu, mbar_wait_slow<kBehind>(bar, parity, abort_flag, p.wait_ns)) != 0;
  };
  long long w0 = 0, w1 = 0;                            // waiting clocks (profiling build)

  if (warp == kTmaWarp) {
    // ------------------------------------------------------------ TMA producer (one thread)
    if (lane == 0) {
      int nq = 0, nk = 0;                              // Q operands and K tiles requested so far
      bool ok = true;
      while (ok && walk.next(sg)) {
        const int l = sg.u / p.Hkv, g = sg.u - l * p.Hkv, qs = nq % p.q_bufs;
        ok = mbar_wait<kBehind>(bar_qempty(qs), (uint32_t)(((nq / p.q_bufs) & 1) ^ 1), abort_flag, p.wait_ns, 100u);
        if (!ok) break;
        ++nq;
        mbar_arrive_expect_tx(bar_qfull(qs), (uint32_t)((kTwice ? 2 : 1) * kSub * p.G * p.W * 128));
#pragma unroll
        for (int dc = 0; dc < kSub; ++dc)
          for (int at = 0; at <= (kTwice ? 64 : 0); at += 64)
            tma_load_4d(smem_u32(q_smem + qs * q_buf_bytes + dc * q_sub_bytes + at * 128), &tmap_q, bar_qfull(qs), dc * 64, g * p.G, 0, l * p.B + sg.b);
        const int tiles = sg.tile_end - sg.tile_beg;
        for (int i = 0; i < tiles; ++i) {
          const int tile = tile_at<PASS>(sg, i), ks = nk % p.k_stages;
          ok = mbar_wait<kBehind>(bar_kempty(ks), (uint32_t)(((nk / p.k_stages) & 1) ^ 1), abort_flag, p.wait_ns, 100u);
          if (!ok) break;
          ++nk;
          SG_CHECK(sg.c0 + tile * kTileKeys < p.T && g < p.Hkv && sg.b < p.B);
          mbar_arrive_expect_tx(bar_kfull(ks), (uint32_t)kKStageBytes);
#pragma unroll
          for (int dc = 0; dc < kSub; ++dc)
            tma_load_4d(smem_u32(k_smem + ks * kKStageBytes + dc * kKSubBytes), &tmap_k, bar_kfull(ks), dc * 64, g, sg.c0 + tile * kTileKeys, l);
        }
      }
      // No copy and no barrier arrival of this CTA may be pending when it exits: wait until the MMAs have released every
      // buffer, or, on an aborted run (nobody consumes what was requested), for the copies themselves.
      for (int i = 0; i < p.k_stages && ok; ++i)
        ok = mbar_wait<kBehind>(bar_kempty((nk + i) % p.k_stages), (uint32_t)((((nk + i) / p.k_stages) & 1) ^ 1), abort_flag, p.wait_ns, 100u);
      for (int i = 0; i < p.q_bufs && ok; ++i)
        ok = mbar_wait<kBehind>(bar_qempty((nq + i) % p.q_bufs), (uint32_t)((((nq + i) / p.q_bufs) & 1) ^ 1), abort_flag, p.wait_ns, 100u);
      if (!ok) {
        for (int n = max(0, nk - p.k_stages); n < nk; ++n)
          mbar_wait<kBehind>(bar_kfull(n % p.k_stages), (uint32_t)((n / p.k_stages) & 1), &never, p.wait_ns, 100u);
        for (int n = max(0, nq - p.q_bufs); n < nq; ++n)
          mbar_wait<kBehind>(bar_qfull(n % p.q_bufs), (uint32_t)((n / p.q_bufs) & 1), &never, p.wait_ns, 100u);
      }
    }
  } else if (warp == kMmaWarp) {
    // ------------------------------------------------------------ MMA issuer (converged warp, one elected lane issues)
    // The tensor pipe holds about two MMAs (~200 clocks) behind the last one issued, and a single warp retires an
    // instruction every 5-10 clocks: whatever stands between the last MMA of a block and the first of the next is time in
    // which the pipe runs dry.  Hence a converged warp (waits and address arithmetic stay warp-uniform), per-segment
    // constants, and every wait beyond its first attempt out of line: 730 clocks per block, 900 to 1400 with one thread
    // and inline waits (micro-benchmark with streamed key tiles).
    const bool leader = elect_one();
    uint32_t ks = 0, kph = 0, n = 0;
    int nq = 0;
    bool ok = true;
    const uint32_t k_lo0 = smem_desc_lo(smem_u32(k_smem)), k_stages = (uint32_t)p.k_stages, q_sub_lo = (uint32_t)q_sub_bytes >> 4;
    constexpr uint32_t k_stage_lo = (uint32_t)kKStageBytes >> 4, k_sub_lo = (uint32_t)kKSubBytes >> 4, q_blk_lo = (128u * 128u) >> 4;
    const uint32_t idesc = make_idesc(128, 128);
    while (ok && walk.next(sg)) {
      const int qs = nq % p.q_bufs;
      SG_PROF_WAIT(w0, ok = wait(bar_qfull(qs), (uint32_t)((nq / p.q_bufs) & 1)));
      if (!ok) break;
      ++nq;
      const uint32_t q_lo0 = smem_desc_lo(smem_u32(q_smem + qs * q_buf_bytes));
      for (int tile = sg.tile_beg; tile < sg.tile_end && ok; ++tile) {
        SG_PROF_WAIT(w0, ok = wait(bar_kfull(ks), kph));
        if (!ok) break;
        const uint32_t k_lo = k_lo0 + ks * k_stage_lo;
        uint32_t q_lo = q_lo0;
        for (int blk = 0; blk < nblk; ++blk, q_lo += q_blk_lo, ++n) {
          const uint32_t st = n & (kStages - 1);
          SG_PROF_WAIT(w1, ok = wait(bar_aempty(st), ((n / kStages) & 1u) ^ 1u));
          if (!ok) break;
          tc_fence_after();
          if (leader) {
            if (PASS == 1) umma_block<4 * kSub>(tmem_base + st * 128u, q_lo, k_lo, q_sub_lo, k_sub_lo, idesc);
            else umma_block<4 * kSub>(tmem_base + st * 128u, k_lo, q_lo, k_sub_lo, q_sub_lo, idesc);
            umma_commit(bar_afull(st));
            if (blk == nblk - 1) umma_commit(bar_kempty(ks));
          }
          __syncwarp();
        }
        if (++ks == k_stages) { ks = 0; kph ^= 1u; }
      }
      if (ok && leader) umma_commit(bar_qempty(qs));
      __syncwarp();
    }
    // Every MMA this warp issued has completed before the CTA frees its tensor memory, also on an aborted run
    // (the commit arrives when all earlier MMAs are done; the wait ignores the abort flag and is bounded).
    if (leader) {
      umma_commit(bar_drain);
      mbar_wait<kBehind>(bar_drain, 0u, &never, p.wait_ns, 0u);
    }
    __syncwarp();
    SG_PROF_STORE(4, w0); SG_PROF_STORE(5, w1);
  } else if (warp < kEpiWarps) {
    // ------------------------------------------------------------ epilogue warps
    // Block n of the CTA's running count is in stage n mod 4 and belongs to warpgroup n mod 3; one stage more than there are
    // warpgroups, so the MMAs of a warpgroup's next block need not wait for its current one.
    const int wg = warp >> 2, quarter = warp & 3;
    const int row_in_tile = quarter * 32 + lane;       // this thread's TMEM lane: its row of the block (pass 1), its key (pass 2)
    const uint32_t t_lane = tmem_base + ((uint32_t)(quarter * 32) << 16);
    const uint64_t scale2 = pack2(p.scale_log2, p.scale_log2);
    uint32_t n0 = 0;                                   // blocks of the CTA before this segment
    int tiles0 = 0;                                    // tiles of the CTA before this segment
    int blocks_before = 0;                             // blocks of the segment before this one
    uint32_t merges = 0;                               // pass 2: parities of the helper's merges (bit per buffer) and of these warps' (bit 2)
    bool ok = true;
    auto release = [&](uint32_t st) {
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(bar_aempty(st));
    };
    for (int sidx = 0; ok && walk.next(sg); ++sidx) {
      const int Weff = min(p.W, sg.N), first_win = sg.N - Weff;      // position of window row 0; keys <= it are visible to all rows
      const int vis_end = (first_win + 1) / kTileKeys;               // tiles [0, vis_end) are visible to every window row
      const uint32_t buf = (uint32_t)sidx & 1u, use = (uint32_t)sidx >> 1;
      const uint32_t n_end = n0 + (uint32_t)((sg.tile_end - sg.tile_beg) * nblk);
      uint32_t n = n0 + (kGroups + (uint32_t)wg - n0 % kGroups) % kGroups;     // this warpgroup's first block of the segment
      int ti = 0, blk = (int)(n - n0);                                // its tile, counted in the segment, and its row block
      while (blk >= nblk) { blk -= nblk; ++ti; }
      if (PASS == 1) {
        // The buffer's previous segment has been merged and published by the helpers (practically always true already).
        // Slot (wg, row) is only ever touched by this thread during the segment, so the statistics need no barrier.
        if (use > 0) ok = wait(bar_tab_free(buf), (use - 1u) & 1u);
        if (!ok) break;
        float* const sm_m = stat + (size_t)(buf * kGroups + wg) * 2 * p.Ralloc + row_in_tile;
        float* const sm_l = sm_m + p.Ralloc;
        for (int i = 0; i < nblk; ++i) { sm_m[i * 128] = -INFINITY; sm_l[i * 128] = 0.f; }
        const bool all_rows = Weff == p.W;
        for (; n < n_end; n += kGroups) {
          const uint32_t st = n & (kStages - 1), col0 = kTwice && quarter >= 2 ? 64u : 0u, t_acc = t_lane + st * 128u + col0;
          SG_PROF_WAIT(w0, ok = wait(bar_afull(st), (n / kStages) & 1u));
          if (!ok) break;
          tc_fence_after();
          float m = sm_m[blk * 128], l = sm_l[blk * 128];
          // The running reference m need not be the row maximum: fp32 keeps its relative precision for any exponent, so
          // the sum of exp2(x - m) is as accurate with a stale (lower) m as with the true maximum, as long as nothing
          // overflows.  A segment starts from the maximum of the block's first 32 columns; a block whose sum leaves the safe
          // range (a value far above m) and a block with hidden scores are done carefully: true maximum first.
          const int tile = tile_at<PASS>(sg, ti);
          bool careful = tile >= vis_end || !all_rows;
          if (!careful) {
            uint32_t a[32], b[32];
            tmem_ld32_issue(a, t_acc);
            tmem_ld_wait(a);
            tmem_ld32_issue(b, t_acc + 32u);
            if (m == -INFINITY) {                      // (a row block's rows start together)
              float x = fmaxf(__uint_as_float(a[0]), __uint_as_float(a[1]));
#pragma unroll
              for (int c = 2; c < 32; c += 2) x = max3(x, __uint_as_float(a[c]), __uint_as_float(a[c + 1]));
              m = x * p.scale_log2;
            }
            const uint64_t nm2 = pack2(-m, -m);
            uint64_t s0 = 0ull, s1 = 0ull;
            chunk_rows(a, scale2, nm2, s0, s1);
            tmem_ld_wait(b);
            if (!kTwice) {
              tmem_ld32_issue(a, t_acc + 64u);
              chunk_rows(b, scale2, nm2, s0, s1);
              tmem_ld_wait(a);
              tmem_ld32_issue(b, t_acc + 96u);
              chunk_rows(a, scale2, nm2, s0, s1);
              tmem_ld_wait(b);
            }
            chunk_rows(b, scale2, nm2, s0, s1);
            float lo, hi;
            unpack2(add2(s0, s1), lo, hi);
            const float s = lo + hi;
            careful = !__all_sync(0xffffffffu, s < 0x1p60f);
            if (!careful) l += s;
          }
          if (careful) {
            const int r = kTwice ? row_in_tile & 63 : blk * 128 + row_in_tile, chunks = kTwice ? 2 : 4;
            // last visible column of this tile, counted from the first one that the thread takes
            const int cmax = r < p.R && r / p.G < Weff ? first_win + r / p.G - tile * kTileKeys - (int)col0 : -1;
            float mx = -INFINITY;
            uint32_t cur[32];
#pragma unroll 1
            for (int j = 0; j < chunks; ++j) {
              tmem_ld32_issue(cur, t_acc + (uint32_t)(j * 32));
              tmem_ld_wait(cur);
#pragma unroll
              for (int c = 0; c < 32; ++c)
                if (j * 32 + c <= cmax) mx = fmaxf(mx, __uint_as_float(cur[c]));
            }
            const float mn = fmaxf(m, mx * p.scale_log2);
            if (mn != -INFINITY) { l *= exp2f(m - mn); m = mn; }
            const float ref = mn == -INFINITY ? 0.f : mn;
#pragma unroll 1
            for (int j = 0; j < chunks; ++j) {
              tmem_ld32_issue(cur, t_acc + (uint32_t)(j * 32));
              tmem_ld_wait(cur);
              float s0 = 0.f, s1 = 0.f;
#pragma unroll
              for (int c = 0; c < 32; c += 2) {
                s0 += j * 32 + c <= cmax ? exp2f(fmaf(__uint_as_float(cur[c]), p.scale_log2, -ref)) : 0.f;
                s1 += j * 32 + c + 1 <= cmax ? exp2f(fmaf(__uint_as_float(cur[c + 1]), p.scale_log2, -ref)) : 0.f;
              }
              l += s0 + s1;
            }
          }
          release(st);
          sm_m[blk * 128] = m;
          sm_l[blk * 128] = l;
          blk += kGroups;
          while (blk >= nblk) { blk -= nblk; ++ti; }
        }
        // This warp's statistics of the segment are complete; the helpers merge the warpgroups' slots and publish them.
        __syncwarp();
        if (lane == 0 && ok && sg.u != p.withhold_unit) mbar_arrive(bar_tab_full(buf));
      } else {
        if (sidx == 0 || (kOwn && epilogue_merges(p, s_prefix[sg.b + 1] - s_prefix[sg.b], *s_per16, blocks_before))) {
          // The first segment's log-sum-exps, and those of a part that the helper would be late with, are what the whole
          // CTA waits for: all epilogue threads merge its records.
          if (sidx == 0) pdl_wait();
          else if (kOwn && use > 0) ok = wait(bar_tab_free(buf), (use - 1u) & 1u);
          if (!ok) break;
          merge_records<12, 1>(p, sg, s_prefix, C, kOwn ? neg_lse + buf * p.Ralloc : neg_lse, tid, 32 * kEpiWarps);
          __syncwarp();
          if (lane == 0) mbar_arrive(bar_own);
          ok = wait(bar_own, kOwn ? merges >> 2 : 0u);
          merges ^= 4u;
        } else {
          // A helper has merged the part's records one segment ahead.  Every warp waits here, also one that gets no block of
          // the segment: that keeps the arrivals below in step with the barrier's phases.
          const uint32_t phase = kOwn ? (merges >> buf) & 1u : buf == 0u ? (use - 1u) & 1u : use & 1u;
          SG_PROF_WAIT(w1, ok = wait(bar_tab_full(buf), phase));
          merges ^= 1u << buf;
        }
        if (!ok) break;
        const float* nl = neg_lse + buf * p.Ralloc;
        const int G = p.G;
        uint64_t s0 = 0ull, s1 = 0ull;
        while (n < n_end) {
          const uint32_t st = n & (kStages - 1), t_acc = t_lane + st * 128u;
          SG_PROF_WAIT(w0, ok = wait(bar_afull(st), (n / kStages) & 1u));
          if (!ok) break;
          tc_fence_after();
          const int tile = tile_at<PASS>(sg, ti), t = tile * kTileKeys + row_in_tile;      // t: this thread's key
          const float* ls = nl + blk * 128;
          if (tile < vis_end && (blk + 1) * 128 <= p.R) {
            uint32_t a[32], b[32];
            tmem_ld32_issue(a, t_acc);
            tmem_ld_wait(a);
            tmem_ld32_issue(b, t_acc + 32u);
            chunk_cols(a, scale2, ls, s0, s1);
            tmem_ld_wait(b);
            tmem_ld32_issue(a, t_acc + 64u);
            chunk_cols(b, scale2, ls + 32, s0, s1);
            tmem_ld_wait(a);
            tmem_ld32_issue(b, t_acc + 96u);
            chunk_cols(a, scale2, ls + 64, s0, s1);
            tmem_ld_wait(b);
            release(st);
            chunk_cols(b, scale2, ls + 96, s0, s1);
          } else {
            const int nchk = (min(128, p.R - blk * 128) + 31) >> 5;       // 32-row chunks (rows past R have log-sum-exp +inf)
            const int rmin = (t - first_win) * G;                          // rows below rmin cannot see key t
            uint32_t cur[32];
#pragma unroll 1
            for (int j = 0; j < nchk; ++j) {
              tmem_ld32_issue(cur, t_acc + (uint32_t)(j * 32));
              tmem_ld_wait(cur);
              if (j == nchk - 1) release(st);
              const int c_lo = rmin - blk * 128 - j * 32;
#pragma unroll
              for (int c = 0; c < 32; ++c) cur[c] = c >= c_lo ? cur[c] : 0xff800000u;
              chunk_cols(cur, scale2, ls + j * 32, s0, s1);
            }
          }
          const int ti_now = ti;
          n += kGroups;
          blk += kGroups;
          while (blk >= nblk) { blk -= nblk; ++ti; }
          if (ti == ti_now && n < n_end) continue;                     // more of this tile's row blocks are this warpgroup's
          float lo, hi;
          unpack2(add2(s0, s1), lo, hi);
          s0 = s1 = 0ull;
          if (nblk == 1) {
            if (t < sg.N) p.importance[(size_t)sg.u * p.T + sg.c0 + t] = lo + hi;
          } else {
            // The tile's row blocks went to different warpgroups: leave the partial column sums for the helper.
            const uint32_t ts = (uint32_t)(tiles0 + ti_now), cs = ts % kColSlots, cu = ts / kColSlots;
            if (cu > 0) ok = wait(bar_cols_free(cs), (cu - 1u) & 1u);
            if (!ok) break;
            cols[(cs * kGroups + wg) * 128 + row_in_tile] = lo + hi;
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_cols_full(cs));
          }
        }
        __syncwarp();
        if (lane == 0 && ok) mbar_arrive(bar_tab_free(buf));
      }
      blocks_before = (int)(n_end - n0);
      n0 = n_end;
      tiles0 += sg.tile_end - sg.tile_beg;
    }
    if (quarter == 0) { SG_PROF_STORE(8 + 2 * wg, w0); SG_PROF_STORE(9 + 2 * wg, w1); SG_PROF_STORE(20, n0); }
  } else {
    // ------------------------------------------------------------ helper warps
    const int hw = warp - kHelperWarp;
    // Everything below touches what the launch before this one wrote or reads: wait until that has completed.
    pdl_wait();
    bool ok = true;
    if (PASS == 1) {
      // merge the warpgroups' statistics of a finished segment and publish its record (half of the rows each)
      for (int sidx = 0; ok && walk.next(sg); ++sidx) {
        const uint32_t buf = (uint32_t)sidx & 1u, use = (uint32_t)sidx >> 1;
        ok = wait(bar_tab_full(buf), use & 1u);
        if (!ok) break;
        const float* sm = stat + (size_t)buf * kGroups * 2 * p.Ralloc;
        float2* rec = p.records + (size_t)(sg.part + (int)blockIdx.x) * p.Ralloc;
        for (int r = hw * 32 + lane; r < (kTwice ? 64 : p.Ralloc); r += 64) {
          float m[2 * kGroups], M = -INFINITY, L = 0.f;
#pragma unroll
          for (int w = 0; w < 2 * kGroups; ++w) {      // (the second half only where the rows stand twice)
            m[w] = w < kGroups || kTwice ? sm[w % kGroups * 2 * p.Ralloc + r + w / kGroups * 64] : -INFINITY;
            M = fmaxf(M, m[w]);
          }
          const float Mu = M == -INFINITY ? 0.f : M;
#pragma unroll
          for (int w = 0; w < 2 * kGroups; ++w)
            if (w < kGroups || kTwice) L += sm[(w % kGroups * 2 + 1) * p.Ralloc + r + w / kGroups * 64] * exp2f(m[w] - Mu);
          rec[r] = make_float2(M, L);
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(bar_tab_free(buf));
      }
    } else if (hw == 0 || nblk == 1) {
      // Merge the records of every segment but the first, one segment ahead of the epilogue.  Both helpers, half of the rows
      // each, when there are no column sums to add up; 24 records in flight: the CTAs at the part boundaries of a one-layer
      // call have a segment or two of a tile each, and parts of twenty records (8192 keys:
      // 28.8 -> 26.6 us for the whole call; one helper, 16 in flight, took eight L2 round trips per segment).
      int blocks_before = 0;
      for (int sidx = 0; ok && walk.next(sg); ++sidx) {
        const int blocks = (sg.tile_end - sg.tile_beg) * nblk, before = blocks_before;
        blocks_before = blocks;
        if (sidx == 0) continue;
        const uint32_t buf = (uint32_t)sidx & 1u, use = (uint32_t)sidx >> 1;
        if (use > 0) ok = wait(bar_tab_free(buf), (use - 1u) & 1u);        // (in every segment: the barrier's phases alternate)
        if (!ok) break;
        if (kOwn && epilogue_merges(p, s_prefix[sg.b + 1] - s_prefix[sg.b], *s_per16, before)) continue;
        merge_records<24, 4>(p, sg, s_prefix, C, neg_lse + buf * p.Ralloc, nblk == 1 ? hw * 32 + lane : lane, nblk == 1 ? 64 : 32);
        __syncwarp();
        if (lane == 0) mbar_arrive(bar_tab_full(buf));
      }
    } else if (nblk > 1) {
      // add up the warpgroups' column sums of a tile, in the order of its row blocks (bitwise reproducible)
      uint32_t n = 0, ts = 0;
      const int nwg = min(nblk, kGroups);
      while (ok && walk.next(sg)) {
        const int tiles = sg.tile_end - sg.tile_beg;
        for (int i = 0; i < tiles; ++i, ++ts, n += (uint32_t)nblk) {
          const int tile = tile_at<PASS>(sg, i);
          const uint32_t cs = ts % kColSlots;
          ok = wait(bar_cols_full(cs), (ts / kColSlots) & 1u);
          if (!ok) break;
          const float* c = cols + cs * kGroups * 128;
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const int t = tile * kTileKeys + q * 32 + lane;
            float s = 0.f;
            for (int w = 0; w < nwg; ++w) s += c[(n + w) % kGroups * 128 + q * 32 + lane];
            if (t < sg.N) p.importance[(size_t)sg.u * p.T + sg.c0 + t] = s;
          }
          __syncwarp();
          if (lane == 0) mbar_arrive(bar_cols_free(cs));
        }
      }
    }
  }
  // ---------------------------------------------------------------- teardown
  // This CTA has no work left: a kernel queued behind this one with programmatic stream serialization (the selection) may
  // have its CTAs placed from now on; it still waits for this whole grid's completion before it reads anything.
  pdl_launch_dependents();
  tc_fence_before();
  __syncthreads();
  if (warp == kMmaWarp) {
    tc_fence_after();
    tmem_dealloc(tmem_base, 512);
  }
  if (tid == 0 && *abort_flag) raise(p.dev_status, SG_ERR_TIMEOUT);
  if (p.clock_out && tid == 0) {
    unsigned long long* o = p.clock_out + kClockWords * (size_t)blockIdx.x;
    o[0] = clk0; o[1] = (unsigned long long)clock64(); o[2] = gt0; o[3] = global_timer_ns();
  }
}

// ---------------------------------------------------------------- host side
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                  const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_tiled_fn() {
  static EncodeTiledFn fn = []() -> EncodeTiledFn {
    void* ptr = nullptr;
    cudaDriverEntryPointQueryResult qres;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &ptr, cudaEnableDefault, &qres) != cudaSuccess) return nullptr;
    if (qres != cudaDriverEntryPointSuccess) return nullptr;
    return reinterpret_cast<EncodeTiledFn>(ptr);
  }();
  return fn;
}

// Testing hooks (sg_testing_score_fault, sg_testing_score_clock): process-wide, off by default.
std::atomic<int> g_test_withhold_unit{-1};
std::atomic<int> g_test_wait_limit_ms{0};
std::atomic<unsigned long long*> g_test_clock_out{nullptr};

struct ScorePlan {
  int R, Ralloc, k_stages, q_bufs, smem_bytes, U, grid;
  bool own;                // pass 2 with kOwn
  size_t workspace_bytes;
  bool ok;
};

// `limit`: the most workspace there is (0 = whatever the plan needs).  Fewer CTAs need fewer records, but a call is not squeezed
// onto fewer than kFewestCtas.
constexpr int kFewestCtas = 32;
ScorePlan plan_score(const sg_shape* s, size_t limit = 0) {
  ScorePlan pl{};
  const int D = s->head_dim;
  const int G = s->num_q_heads / s->num_kv_heads;
  pl.R = G * s->window;
  pl.Ralloc = (pl.R + 127) & ~127;
  const int q_bytes = pl.Ralloc * D * 2;
  const int k_stage = kTileKeys * D * 2;
  const int table1 = 4 * kGroups * pl.Ralloc * 4, table2 = 2 * pl.Ralloc * 4 + kColSlots * kGroups * 128 * 4;
  const int tail = (40 * 8 + (table1 > table2 ? table1 : table2) + 2 * (s->batch + 1) * 4 + 15) & ~15;
  const int avail = kSmemLimit - 1024 - tail;
  // Two Q buffers let the next segment's queries load while the current one computes; fall back to one
  // when that would leave fewer than three K stages.
  pl.q_bufs = 2;
  pl.k_stages = (avail - 2 * q_bytes) / k_stage;
  if (pl.k_stages < 3) { pl.q_bufs = 1; pl.k_stages = (avail - q_bytes) / k_stage; }
  if (pl.k_stages > kMaxKStages) pl.k_stages = kMaxKStages;
  pl.ok = pl.k_stages >= 2 && s->window <= 256 && pl.R <= 1024 && s->batch <= kMaxBatchSmem;
  pl.smem_bytes = 1024 + pl.q_bufs * q_bytes + pl.k_stages * k_stage + tail;
  if (pl.smem_bytes < 120 * 1024) pl.smem_bytes = 120 * 1024;     // one CTA per SM: each CTA takes the whole TMEM
  pl.U = s->num_layers * s->num_kv_heads;
  const int64_t tiles = (int64_t)pl.U * ((int64_t)s->total_tokens / kTileKeys + s->batch);      // upper bound
  pl.grid = (int)(tiles < kNumSMs ? tiles : kNumSMs);
  // records: a CTA adds at most one segment to the parts
  const int64_t record = (int64_t)pl.Ralloc * sizeof(float2), parts = (int64_t)pl.U * s->batch;
  if (limit > 0) {
    const int64_t most = (int64_t)limit / record - parts;
    if (most >= kFewestCtas && most < pl.grid) pl.grid = (int)most;
  }
  pl.workspace_bytes = (size_t)((parts + pl.grid) * record);
  // The code for the epilogue's own merges costs the hot loop 1 to 3 % (registers), so it is there only where CTAs have more than a
  // tile and the helper's merge of the longest part would take clearly longer than all blocks of a CTA.  (Of 330 random shapes of 129
  // to 1024 rows 14 get 3 to 49 % faster, the others run as before; without the 8 trips more of them gained up to 20 %, but
  // some thirty with a tile or two per CTA lost 1 to 5 %.)
  const int64_t per16 = pl.grid > 0 ? tiles * 16 / pl.grid : 0;
  const int64_t nrec = per16 > 16 ? ((int64_t)s->max_seqlen / kTileKeys + 1) * 16 / per16 + 1 : 0;
  pl.own = pl.Ralloc > 128 && nrec > 0 && helper_trips(pl.Ralloc, (int)nrec) * 16 > per16 * (pl.Ralloc >> 7) + 8 * 16;
  return pl;
}

template <int D, int PASS, bool kVariant>
sg_status launch_pass(const CUtensorMap& q, const CUtensorMap& k, const ScoreParams& p, const ScorePlan& pl, cudaStream_t s) {
  SG_ENSURE_SMEM((score_kernel<D, PASS, kVariant>), pl.smem_bytes);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)pl.grid);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = (size_t)pl.smem_bytes;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  SG_CUDA_TRY(cudaLaunchKernelEx(&cfg, score_kernel<D, PASS, kVariant>, q, k, p));
  return SG_OK;
}

}  // namespace

size_t score_workspace_bytes(const sg_shape* s) {
  if (s->num_kv_heads < 1 || s->num_q_heads < 1 || s->window < 1 || s->num_layers < 1) return 0;
  if (s->num_q_heads % s->num_kv_heads != 0) return 0;
  return plan_score(s).workspace_bytes;
}

}  // namespace sg

extern "C" void sg_testing_score_fault(int32_t withhold_unit, int32_t wait_limit_ms) {
  sg::g_test_withhold_unit.store(withhold_unit, std::memory_order_relaxed);
  sg::g_test_wait_limit_ms.store(wait_limit_ms, std::memory_order_relaxed);
}

extern "C" void sg_testing_score_clock(void* dev_buffer) {
  sg::g_test_clock_out.store(static_cast<unsigned long long*>(dev_buffer), std::memory_order_relaxed);
}

extern "C" int32_t sg_testing_score_grid(const sg_shape* shape) {
  using namespace sg;
  if (check_shape(shape, true) != SG_OK) return 0;
  const ScorePlan pl = plan_score(shape);
  return pl.ok ? pl.grid : 0;
}

extern "C" int32_t sg_testing_score_cluster(const sg_shape* shape) {
  using namespace sg;
  if (check_shape(shape, true) != SG_OK) return 0;
  return plan_score(shape).ok ? score_cluster_size(shape, true) : 0;
}

namespace sg {
namespace {

// `limit`: as in plan_score, and the two passes whatever the shape.  `pack`: only where one kernel does it all, else SG_ERR_UNSUPPORTED
// with nothing launched.
sg_status run_score(const sg_shape* shape, const void* q_win, const void* k_cache, float* importance, void* workspace,
                    size_t workspace_bytes, size_t limit, const PackLaunch* pack, int32_t* dev_status, void* stream) {
  sg_status st = check_shape(shape, true);
  if (st != SG_OK) return st;
  if (shape->total_tokens == 0) return SG_OK;
  if (!q_win || !k_cache || !importance) return SG_ERR_INVALID;
  if (!aligned16(q_win) || !aligned16(k_cache) || !aligned16(importance) || !aligned16(workspace)) return SG_ERR_INVALID;
  const ScorePlan pl = plan_score(shape, limit);
  if (!pl.ok) return SG_ERR_UNSUPPORTED;
  if (!workspace || workspace_bytes < pl.workspace_bytes) return SG_ERR_WORKSPACE;
  unsigned long long* const clock_out = g_test_clock_out.load(std::memory_order_relaxed);
  const bool cluster = limit == 0 && !clock_out && score_cluster_size(shape, pack != nullptr) > 0;
  if (pack && !cluster) return SG_ERR_UNSUPPORTED;
  EncodeTiledFn encode = encode_tiled_fn();
  if (!encode) return cuda_fail((int)cudaErrorUnknown);

  const int D = shape->head_dim;
  const int G = shape->num_q_heads / shape->num_kv_heads;
  CUtensorMap tmap_q, tmap_k;
  {
    // q_win [L*B][W][H_q][d]; box = (64 of d, G heads, W rows, 1) -> rows ordered (window row, head in group)
    const cuuint64_t dims[4] = {(cuuint64_t)D, (cuuint64_t)shape->num_q_heads, (cuuint64_t)shape->window,
                                (cuuint64_t)shape->num_layers * shape->batch};
    const cuuint64_t strides[3] = {(cuuint64_t)D * 2, (cuuint64_t)shape->num_q_heads * D * 2,
                                   (cuuint64_t)shape->window * shape->num_q_heads * D * 2};
    const cuuint32_t box[4] = {64, (cuuint32_t)G, (cuuint32_t)shape->window, 1};
    const cuuint32_t estr[4] = {1, 1, 1, 1};
    const CUresult r = encode(&tmap_q, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(q_win), dims, strides, box, estr,
                              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return cuda_fail((int)r);
  }
  {
    // k_cache viewed as (d, H_kv, T, L) with the caller's strides; box = 64 of d x 1 head x 128 tokens
    const cuuint64_t dims[4] = {(cuuint64_t)D, (cuuint64_t)shape->num_kv_heads, (cuuint64_t)shape->total_tokens,
                                (cuuint64_t)shape->num_layers};
    const cuuint64_t hs = shape->num_kv_heads > 1 ? (cuuint64_t)shape->cache_head_stride * 2 : (cuuint64_t)D * 2;
    const cuuint64_t ls = shape->num_layers > 1 ? (cuuint64_t)shape->cache_layer_stride * 2
                                                : (cuuint64_t)shape->cache_token_stride * 2 * shape->total_tokens;
    const cuuint64_t strides[3] = {hs, (cuuint64_t)shape->cache_token_stride * 2, ls};
    const cuuint32_t box[4] = {64, 1, (cuuint32_t)kTileKeys, 1};
    const cuuint32_t estr[4] = {1, 1, 1, 1};
    const CUresult r = encode(&tmap_k, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(k_cache), dims, strides, box, estr,
                              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return cuda_fail((int)r);
  }

  ScoreParams p;
  p.cu = shape->cu_seqlens;
  p.importance = importance;
  p.dev_status = dev_status;
  p.T = shape->total_tokens;
  p.B = shape->batch;
  p.Hkv = shape->num_kv_heads;
  p.G = G;
  p.W = shape->window;
  p.R = pl.R;
  p.Ralloc = pl.Ralloc;
  p.k_stages = pl.k_stages;
  p.q_bufs = pl.q_bufs;
  p.smem_bytes = pl.smem_bytes;
  p.withhold_unit = g_test_withhold_unit.load(std::memory_order_relaxed);
  const int limit_ms = g_test_wait_limit_ms.load(std::memory_order_relaxed);
  p.wait_ns = limit_ms > 0 ? (uint32_t)limit_ms * 1000000u : 1000000000u;
  p.clock_out = clock_out;
  p.scale_log2 = kLog2e / sqrtf((float)D);

  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if (cluster) return score_cluster_launch(shape, tmap_q, tmap_k, ScoreLaunch{importance, dev_status, p.withhold_unit, p.wait_ns, s}, pack);
  p.units = pl.U;
  p.records = static_cast<float2*>(workspace);
  if (p.R <= 64) st = D == 128 ? launch_pass<128, 1, true>(tmap_q, tmap_k, p, pl, s) : launch_pass<64, 1, true>(tmap_q, tmap_k, p, pl, s);
  else st = D == 128 ? launch_pass<128, 1, false>(tmap_q, tmap_k, p, pl, s) : launch_pass<64, 1, false>(tmap_q, tmap_k, p, pl, s);
  if (st != SG_OK) return st;
  if (pl.own) return D == 128 ? launch_pass<128, 2, true>(tmap_q, tmap_k, p, pl, s) : launch_pass<64, 2, true>(tmap_q, tmap_k, p, pl, s);
  return D == 128 ? launch_pass<128, 2, false>(tmap_q, tmap_k, p, pl, s) : launch_pass<64, 2, false>(tmap_q, tmap_k, p, pl, s);
}

}  // namespace
}  // namespace sg

extern "C" sg_status sg_score(const sg_shape* shape, const void* q_win, const void* k_cache, float* importance,
                              void* workspace, size_t workspace_bytes, int32_t* dev_status, void* stream) {
  return sg::run_score(shape, q_win, k_cache, importance, workspace, workspace_bytes, 0, nullptr, dev_status, stream);
}

extern "C" sg_status sg_internal_score_select_pack(const sg_shape* shape, const void* q_win, const void* k_cache, const void* v_cache,
                                                   float* importance, void* workspace, size_t workspace_bytes, const int32_t* cu_k,
                                                   int32_t total_sel, int32_t* sel_idx, void* packed_k, void* packed_v,
                                                   int32_t* dev_status, void* stream) {
  using namespace sg;
  if (total_sel <= 0 || !cu_k || !v_cache || !sel_idx || !packed_k || !packed_v) return SG_ERR_UNSUPPORTED;
  if (!aligned16(cu_k) || !aligned16(v_cache) || !aligned16(sel_idx) || !aligned16(packed_k) || !aligned16(packed_v)) return SG_ERR_UNSUPPORTED;
  const PackLaunch pack{cu_k, total_sel, k_cache, v_cache, sel_idx, packed_k, packed_v};
  const sg_status st = run_score(shape, q_win, k_cache, importance, workspace, workspace_bytes, 0, &pack, dev_status, stream);
  return st == SG_ERR_CUDA || (st == SG_OK && shape->total_tokens > 0) ? st : SG_ERR_UNSUPPORTED;
}


// ---------------------------------------------------------------------------------------------
// sg_score_static: sg_score for callers that cannot allocate device memory.
//
// The row statistics that pass 1 hands to pass 2 normally live in a caller-provided workspace.
// Here they live in a fixed array that is part of the library image, so the caller needs no
// allocator at all.  The array is shared by every call on a device and keeps the previous call's
// contents; every word of it is written by pass 1 before pass 2 reads it.
namespace sg {
namespace {
static __device__ __align__(256) unsigned char g_score_static_scratch[SG_SCORE_STATIC_SCRATCH_BYTES];
}  // namespace
}  // namespace sg

extern "C" sg_status sg_score_static(const sg_shape* shape, const void* q_win, const void* k_cache,
                                     float* importance, int32_t* dev_status, void* stream) {
  using namespace sg;
  sg_status st = check_shape(shape, true);
  if (st != SG_OK) return st;
  if (shape->total_tokens == 0) return SG_OK;
  if (!plan_score(shape).ok) return SG_ERR_UNSUPPORTED;      // same answer as sg_score for shapes no kernel covers
  if (plan_score(shape, SG_SCORE_STATIC_SCRATCH_BYTES).workspace_bytes > (size_t)SG_SCORE_STATIC_SCRATCH_BYTES) return SG_ERR_WORKSPACE;
  // In host code the array's name is only a handle; the device address has to be asked for, once per
  // device, with that device current.
  static std::atomic<void*> scratch_of_device[64];
  int dev = 0;
  SG_CUDA_TRY(cudaGetDevice(&dev));
  void* scratch = (dev >= 0 && dev < 64) ? scratch_of_device[dev].load(std::memory_order_acquire) : nullptr;
  if (!scratch) {
    SG_CUDA_TRY(cudaGetSymbolAddress(&scratch, g_score_static_scratch));
    if (dev >= 0 && dev < 64) scratch_of_device[dev].store(scratch, std::memory_order_release);
  }
  return run_score(shape, q_win, k_cache, importance, scratch, (size_t)SG_SCORE_STATIC_SCRATCH_BYTES, (size_t)SG_SCORE_STATIC_SCRATCH_BYTES,
                   nullptr, dev_status, stream);
}
