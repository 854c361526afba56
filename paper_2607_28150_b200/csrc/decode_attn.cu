// sg_sparse_decode_attn: split-KV decode attention over a packed source plus an index-gathered source.
//
// Every attended token costs 2*d*2 bytes of K+V per KV head and only 4*G*d flops: large batches are bound by HBM, small
// ones by the chain of launch, first loads, a slice or two per warp, and merge.  In between a warp's instructions are what
// takes the time: they issue one by one, four to five clocks each, with few warps per scheduler.
// The token list of a (sequence, KV head) -- packed rows first, then local rows addressed through
// local_idx -- is cut into slices of 16 tokens.  The slices are dealt out round robin over all warps of all
// CTAs that share a (sequence, KV head), so every CTA gets the same mix of packed and gathered slices; a warp
// streams its slices through a ring of its own in shared memory, half a slice (16 rows of K, or of V) per slot
// (16-byte cp.async copies, XOR-swizzled rows so ldmatrix is conflict-free; gathered rows are whole 2*d-byte lines, so
// sector efficiency stays 100 %).  The ring is private to the warp, so the loop has no block-wide barrier: a warp waits
// only for its own copies.
// S^T = K Q^T and O^T += V^T P^T run on bf16 tensor-core MMAs with the tokens (or the head dimension) on the 16-row side and
// the G query rows of the KV head on the 8-column side: no row is padding at G = 8, half are at G = 4, and the accumulator
// takes d/4 registers.  (With the queries on the 16-row side: twice the MMAs and accumulators, 420 instructions per slice
// instead of 200, and so many registers and so deep a ring that an SM held one CTA of eight warps; it holds two now, and
// consecutive calls overlap on it.  32 layers of 819 entries: 48.5 -> 39.7 us, 4 layers of 32 x 820 entries 78.7 -> 73.4,
// one layer of 128 x 4096 entries 342 -> 305 us, 7.1 TB/s.)
// The online softmax (base 2) stays in registers.
// The split-KV partials (m, l, unnormalised O) never leave the chip: the warps of a CTA merge through
// shared memory, and the CTAs of a (sequence, KV head) form a thread-block cluster (1, 2, 4 or 8 CTAs);
// every CTA owns a slice of the G*d outputs and receives the other CTAs' partials of that slice in its own
// shared memory (remote stores that report their bytes to an mbarrier of the owner, so only the owner's merging
// threads wait, and only for what is addressed to them), then merges them with the log-sum-exp rule
// (m = max m_j, l = sum l_j 2^(m_j-m), o = sum o_j 2^(m_j-m) / l) and writes bf16 out and fp32 lse.
// One launch, no workspace.
// (Measured and dropped: a two-kernel variant with partials in HBM, 2x slower on long single-sequence
// lists; clusters of 16, few of which can be co-scheduled; a block-wide ring of 64-token tiles with a
// barrier per tile, 10-25 % slower at every size.)
// The launch uses programmatic dependent launch, so back-to-back decode calls overlap their launch
// latency and prologue with the previous call's tail.
#include "common.cuh"
#include "launch.h"

namespace sg {
namespace {

constexpr int kSlice = 16;         // tokens per warp step (one m16n8k16 k-extent of V^T P^T)
constexpr float kLog2e = 1.4426950408889634f;
constexpr float kLn2 = 0.6931471805599453f;

struct DecParams {
  const uint16_t* q;
  const uint16_t* packed_k;
  const uint16_t* packed_v;
  const uint16_t* local_k;
  const uint16_t* local_v;
  const int32_t* cu;
  const int32_t* cu_k;
  const int32_t* cu_nloc;
  const int32_t* local_idx;
  const int32_t* packed_count;   // [B][Hkv] packed rows of a (sequence, KV head) that are in the list, or null: all k_b
  const int32_t* local_skip;     // [B][Hkv] leading entries of the head's local-index row that are not in the list, or null
  uint16_t* out;
  float* lse;
  int32_t* dev_status;
  int64_t ts, hs;
  uint32_t ts_bytes;  // token stride in bytes, or 0 when it does not fit
  int32_t B, Hq, Hkv, G, K_tot, NL_tot;
  int32_t n_tokens;  // total tokens of the batch: with one sequence every prefix array is {0, total}, known on the host
  int32_t csize;     // CTAs per (sequence, KV head) = cluster size
  float scale_log2;
};

__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async16_zfill(uint32_t dst, const void* src, int src_bytes) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(dst), "l"(src), "r"(src_bytes) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory"); }

__device__ __forceinline__ void ldmatrix_x4(uint32_t (&r)[4], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}
__device__ __forceinline__ void ldmatrix_x4_trans(uint32_t (&r)[4], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}
__device__ __forceinline__ void mma_bf16(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                         uint32_t b0, uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
               : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t*>(&v);
}

__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;\n" ::: "memory"); }
// Remote stores that report their bytes to an mbarrier of the destination CTA: the owner of an output slice waits on
// its own barrier for everybody's partials instead of the whole cluster meeting at a barrier.
__device__ __forceinline__ void st_async_f32(float* local_ptr, uint64_t* local_bar, uint32_t cta_rank, float v) {
  uint32_t raddr, rbar;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;\n" : "=r"(raddr) : "r"(smem_u32(local_ptr)), "r"(cta_rank));
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;\n" : "=r"(rbar) : "r"(smem_u32(local_bar)), "r"(cta_rank));
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.f32 [%0], %1, [%2];\n" ::"r"(raddr), "f"(v), "r"(rbar) : "memory");
}
__device__ __forceinline__ void st_async_f32x2(float* local_ptr, uint64_t* local_bar, uint32_t cta_rank, float a, float b) {
  uint32_t raddr, rbar;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;\n" : "=r"(raddr) : "r"(smem_u32(local_ptr)), "r"(cta_rank));
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;\n" : "=r"(rbar) : "r"(smem_u32(local_bar)), "r"(cta_rank));
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v2.f32 [%0], {%1, %2}, [%3];\n" ::"r"(raddr), "f"(a), "f"(b), "r"(rbar) : "memory");
}
__device__ __forceinline__ void cluster_arrive_release() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n" ::: "memory");
}
// Bounded wait for phase 0 of an mbarrier whose bytes come from other CTAs of the cluster; false when it gave up.
__device__ __forceinline__ bool mbar_wait_cluster_bounded(uint64_t* bar) {
  const uint32_t addr = smem_u32(bar);
  const long long t0 = clock64();
  do {                                                      // the senders run concurrently (same cluster): microseconds; the limit is ~0.5 s
    uint32_t done;
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], 0;\n\tselp.u32 %0, 1, 0, p;\n\t}\n"
                 : "=r"(done) : "r"(addr) : "memory");
    if (done) return true;
  } while (clock64() - t0 < 1000000000LL);
  return false;
}
// Exchanges rows and columns of an 8 x 8 matrix of 16-bit values held as an MMA accumulator holds one (lane / 4 = row).
__device__ __forceinline__ uint32_t movmatrix_trans(uint32_t v) {
  uint32_t r;
  asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;\n" : "=r"(r) : "r"(v));
  return r;
}

// kTwoLane: a counted call with local_skip; a kernel of its own, because a branch on the pointer in front of the first loads cost
// the plain calls 0.5 to 1 % (a decode step of 32 layers of 820 entries at batch 1 39.8 us, without it 39.5).  kN: 8-row tiles of the KV head's query rows (1 for G <= 8, 2 up to 16).  kDecWarps warps per CTA, each with a private ring
// of kSlots half slices: three leave room for two 8-warp CTAs per SM (d = 128), six for one.
template <int D, int kN, int kDecWarps, int kSlots, bool kTwoLane>
__global__ void __launch_bounds__(kDecWarps * 32, (kN == 1 && kSlots * D <= 384 ? 16 : 8) / kDecWarps) decode_partial_kernel(const DecParams p) {
  constexpr int kDecThreads = kDecWarps * 32;
  constexpr int kRowBytes = D * 2;
  constexpr int kChunksPerRow = D / 8;                       // 16-byte chunks
  constexpr int kHalfBytes = kSlice * kRowBytes;             // K (or V) rows of one slice
  constexpr int kCopiesPerLane = kSlice * kChunksPerRow / 32;
  constexpr uint32_t kFull = 0xffffffffu;
  extern __shared__ __align__(1024) uint8_t smem_raw[];       // per warp: kSlots half slices, rows XOR-swizzled
  // Receive area for the cluster merge, never aliased by the rings: the slice of the G*d outputs this CTA
  // owns, as every rank's partial: rx_o [8][per], rx_m [8][16], rx_l [8][16].
  float* rx_m = reinterpret_cast<float*>(smem_raw + kDecWarps * kSlots * kHalfBytes);
  float* rx_l = rx_m + 8 * 16;
  float* rx_o = rx_l + 8 * 16;
  uint64_t* rx_bar = reinterpret_cast<uint64_t*>(rx_o + 16 * D);   // counts the bytes of the partials pushed into the three arrays

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int g = blockIdx.y;
  pdl_launch_dependents();
  if (p.csize > 1) {
    if (tid == 0) {
      // every rank sends this CTA its partial of the slice owned here and its (M, L) of the G rows
      const int per0 = (p.G * D + p.csize - 1) / p.csize;
      const int c_rank = blockIdx.x % p.csize;
      const int own = max(0, min(p.G * D, (c_rank + 1) * per0) - c_rank * per0);
      const uint32_t bytes = (uint32_t)p.csize * (uint32_t)(own + 2 * p.G) * 4u;
      const uint32_t bar = smem_u32(rx_bar);
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(bar) : "memory");
      asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
      asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(bar), "r"(bytes) : "memory");
    }
    cluster_arrive_release();                                  // "this CTA runs, its barrier is set up": awaited before the first remote store
  }
  // The counts, rows and index lists of a two-lane call come from the calls right in front of it (split, pack): it reads
  // nothing before they are complete and visible.  (They have ended when its CTAs are placed, so the wait is short.)
  // Everything it reads is read with plain loads: the compiler may move read-only-cache loads across the wait.  Calls
  // without a skip are those of a decode loop over rows selected and packed long before: one behind another they overlap as
  // plain calls do (one sequence of 820 entries: 1.7 us per call, 4.5 if each waits; 14 of 3277: 17 and 40).
  if (kTwoLane) pdl_wait();
  const int b = blockIdx.x / p.csize;                          // grid.x = B * cluster size
  const int c = blockIdx.x - b * p.csize;                      // rank in the cluster
  // A single sequence (the latency-critical case) needs no prefix loads: a dependent round trip to L2 less before the
  // first copy can be issued.
  const bool one = p.B == 1;
  const int ck0 = one ? 0 : p.cu_k[b];
  const int kb = one ? p.K_tot : p.cu_k[b + 1] - ck0;          // packed rows per KV head (the slot size in the buffer)
  const int kbe = p.packed_count ? min(kb, max(0, p.packed_count[(int64_t)b * p.Hkv + g])) : kb;   // ... of which in the list
  const int cl0 = one ? 0 : p.cu_nloc[b];
  const int nl_row = one ? p.NL_tot : p.cu_nloc[b + 1] - cl0;
  const int lskip = kTwoLane ? min(nl_row, max(0, p.local_skip[(int64_t)b * p.Hkv + g])) : 0;
  const int nl = nl_row - lskip;
  const int c0 = one ? 0 : p.cu[b];
  const int nseq = one ? p.n_tokens : p.cu[b + 1] - c0;

  const uint16_t* pk_base = p.packed_k + ((int64_t)ck0 * p.Hkv + (int64_t)g * kb) * D;
  const uint16_t* pv_base = p.packed_v + ((int64_t)ck0 * p.Hkv + (int64_t)g * kb) * D;
  const uint16_t* lk_base = p.local_k + (int64_t)c0 * p.ts + (int64_t)g * p.hs;
  const uint16_t* lv_base = p.local_v + (int64_t)c0 * p.ts + (int64_t)g * p.hs;
  const uint32_t ring = smem_u32(smem_raw) + warp * (kSlots * kHalfBytes);        // this warp's ring

  // The slices of the list [packed rows ++ local rows] of (b, g) are dealt out round robin over all warps of all CTAs of
  // the cluster (slice s goes to rank s % csize, warp (s / csize) % warps): every CTA gets the same mix of contiguous
  // packed slices and slower gathered ones, whatever the split of the list.
  const int ntok = kbe + nl;
  const int step = kDecWarps * p.csize * kSlice;               // list positions from a slice of this warp to its next
  int li0 = (warp * p.csize + c) * kSlice;                     // first list position of the warp's slice
  const int32_t* idx_base = p.local_idx + (int64_t)g * p.NL_tot + cl0 + lskip - kbe + (lane & 15);   // indexed by list position
  // Lane r (and r + 16) holds the local index of row r of a slice, read ahead of its use.
  auto fetch_idx = [&](int at) -> int {
    const int li = at + (lane & 15);
    return (li < ntok && li >= kbe) ? idx_base[at] : 0;
  };
  // A warp is alone on its scheduler or shares it with a few others, and its instructions issue one by one: what a slice takes
  // is its instruction count (a first form with 600 of them took 2500 clocks, this one has about 200).  So the copies' addresses are built from per-lane constants and
  // immediate offsets, with one multiplication per gathered row; what does not occur in the bulk of a list (the slice where
  // packed rows end, the last slice, bad indices, very large strides) goes through a loop.
  constexpr int kRowsPerCopy = 32 / kChunksPerRow;
  const int row0 = lane / kChunksPerRow, col0 = lane % kChunksPerRow;
  const uint32_t dst0 = ring + row0 * kRowBytes + ((col0 ^ row0) << 4);
  pk_base += lane * 8;
  pv_base += lane * 8;
  const uint8_t* const lk_lane = reinterpret_cast<const uint8_t*>(lk_base + col0 * 8);
  const uint8_t* const lv_lane = reinterpret_cast<const uint8_t*>(lv_base + col0 * 8);
  // Copies the K or V rows of the slice at list position `at` into a slot; returns the rows that hold a real token (bit r: row r).
  auto load_half = [&](int at, bool is_v, int slot, int idx_reg) -> uint32_t {
    const uint32_t dst = dst0 + slot * kHalfBytes;
    auto dst_of = [&](int i) { return (dst ^ (((i * kRowsPerCopy) & 7) << 4)) + i * (kRowsPerCopy * kRowBytes); };
    if (at + kSlice <= kbe) {
      // the whole slice lies in the packed buffer: 16 consecutive rows are one contiguous run of 16-byte pieces
      const uint16_t* src = (is_v ? pv_base : pk_base) + (int64_t)at * D;
#pragma unroll
      for (int i = 0; i < kCopiesPerLane; ++i) cp_async16(dst_of(i), src + i * 256);
      return 0xffffu;
    }
    const uint8_t* local = is_v ? lv_lane : lk_lane;
    if (at >= kbe && at + kSlice <= ntok && p.ts_bytes && __all_sync(kFull, (uint32_t)idx_reg < (uint32_t)nseq)) {
#pragma unroll
      for (int i = 0; i < kCopiesPerLane; ++i) {
        const uint32_t t = (uint32_t)__shfl_sync(kFull, idx_reg, row0 + i * kRowsPerCopy);
        cp_async16(dst_of(i), local + (uint64_t)t * p.ts_bytes);
      }
      return 0xffffu;
    }
    const int li = at + (lane & 15);
    const bool ok = li < kbe || (li < ntok && (uint32_t)idx_reg < (uint32_t)nseq);
    if (li < ntok && !ok && !is_v && lane < 16) raise(p.dev_status, SG_ERR_INDEX);
    const uint32_t good = __ballot_sync(kFull, ok) & 0xffffu;
    // lane r finds row r's source, its copiers ask it
    const uint64_t mine = li < kbe ? (uint64_t)((is_v ? pv_base : pk_base) - lane * 8 + (int64_t)li * D) : (uint64_t)(local - col0 * 16 + (int64_t)idx_reg * p.ts * 2);
#pragma unroll
    for (int i = 0; i < kCopiesPerLane; ++i) {
      const int row = row0 + i * kRowsPerCopy;
      const uint64_t src = __shfl_sync(kFull, mine, row) + col0 * 16;
      cp_async16_zfill(dst_of(i), reinterpret_cast<const void*>(src), (good >> row) & 1u ? 16 : 0);   // rows without a token are zero
    }
    return good;
  };

  float o_acc[kN][D / 16][4], m_run[kN][2], l_run[kN][2];
#pragma unroll
  for (int t = 0; t < kN; ++t) {
#pragma unroll
    for (int i = 0; i < D / 16; ++i) { o_acc[t][i][0] = o_acc[t][i][1] = o_acc[t][i][2] = o_acc[t][i][3] = 0.f; }
    m_run[t][0] = m_run[t][1] = -INFINITY;
    l_run[t][0] = l_run[t][1] = 0.f;
  }

  // The halves K0 V0 K1 V1 ... go through the ring in order, half h into slot h mod kSlots; a slot is refilled, with half
  // h + kSlots, as soon as its fragments are in registers.
  static_assert(kSlots == 3 || kSlots == 6, "the order of the refills below");
  constexpr int kAhead = kSlots == 3 ? 2 : 3;                 // slices that are asked for ahead of the current one
  uint32_t mask[kAhead + 1] = {};                             // real rows of this slice and the next ones
  int idx[kAhead];                                            // local indices of the next slices
  {
    const int idx0 = fetch_idx(li0);
#pragma unroll
    for (int i = 0; i < kAhead; ++i) idx[i] = fetch_idx(li0 + (i + 1) * step);
#pragma unroll 1
    for (int h = 0; h < kSlots; ++h) {                        // not unrolled: this code runs once per call, from a cold instruction cache
      const int at = li0 + (h >> 1) * step;
      const uint32_t got = at < ntok ? load_half(at, h & 1, h, h < 2 ? idx0 : h < 4 ? idx[0] : idx[1]) : 0u;
#pragma unroll
      for (int i = 0; i < kAhead; ++i) mask[i] = h == 2 * i ? got : mask[i];
      cp_async_commit();
    }
  }

  // Everything in this kernel up to its output stores reads only inputs of the decode step -- the KV sources, the
  // index lists, the prefix arrays and the query rows -- which the contract of the plain call treats as stable: they must
  // not be written by a kernel that itself lets its dependents start early (such as the previous layer's call of this
  // kernel).  So nothing waits here: the dependency wait sits in front of the stores of out / lse, and consecutive
  // calls overlap everything but those stores.
  // Q fragments (B operand, D x 8 per tile; rows >= G are zero).
  const int r8 = lane >> 2, c2 = 2 * (lane & 3);
  uint32_t qf[kN][D / 16][2];
  {
    const uint16_t* qb = p.q + ((int64_t)b * p.Hq + (int64_t)g * p.G) * D;
#pragma unroll
    for (int t = 0; t < kN; ++t) {
      const int r = t * 8 + r8;
#pragma unroll
      for (int kk = 0; kk < D / 16; ++kk) {
        qf[t][kk][0] = r < p.G ? *reinterpret_cast<const uint32_t*>(qb + r * D + kk * 16 + c2) : 0u;
        qf[t][kk][1] = r < p.G ? *reinterpret_cast<const uint32_t*>(qb + r * D + kk * 16 + c2 + 8) : 0u;
      }
    }
  }

  // The ring is private to the warp: no block-wide barrier inside the loop, the warps drift freely.
  // K fragments (A operand): matrices of tokens 0-7 and 8-15 x two column pieces; V^T: two column pieces x tokens 0-7 and 8-15
  const int mi = lane >> 3, r7 = lane & 7;
  const uint32_t k_lane = ring + ((mi & 1) * 8 + r7) * kRowBytes + (((mi >> 1) ^ r7) << 4);
  const uint32_t v_lane = ring + ((mi >> 1) * 8 + r7) * kRowBytes + (((mi & 1) ^ r7) << 4);
  int slot = 0;                                               // of K of slice j; V is in the next one
#pragma unroll 1
  for (; li0 < ntok; li0 += step) {
    const int vslot = slot == kSlots - 1 ? 0 : slot + 1;
    cp_async_wait<kSlots - 1>();
    __syncwarp();
    uint32_t f[D / 16][4];                                    // all fragment loads of a half before its MMAs
    {
      const uint32_t at = k_lane + slot * kHalfBytes;
#pragma unroll
      for (int kk = 0; kk < D / 16; ++kk) ldmatrix_x4(f[kk], at ^ (kk << 5));
    }
    __syncwarp();
    // S^T = K Q^T: 16 tokens x 8 query rows per tile, even and odd k-steps in chains of their own (a warp has only one or
    // two slices at small batch: the length of the chain is what it waits for)
    float s_acc[kN][4], s_odd[kN][4];
#pragma unroll
    for (int t = 0; t < kN; ++t) {
      s_odd[t][0] = s_odd[t][1] = s_odd[t][2] = s_odd[t][3] = 0.f;
      s_acc[t][0] = s_acc[t][1] = s_acc[t][2] = s_acc[t][3] = 0.f;
#pragma unroll
      for (int kk = 0; kk < D / 16; ++kk)
        mma_bf16((kk & 1) ? s_odd[t] : s_acc[t], f[kk][0], f[kk][1], f[kk][2], f[kk][3], qf[t][kk][0], qf[t][kk][1]);
    }
    // The tensor cores are busy with S: refill K's slot, fetch the V fragments (into the registers of K's), refill V's slot.
    if (kSlots == 3) {
      if (li0 + step < ntok) load_half(li0 + step, true, slot, idx[0]);
    } else {
      if (li0 + 3 * step < ntok) mask[kAhead] = load_half(li0 + 3 * step, false, slot, idx[kAhead - 1]);
    }
    cp_async_commit();
    const uint32_t rows = mask[0];
    cp_async_wait<kSlots - 1>();
    __syncwarp();
    {
      const uint32_t at = v_lane + vslot * kHalfBytes;
#pragma unroll
      for (int dc = 0; dc < D / 16; ++dc) ldmatrix_x4_trans(f[dc], at ^ (dc << 5));
    }
    __syncwarp();
    if (kSlots == 3) {
      if (li0 + 2 * step < ntok) mask[kAhead] = load_half(li0 + 2 * step, false, vslot, idx[kAhead - 1]);
    } else {
      if (li0 + 3 * step < ntok) load_half(li0 + 3 * step, true, vslot, idx[kAhead - 1]);
    }
    cp_async_commit();
#pragma unroll
    for (int i = 0; i < kAhead; ++i) mask[i] = mask[i + 1];
#pragma unroll
    for (int i = 0; i + 1 < kAhead; ++i) idx[i] = idx[i + 1];
    idx[kAhead - 1] = fetch_idx(li0 + (kAhead + 1) * step);
    // online softmax in base 2; padding and skipped indices are masked.  The lane holds tokens r8 and r8 + 8 of query rows c2
    // and c2 + 1 of a tile.
    const bool ok0 = (rows >> r8) & 1u, ok1 = (rows >> (r8 + 8)) & 1u;
    uint32_t pf[kN][2];
    bool rescale = false;
    float al[kN][2];
#pragma unroll
    for (int t = 0; t < kN; ++t) {
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const float a = ok0 ? s_acc[t][e] + s_odd[t][e] : -INFINITY, c = ok1 ? s_acc[t][2 + e] + s_odd[t][2 + e] : -INFINITY;
        float mx = fmaxf(a, c);
        mx = fmaxf(mx, __shfl_xor_sync(kFull, mx, 4));
        mx = fmaxf(mx, __shfl_xor_sync(kFull, mx, 8));
        mx = fmaxf(mx, __shfl_xor_sync(kFull, mx, 16));
        const float mn = fmaxf(m_run[t][e], mx * p.scale_log2), mu = mn == -INFINITY ? 0.f : mn;
        al[t][e] = exp2f(m_run[t][e] - mu);
        m_run[t][e] = mn;
        const float p0 = exp2f(fmaf(a, p.scale_log2, -mu)), p1 = exp2f(fmaf(c, p.scale_log2, -mu));
        // every lane keeps the part of the row sum that its own tokens make; the parts are added up once, after the last slice
        l_run[t][e] = l_run[t][e] * al[t][e] + (p0 + p1);
        s_acc[t][e] = p0;
        s_acc[t][2 + e] = p1;
        rescale = rescale || al[t][e] != 1.f;
      }
      pf[t][0] = movmatrix_trans(pack_bf16(s_acc[t][0], s_acc[t][1]));
      pf[t][1] = movmatrix_trans(pack_bf16(s_acc[t][2], s_acc[t][3]));
    }
    if (__any_sync(kFull, rescale)) {
#pragma unroll
      for (int t = 0; t < kN; ++t) {
#pragma unroll
        for (int i = 0; i < D / 16; ++i) {
          o_acc[t][i][0] *= al[t][0]; o_acc[t][i][1] *= al[t][1];
          o_acc[t][i][2] *= al[t][0]; o_acc[t][i][3] *= al[t][1];
        }
      }
    }
    // O^T += V^T P^T
#pragma unroll
    for (int t = 0; t < kN; ++t) {
#pragma unroll
      for (int dc = 0; dc < D / 16; ++dc) mma_bf16(o_acc[t][dc], f[dc][0], f[dc][1], f[dc][2], f[dc][3], pf[t][0], pf[t][1]);
    }
    slot = slot >= kSlots - 2 ? slot + 2 - kSlots : slot + 2;
  }
#pragma unroll
  for (int t = 0; t < kN; ++t) {
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      l_run[t][e] += __shfl_xor_sync(kFull, l_run[t][e], 4);
      l_run[t][e] += __shfl_xor_sync(kFull, l_run[t][e], 8);
      l_run[t][e] += __shfl_xor_sync(kFull, l_run[t][e], 16);
    }
  }
  cp_async_wait<0>();
  __syncthreads();

  // merge the warps through shared memory (the rings are free now)
  constexpr int kOStride = D + 4;                             // row stride of the partials: the lanes of a store hit 32 different banks
  float* sm_o = reinterpret_cast<float*>(smem_raw);           // [kDecWarps][8 kN][kOStride]
  float* sm_m = sm_o + kDecWarps * 8 * kN * kOStride;         // [kDecWarps][16]
  float* sm_l = sm_m + kDecWarps * 16;
#pragma unroll
  for (int t = 0; t < kN; ++t) {
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const int r = t * 8 + c2 + e;                           // rows >= G are padding and never read
      if (r < p.G) {
        if (r8 == 0) { sm_m[warp * 16 + r] = m_run[t][e]; sm_l[warp * 16 + r] = l_run[t][e]; }
        float* dst = sm_o + (warp * 8 * kN + r) * kOStride + r8;
#pragma unroll
        for (int i = 0; i < D / 16; ++i) { dst[i * 16] = o_acc[t][i][e]; dst[i * 16 + 8] = o_acc[t][i][2 + e]; }
      }
    }
  }
  __syncthreads();
  // CTA-level partial of every output; with a cluster, each rank owns a slice of the G*d outputs and
  // every CTA pushes its partial of a slice into the owner's receive area (distributed shared memory).
  const int cs = p.csize;
  const int per = (p.G * D + cs - 1) / cs;
  __nv_bfloat16* outp = reinterpret_cast<__nv_bfloat16*>(p.out) + ((int64_t)b * p.Hq + (int64_t)g * p.G) * D;
  float* lsep = p.lse ? p.lse + (int64_t)b * p.Hq + (int64_t)g * p.G : nullptr;
  if (cs > 1) cluster_wait();                                  // every CTA of the cluster has started
  if (cs == 1) pdl_wait();                                     // out / lse are written below: all earlier work in the stream first
  // two neighbouring outputs per thread (same row, same owner: D and the owners' slices are even)
  for (int e = 2 * tid; e < p.G * D; e += 2 * kDecThreads) {
    const int r = e / D, col = e - r * D;
    float M = -INFINITY;
#pragma unroll
    for (int w = 0; w < kDecWarps; ++w) M = fmaxf(M, sm_m[w * 16 + r]);
    const float Mu = M == -INFINITY ? 0.f : M;
    float L = 0.f, O0 = 0.f, O1 = 0.f;
#pragma unroll
    for (int w = 0; w < kDecWarps; ++w) {
      const float f = exp2f(sm_m[w * 16 + r] - Mu);
      const float2 o = *reinterpret_cast<const float2*>(sm_o + (w * 8 * kN + r) * kOStride + col);
      L += sm_l[w * 16 + r] * f;
      O0 += o.x * f;
      O1 += o.y * f;
    }
    if (cs == 1) {
      *reinterpret_cast<__nv_bfloat162*>(outp + e) = __floats2bfloat162_rn(L > 0.f ? O0 / L : 0.f, L > 0.f ? O1 / L : 0.f);
      if (lsep && col == 0) lsep[r] = L > 0.f ? (M + log2f(L)) * kLn2 : -INFINITY;
    } else {
      const int owner = e / per;
      st_async_f32x2(rx_o + c * per + (e - owner * per), rx_bar, owner, O0, O1);
      if ((col >> 1) < cs) {                                  // the row's (M, L) goes to every rank: one thread per rank
        st_async_f32(rx_m + c * 16 + r, rx_bar, col >> 1, M);
        st_async_f32(rx_l + c * 16 + r, rx_bar, col >> 1, L);
      }
    }
  }
  if (cs > 1) {
    // Only the threads that merge wait, and only for the bytes addressed to this CTA.  Once they are all here nobody
    // writes into this CTA's shared memory any more, so it may finish without meeting the others again.
    const int e_beg = c * per, e_end = min(p.G * D, e_beg + per);
    if ((e_beg + tid < e_end || tid == 0) && !mbar_wait_cluster_bounded(rx_bar)) {   // thread 0 keeps the CTA alive for its senders in any case
      raise(p.dev_status, SG_ERR_TIMEOUT);
      return;
    }
    pdl_wait();                                                // out / lse are written below: all earlier work in the stream first
    for (int e = e_beg + tid; e < e_end; e += kDecThreads) {
      const int r = e / D, col = e - r * D;
      float mj[8], lj[8], oj[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const bool on = j < cs;
        mj[j] = on ? rx_m[j * 16 + r] : -INFINITY;
        lj[j] = on ? rx_l[j * 16 + r] : 0.f;
        oj[j] = on ? rx_o[j * per + (e - e_beg)] : 0.f;
      }
      float M = -INFINITY;
#pragma unroll
      for (int j = 0; j < 8; ++j) M = fmaxf(M, mj[j]);
      const float Mu = M == -INFINITY ? 0.f : M;
      float L = 0.f, O = 0.f;
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const float f = exp2f(mj[j] - Mu);
        L += lj[j] * f;
        O += oj[j] * f;
      }
      outp[e] = __float2bfloat16_rn(L > 0.f ? O / L : 0.f);
      if (lsep && col == 0) lsep[r] = L > 0.f ? (M + log2f(L)) * kLn2 : -INFINITY;
    }
  }
}

// rings, and with a cluster the receive area and its barrier
constexpr int decode_smem_bytes(int D, int warps, int slots, bool cluster) {
  return warps * slots * kSlice * D * 2 + (cluster ? (2 * 8 * 16 + 16 * D) * 4 + 16 : 0);
}

}  // namespace

// Launch shape, from a sweep over 1 to 64 sequences of 8 KV heads and lists of 30 to 6400 entries, each timed as calls that
// follow one another at once (a decode step replayed from a graph) and as a call behind an unrelated kernel.  A
// (sequence, KV head) pair is split over a cluster of 1, 2, 4 or 8 CTAs; two 8-warp or four 4-warp CTAs fit on an SM.
//  * pairs <= SMs: the clusters are spread one CTA per SM, which leaves room on every SM for the next call; the cluster size is
//    the smallest power of two (<= 8, the portable limit) that gives each warp about one slice, or the largest that fits.
//  * more pairs: one CTA each; eight warps once a list has 1024 entries (24 sequences of 1600: 30.2 us alone against 32.8 with
//    four), else four, whose merge is half as wide (64 sequences of 200: 9.8 against 11.3 us).
// Rings of three slots, two CTAs per SM and so two calls overlapped, are faster wherever rows are gathered (14 sequences of 1600
// entries, half of them gathered, 12 layers: 186 us against 199 with six slots) and for short lists.  Lists that are all
// packed stream at HBM rate once every warp has six slices or more; six slots then keep more bytes under way (a call behind an
// unrelated kernel / calls in sequence, three slots -> six: 14 sequences of 820 entries 11.3 -> 10.5 / 7.2 -> 7.0 us, 8 of 1640
// 12.6 -> 11.8 / 8.3 -> 8.1, 14 of 4096 38.4 -> 37.7 / 32.2 -> 32.1; with five slices per warp 10 of 600 8.35 -> 8.18 / 4.0 -> 4.4).
// Clusters have to fill three quarters of the SMs for that (96 CTAs of 6 x 4096 entries: 20.1 -> 19.4 / 13.5 -> 14.1).
// With more pairs than SMs six slots at d = 128 mean one CTA per SM, and up to one and a half CTAs per SM that is a second wave
// nearly empty: there four warps and three slots, all CTAs resident at once (19 sequences of 1640 entries 29.8 -> 25.5 / 18.3 ->
// 15.5 us, 24 of 4096 66.4 -> 62.6 / 54.5 -> 53.7; equal at 28 sequences; at d = 64 two six-slot CTAs fit and stay ahead: 19
// of 1640 14.7 against 17.0).  With more than eight query rows per KV head the registers allow one 8-warp CTA per SM
// anyway: six slots.
// A two-lane call names one row of the KV index as its packed and as its indexed list, so avg_tokens is up to twice what it
// attends.  Planned for the row's length, the chain of split, pack and attention is slower more often than faster
// (19 sequences of 820 entries 30.2 -> 32.7 us, 1 of 820 11.8 -> 12.3, 64 of 820 87.9 -> 83.4): it stays.
// It does not overlap the next call, so its clusters may fill both CTAs of every SM, where two fit (up to eight query rows per KV head; with
// sixteen the listed chain below took 36.8 -> 40.1 us, a second wave).  That pays where the longest row is well above the
// average and its warps have five slices or more: the call lasts as long as that row.  Whole chains of split, pack and attention, 8
// sequences of 6321 to 32061 tokens, a tenth of them required: 33.0 -> 30.6 us, four tenths 106 -> 90, d = 64 24.8 -> 21.5, 2 heads of 64
// 14.9 -> 13.3; but 8 of 500 to 4000 tokens 11.8 -> 12.6 and, of equal lengths, 16 of 1638 entries 40.2 -> 41.1, 4 of
// 1638 18.1 -> 18.5, which the rule leaves as they are.
void decode_plan(const sg_shape* shape, int32_t total_sel, int32_t total_loc, bool two_lane, int* csize, int* warps, int* slots) {
  const int64_t pairs = (int64_t)shape->batch * shape->num_kv_heads;
  const int64_t avg_tokens = ((int64_t)total_sel + total_loc) / shape->batch;
  const bool packed_only = total_loc == 0;
  int W = 8, cs = 1;
  if (pairs > kNumSMs) {
    W = avg_tokens < 1024 || (packed_only && shape->head_dim == 128 && 2 * pairs <= 3 * kNumSMs) ? 4 : 8;
  } else if (avg_tokens > (pairs >= 64 ? 14 : 8) * kSlice) {   // else a slice or two per warp of one CTA already: no cluster to merge
    int fit = 1;
    while (fit < 8 && pairs * fit * 2 <= kNumSMs) fit *= 2;
    // clusters of eight only while those of two calls fit side by side: one that cannot be placed waits for a whole call (2x)
    if (fit == 8 && pairs * 16 > kNumSMs) fit = 4;
    // short lists: four warps per CTA already give every warp at most ~1.75 slices, and the merge is half as wide
    W = 4 * avg_tokens <= 7 * 4 * kSlice * fit ? 4 : 8;
    while (cs < fit && (int64_t)cs * W * kSlice < avg_tokens) cs *= 2;
  }
  const bool wide_group = shape->num_q_heads / shape->num_kv_heads > 8;
  if (two_lane && !wide_group && pairs <= kNumSMs && W == 8 && shape->total_tokens > 0) {
    const int64_t longest = (int64_t)total_sel * shape->max_seqlen / shape->total_tokens, average = total_sel / shape->batch;
    if (4 * longest >= 5 * average && longest >= 5 * kSlice * W * cs && cs < 8 && pairs * cs <= kNumSMs) cs *= 2;
  }
  *csize = cs;
  *warps = W;
  const bool streams = packed_only && W == 8 && avg_tokens >= 6 * kSlice * W * cs && (cs == 1 ? 2 * pairs > kNumSMs : 4 * pairs * cs > 3 * kNumSMs);
  *slots = wide_group || streams ? 6 : 3;
}

size_t decode_workspace_bytes(const sg_shape*, int32_t, int32_t) { return 0; }   // partials stay on chip

}  // namespace sg

namespace sg {
namespace {
// Testing hook (sg_testing_decode_overlap): 0 launches the decode kernel fully ordered behind earlier work.
std::atomic<int> g_test_decode_overlap{1};
sg_status decode_launch(const sg_shape* shape, const void* q, const void* packed_k, const void* packed_v, const int32_t* cu_k,
                        int32_t total_sel, const int32_t* packed_count, const int32_t* local_skip, const void* local_k,
                        const void* local_v, const int32_t* local_idx, const int32_t* cu_nloc, int32_t total_loc,
                        float softmax_scale, void* out, float* lse, void* workspace, size_t workspace_bytes,
                        int32_t* dev_status, void* stream);
}
}  // namespace sg

extern "C" int32_t sg_testing_decode_cluster(const sg_shape* shape, int32_t total_sel, int32_t total_loc, int32_t two_lane) {
  using namespace sg;
  if (check_shape(shape, false) != SG_OK || total_sel < 0 || total_loc < 0) return 0;
  int csize = 0, warps = 0, slots = 0;
  decode_plan(shape, total_sel, total_loc, two_lane != 0, &csize, &warps, &slots);
  return csize;
}

extern "C" void sg_testing_decode_overlap(int32_t allowed) {
  sg::g_test_decode_overlap.store(allowed, std::memory_order_relaxed);
}

extern "C" sg_status sg_sparse_decode_attn(const sg_shape* shape, const void* q, const void* packed_k,
                                           const void* packed_v, const int32_t* cu_k, int32_t total_sel,
                                           const void* local_k, const void* local_v, const int32_t* local_idx,
                                           const int32_t* cu_nloc, int32_t total_loc, float softmax_scale,
                                           void* out, float* lse, void* workspace, size_t workspace_bytes,
                                           int32_t* dev_status, void* stream) {
  return sg::decode_launch(shape, q, packed_k, packed_v, cu_k, total_sel, nullptr, nullptr, local_k, local_v, local_idx,
                           cu_nloc, total_loc, softmax_scale, out, lse, workspace, workspace_bytes, dev_status, stream);
}

extern "C" sg_status sg_sparse_decode_attn_counted(const sg_shape* shape, const void* q, const void* packed_k,
                                                   const void* packed_v, const int32_t* cu_cap, int32_t total_cap,
                                                   const int32_t* packed_count, const void* local_k, const void* local_v,
                                                   const int32_t* local_idx, const int32_t* cu_nloc, int32_t total_loc,
                                                   const int32_t* local_skip, float softmax_scale, void* out, float* lse,
                                                   int32_t* dev_status, void* stream) {
  if ((!packed_count && !local_skip) || !sg::aligned16(packed_count) || !sg::aligned16(local_skip)) return SG_ERR_INVALID;
  return sg::decode_launch(shape, q, packed_k, packed_v, cu_cap, total_cap, packed_count, local_skip, local_k, local_v,
                           local_idx, cu_nloc, total_loc, softmax_scale, out, lse, nullptr, 0, dev_status, stream);
}

namespace sg {
namespace {
sg_status decode_launch(const sg_shape* shape, const void* q, const void* packed_k, const void* packed_v, const int32_t* cu_k,
                        int32_t total_sel, const int32_t* packed_count, const int32_t* local_skip, const void* local_k,
                        const void* local_v, const int32_t* local_idx, const int32_t* cu_nloc, int32_t total_loc,
                        float softmax_scale, void* out, float* lse, void* workspace, size_t workspace_bytes,
                        int32_t* dev_status, void* stream) {
  using namespace sg;
  sg_status st = check_shape(shape, false);
  if (st != SG_OK) return st;
  if (shape->num_layers != 1 || total_sel < 0 || total_loc < 0) return SG_ERR_INVALID;
  if (!q || !out || !cu_k || !cu_nloc) return SG_ERR_INVALID;
  if (total_sel > 0 && (!packed_k || !packed_v)) return SG_ERR_INVALID;
  if (total_loc > 0 && (!local_k || !local_v || !local_idx)) return SG_ERR_INVALID;
  if (!aligned16(q) || !aligned16(out) || !aligned16(cu_k) || !aligned16(cu_nloc) || !aligned16(packed_k) ||
      !aligned16(packed_v) || !aligned16(local_k) || !aligned16(local_v) || !aligned16(local_idx) ||
      !aligned16(workspace) || (lse && (reinterpret_cast<uintptr_t>(lse) & 3u)))
    return SG_ERR_INVALID;
  if (!(softmax_scale >= 0.f)) return SG_ERR_INVALID;
  (void)workspace_bytes;                                      // no workspace is needed: partials stay on chip
  const int D = shape->head_dim;
  const int G = shape->num_q_heads / shape->num_kv_heads;
  DecParams p;
  p.q = static_cast<const uint16_t*>(q);
  p.packed_k = static_cast<const uint16_t*>(packed_k ? packed_k : q);
  p.packed_v = static_cast<const uint16_t*>(packed_v ? packed_v : q);
  p.local_k = static_cast<const uint16_t*>(local_k ? local_k : q);
  p.local_v = static_cast<const uint16_t*>(local_v ? local_v : q);
  p.cu = shape->cu_seqlens;
  p.cu_k = cu_k;
  p.cu_nloc = cu_nloc;
  p.local_idx = local_idx ? local_idx : cu_nloc;
  p.packed_count = packed_count;
  p.local_skip = local_skip;
  p.out = static_cast<uint16_t*>(out);
  p.lse = lse;
  p.dev_status = dev_status;
  p.ts = shape->cache_token_stride;
  p.ts_bytes = p.ts > 0 && p.ts < (1 << 30) ? (uint32_t)p.ts * 2u : 0u;
  p.hs = shape->cache_head_stride;
  p.B = shape->batch;
  p.Hq = shape->num_q_heads;
  p.Hkv = shape->num_kv_heads;
  p.G = G;
  p.K_tot = total_sel;
  p.NL_tot = total_loc;
  p.n_tokens = shape->total_tokens;
  int warps = 4, slots = 3;
  decode_plan(shape, total_sel, total_loc, local_skip != nullptr, &p.csize, &warps, &slots);
  p.scale_log2 = (softmax_scale > 0.f ? softmax_scale : 1.0f / sqrtf((float)D)) * kLog2e;
  const int64_t grid_x = (int64_t)shape->batch * p.csize;
  if (grid_x > 0x7fffffffLL || shape->num_kv_heads > 65535) return SG_ERR_UNSUPPORTED;

  cudaLaunchAttribute attrs[2];
  attrs[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attrs[0].val.programmaticStreamSerializationAllowed = g_test_decode_overlap.load(std::memory_order_relaxed) ? 1 : 0;
  attrs[1].id = cudaLaunchAttributeClusterDimension;
  attrs[1].val.clusterDim.x = (unsigned)p.csize;
  attrs[1].val.clusterDim.y = 1;
  attrs[1].val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.stream = static_cast<cudaStream_t>(stream);
  cfg.attrs = attrs;
  cfg.numAttrs = p.csize > 1 ? 2 : 1;
  cfg.blockDim = dim3((unsigned)warps * 32);
  // one launch: sequences with empty lists still get out = 0 and lse = -inf
  cfg.gridDim = dim3((unsigned)grid_x, (unsigned)shape->num_kv_heads);
  cfg.dynamicSmemBytes = (size_t)decode_smem_bytes(D, warps, slots, p.csize > 1);
#define SG_LAUNCH_DECODE(DD, NN, WW, SS, TL)                                                         \
  do {                                                                                               \
    SG_ENSURE_SMEM((decode_partial_kernel<DD, NN, WW, SS, TL>), decode_smem_bytes(DD, WW, SS, true)); \
    SG_CUDA_TRY(cudaLaunchKernelEx(&cfg, decode_partial_kernel<DD, NN, WW, SS, TL>, p));             \
  } while (0)
#define SG_LAUNCH_DECODE_D(DD, TL)                                            \
  do {                                                                        \
    if (G > 8 && warps == 8) SG_LAUNCH_DECODE(DD, 2, 8, 6, TL);               \
    else if (G > 8) SG_LAUNCH_DECODE(DD, 2, 4, 6, TL);                        \
    else if (warps == 4) SG_LAUNCH_DECODE(DD, 1, 4, 3, TL);                   \
    else if (slots == 6) SG_LAUNCH_DECODE(DD, 1, 8, 6, TL);                   \
    else SG_LAUNCH_DECODE(DD, 1, 8, 3, TL);                                   \
  } while (0)
  if (local_skip) {
    if (D == 128) SG_LAUNCH_DECODE_D(128, true);
    else SG_LAUNCH_DECODE_D(64, true);
  } else if (D == 128) {
    SG_LAUNCH_DECODE_D(128, false);
  } else {
    SG_LAUNCH_DECODE_D(64, false);
  }
#undef SG_LAUNCH_DECODE_D
#undef SG_LAUNCH_DECODE
  return SG_OK;
}
}  // namespace
}  // namespace sg
