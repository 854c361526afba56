// PTX wrappers of the scoring kernel: mbarriers with bounded waits, TMA tile loads, tcgen05 MMAs and tensor memory.
#pragma once

#include <cuda.h>
#include <stdint.h>

#include "common.cuh"

namespace sg {

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ uint64_t global_timer_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
// One try_wait: true when the phase has completed.
__device__ __forceinline__ bool mbar_test(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
  return ok != 0;
}
// Bounded wait: gives up after `limit_ns` (about one second in normal use), or once another thread has set
// *abort_flag.  try_wait comes back after a short, hardware-chosen time whether or not the phase has completed, so a
// thread that simply retries spins through a dozen instructions per attempt -- issue slots and, worse, entries of the
// queue that the SFU instructions of the working warps go through (measured: one retry per 11 clocks and SM, 60 % of
// all executed instructions, SFU pipe at 51 %).  A waiter therefore sleeps `sleep_ns` between attempts (chosen per
// role: short on the MMA thread's critical path, long for the producer that runs ahead) and looks at the clock and the
// abort flag only every 64th attempt.
// kBehind: the thread has executed pdl_wait().  Otherwise the work it waits for may itself be waiting for the kernel in
// front of this one, whose time does not count: when the limit first runs out, the thread waits for that kernel and
// starts its limit again.
template <bool kBehind>
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag, uint32_t limit_ns,
                                          uint32_t sleep_ns) {
  if (mbar_test(bar, parity)) return true;
  bool behind = kBehind;
  uint64_t t0 = 0;
  for (uint32_t it = 0;; ++it) {
    if (sleep_ns) __nanosleep(sleep_ns);
    if (mbar_test(bar, parity)) return true;
    if ((it & 63u) == 63u) {
      if (*abort_flag) return false;
      const uint64_t now = global_timer_ns();
      if (t0 == 0) {
        t0 = now;
      } else if (now - t0 > (uint64_t)limit_ns) {
        if (behind) { *abort_flag = 1; return false; }
        pdl_wait();
        behind = true;
        t0 = global_timer_ns();
      }
    }
  }
}
// The same wait for code that issues work on its critical path: everything but a first attempt stays out of line.
template <bool kBehind>
static __device__ __noinline__ bool mbar_wait_slow(uint32_t bar, uint32_t parity, volatile int* abort_flag, uint32_t limit_ns) {
  return mbar_wait<kBehind>(bar, parity, abort_flag, limit_ns, 0u);
}
__device__ __forceinline__ void fence_barrier_init() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

__device__ __forceinline__ void tma_prefetch_map(const CUtensorMap* map) {
  asm volatile("prefetch.tensormap [%0];" ::"l"(map) : "memory");
}
__device__ __forceinline__ void tma_load_4d(uint32_t dst, const CUtensorMap* map, uint32_t bar, int c0, int c1, int c2, int c3) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], [%2];"
      ::"r"(dst), "l"(map), "r"(bar), "r"(c0), "r"(c1), "r"(c2), "r"(c3) : "memory");
}
__device__ __forceinline__ void tmem_alloc(uint32_t smem_dst, uint32_t cols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_dst), "r"(cols) : "memory");
}
__device__ __forceinline__ void tmem_relinquish() {
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t cols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(cols) : "memory");
}
__device__ __forceinline__ void umma_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
// TMEM load of 32 consecutive fp32 columns of this thread's lane, issued without waiting: the registers hold
// the data only after tmem_ld_wait().  A warp issues the load of its next 32 columns before it works on the
// current ones, so the load's latency is covered by arithmetic.
__device__ __forceinline__ void tmem_ld32_issue(uint32_t (&r)[32], uint32_t taddr) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
        "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
        "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr) : "memory");
}
// The same with 16 columns.
__device__ __forceinline__ void tmem_ld16_issue(uint32_t (&r)[16], uint32_t taddr) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
                 "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
               : "r"(taddr) : "memory");
}
// Waits for the thread's outstanding TMEM loads.  The empty statements that follow tie the registers of the
// load that has just completed to this point of the program: volatile statements keep their order, and every
// later use of the registers depends on them, so the compiler cannot schedule arithmetic on the data ahead of the wait.
template <int N>
__device__ __forceinline__ void tmem_ld_tie(uint32_t (&r)[N]) {
#pragma unroll
  for (int i = 0; i < N; i += 8)
    asm volatile("" : "+r"(r[i]), "+r"(r[i + 1]), "+r"(r[i + 2]), "+r"(r[i + 3]), "+r"(r[i + 4]), "+r"(r[i + 5]),
                      "+r"(r[i + 6]), "+r"(r[i + 7]) :: "memory");
}
template <int N>
__device__ __forceinline__ void tmem_ld_wait(uint32_t (&r)[N]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
  tmem_ld_tie(r);
}

// Shared-memory matrix descriptor of a K-major bf16 tile stored as rows of 128 bytes with the
// 128-byte swizzle (what TMA writes with CU_TENSOR_MAP_SWIZZLE_128B).  High word: 8-row groups are 1024
// bytes apart (stride byte offset, bits [32,46)), descriptor version 1 for sm_100 (bit 46), layout type
// SWIZZLE_128B = 2 (bits [61,64)); the leading byte offset is unused for this layout.  Low word: the start
// address in 16-byte units (bits [0,14)); advancing 16 elements along K inside the 128-byte span adds 2.
constexpr uint32_t kSmemDescHi = (1024u >> 4) | (1u << 14) | (2u << 29);
__device__ __forceinline__ uint32_t smem_desc_lo(uint32_t addr) { return (addr & 0x3FFFFu) >> 4; }
// Instruction descriptor: bf16 x bf16 -> fp32, both operands K-major, M x N tile.
__device__ __forceinline__ uint32_t make_idesc(int M, int N) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// D[tmem] = A[smem] * B[smem], bf16 x bf16 -> fp32, issued by one thread; the operands are shared-memory matrix
// descriptors given as their low words (address field), the high word is the same for every operand.
__device__ __forceinline__ void umma_step(uint32_t tmem_d, uint32_t a_lo, uint32_t b_lo, uint32_t idesc, bool accumulate) {
  asm volatile(
      "{\n\t.reg .b64 da, db;\n\t.reg .pred p;\n\t"
      "setp.ne.u32 p, %5, 0;\n\t"
      "mov.b64 da, {%1, %3};\n\tmov.b64 db, {%2, %3};\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %4, p;\n\t}"
      ::"r"(tmem_d), "r"(a_lo), "r"(b_lo), "r"(kSmemDescHi), "r"(idesc), "r"((uint32_t)accumulate) : "memory");
}
// All MMAs of one accumulator block: NK k-steps of 16 elements, four per 128-byte sub-tile (descriptor low word += 2 per
// step inside a sub-tile, += a_sub / b_sub to the next sub-tile).  The first MMA overwrites the accumulator, the others
// add to it.
template <int NK>
__device__ __forceinline__ void umma_block(uint32_t tmem_d, uint32_t a_lo, uint32_t b_lo, uint32_t a_sub, uint32_t b_sub, uint32_t idesc) {
#pragma unroll
  for (int i = 0; i < NK; ++i) umma_step(tmem_d, a_lo + (i >> 2) * a_sub + (i & 3) * 2, b_lo + (i >> 2) * b_sub + (i & 3) * 2, idesc, i > 0);
}
// One lane of a converged warp.
__device__ __forceinline__ bool elect_one() {
  uint32_t e;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(e));
  return e != 0;
}

}  // namespace sg
