/*
 * smartgen_testing.h -- test and measurement hooks of libsmartgen.so.  Not part of the hot path: nothing
 * here computes anything of the method, and a production caller never needs these calls.  They exist so
 * that tests can make a bounded device-side wait run out without hanging or faulting anything, and so
 * that the benchmark can read the SM clock a scoring kernel actually ran at.  The paper has no counterpart.
 *
 * All are process-wide switches read by the next call of the named entry point on any thread.
 */
#ifndef SMARTGEN_TESTING_H_
#define SMARTGEN_TESTING_H_

#include <stdint.h>

#include "smartgen.h"

#ifdef __cplusplus
extern "C" {
#endif

/*
 * sg_testing_score_fault -- make the scoring kernel's bounded waits observable.
 *   withhold_unit   >= 0: the row statistics that pass 1 gathers for this (layer * H_kv + kv_head) unit are computed
 *                   but never handed to the warps that publish them, whose wait runs out (calls that run as one kernel: one
 *                   CTA of each of the unit's clusters does not send its own to the others); -1: off.
 *   wait_limit_ms   > 0: every bounded wait in the kernels gives up after this many milliseconds instead of about a
 *                   second; 0: the normal limit.  The time of earlier kernels does not count: a wait of the second kernel that
 *                   runs out first waits for the first kernel and then starts its limit once more.
 * A wait that gives up sets the SG_ERR_TIMEOUT bit in the call's device status word; its CTA stops taking work,
 * waits (bounded) for its own outstanding copies and MMAs, frees its tensor memory and returns.  The importance
 * array is then only partly written (and where one kernel also selects and packs, the entries and rows of the parts that
 * gave up are -1 and zero).  Nothing traps and nothing spins without a limit.
 */
void sg_testing_score_fault(int32_t withhold_unit, int32_t wait_limit_ms);

/*
 * sg_testing_score_clock -- record the clock of the scoring kernels.  dev_buffer: device memory of at least
 * sg_testing_score_grid(shape) * 32 uint64 words (NULL switches the recording off).  CTA c of the next scoring
 * kernels (of the two of a call, the later one's record stays) writes words [32c .. 32c+3] (a library built without -DSG_SCORE_PROFILE packs them as [4c .. 4c+3]):
 * clock64() at its start and end, %globaltimer (ns) at its start and end.  (end - start) cycles / nanoseconds is
 * the SM clock in GHz the kernel really ran at, which a 200 ms nvidia-smi sample cannot show for a 0.2 ms kernel.
 */
void sg_testing_score_clock(void* dev_buffer);

/* Number of CTAs of each of sg_score's launches for this shape on a 148-SM device. */
int32_t sg_testing_score_grid(const sg_shape* shape);

/* CTAs per (layer, sequence, KV head) of the kernel that scores, selects and packs in one launch, where the prefill sequences take
 * it for this shape on the current device; else 0. */
int32_t sg_testing_score_cluster(const sg_shape* shape);

/* CTAs per (sequence, KV head) of an attention call with these totals; two_lane != 0: a counted call with local_skip. */
int32_t sg_testing_decode_cluster(const sg_shape* shape, int32_t total_sel, int32_t total_loc, int32_t two_lane);

/*
 * sg_testing_decode_overlap -- allowed = 0: the following sg_sparse_decode_attn calls are launched without
 * programmatic stream serialization, i.e. fully ordered behind everything earlier in the stream, so that the
 * benchmark can report the time of a call that may not overlap its predecessor; 1 (the default) restores the
 * documented behaviour (a call overlaps the previous call up to its own output stores).
 */
void sg_testing_decode_overlap(int32_t allowed);

#ifdef __cplusplus
}
#endif
#endif /* SMARTGEN_TESTING_H_ */
