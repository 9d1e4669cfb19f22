/*
 * argus_testing.h — test, tuning and measurement aids of the region-trace library. Not part of
 * the product ABI (argus.h): nothing here changes a result, and production callers need none
 * of it. The switches are process-wide.
 */
#ifndef ARGUS_TESTING_H_
#define ARGUS_TESTING_H_

#include "argus.h"

#ifdef __cplusplus
extern "C" {
#endif

/* argus_pair_intervals (Section 3.2, the nested region context stack per warp) with an explicit
 * kernel choice: 0 = automatic, 1 = one thread per stream (sequential stack, any input),
 * 2 = tiled kernel (CTAs walk streams tile by tile, may hand a stream on to one another, and hand
 * the markers that break the nesting to the sequential stack). Arguments, ownership and errors
 * as argus_pair_intervals; all choices produce identical output. */
int argus_pair_intervals_ex(const argus_event_t* events /*device*/, uint64_t num_events,
                            const uint64_t* stream_offsets /*device [S+1]*/,
                            uint32_t num_streams, uint32_t num_regions,
                            argus_interval_t* intervals /*device*/, uint64_t interval_capacity,
                            uint64_t* interval_offsets /*device [S+1] out*/,
                            argus_ambiguity_t* ambig /*device*/, uint64_t ambig_capacity,
                            uint64_t* ambig_offsets /*device [S+1] out*/,
                            argus_status_t* status /*device*/, void* workspace /*device*/,
                            size_t workspace_bytes, void* cuda_stream, int kernel_choice);

/* Measurement helpers (host-side bookkeeping only).
 * argus_launch_count: kernels this library has launched since it was loaded.
 * argus_profile_enable(1): from now on each operation records a CUDA event pair on its stream
 * around its dominant kernel (slot 0 = pairing kernel of argus_pair_intervals, 1 = per-stream
 * accumulation kernel of argus_aggregate, 2 = per-(pair, SM) kernel of argus_overlap, 3 = reserved).
 * argus_profile_read: waits for the recorded events, writes per slot the summed kernel time in
 * milliseconds and the number of recorded launches (arrays of 4), and forgets them. */
unsigned long long argus_launch_count(void);
void argus_profile_enable(int on);
int argus_profile_read(double* ms_total /*host [4]*/, unsigned long long* launches /*host [4]*/);

/* argus_set_synthesize_mode: where argus_synthesize aggregates and selects overlap spans: -1 automatic,
 * 1 in one pass over the intervals' digests, 2 and 3 the three plain operations. A mode the inputs do not allow falls back to the automatic choice.
 * argus_set_tile_variant: shape of the tiled pairing kernel, 0 = the default <128 threads, 5 events per
 * thread, 7 blocks per SM>, 1..3 = <192,5,4>, <64,5,8>, <256,7,2> (tiles end at other places).
 * argus_testing_set_poll_limit: polls after which a block of the tiled pairing kernel that waits for a
 * hand-over gives up with ARGUS_ERR_TIMEOUT (default 2^19, about a second; 0 restores the default). A test
 * sets it to a few polls to see the bounded wait run out and the call return with the status set.
 * argus_testing_pair_passes: after a pairing call (or argus_synthesize) in this workspace is complete, whether the
 * trace's markers were counted before pairing and whether its second pass rewrote intervals. Waits for the device.
 * argus_testing_record_blocks: blocks of this many threads (256, 192 or 128) of argus_aggregate's pass over the records that an SM holds
 * with this many regions (400 at most): as the library's choice between the three takes it, and as the device says.
 * argus_testing_set_hand_overs: 1 = a block of the tiled pairing kernel hands its stream on whenever it looks whether to, whatever the others
 * have left; 0 = the default. Results do not depend on it.
 * argus_testing_hand_overs: after a pairing call (or argus_synthesize) in this workspace is complete, how many times its two
 * passes handed a stream on. Waits for the device.
 * argus_testing_limit_requests: how many times since the library was loaded a launch needed more shared memory than a kernel gets without
 * asking, and asked for it.
 * argus_testing_hold_sms: a kernel on the stream that holds this many SMs (148 at most; 200 KB of shared memory each, so that no block of the
 * pairing kernel fits beside it) for this many microseconds (a second at most), and then ends by itself: what another stream's long
 * kernel does to a call. */
void argus_set_synthesize_mode(int mode);
void argus_set_tile_variant(int variant);
void argus_testing_set_poll_limit(unsigned int polls);
int argus_testing_pair_passes(const void* workspace /*device*/, uint32_t* counted /*host*/, uint32_t* second_pass /*host*/);
int argus_testing_record_blocks(uint32_t num_regions, uint32_t threads, uint32_t* by_rule /*host*/, uint32_t* by_device /*host*/);
void argus_testing_set_hand_overs(int always);
int argus_testing_hand_overs(const void* workspace /*device*/, uint64_t* first_pass /*host*/, uint64_t* second_pass /*host*/);
unsigned long long argus_testing_limit_requests(void);
int argus_testing_hold_sms(unsigned int sms, unsigned int microseconds, void* cuda_stream);

#ifdef __cplusplus
}
#endif
#endif /* ARGUS_TESTING_H_ */
