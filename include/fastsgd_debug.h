/*
 * fastsgd_debug.h -- profiling and test aids of libfastsgd_b200.so.
 *
 * Nothing here is part of the codec (the paper has no counterpart for any of
 * it): per-kernel event timing and a launch counter for the benchmark, a way
 * for tests to shorten the kernels' bounded waits, and the byte offsets of a few
 * workspace fields that tests and the benchmark read or set.
 */
#ifndef FASTSGD_DEBUG_H
#define FASTSGD_DEBUG_H

#include <stdint.h>

#ifdef __cplusplus
extern "C" {
#endif

/* While enabled, every kernel launch is bracketed by a pair of CUDA events
 * recorded on its stream.  fastsgd_kernel_timing_read synchronises those
 * events, adds up the elapsed milliseconds and the launches per kernel (index
 * 0 abs-sum, 1 encode, 2 decode-accumulate) since the last read, and forgets
 * them.  Off by default; the events add a little launch overhead. */
int fastsgd_kernel_timing_enable(int enable);
int fastsgd_kernel_timing_read(double ms_total[3], uint64_t launches[3]);

/* number of kernels the library has launched since it was loaded */
uint64_t fastsgd_launch_count(void);

/* Iteration limits of the kernels' bounded waits, for the launches that follow:
 *   block_polls  polls of a flag, descriptor or prefix another thread block writes
 *   copy_tries   tries (about 10 us each) of a wait on a bulk copy
 *   queue_polls  polls of the decoder's queue of large groups (0xFFFFFFFF: give
 *                up at the first poll that finds the slot empty)
 * 0 restores a default.  Tests shorten them so that a wait that cannot complete
 * (a counter they have set beyond reach) ends in FASTSGD_ST_TIMEOUT within
 * milliseconds; production code never calls this. */
int fastsgd_debug_set_wait_limits(uint32_t block_polls, uint32_t copy_tries, uint32_t queue_polls);

/* Caps the number of thread blocks of the encoders' launches (fastsgd_compress,
 * _batch, _kv) that follow; 0 restores the default (as many as are resident at
 * once).  The stream never depends on the grid: tests use this to show it. */
int fastsgd_debug_set_grid(uint32_t blocks);

/* Who decodes one group, by the rules of the decoder's launch (a pure function: no GPU is used):
 *   mode        0 aggregation, 1 update as a pass of its own, 2 update in one launch, 3 the same on the packed state
 *   streams     1..8, of the launch
 *   n           entries of the gradient
 *   owned       groups of the thread block that holds the group
 *   alike_mean  keys of a group on average where most groups of the block have about as many; else 0
 *   keys, words keys of the group over all streams, 32-bit words of its blobs
 *   bulk        dense_out (mode 2: theta, m and v) is 16-byte aligned
 * Returns 0, 1, 2: one, two, four warps (several streams: by a table of keys); 3: four warps by ranks; 4: the block, entry by
 * entry (the update: or over its slice of g); 5: the block over the group's slice of dense_out; 6: the block, a group wider than that slice;
 * 7: one warp with two entries a lane in flight; -1: bad arguments. */
int fastsgd_debug_decoder_route(uint32_t mode, uint32_t streams, uint64_t n, uint32_t group_log2, uint32_t owned, uint32_t alike_mean, uint32_t keys, uint32_t words, int bulk);

/* Byte offsets inside the registered workspace (all of them in its fixed first
 * part): [0] u32 bar_count[8], arrivals (k_resident: per gradient);
 * [1] u32 ne_count[8], tiles the last encoder launch read a second time, per
 * gradient; [2] u32 error; [3] u32 tiles or groups the last encoder launch had no place for until its last step, which
 * packed them anew; [4], [5] unused; [6] u32 decoder queue slots; [7] u32 decoder queue counters[6]. */
#define FASTSGD_DEBUG_LAYOUT_FIELDS 8
int fastsgd_debug_layout(uint64_t* offsets, uint32_t count);

#ifdef __cplusplus
}
#endif
#endif /* FASTSGD_DEBUG_H */
