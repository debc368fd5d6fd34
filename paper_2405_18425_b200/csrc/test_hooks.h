/* Hooks for the library's own tests (exported from libvig_bigla.so, not part of the public C ABI:
 * include/vig_bigla.h does not declare them and applications must not call them).
 *
 * vig_test_set_kernel_preference: which kernel family the bf16 forward entry points use from now on,
 * process-wide and without any synchronisation against calls in flight on other threads.
 *   VIG_TEST_KERNEL_AUTO   the default dispatch
 *   VIG_TEST_KERNEL_SIMT   always the fp32 SIMT recurrence kernel
 *   VIG_TEST_KERNEL_CHUNK_TASKS  sequences of more than 256 tokens always take the three chunk-task launches
 *   VIG_TEST_KERNEL_SEGMENTS     sequences of 257 .. 8192 tokens always take the segmented single launch
 *   VIG_TEST_KERNEL_TCGEN05      always the tcgen05 kernels: the single-block one up to 256 tokens, chunk tasks or segments beyond
 *   VIG_TEST_KERNEL_WARP_TILES   always the kernels of one warp per 16 tokens, one block per unit or per chunk
 *   VIG_TEST_KERNEL_CLUSTERS     129 .. 1024 tokens: the blocks of up to 128 tokens of a unit always as one cluster
 * The default chooses between all of these but SIMT by head size, length and unit count.  vig_bigla_workspace_bytes follows the
 * setting: query it under the setting the call will run with.
 * Returns VIG_OK, or VIG_ERR_UNSUPPORTED for an unknown value (the setting is then unchanged). */
#ifndef VIG_TEST_HOOKS_H
#define VIG_TEST_HOOKS_H

#include <stddef.h>

#ifdef __cplusplus
extern "C" {
#endif

enum vig_test_kernel { VIG_TEST_KERNEL_AUTO = 0, VIG_TEST_KERNEL_SIMT = 2, VIG_TEST_KERNEL_CHUNK_TASKS = 3, VIG_TEST_KERNEL_SEGMENTS = 4,
                       VIG_TEST_KERNEL_TCGEN05 = 5, VIG_TEST_KERNEL_WARP_TILES = 6, VIG_TEST_KERNEL_CLUSTERS = 8 };
int vig_test_set_kernel_preference(int preference);

/* Synchronises `stream`, then returns and clears the number of (batch, head) units that the tensor-core kernels of the
 * current device handed to their in-kernel fp32 recurrence because a gate left the range of the factorised tiles
 * (negative: a vig_status error). */
int vig_test_take_fallback_count(void* stream);

/* In the next call of the forward pass (one launch for units of at most 256 tokens, the warp-tile launches beyond) or of the
 * tensor-core gradient, the blocks of the first launch wait, with a limit of a few dozen polls, on an mbarrier that nothing
 * ever completes: the bounded wait runs out within microseconds, nothing is stored, and vig_last_device_status reports
 * VIG_ERR_DEVICE_TIMEOUT.  Nothing faults and nothing spins beyond that limit.
 * vig_test_expire_next_exchange: the same for the last wait of a gradient of two chunks, the left one's for the right one's
 * sums: the gate gradients of the left chunk are not stored. */
void vig_test_expire_next_wait(void);
void vig_test_expire_next_exchange(void);

/* 1 if the host entry point would let a kernel read or write these bytes of host memory (all of them pinned and mapped,
 * both ends 16-byte aligned), 0 if it would leave them to a copy engine.  Launches nothing. */
int vig_test_host_copy_usable(const void* host, size_t bytes);

#ifdef __cplusplus
}
#endif
#endif /* VIG_TEST_HOOKS_H */
