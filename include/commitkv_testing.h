/*
 * commitkv_testing.h — test support of libcommitkv.so (not part of the hot
 * path).
 *
 * The greedy joint test (Section 3.3, Eq. 11) runs as one cooperative kernel
 * whose blocks meet at a grid barrier once per candidate; every wait at that
 * barrier is bounded (about one second), after which the kernel records
 * COMMITKV_ERR_TIMEOUT in the workspace status word and returns, leaving the
 * CUDA context usable.  This entry point makes that wait run out on purpose:
 * it launches `blocks` blocks at the same barrier code but tells it to
 * expect blocks + 1 arrivals, so the wait can only end by its limit.
 *
 *   workspace  an initialised CommitKV workspace (>= 256 bytes).
 *   blocks     1..64 co-resident blocks.
 * Returns COMMITKV_OK if the kernel was launched; the timeout is then read
 * with commitkv_workspace_status (expected: COMMITKV_ERR_TIMEOUT).
 */
#ifndef COMMITKV_TESTING_H
#define COMMITKV_TESTING_H

#include "commitkv.h"

#ifdef __cplusplus
extern "C" {
#endif

commitkv_status commitkv_test_barrier_timeout(void *workspace, size_t workspace_bytes,
                                              int32_t blocks, cudaStream_t stream);

/*
 * What the last scoring launch on this workspace left to its page passes:
 * pages_out[0] and pages_out[1] (host) receive the (row tile, page) pairs
 * that the two list passes of the pruned page pass scored, both 0 where the
 * full page pass ran.  Waits for the stream.
 */
commitkv_status commitkv_test_pruned_pages(const void *workspace, size_t workspace_bytes, uint64_t *pages_out,
                                           cudaStream_t stream);

/* Kernels that the calling thread's calls have launched so far (a counter per
 * thread, which nothing else reads). */
uint64_t commitkv_test_launches(void);

#ifdef __cplusplus
}
#endif

#endif /* COMMITKV_TESTING_H */
