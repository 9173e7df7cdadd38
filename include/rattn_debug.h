/*
 * rattn_debug.h -- the one extra entry point of the DEBUG build of the library
 * (librattn_dbg.so: the same sources compiled with -DRATTN_DEBUG_KNOBS; librattn.so does
 * not export it and contains none of its code).
 *
 * Every device-side wait of the kernels is bounded: when one expires the kernel raises an
 * abort flag, every role stops, the CTA frees its tensor memory and returns, and the status
 * word of the workspace reads RATTN_ERR_TIMEOUT.  That path cannot be reached by valid
 * input, so the debug build offers host-selected ways to reach it without faulting
 * anything, and its waits give up after 2^15 polls instead of 2^21:
 *   1  the tensor-core forward's first row group leaves out ONE mbarrier arrival (a plain
 *      arrive with no asynchronous copy behind it) in the first work unit of every CTA, so
 *      that a wait does run out;
 *   2  in every tensor-core kernel whose threads share named barriers, some of these threads
 *      treat their first wait as run out while the others have passed the same wait.
 *   3  rattn_forward_status finds that the scratch pool cannot be given back;
 *   4  in the chunk-state kernel alone, some of the threads that take the sums treat their wait
 *      for the last one as run out.
 * The paper has no counterpart; this exists for the failure-detection test.
 */
#ifndef RATTN_DEBUG_H_
#define RATTN_DEBUG_H_

#ifdef __cplusplus
extern "C" {
#endif

/* on = 1 .. 4: what is called from now on fails in that way; 0: normal operation.
 * Process-wide switch, host side only.  Returns RATTN_OK. */
int rattn_debug_withhold_arrival(int on);

#ifdef __cplusplus
}
#endif
#endif /* RATTN_DEBUG_H_ */
