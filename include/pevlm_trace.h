/*
 * pevlm_trace.h -- optional tracing facility of libpevlm.so (not part of the product ABI).
 *
 * A library built with -DPEVLM_TRACE (PEVLM_TRACE=1 python -m paper_2506_19651_b200.build --force) adds up, for the
 * first pair of thread blocks of a launch of the attention kernel, the clock64 cycles that every warp spends in each
 * kind of barrier wait, and exports the read-back call below; `python -m paper_2506_19651_b200.timeline` prints the
 * table.  A library built without the flag has neither the accounting nor this symbol.
 */
#ifndef PEVLM_TRACE_H_
#define PEVLM_TRACE_H_
#ifdef __cplusplus
extern "C" {
#endif

/* host_out: 2 x 16 x 32 words, [thread block][warp][wait id]; id 0 holds the cycles of the warp's whole role, id 1 the
 * key tiles a softmax warp handled, ids from 11 on are those of a reported timeout.  Returns 0 or -1. */
int pevlm_debug_waits(unsigned* host_out);

#ifdef __cplusplus
}
#endif
#endif /* PEVLM_TRACE_H_ */
