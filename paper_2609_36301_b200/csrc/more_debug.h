/*
 * Diagnostic entry points of libmore_route.so.  Not part of the public interface (include/more_route.h): they exist
 * for the test-suite and for the instrumented builds, and may change without notice.
 */
#ifndef MORE_DEBUG_H_
#define MORE_DEBUG_H_

#ifdef __cplusplus
extern "C" {
#endif

/*
 * more_route_debug_counters -- synchronise `stream`, copy the current device's 16 epilogue event counters to out16
 * (host) and clear them.  The kernels only maintain the counters when the library was built with -DMORE_STATS;
 * otherwise they read zero.
 */
int more_route_debug_counters(unsigned long long* out16, void* stream);

/*
 * more_debug_expire_wait -- launch a one-warp kernel that waits, with the library's bounded mbarrier wait, on a barrier
 * nobody ever arrives at, with a budget of `budget_cycles` SM clocks (a millisecond or so is plenty).  The wait runs out
 * by construction, the kernel records MORE_ERR_TIMEOUT in the device status word exactly as the router kernels would,
 * and returns normally: nothing hangs, traps or faults.  The next more_route_status() must report MORE_ERR_TIMEOUT once.
 * No TMA, no tensor memory.  Asynchronous on `stream`.
 */
int more_debug_expire_wait(long long budget_cycles, void* stream);

/*
 * more_debug_scratch_guard -- the library's cached scratch allocation carries a 256-byte guard region behind the bytes
 * the last plan asked for, filled with a pattern when the plan is made.  This call synchronises `stream` and returns 1
 * if the guard still holds the pattern, 0 if something wrote into it, or a negative MORE_ERR_* code.
 */
int more_debug_scratch_guard(void* stream);

/*
 * more_debug_scratch_bytes -- device memory, in bytes, that more_route_ex with these arguments makes the library's cached
 * scratch allocation hold (the plan for 148 SMs), or a negative MORE_ERR_* code.  Host-only; needs no device.
 */
long long more_debug_scratch_bytes(int T, int h, int r, int M, int k, int gate_mode, int want_lse, int path, int msplit);

/*
 * more_debug_chain_lists -- where the sweep's lists of such a call lie if the scratch allocation is at address `scratch` (the
 * plan for 148 SMs): out4 = address of the first area, number of areas, places of a list, bytes from one place to the next; an
 * area is places x bytes long.  MORE_ERR_SHAPE if the chain does not serve the call.  Host-only; needs no device.
 */
int more_debug_chain_lists(int T, int h, int r, int M, int k, int gate_mode, int want_lse, int msplit, unsigned long long scratch,
                           unsigned long long* out4);

/*
 * more_debug_join_lists -- the second half of a standard router whose experts are split into `parts` (2 ... 256): every part's
 * list of a token, val and id [T][parts][k] (descending, -inf where it is shorter) and mz [T][parts] = (largest logit x log2 e,
 * sum), is left in the library's scratch as the part's CTA leaves it, over a pattern, and joined by the finishing kernels.
 * Where swept [T][parts] is 0 it is left as by a CTA whose wait gave up.  Device pointers; asynchronous on `stream`.
 */
int more_debug_join_lists(int T, int M, int k, int gate_mode, int parts, const float* val, const int32_t* id, const void* mz,
                          const unsigned char* swept, int32_t* out_idx, float* out_gate, int32_t* out_counts, float* out_topval,
                          float* out_lse, void* stream);

/*
 * more_debug_psum_plan -- how more_route_psum cuts a call on its tensor-core path (148 SMs): out2 = tokens of a block, CTAs per
 * block.  Host-only; needs no device.
 */
int more_debug_psum_plan(int T, int h, int M, int* out2);

#ifdef __cplusplus
}
#endif
#endif /* MORE_DEBUG_H_ */
