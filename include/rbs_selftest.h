/*
 * rbs_selftest.h -- operational self-tests of the RBS prefill library (no counterpart in the paper).
 *
 * These entry points exercise the library's own safety machinery without disturbing the GPU: nothing here
 * faults, traps or spins without a limit.
 */
#ifndef RBS_SELFTEST_H_
#define RBS_SELFTEST_H_

#include "rbs.h"

#ifdef __cplusplus
extern "C" {
#endif

/*
 * Host only, needs no GPU.  Checks the table through which per-device values (the device address of the
 * status word, the SM count) are looked up once per device and never shared between devices, using a fake
 * lookup.  Returns 0 when every check passes, otherwise the number of the first failed check.
 */
RBS_API int rbs_selftest_device_table(void);

/*
 * Host only, needs no GPU.  The number of kernels that rbs_select (n_q_tokens = seqlen) or rbs_select_chunk launches for
 * this shape: 2 where the scoring kernel turns its counts into densities itself (short calls at blocks of 64 and 128),
 * else 3; 0 for a shape that is refused.
 */
RBS_API int rbs_selftest_select_launches(const rbs_shape* shape, int n_q_tokens);

/*
 * Launches one single-thread CTA on `stream` that waits, with the library's bounded mbarrier wait, on a barrier
 * that nothing ever arrives on, with `spin_limit` probes (1 .. 65536) instead of the production limit.  The wait
 * runs out, records its code in the device status word and the kernel returns normally: afterwards
 * rbs_device_status() reports RBS_ERR_TIMEOUT until cleared, *gave_up (device, one uint32) is 1, and the CUDA
 * context is fully usable.  Returns RBS_ERR_INVALID_ARG for a null pointer or a limit outside the range.
 */
RBS_API rbs_status rbs_selftest_wait_timeout(unsigned int spin_limit, unsigned int* gave_up, void* stream);

/*
 * Launches one warp on `stream` that runs the attention kernel's two forms of the bounded wait, with 1,024 probes each
 * (about 4 ms), on a barrier whose phase is complete and on one that nothing arrives on.  answers (device, four
 * uint32): the lanes that saw the first barrier (all of them) and the second (none), then the same two answers of one
 * lane waiting alone (1, 0).  Afterwards rbs_device_status() reports RBS_ERR_TIMEOUT until cleared, and the CUDA context
 * is fully usable.  Returns RBS_ERR_INVALID_ARG for a null pointer.
 */
RBS_API rbs_status rbs_selftest_warp_wait(unsigned int* answers, void* stream);

/*
 * Debug build only (the library compiled with -DRBS_DEBUG; rbs_version() says "debug checks"): launches one thread
 * on `stream` that runs one of the kernels' index checks with an index equal to its bound.  The check fails, records
 * 0x100 + 0xff in the device status word and the guarded access is skipped: afterwards *skipped (device, one
 * uint32) is 1, rbs_device_status() reports RBS_ERR_DEBUG_CHECK until cleared, and the CUDA context is fully usable
 * (nothing traps or faults).  The release build has no such checks and returns RBS_ERR_UNSUPPORTED without a launch.
 */
RBS_API rbs_status rbs_selftest_debug_check(unsigned int* skipped, void* stream);

/*
 * Debug build only: makes one wait of the attention kernel run out in every thread block of the attention calls that
 * follow.  Softmax warp `warp` (0 .. 15; negative: no wait any more) does its wait of the kind `which` (0: the next tile's
 * announcement, 1: S of a step, 2: P free, 3: O before it is rescaled, 4: O of a tile) that has `before` waits of that
 * kind in front of it on a barrier that nothing arrives on, with 64 probes.  Such a call ends within seconds with its
 * outputs undefined and code 7 in the status word; nothing traps or faults, and once the switch is back at -1 and the
 * word cleared, calls are as before.  Synchronous; not for use beside running attention calls.  The release build
 * returns RBS_ERR_UNSUPPORTED.
 */
RBS_API rbs_status rbs_selftest_attention_wait(int warp, int which, int before);

/*
 * Debug build only: the same for the selections that follow: epilogue warp `warp` (0 .. 15; negative: none any more) of the
 * two-head scoring kernel does its wait for an accumulator that has `before` such waits in front of it on a barrier that
 * nothing arrives on, with 64 probes.
 */
RBS_API rbs_status rbs_selftest_select_wait(int warp, int before);

#ifdef __cplusplus
}
#endif
#endif /* RBS_SELFTEST_H_ */
