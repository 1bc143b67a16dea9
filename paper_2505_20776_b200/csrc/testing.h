/*
 * Entry points of the TEST library (libspecext_testing.so, built with -DSPECEXT_TESTING).  They are
 * not part of the product ABI (include/specext.h) and the product library does not export them.
 */
#ifndef SPECEXT_TESTING_H_
#define SPECEXT_TESTING_H_

#include <stdint.h>

#include "../../include/specext.h"

#ifdef __cplusplus
extern "C" {
#endif

/*
 * Forces, for every later call in the process, which attention kernel specext_verify_attn launches
 * and a lower bound on the 128-key tiles per worker:
 *   attn_kernel       : 0 = the product's choice; 1 = the CUDA-core cross-check kernel; 2 / 3 = the
 *                       one-CTA / paired-CTA tensor-core kernel (3 falls back to 2 for shapes the
 *                       paired kernel is not built for).
 *   min_tiles_per_cta : > 0 to change (fewer, longer splits).
 * Both change the workspace size: query specext_verify_attn_workspace after setting them.
 */
int specext_test_set_tuning(int32_t attn_kernel, int32_t min_tiles_per_cta);

/*
 * The form that a call takes (length_on_device: a draft call), without running it.  out[4]: the kernel
 * (2 / 3 as above), the size of its clusters or 0, the rows of Q that a CTA keeps (one-CTA kernel), the
 * key tiles per worker, rounded down.  Returns a specext_status.
 */
int specext_test_plan(const specext_attn_desc* desc, int32_t length_on_device, int32_t* out);

/*
 * Launches a one-CTA kernel that waits, with the library's bounded mbarrier wait and the given limit
 * in SM cycles, on a barrier whose last arrival never comes.  The wait must run out, the kernel must
 * OR (1 << SPECEXT_ERR_TIMEOUT) into *device_status and return normally (no trap), leaving the
 * context usable.  Returns a specext_status for the launch.
 */
int specext_test_wait_timeout(int64_t limit_cycles, int32_t* device_status, void* cuda_stream);

/*
 * Launches a kernel of one CTA that lets the kernels behind it be set up at once, runs for `cycles` SM
 * cycles (1 .. 4e9) and then stores `value` to *dst.  Returns a specext_status for the launch.
 */
int specext_test_slow_kernel(int64_t cycles, int32_t* dst, int32_t value, void* cuda_stream);

/*
 * Launches a kernel of one warp that runs the end of a role that has given up (see settle in sm100.cuh)
 * with a copy of 16 KB from `src` (16-byte aligned) on its way.  out[2] (device): the cycles it took,
 * and whether the copy had landed then.
 */
int specext_test_settle(const void* src, int64_t* out, void* cuda_stream);
int64_t specext_test_settle_cycles(void);

/* The library's limit of a bounded wait, in SM cycles. */
int64_t specext_test_wait_limit(void);

#ifdef __cplusplus
}
#endif
#endif /* SPECEXT_TESTING_H_ */
