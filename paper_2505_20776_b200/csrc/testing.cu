// Kernels and entry points that exist only in the test library (see testing.h).
#ifdef SPECEXT_TESTING
#include "common.cuh"
#include "sm100.cuh"
#include "testing.h"

namespace {

// The waiting path of the attention kernels, exercised in isolation: a barrier that expects two
// arrivals gets one, so the phase never completes and the bounded wait has to give up.
__global__ void __launch_bounds__(32) wait_timeout_kernel(long long limit_cycles, int32_t* status) {
  __shared__ uint64_t bar;
  __shared__ int abort_flag;
  if (threadIdx.x == 0) {
    abort_flag = 0;
    sm100::mbar_init(&bar, 2);
    sm100::fence_mbar_init();
  }
  __syncwarp();
  if (threadIdx.x == 0) sm100::mbar_arrive(&bar);
  __syncwarp();
  const bool ok = sm100::mbar_wait(&bar, 0, &abort_flag, limit_cycles);
  if (!ok && threadIdx.x == 0) spx_raise(status, SPECEXT_ERR_TIMEOUT);
}

// A kernel that lets its dependents be set up at once and then takes its time, as one of another library may: at its end it
// writes `value` to *dst.  It ends by itself after `cycles`.
__global__ void __launch_bounds__(32) slow_kernel(long long cycles, int32_t* dst, int32_t value) {
  sm100::pdl_launch_dependents();
  if (threadIdx.x != 0) return;
  const long long t0 = clock64();
  while (clock64() - t0 < cycles) __nanosleep(1000);
  *dst = value;
}

// The end of a role that gives up while a copy is on its way.  out: the cycles it took and whether the copy had landed then.
__global__ void __launch_bounds__(32) settle_kernel(const unsigned char* src, long long* out) {
  __shared__ __align__(128) unsigned char dst[16384];
  __shared__ uint64_t bar;
  if (threadIdx.x != 0) return;
  sm100::mbar_init(&bar, 1);
  sm100::fence_mbar_init();
  sm100::mbar_arrive_expect_tx(&bar, sizeof(dst));
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               ::"r"(sm100::smem_u32(dst)), "l"(src), "r"((uint32_t)sizeof(dst)), "r"(sm100::smem_u32(&bar))
               : "memory");
  const long long t0 = clock64();
  sm100::settle();
  out[0] = clock64() - t0;
  out[1] = sm100::mbar_test_wait(&bar, 0);
}

}  // namespace

extern "C" int specext_test_settle(const void* src, int64_t* out, void* cuda_stream) {
  if (!src || !out || (reinterpret_cast<uintptr_t>(src) & 15u) != 0) return SPECEXT_ERR_INVALID_ARG;
  settle_kernel<<<1, 32, 0, static_cast<cudaStream_t>(cuda_stream)>>>(static_cast<const unsigned char*>(src),
                                                                     reinterpret_cast<long long*>(out));
  if (cudaGetLastError() != cudaSuccess) return SPECEXT_ERR_CUDA;
  return SPECEXT_OK;
}

extern "C" int64_t specext_test_settle_cycles(void) { return sm100::kSettleCycles; }

extern "C" int specext_test_slow_kernel(int64_t cycles, int32_t* dst, int32_t value, void* cuda_stream) {
  if (!dst || cycles < 1 || cycles > 4000000000ll) return SPECEXT_ERR_INVALID_ARG;
  slow_kernel<<<1, 32, 0, static_cast<cudaStream_t>(cuda_stream)>>>((long long)cycles, dst, value);
  if (cudaGetLastError() != cudaSuccess) return SPECEXT_ERR_CUDA;
  return SPECEXT_OK;
}

extern "C" int64_t specext_test_wait_limit(void) { return sm100::kWaitLimitCycles; }

extern "C" int specext_test_wait_timeout(int64_t limit_cycles, int32_t* device_status, void* cuda_stream) {
  if (!device_status || limit_cycles < 1 || limit_cycles > 4000000000ll) return SPECEXT_ERR_INVALID_ARG;
  wait_timeout_kernel<<<1, 32, 0, static_cast<cudaStream_t>(cuda_stream)>>>((long long)limit_cycles, device_status);
  if (cudaGetLastError() != cudaSuccess) return SPECEXT_ERR_CUDA;
  return SPECEXT_OK;
}
#endif  // SPECEXT_TESTING
