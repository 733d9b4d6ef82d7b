// selftest.cu -- exercises the bounded waits of the kernels without a fault:
// one warp waits on an mbarrier phase that nothing completes and for a
// shared-memory count that nothing adds to, each with a short limit, and
// HPD_DEVERR_TIMEOUT is recorded in the workspace error word when a wait gives
// up (for the count by the wait itself, which sets the abort word too).  The
// kernel then returns normally, so the context stays usable.
#include "common.cuh"
#include "sm100.cuh"

namespace hpd {
namespace {

using namespace sm100;

__global__ void __launch_bounds__(32, 1) wait_selftest_kernel(uint32_t *err, uint64_t limit_ns) {
  __shared__ __align__(8) uint64_t never;
  __shared__ int count, abort;
  const int lane = threadIdx.x & 31;
  if (lane == 0) {
    mbar_init(smem_u32(&never), 1);
    fence_mbar_init();
    count = 0;
    abort = 0;
  }
  __syncwarp();
  // nothing arrives: the phase with parity 0 never completes
  if (!__all_sync(0xffffffffu, mbar_wait(smem_u32(&never), 0, nullptr, limit_ns)) && lane == 0)
    flag_error(err, HPD_DEVERR_TIMEOUT);
  // nothing adds to the count: that wait gives up as well, and sets its error
  // bit and the abort word (without the one, the other does not count)
  const bool seen = __all_sync(0xffffffffu, await_count(smem_u32(&count), 1, &abort, err,
                                                        HPD_DEVERR_TIMEOUT << 8, limit_ns));
  __syncwarp();
  if (lane == 0 && (seen || *static_cast<volatile int *>(&abort) == 0))
    atomicAnd(err, ~(HPD_DEVERR_TIMEOUT << 8));
}

}  // namespace

cudaError_t launch_wait_selftest(uint32_t *err, uint64_t limit_ns, cudaStream_t s) {
  wait_selftest_kernel<<<1, 32, 0, s>>>(err, limit_ns);
  return cudaGetLastError();
}

}  // namespace hpd
