// Bounded-wait self-test: the time-out path of the tensor-core kernels, exercised on its own.
// A warp waits with ptx::mbar_wait_warp (the routine of every role that runs warp-collective code) on an mbarrier
// that completes only after the wait has run out: lane 0 has the caller's budget and the other lanes that of the product
// kernels beyond it, and a second warp completes the barrier as soon as lane 0 has given up (it waits for that in turn with
// a limit). Lane by lane the outcomes would then differ, expired in lane 0 and complete in the others; the warp has to
// leave as one. If every lane was told that the wait failed, the kernel raises the status word exactly as the product
// kernels do in their teardown, and returns.
#include "sf_common.cuh"
#include "tc_ptx.cuh"

namespace sf {
namespace {

__global__ void __launch_bounds__(64) wait_expiry_kernel(int* status, long long budget) {
  __shared__ uint64_t bar;
  __shared__ int abort_flag;
  if (threadIdx.x == 0) {
    ptx::mbar_init(&bar, 1);
    abort_flag = 0;
    ptx::fence_mbar_init();
  }
  __syncthreads();
  volatile int* flag = &abort_flag;
  if (threadIdx.x < 32) {
    const bool ok = ptx::mbar_wait_warp(&bar, 0, flag, threadIdx.x == 0 ? budget : budget + ptx::kWaitBudgetClocks);
    if (__ballot_sync(0xFFFFFFFFu, !ok) == 0xFFFFFFFFu && threadIdx.x == 0) atomicExch(status, 1);
  } else if (threadIdx.x == 32) {
    const long long t0 = clock64();
    while (!*flag && clock64() - t0 < budget + 2 * ptx::kWaitBudgetClocks) {}
    ptx::mbar_arrive(&bar);
  }
}

}  // namespace
}  // namespace sf

extern "C" int sf_selftest_wait_expiry(void* workspace, int64_t budget_clocks, void* stream) {
  if (!workspace) return SF_ERR_NULL;
  if (budget_clocks < 1 || budget_clocks > (int64_t(1) << 31)) return SF_ERR_SHAPE;
  if (!sf::aligned16(workspace)) return SF_ERR_ALIGN;
  int st = sf::check_arch();
  if (st != SF_OK) return st;
  sf::wait_expiry_kernel<<<1, 64, 0, (cudaStream_t)stream>>>((int*)workspace, (long long)budget_clocks);
  SF_LAUNCH_CHECK();
  return SF_OK;
}
