// Self-test of the bounded device waits used by the FFN kernels.
//
// A kernel waits on an mbarrier that nothing ever arrives at, through the
// same bounded wait (mbar_wait_warp) that the pipeline waits of the library
// use.  The wait must give up after its time budget, the kernel must report
// XS_DEV_TIMEOUT in the caller's xs_stats and return, and the CUDA context
// must stay usable.  A second wait runs out for half of the warp's lanes only:
// all of them must be told so.  No fault, trap or unbounded loop is involved.
#include <cuda_runtime.h>

#include "tc_ptx.cuh"
#include "xs_internal.cuh"

namespace xs {
namespace {

constexpr int kWaitThreads = 64;

__global__ void wait_timeout_kernel(xs_stats *stats, unsigned long long budget_ns) {
  __shared__ __align__(8) uint64_t bars[2];
  __shared__ int abort_flag;
  const uint32_t bar = ptx::smem_u32(&bars[0]), late = ptx::smem_u32(&bars[1]);
  if (threadIdx.x == 0) {
    ptx::mbar_init(bar, 1);
    ptx::mbar_init(late, 1);
    abort_flag = 0;
    ptx::fence_mbar_init();
  }
  __syncthreads();
  if (threadIdx.x < 32) {
    const uint64_t t0 = ptx::globaltimer();
    const bool ok = ptx::mbar_wait_warp(bar, 0, budget_ns, &abort_flag);
    const uint64_t waited = ptx::globaltimer() - t0;
    if (threadIdx.x == 0) {
      stats->status = ok ? XS_DEV_OK : XS_DEV_TIMEOUT;
      stats->reserved[0] = static_cast<int32_t>(waited / 1000000ull);  // milliseconds waited
      // Complete the barrier's phase so that nothing is left pending.
      ptx::mbar_arrive(bar);
    }
  }
  __syncthreads();
  // The other warp arrives after budget_ns: too late for the even lanes,
  // which gave up at half of it, in time for the odd ones.
  if (threadIdx.x < 32) {
    const bool ok = ptx::mbar_wait_warp(late, 0, threadIdx.x & 1 ? 2 * budget_ns : budget_ns / 2, &abort_flag);
    const unsigned told = __ballot_sync(0xffffffffu, ok);
    if (threadIdx.x == 0) stats->reserved[1] = __popc(told);
  } else if (threadIdx.x == 32) {
    const uint64_t t0 = ptx::globaltimer();
    while (ptx::globaltimer() - t0 < budget_ns) __nanosleep(1000);
    ptx::mbar_arrive(late);
  }
}

}  // namespace
}  // namespace xs

extern "C" int xshare_selftest_wait_timeout(xs_stats *stats, uint64_t budget_ns,
                                            xs_stream_t stream) {
  if (stats == nullptr) return XS_ERR_NULL;
  if (budget_ns == 0 || budget_ns > 2000000000ull) return XS_ERR_PARAM;
  xs::wait_timeout_kernel<<<1, xs::kWaitThreads, 0, reinterpret_cast<cudaStream_t>(stream)>>>(
      stats, static_cast<unsigned long long>(budget_ns));
  return cudaGetLastError() == cudaSuccess ? XS_OK : XS_ERR_CUDA;
}
