// Self-test of the bounded barrier waits that the TMA kernels use: one small CTA waits, with a
// probe bound of 2^10 (about a millisecond), on a barrier that nobody ever arrives at, first in the one form and
// then in the other.  Each must give up, make the other
// threads' waits return at once, leave RECACHE_DEV_TIMEOUT (the first: and where) in its status word, take the same drain as
// the real kernels and end normally, so that the context stays usable.  Nothing here hangs or faults: the waits are
// bounded by construction.
#include "common.cuh"

namespace {

constexpr uint32_t SELFTEST_PROBES = 1u << 10;

__global__ void __launch_bounds__(64) wait_selftest_kernel(int32_t* status, int32_t* report) {
  __shared__ __align__(8) uint64_t barrier_word;
  __shared__ int abort_word, gave_up_word;
  const uint32_t bar = (uint32_t)__cvta_generic_to_shared(&barrier_word);
  volatile int* abort_flag = &abort_word;
  if (threadIdx.x == 0) {
    abort_word = gave_up_word = 0;
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(1u) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  const long long t0 = clock64();
  // warp 0 runs into the bound; warp 1 starts later and must be released by the abort flag
  if (threadIdx.x >= 32) { while (clock64() - t0 < 20000ll) { } }
  rc_mbar_wait<SELFTEST_PROBES, RC_WHERE_SELFTEST>(bar, 0u, abort_flag, status);
  const long long t1 = clock64();
  if (*abort_flag) rc_timeout_drain();
  __syncthreads();
  // the other form, as a kernel with it ends; its status word is one of its own here, as the first error wins
  volatile int* gave_up = &gave_up_word;
  const long long t2 = clock64();
  if (threadIdx.x >= 32) { while (clock64() - t2 < 20000ll) { } }
  rc_mbar_wait_small<SELFTEST_PROBES>(bar, 0u, (uint32_t)__cvta_generic_to_shared(&gave_up_word));
  if (*gave_up) {
    rc_set_status(status + 2, RECACHE_DEV_TIMEOUT);
    rc_timeout_drain();
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    const int other = atomicExch(status + 2, 0);
    report[0] = *abort_flag && *gave_up && other == RECACHE_DEV_TIMEOUT;   // 1: both gave up
    report[1] = (int32_t)min((t1 - t0) >> 10, 0x7fffffffll);   // kilo-cycles spent waiting
  }
}

}  // namespace

cudaError_t rc_launch_wait_selftest(const recache_ctx* ctx, int32_t* report, cudaStream_t st) {
  wait_selftest_kernel<<<1, 64, 0, st>>>(ctx->status, report);
  return cudaGetLastError();
}
