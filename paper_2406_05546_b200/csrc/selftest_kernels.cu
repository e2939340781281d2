// A check of the give-up path that every tensor-core kernel shares: a bounded wait on an mbarrier runs out in one of four
// warps while the other three find theirs complete, all four settle that they stop (as the warps of a kernel's write-out do
// before they exchange sums), the kernel records STATUS_WAIT_TIMEOUT in the context's status word and returns normally, and
// the host reads the word back through ps_stats().  The probe kernel touches nothing but two barriers of its own in shared
// memory: no copy is in flight, no tensor memory is held, nothing faults or hangs.
#include "kernels.h"
#include "tc5_common.cuh"

namespace psk {

namespace {

__global__ void __launch_bounds__(128) wait_timeout_probe(uint32_t* status, long long limit_cycles) {
  __shared__ uint64_t never, complete;
  __shared__ int stopped;
  if (threadIdx.x == 0) {
    mbar_init(&never, 1);                   // one arrival expected; nobody ever arrives
    mbar_init(&complete, 1);
    stopped = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    mbar_arrive(&complete);
  }
  __syncthreads();
  const bool ok = mbar_wait(threadIdx.x < 96 ? &complete : &never, 0, limit_cycles);
  if (!warps_agree<1, 128>(ok)) atomicAdd(&stopped, 1);
  __syncthreads();
  if (threadIdx.x == 0 && stopped == 128) atomicOr(status, STATUS_WAIT_TIMEOUT);
}

}  // namespace

int launch_wait_timeout_probe(uint32_t* status, long long limit_cycles, cudaStream_t st) {
  wait_timeout_probe<<<1, 128, 0, st>>>(status, limit_cycles);
  return cudaGetLastError() == cudaSuccess ? 1 : -1;
}

}  // namespace psk
