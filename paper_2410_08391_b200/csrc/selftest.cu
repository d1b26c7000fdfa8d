// Self-test of the bounded device-side waits: a one-block kernel waits on a barrier that nothing will ever complete, with a
// limit of a few thousand polls.  The wait must run out, the kernel must return, and the status word must read DEV_TIMEOUT,
// which kvp_poll_status reports as KVP_ERR_TIMEOUT.  A further warp plays a loader of the barrier-free step kernel whose slot is
// free but whose consumers have given up: its wait must say so (word 3 of the status block then reads 1).
#include "kvp_internal.h"
#include "step_waits.cuh"

namespace {
using namespace tcp;

__global__ void __launch_bounds__(96) wait_timeout_kernel(int* status, uint32_t limit) {
  __shared__ __align__(8) unsigned long long bar, free_bar;
  __shared__ int abort_mem, given_up;
  volatile int* abort_flag = &abort_mem;
  if (threadIdx.x == 0) {
    mbar_init(smem_u32(&bar), 1);
    mbar_init(smem_u32(&free_bar), 1);
    *abort_flag = 0;
    given_up = 1;
    status[1] = status[2] = status[3] = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  // thread 0 plays a consumer whose producer never arrives; thread 32 a second role that watches the abort flag
  if (threadIdx.x == 0 || threadIdx.x == 32) mbar_wait(smem_u32(&bar), 0, abort_flag, status, limit);
  if (threadIdx.x >= 64) {       // phase "minus one" of a fresh barrier counts as complete: a loader's first wait
    const bool go = lazy_wait(smem_u32(&free_bar), 1, &given_up, status + 2);
    if (threadIdx.x == 64) status[3] = go ? 2 : 1;
  }
  __syncthreads();
}
}  // namespace

extern "C" kvp_status kvp_selftest_wait_timeout(kvp_handle* h, void* workspace, void* stream) {
  if (!h || !workspace) return KVP_ERR_INVALID_ARG;
  h->err.clear();
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev != h->device) {
    cudaGetLastError();
    h->err = "current device is not the handle's device";
    return KVP_ERR_INVALID_ARG;
  }
  ++h->n_launch;
  wait_timeout_kernel<<<1, 96, 0, (cudaStream_t)stream>>>((int*)workspace, 4096u);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    h->err = std::string("kvp_selftest_wait_timeout: ") + cudaGetErrorString(e);
    return KVP_ERR_CUDA;
  }
  return KVP_OK;
}
