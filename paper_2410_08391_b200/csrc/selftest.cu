// Self-test of the bounded device-side waits: a one-block kernel waits, with a 64th of each kind's limit, for what never comes.
// Every wait must run out, the kernel must return, and the status word must read DEV_TIMEOUT, which kvp_poll_status reports as
// KVP_ERR_TIMEOUT.  The kinds: the mbarrier wait of most kernels (status word), the tagged value (word 1) and the sleeping loader
// (word 2) of the barrier-free step kernel.
#include "kvp_internal.h"
#include "step_waits.cuh"

namespace {
using namespace tcp;

__global__ void __launch_bounds__(128) wait_timeout_kernel(int* status) {
  __shared__ __align__(8) unsigned long long bar;
  __shared__ int abort_mem, abort_tag, abort_lazy;
  volatile int* abort_flag = &abort_mem;
  if (threadIdx.x == 0) {
    mbar_init(smem_u32(&bar), 1);
    *abort_flag = 0;
    abort_tag = abort_lazy = 0;
    status[1] = status[2] = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  // thread 0 plays a consumer whose producer never arrives; thread 32 a second role that watches the abort flag
  if (threadIdx.x == 0 || threadIdx.x == 32) mbar_wait(smem_u32(&bar), 0, abort_flag, status, TRY_WAIT_LIMIT / 64);
  if (threadIdx.x == 64) {       // a value whose tag never arrives: the tag would be the upper half of the first two words
    bool dead = false;
    ll_wait(reinterpret_cast<const u64*>(status), 0xffffffffu, dead, &abort_tag, status + 1, L2_POLL_LIMIT / 64);
  }
  if (threadIdx.x >= 96) lazy_wait(smem_u32(&bar), 0, &abort_lazy, status + 2, LAZY_LIMIT / 64);
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
  wait_timeout_kernel<<<1, 128, 0, (cudaStream_t)stream>>>((int*)workspace);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    h->err = std::string("kvp_selftest_wait_timeout: ") + cudaGetErrorString(e);
    return KVP_ERR_CUDA;
  }
  return KVP_OK;
}
