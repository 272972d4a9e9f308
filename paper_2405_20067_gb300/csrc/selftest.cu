// selftest.cu -- failure-detection self-test of the bounded device waits
// (ndg_selftest_timeout): one CTA waits on an mbarrier that nothing ever
// completes, with the same wait helpers as the tensor-core kernels.  When
// the bound runs out the CTA records NDG_ERR_TIMEOUT in the workspace status
// word and returns, so the context stays usable; nothing faults or traps.
// And the preparation's FP64 functions beside CUDA's (ndg_selftest_math).
#include <cuda_runtime.h>

#include "common.cuh"
#include "internal.h"
#include "kernels.h"
#include "prep_math.cuh"
#include "tcgen05.cuh"

namespace ndg {

__device__ __forceinline__ unsigned long long selftest_ns() {
  unsigned long long v;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(v));
  return v;
}

// which = 0: the roles' waits, a warp's (warp_wait) by warp 0 and the issuer's
// (lane_wait) by a lane of warp 1 at the same time; which = 1: the spinning
// wait of the kernels' final drain (mbar_wait_bounded, kWaitLimit polls).  The
// timeout is recorded if every wait ran out, none of them within 0.2 s (a
// shorter bound would end kernels that are only delayed).
__global__ void selftest_wait_kernel(int* status, int which) {
  __shared__ uint64_t bar;
  __shared__ int abort_flag, good;
  if (threadIdx.x == 0) {
    mbar_init(&bar, 1);  // one arrival expected; none is ever made
    abort_flag = 0;
    good = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  const unsigned long long t0 = selftest_ns();
  bool ok = true;
  if (threadIdx.x < 32) {
    if (which == 0) {
      ok = warp_wait(&bar, 0, &abort_flag);
    } else {
      int r = 1;
      if (threadIdx.x == 0) r = mbar_wait_bounded(&bar, 0, kWaitLimit) ? 1 : 0;
      ok = __shfl_sync(0xffffffffu, r, 0) != 0;
    }
  } else if (which == 0) {
    int r = 1;
    if (threadIdx.x == 32) r = lane_wait(&bar, 0, &abort_flag) ? 1 : 0;
    ok = __shfl_sync(0xffffffffu, r, 0) != 0;
  }
  const bool waited = which == 0 || threadIdx.x < 32;
  if ((threadIdx.x & 31) == 0 && (!waited || (!ok && selftest_ns() - t0 >= 200000000ull)))
    atomicAdd(&good, 1);
  __syncthreads();
  if (threadIdx.x == 0 && good == 2 && status) set_status(status, NDG_ERR_TIMEOUT);
}

int launch_selftest_wait(int* status, int which, cudaStream_t s) {
  selftest_wait_kernel<<<1, 64, 0, s>>>(status, which);
  return 1;
}

// Functions as in prep_math.cuh; arguments of 0 to 2 are rounded to FP32.
__global__ void selftest_math_kernel(int which, long long n, const double* __restrict__ a,
                                     const double* __restrict__ b, double* __restrict__ own,
                                     double* __restrict__ cuda) {
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x) {
    const float v = (float)a[i];
    if (which == 0) {
      own[i] = exp_f32(v);
      cuda[i] = exp((double)v);
    } else if (which == 1) {
      own[i] = sigmoid(v);
      cuda[i] = 1.0 / (1.0 + exp(-(double)v));
    } else if (which == 2) {
      own[i] = off_diagonal(v);
      cuda[i] = 2.0 / (1.0 + exp(-(double)v)) - 1.0;
    } else {
      own[i] = quotient(a[i], b[i], 1.0 / b[i]);
      cuda[i] = a[i] / b[i];
    }
  }
}

int launch_selftest_math(int which, long long n, const double* a, const double* b, double* own,
                         double* cuda, cudaStream_t s) {
  if (n <= 0) return 0;
  const long long blocks = ceil_div<long long>(n, 256);
  selftest_math_kernel<<<(unsigned)(blocks < 4096 ? blocks : 4096), 256, 0, s>>>(which, n, a, b, own, cuda);
  return 1;
}

}  // namespace ndg
