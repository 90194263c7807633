// Test hooks for the fault paths, exercised without faulting the GPU: a bounded device-side
// wait that runs out (an mbarrier that nothing arrives at) and reports through the context's
// status word, and host-side injection of workspace allocation failures.  Also the plan of a single
// call, for tests and benchmarks that name the kernel a call runs on.
#include <algorithm>

#include "ozg_context.h"
#include "ozg_device.cuh"

namespace ozg {
namespace {

// One thread waits on an mbarrier that no thread arrives at.  The wait is bounded at `limit`
// clock cycles; when it runs out the thread raises the timeout status (sticky until ozg_sync),
// as every wait of the GEMM kernels does, and the kernel returns normally.
__global__ void debug_wait_kernel(int* status, long long limit) {
  __shared__ __align__(8) uint64_t bar;
  if (threadIdx.x == 0) {
    mbar_init(&bar, 1);
    mbar_fence_init();
    const long long t0 = clock64();
    while (!mbar_try_wait(&bar, 0)) {
      if (clock64() - t0 > limit) {
        atomicExch(status, kDevTimeout);
        break;
      }
    }
  }
}

}  // namespace
}  // namespace ozg

extern "C" int ozg_debug_wait(ozg_ctx* c, long long cycles) {
  if (!c || cycles < 1000 || cycles > 4000000000ll) return OZG_ERR_INVALID;
  cudaSetDevice(c->device);
  { ozg::debug_wait_kernel<<<1, 32, 0, c->stream>>>(c->dflags, cycles); ozg::note_launch(); }
  return cudaGetLastError() == cudaSuccess ? OZG_OK : OZG_ERR_CUDA;
}

extern "C" int ozg_debug_fail_allocs(ozg_ctx* c, int n) {
  if (!c || n < 0) return OZG_ERR_INVALID;
  c->fail_allocs = n;
  return OZG_OK;
}

extern "C" int ozg_debug_single_plan(int num_sms, int cplx, int64_t m, int64_t n, int64_t k, int slices, int sel_max,
                                     int fallback, int* plan) {
  if (!plan || num_sms < 2 || m < 1 || n < 1 || k < 1 || slices < 0 || slices > OZG_MAX_SLICES) return OZG_ERR_INVALID;
  const bool autos = slices == 0;
  if (autos && (sel_max < 1 || sel_max > OZG_MAX_SLICES || fallback < 1 || fallback > OZG_MAX_SLICES)) return OZG_ERR_INVALID;
  const int64_t w = cplx ? 2 : 1;
  const int planes = autos ? std::max(sel_max, fallback) : slices;
  const ozg::host::SinglePlan P =
      ozg::host::plan_single(num_sms, cplx != 0, w * m, w * n, k, autos, autos ? std::min(sel_max, ozg::kKdMax) : slices, planes);
  plan[0] = P.kd;
  plan[1] = P.kd ? 1 : P.parts;
  plan[2] = P.part_kb;
  plan[3] = P.part_windows;
  return OZG_OK;
}
