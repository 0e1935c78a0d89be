// selftest.cu -- a bounded device wait that runs out is counted and reported to the
// host, and the device stays usable. The probe stands for itself: no kernel of the
// solver waits on a copy or on another block.
#include "../../include/reg.h"
#include "internal.h"

namespace reg {
namespace {

__device__ int g_timeouts;

__device__ __forceinline__ unsigned smem_addr(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t* bar, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(smem_addr(bar)), "r"(count) : "memory");
}
// wait for the phase with parity `parity`; false when the bound runs out
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, unsigned parity, int tries = 1 << 20) {
  for (int i = 0; i < tries; ++i) {
    unsigned done;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(smem_addr(bar)), "r"(parity)
        : "memory");
    if (done) return true;
  }
  return false;
}
// Failure-path check: one block waits on an mbarrier that nothing completes,
// gives up after `tries` polls and counts the timeout.
__global__ void k_wait_timeout_probe(int tries) {
  __shared__ __align__(8) uint64_t bar;
  if (threadIdx.x == 0) {
    mbar_init(&bar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  __syncthreads();
  if (!__syncthreads_and(mbar_wait(&bar, 0, tries)) && threadIdx.x == 0) atomicAdd(&g_timeouts, 1);
}

}  // namespace
}  // namespace reg

extern "C" reg_status reg_selftest_copy_timeout(int* counted) {
  if (!counted) return REG_EINVAL;
  try {
    reg::k_wait_timeout_probe<<<1, 32>>>(1 << 12);
    REG_CUDA(cudaGetLastError());
    REG_CUDA(cudaDeviceSynchronize());
    REG_CUDA(cudaMemcpyFromSymbol(counted, reg::g_timeouts, sizeof(int)));
    const int zero = 0;
    REG_CUDA(cudaMemcpyToSymbol(reg::g_timeouts, &zero, sizeof(int)));
  } catch (const reg::CudaError& e) {
    reg::set_thread_error(e.what);
    return REG_ECUDA;
  }
  return REG_OK;
}
