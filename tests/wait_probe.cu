// Waits whose barrier nobody completes, and one whose barrier somebody does: what they return, and after how long.
#include "waits.cuh"

using namespace dslide;

// out: [0] the wait that nothing ends, [1] a wait after it, [2] the flag, [3] a completed phase; cycles: of the first two
__global__ void k_waits(int* out, long long* cycles) {
  __shared__ __align__(8) uint64_t never, done;
  __shared__ int flag;
  if (threadIdx.x == 0) {
    flag = 0;
    for (uint64_t* b : {&never, &done}) asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(tc_smem(b)) : "memory");
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(tc_smem(&done)) : "memory");
    const long long t0 = clock64();
    out[0] = tc_bar_wait(&never, 0, &flag);
    const long long t1 = clock64();
    out[1] = tc_bar_wait(&never, 0, &flag);
    cycles[0] = t1 - t0;
    cycles[1] = clock64() - t1;
    out[2] = flag;
    out[3] = tc_bar_wait(&done, 0, &flag);
  }
}

extern "C" int run_waits(int* out, long long* cycles) {      // host arrays of 4 and 2
  int* d = nullptr;
  long long* c = nullptr;
  cudaError_t e = cudaMalloc(&d, 16);
  if (e == cudaSuccess) e = cudaMalloc(&c, 16);
  if (e == cudaSuccess) {
    k_waits<<<1, 32>>>(d, c);
    e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaMemcpy(out, d, 16, cudaMemcpyDeviceToHost);
    if (e == cudaSuccess) e = cudaMemcpy(cycles, c, 16, cudaMemcpyDeviceToHost);
  }
  cudaFree(d);
  cudaFree(c);
  return (int)e;
}
