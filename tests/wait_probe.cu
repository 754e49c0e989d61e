// Waits whose barrier nobody completes, and one whose barrier somebody does: what they return, and after how long.
#include "waits.cuh"

using namespace dslide;

__device__ __forceinline__ void init_bar(uint64_t* b) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(tc_smem(b)) : "memory");
}

// out: [0] the wait that nothing ends, [1] a wait after it, [2] the flag, [3] a completed phase; cycles: of the first two
__global__ void k_waits(int* out, long long* cycles) {
  __shared__ __align__(8) uint64_t never, done;
  __shared__ int flag;
  if (threadIdx.x == 0) {
    flag = 0;
    init_bar(&never);
    init_bar(&done);
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(tc_smem(&done)) : "memory");
    const long long t0 = clock64();
    out[0] = tc_bar_wait<false>(&never, 0, &flag);
    const long long t1 = clock64();
    out[1] = tc_bar_wait<false>(&never, 0, &flag);
    cycles[0] = t1 - t0;
    cycles[1] = clock64() - t1;
    out[2] = flag;
    out[3] = tc_bar_wait<false>(&done, 0, &flag);
  }
}

// Two blocks of a cluster: the first waits for what nobody completes, the second learns of it.  out: [0] the first's wait, [1] the
// first's flag, [2] the second's flag, [3] the second's wait after that; cycles: [0] the second's wait, [1] a drain in the first
__global__ void __cluster_dims__(2, 1, 1) k_pair(int* out, long long* cycles) {
  __shared__ __align__(8) uint64_t never;
  __shared__ int flag;
  if (threadIdx.x == 0) { flag = 0; init_bar(&never); }
  asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
  if (threadIdx.x == 0 && blockIdx.x == 0) {
    out[0] = tc_bar_wait<true>(&never, 0, &flag);
    out[1] = flag;
    const long long t0 = clock64();
    tc_bar_drain(&never, 0, t0 + DRAIN_CYCLES);
    cycles[1] = clock64() - t0;
  }
  if (threadIdx.x == 0 && blockIdx.x == 1) {
    const long long t0 = clock64();
    while (*(volatile int*)&flag == 0 && clock64() - t0 < 2 * WAIT_CYCLES) __nanosleep(1000);
    out[2] = *(volatile int*)&flag;
    const long long t1 = clock64();
    out[3] = tc_bar_wait<true>(&never, 0, &flag);
    cycles[0] = clock64() - t1;
  }
  asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}

// A warp whose block has given up waits, half of its lanes for a phase that has completed and half for one that nobody completes: all
// lanes get the same answer, and one of them is elected after it.  Then all for the completed one, with the flag set.
// out: [0] lanes told that the mixed phase has completed, [1] lanes elected after it, [2] and [3] the same of the second wait
__global__ void k_warp(int* out, long long* cycles) {
  __shared__ __align__(8) uint64_t never, done;
  __shared__ int flag;
  if (threadIdx.x == 0) {
    flag = 1;
    init_bar(&never);
    init_bar(&done);
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(tc_smem(&done)) : "memory");
  }
  __syncthreads();
  const long long t0 = clock64();
  for (int i = 0; i < 2; ++i) {
    const bool ok = tc_bar_wait_warp<false>(i == 0 && (threadIdx.x & 1) ? &never : &done, 0, &flag);
    uint32_t one;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(one));
    const int told = __popc(__ballot_sync(0xffffffffu, ok)), elected = __popc(__ballot_sync(0xffffffffu, one != 0u));
    if (threadIdx.x == 0) { out[2 * i] = told; out[2 * i + 1] = elected; }
    if (threadIdx.x == 0) cycles[i] = clock64() - t0;
  }
}

// The same of a wait without a flag, whose lanes give up by the clock.  out: [0] lanes told that the mixed phase has completed, [1] that
// the completed one has; cycles: of the first
__global__ void k_warp_limited(int* out, long long* cycles) {
  __shared__ __align__(8) uint64_t never, done;
  if (threadIdx.x == 0) {
    init_bar(&never);
    init_bar(&done);
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(tc_smem(&done)) : "memory");
  }
  __syncthreads();
  const long long t0 = clock64();
  for (int i = 0; i < 2; ++i) {
    const bool ok = bar_wait_limited_warp(i == 0 && (threadIdx.x & 1) ? &never : &done, 0);
    const int told = __popc(__ballot_sync(0xffffffffu, ok));
    if (threadIdx.x == 0) { out[i] = told; cycles[i] = clock64() - t0; }
  }
}

extern "C" int run_waits(int which, int* out, long long* cycles) {      // host arrays of 4 and 2
  int* d = nullptr;
  long long* c = nullptr;
  cudaError_t e = cudaMalloc(&d, 16);
  if (e == cudaSuccess) e = cudaMalloc(&c, 16);
  if (e == cudaSuccess) {
    if (which == 3) k_warp_limited<<<1, 32>>>(d, c);
    else if (which == 2) k_warp<<<1, 32>>>(d, c);
    else if (which == 1) k_pair<<<2, 32>>>(d, c);
    else k_waits<<<1, 32>>>(d, c);
    e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaMemcpy(out, d, 16, cudaMemcpyDeviceToHost);
    if (e == cudaSuccess) e = cudaMemcpy(cycles, c, 16, cudaMemcpyDeviceToHost);
  }
  cudaFree(d);
  cudaFree(c);
  return (int)e;
}
