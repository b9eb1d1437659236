// GPU code that only the tests need.
#include <cuda_runtime.h>

#include <cstdint>

// Holds smem bytes of shared memory per block for about ns nanoseconds.
__global__ void k_hold(unsigned long long ns) {
  extern __shared__ uint8_t held[];
  unsigned long long t0, t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
  if (threadIdx.x == 0) held[0] = 1;
  do {
    __nanosleep(1000);
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  } while (t - t0 < ns);
}

// One block of k_hold per SM (two do not fit) on the stream; 0 or a CUDA error.
extern "C" int helper_hold(uint64_t smem, uint64_t ns, cudaStream_t stream) {
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e == cudaSuccess && (smem <= 114 * 1024 || ns > 1000000000ull)) e = cudaErrorInvalidValue;
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_hold, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  // the whole of the SM's shared memory, so that other kernels' blocks fit beside it
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_hold, cudaFuncAttributePreferredSharedMemoryCarveout,
                             cudaSharedmemCarveoutMaxShared);
  if (e != cudaSuccess) return (int)e;
  k_hold<<<sms, 32, smem, stream>>>(ns);
  return (int)cudaGetLastError();
}
