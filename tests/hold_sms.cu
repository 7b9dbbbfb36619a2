// Other work on the GPU, for tests: blocks that take an SM's shared memory each and leave by themselves
// after a given time.

#include <cuda_runtime.h>

__global__ void k_hold(unsigned long long ns) {
  unsigned long long t0, t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
  do {
    __nanosleep(1000000);
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  } while (t - t0 < ns);
}

// Hold all but `spare` SMs for ms milliseconds (at most 20 s), on a stream of its own; returns at once.
extern "C" int hold_sms(int spare, int ms) {
  const int smem = 200 * 1024;
  int dev = 0, sms = 0;
  cudaStream_t s;
  if (ms < 0 || ms > 20000 || cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
      cudaFuncSetAttribute(k_hold, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess ||
      cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking) != cudaSuccess || spare >= sms)
    return 1;
  k_hold<<<sms - spare, 32, smem, s>>>(1000000ull * ms);
  const cudaError_t e = cudaGetLastError();
  cudaStreamDestroy(s);   // released when its work is done
  return e != cudaSuccess;
}
