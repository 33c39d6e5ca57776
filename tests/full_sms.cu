// Work that fills every SM for a while: three CTAs that hold 63 of its 64 warps and nearly all of its shared memory.
#include <ctime>
#include <cuda_runtime.h>

namespace {
constexpr int kThreads = 672, kShared = 72 * 1024;
cudaStream_t stream;
int *here;                                        // CTAs that have started (pinned)

__global__ void __launch_bounds__(kThreads, 3) k_full(int *started, unsigned long long ns) {
  extern __shared__ volatile unsigned char held[];
  if (threadIdx.x == 0) atomicAdd_system(started, 1);
  unsigned long long t0, t;
  asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t0));
  for (int i = 0; i < (1 << 20); ++i) {           // bounded either way
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
    if (t - t0 > ns) break;
    __nanosleep(1000);
  }
  held[threadIdx.x] = 0;
}
}  // namespace

// Fills the GPU for so many milliseconds; 1 once all of it is there.
extern "C" __attribute__((visibility("default"))) int fill(int ms) {
  int sms = 0;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, 0);
  if (!here && (cudaMallocHost(&here, sizeof(int)) != cudaSuccess || cudaStreamCreateWithFlags(&stream, cudaStreamNonBlocking) != cudaSuccess)) return -1;
  *here = 0;
  cudaFuncSetAttribute(k_full, cudaFuncAttributeMaxDynamicSharedMemorySize, kShared);
  k_full<<<3 * sms, kThreads, kShared, stream>>>(here, ms * 1000000ull);
  for (int i = 0; i < 1000 && *(volatile int *)here < 3 * sms; ++i) { timespec t{0, 10000}; nanosleep(&t, nullptr); }
  return *(volatile int *)here == 3 * sms;
}

extern "C" __attribute__((visibility("default"))) int still_full() { return cudaStreamQuery(stream) == cudaErrorNotReady; }
