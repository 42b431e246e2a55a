// A block whose free is pending on one stream, and an allocation on another that needs it.
#include "common.cuh"

using namespace nne;

__global__ void busy_kernel(long long cycles, const char* block, char* seen) {
  const long long t0 = clock64();
  while (clock64() - t0 < cycles) {
  }
  *seen = *block;
}

// Two blocks of `bytes` from a pool of max_bytes: the first is freed behind `cycles` of work
// on its stream, the second allocated on another.  Returns the second allocation's error, -1
// for a failure before it, -2 if the first block's contents did not last to its free.
extern "C" int alloc_behind_free(size_t bytes, size_t max_bytes, long long cycles) {
  MemPool pool(0, max_bytes);
  if (!pool.handle()) return -1;
  PoolScope scope(&pool);
  cudaStream_t a, b;
  char *first = nullptr, *second = nullptr, *seen = nullptr, got = 0;
  if (cudaStreamCreateWithFlags(&a, cudaStreamNonBlocking) != cudaSuccess) return -1;
  if (cudaStreamCreateWithFlags(&b, cudaStreamNonBlocking) != cudaSuccess) return -1;
  if (cudaMalloc(&seen, 1) != cudaSuccess || dev_alloc(&first, bytes, a) != cudaSuccess) return -1;
  cudaMemsetAsync(first, 1, bytes, a);
  busy_kernel<<<1, 1, 0, a>>>(cycles, first, seen);
  cudaFreeAsync(first, a);
  const cudaError_t e = dev_alloc(&second, bytes, b);
  if (e == cudaSuccess) {
    cudaMemsetAsync(second, 2, bytes, b);
    cudaFreeAsync(second, b);
  }
  cudaGetLastError();
  if (cudaDeviceSynchronize() != cudaSuccess) return -1;
  cudaMemcpy(&got, seen, 1, cudaMemcpyDeviceToHost);
  cudaFree(seen);
  cudaStreamDestroy(a);
  cudaStreamDestroy(b);
  return got == 1 ? (int)e : -2;
}
