// The double-float reduction of host matrices.
#include <vector>

#include "kernels.cuh"

using namespace nne;

// H: batch x n x n complex64; d: batch x n, e: batch x n complex128 (T[k+1][k] = e[k]),
// Vh: batch x n x n complex64 (reflector j conjugated in row j).
extern "C" int tridiag_df_host(int n, int batch, const float* H, double* d, double* e, float* Vh) {
  const size_t nn = (size_t)n * n * batch, nb = (size_t)n * batch;
  char* blk = nullptr;
  const size_t sizes[] = {8 * nn, 16 * nn, 16 * nb, 256 * (size_t)batch, 8 * nb, 16 * nb, 8 * nn};
  size_t at[8] = {0};
  for (int i = 0; i < 7; ++i) at[i + 1] = at[i] + (sizes[i] + 255) / 256 * 256;
  cudaError_t ce = cudaMalloc(&blk, at[7]);
  if (ce == cudaSuccess) ce = cudaMemset(blk, 0, at[7]);
  if (ce == cudaSuccess) ce = cudaMemcpy(blk, H, 8 * nn, cudaMemcpyHostToDevice);
  if (ce == cudaSuccess)
    ce = tridiag_df(nullptr, (const cx<float>*)blk, (long long)n * n, n, (float4*)(blk + at[1]), (float4*)(blk + at[2]),
                    (float2*)(blk + at[3]), (double*)(blk + at[4]), (cx<double>*)(blk + at[5]), (cx<float>*)(blk + at[6]),
                    batch);
  if (ce == cudaSuccess) ce = cudaDeviceSynchronize();
  if (ce == cudaSuccess) ce = cudaMemcpy(d, blk + at[4], 8 * nb, cudaMemcpyDeviceToHost);
  if (ce == cudaSuccess) ce = cudaMemcpy(e, blk + at[5], 16 * nb, cudaMemcpyDeviceToHost);
  if (ce == cudaSuccess) ce = cudaMemcpy(Vh, blk + at[6], 8 * nn, cudaMemcpyDeviceToHost);
  cudaFree(blk);
  return (int)ce;
}
