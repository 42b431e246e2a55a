// The float64 bisection of complex128 states on host arrays.
#include "kernels.cuh"

using namespace nne;

// d, e: batch x n; lamf, lam: batch x r.
extern "C" int bisect64_host(int n, int r, int batch, const double* d, const double* e, const float* lamf, double* lam) {
  const size_t nb = sizeof(double) * (size_t)n * batch, rb = sizeof(double) * (size_t)r * batch;
  char* blk = nullptr;
  cudaError_t ce = cudaMalloc(&blk, 2 * nb + 2 * rb);
  double *dd = (double*)blk, *de = (double*)(blk + nb), *dl = (double*)(blk + 2 * nb);
  float* df = (float*)(blk + 2 * nb + rb);
  if (ce == cudaSuccess) ce = cudaMemcpy(dd, d, nb, cudaMemcpyHostToDevice);
  if (ce == cudaSuccess) ce = cudaMemcpy(de, e, nb, cudaMemcpyHostToDevice);
  if (ce == cudaSuccess) ce = cudaMemcpy(df, lamf, rb / 2, cudaMemcpyHostToDevice);
  if (ce == cudaSuccess) ce = bisect64(nullptr, dd, de, n, r, df, dl, batch, BISECT_C128);
  if (ce == cudaSuccess) ce = cudaMemcpy(lam, dl, rb, cudaMemcpyDeviceToHost);
  cudaFree(blk);
  return (int)ce;
}
