// The reciprocals and reciprocal square roots of recip.cuh and df.cuh on arrays.
#include "df.cuh"
#include "recip.cuh"

using namespace nne;

// which: 0 1/x and 1 1/sqrt(x) in float64, 2 1/sqrt(x) in float32, 3 1/sqrt(x) and 4 1/x in
// double-float (x and y hold hi and lo of each value).
__global__ void recip_kernel(int which, int n, const double* x, double* y) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    if (which == 0) y[i] = rcp_series(x[i]);
    else if (which == 1) y[i] = rsqrt_series(x[i]);
    else if (which == 2) y[i] = (double)rsqrt_series((float)x[i]);
    else {
      const float2 v = make_float2((float)x[2 * i], (float)x[2 * i + 1]);
      const float2 w = which == 3 ? df_rsqrt(v) : df_rcp(v);
      y[2 * i] = w.x;
      y[2 * i + 1] = w.y;
    }
  }
}

extern "C" int recip_host(int which, int n, const double* x, double* y) {
  const size_t b = sizeof(double) * (size_t)n * (which > 2 ? 2 : 1);
  double* d = nullptr;
  cudaError_t ce = cudaMalloc(&d, 2 * b);
  if (ce == cudaSuccess) ce = cudaMemcpy(d, x, b, cudaMemcpyHostToDevice);
  if (ce == cudaSuccess) {
    recip_kernel<<<256, 256>>>(which, n, d, d + b / sizeof(double));
    ce = cudaGetLastError();
  }
  if (ce == cudaSuccess) ce = cudaMemcpy(y, d + b / sizeof(double), b, cudaMemcpyDeviceToHost);
  cudaFree(d);
  return (int)ce;
}
