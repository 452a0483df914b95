// The library's FP64 reciprocal and square root on an array of device values.
#include "cell_math.cuh"

namespace {
__global__ void k_roots(const double* x, double* r, double* s, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  r[i] = fv::recip<double>(x[i]);
  s[i] = fv::root<double>(x[i]);
}
}  // namespace

extern "C" int fp64_roots(const double* x, double* r, double* s, int n, cudaStream_t stream) {
  if (n > 0) k_roots<<<(n + 255) / 256, 256, 0, stream>>>(x, r, s, n);
  return (int)cudaGetLastError();
}
