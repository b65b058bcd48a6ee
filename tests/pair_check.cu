// The functions of tcw_pair.cuh over n values: out[4 n] = near_float, hi, lo (as
// double) and the reciprocal of each.
#include "tcw_pair.cuh"

__global__ void pair_kernel(const double* v, int n, double* out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  float hi, lo;
  tcw::split_float(v[i], hi, lo);
  out[4 * i] = tcw::near_float(v[i]);
  out[4 * i + 1] = hi;
  out[4 * i + 2] = lo;
  out[4 * i + 3] = tcw::reciprocal(v[i]);
}

extern "C" int pair_check(const double* v, int n, double* out) {
  pair_kernel<<<(n + 127) / 128, 128>>>(v, n, out);
  const cudaError_t e = cudaDeviceSynchronize();
  return (int)e;
}
