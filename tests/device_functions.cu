// The scalar device functions of csrc, element by element over arrays, for tests/test_gpu_device_functions.py.
#include "common.cuh"

using namespace gev;

namespace {

template <class F> __global__ void k_map(int n, F f) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) f(i);
}
template <class F> int map(int n, F f) {
  k_map<<<(n + 255) / 256, 256>>>(n, f);
  return (int)cudaDeviceSynchronize();
}

}  // namespace

extern "C" {

int t_norm_low(int n, const double* q, float* out) {
  return map(n, [=] __device__(int i) { out[i] = norm_low(q[i]); });
}

}
