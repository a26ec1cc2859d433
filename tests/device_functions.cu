// The scalar device functions of csrc, element by element over arrays, for tests/test_gpu_device_functions.py.
#include "common.cuh"
#include "int_sums.cuh"

using namespace gev;

namespace {

template <class F> __global__ void k_map(int n, F f) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) f(i);
}
template <int N> __device__ double row_sum(const double* v) {
  double a[N];
  for (int u = 0; u < N; ++u) a[u] = v[u];
  return sum_block(a);
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

int t_recip(int n, const double* x, double* out) {
  return map(n, [=] __device__(int i) { out[i] = recip(x[i]); });
}
int t_divide(int n, const double* x, double* out) {
  return map(n, [=] __device__(int i) { out[i] = 1.0 / x[i]; });
}
int t_recip_sqrt(int n, const double* x, double* out) {
  return map(n, [=] __device__(int i) { out[i] = recip_sqrt(x[i]); });
}
int t_rsqrt(int n, const double* x, double* out) {
  return map(n, [=] __device__(int i) { out[i] = rsqrt(x[i]); });
}
// out: n x 3, tau, beta, scale
int t_house(int n, const double* alpha, const double* xn, double* out) {
  return map(n, [=] __device__(int i) { house(alpha[i], xn[i], out[3 * i], out[3 * i + 1], out[3 * i + 2]); });
}
int t_house_cx(int n, const double* alpha, const double* xn, double* out) {
  return map(n, [=] __device__(int i) {
    zd tau, beta, scale;
    house(make_zd(alpha[2 * i], alpha[2 * i + 1]), xn[i], tau, beta, scale);
    double* o = out + 6 * i;
    o[0] = tau.x; o[1] = tau.y; o[2] = beta.x; o[3] = beta.y; o[4] = scale.x; o[5] = scale.y;
  });
}

// v: n x 20 or n x 40
int t_sum_block_20(int n, const double* v, double* out) {
  return map(n, [=] __device__(int i) { out[i] = row_sum<20>(v + 20 * i); });
}
int t_sum_block_40(int n, const double* v, double* out) {
  return map(n, [=] __device__(int i) { out[i] = row_sum<40>(v + 40 * i); });
}
int t_to_fp64(int n, const long long* acc, const float* sh, const int* e, double* out) {
  return map(n, [=] __device__(int i) { out[i] = to_fp64(acc[i], sh[i], e[i]); });
}
int t_to_fp64_fast(int n, const long long* acc, const float* sh, const int* e, double* out) {
  return map(n, [=] __device__(int i) { out[i] = to_fp64_fast(acc[i], sh[i], e[i], i & 1 ? 0xFFFFFFFFu : 0u); });
}

}
