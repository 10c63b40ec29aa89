// The scalar device functions of frkc2_math.cuh over arrays, for test_gpu_math.py.
#include "frkc2_math.cuh"

using namespace frkc2;

__global__ void k_roots(const double* a, double* s, double* r, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) {
    s[i] = sqrt_h3(a[i]);
    r[i] = rsqrt_h3(a[i]);
  }
}

__global__ void k_kappa64(const double* x, const double* y, double c, double* kr, double* ki, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) kappa_power25_fast<double>(x[i], y[i], c, kr[i], ki[i]);
}

__global__ void k_kappa32(const float* x, const float* y, float c, float* kr, float* ki, int pairs) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= pairs) return;
  float2 r, m;
  kappa25_pair(make_float2(x[2 * i], x[2 * i + 1]), make_float2(y[2 * i], y[2 * i + 1]), c * 0.70710678118654752440f, r, m);
  kr[2 * i] = r.x;
  kr[2 * i + 1] = r.y;
  ki[2 * i] = m.x;
  ki[2 * i + 1] = m.y;
}

__global__ void k_kappa_mixed(const float* x, const float* y, float c, float* kr, float* ki, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) kappa_power25_mixed(x[i], y[i], c, kr[i], ki[i]);
}

__global__ void k_convert(const double* d, const float* f, float* nd, double* wf, unsigned char* slow, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  bool a = false, b = false;
  nd[i] = narrow_fast(d[i], a);
  wf[i] = widen_fast(f[i], b);
  slow[i] = (a ? 1 : 0) + (b ? 2 : 0);
}

extern "C" {
int run_roots(const double* a, double* s, double* r, int n) {
  k_roots<<<(n + 255) / 256, 256>>>(a, s, r, n);
  return cudaDeviceSynchronize();
}
int run_kappa64(const double* x, const double* y, double c, double* kr, double* ki, int n) {
  k_kappa64<<<(n + 255) / 256, 256>>>(x, y, c, kr, ki, n);
  return cudaDeviceSynchronize();
}
int run_kappa32(const float* x, const float* y, float c, float* kr, float* ki, int n) {  // n even
  k_kappa32<<<(n / 2 + 255) / 256, 256>>>(x, y, c, kr, ki, n / 2);
  return cudaDeviceSynchronize();
}
int run_kappa_mixed(const float* x, const float* y, float c, float* kr, float* ki, int n) {
  k_kappa_mixed<<<(n + 255) / 256, 256>>>(x, y, c, kr, ki, n);
  return cudaDeviceSynchronize();
}
int run_convert(const double* d, const float* f, float* nd, double* wf, unsigned char* slow, int n) {
  k_convert<<<(n + 255) / 256, 256>>>(d, f, nd, wf, slow, n);
  return cudaDeviceSynchronize();
}
}
