// Device arithmetic of lbm_math.cuh and lbm_exptab.cuh beside CUDA's own functions,
// for the GPU tests.  Buffers are host arrays of n values.
#include "lbm_math.cuh"

using namespace lbm;

__global__ void rcp32(const float* x, float* got, float* want, int n) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= n) return;
  got[k] = vrcp(x[k]);
  want[k] = __frcp_rn(x[k]);
}
__global__ void rcp64(const double* x, double* got, double* want, int n) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= n) return;
  got[k] = vrcp(x[k]);
  want[k] = __drcp_rn(x[k]);
}
__global__ void exp64(const double* x, double* got, double* want, int n, int one_minus) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= n) return;
  if (!exp_arg_ok(x[k])) {
    got[k] = want[k] = -1.0;
    return;
  }
  got[k] = one_minus ? exp_neg_table<true>(x[k]) : exp_neg_table<false>(x[k]);
  want[k] = one_minus ? -expm1(-x[k]) : exp(-x[k]);
}

template <typename T, typename Launch>
static int run(const T* x, T* got, T* want, int n, Launch launch) {
  T* d = nullptr;
  cudaError_t e = cudaMalloc(&d, 3 * sizeof(T) * (size_t)n);
  if (e != cudaSuccess) return (int)e;
  cudaMemcpy(d, x, sizeof(T) * (size_t)n, cudaMemcpyHostToDevice);
  launch(d, d + n, d + 2 * (size_t)n, (n + 255) / 256);
  e = cudaGetLastError();
  if (e == cudaSuccess) e = cudaMemcpy(got, d + n, sizeof(T) * (size_t)n, cudaMemcpyDeviceToHost);
  if (e == cudaSuccess) e = cudaMemcpy(want, d + 2 * (size_t)n, sizeof(T) * (size_t)n, cudaMemcpyDeviceToHost);
  cudaFree(d);
  return (int)e;
}
extern "C" int run_rcp32(const float* x, float* got, float* want, int n) {
  return run(x, got, want, n, [=](float* a, float* b, float* c, int g) { rcp32<<<g, 256>>>(a, b, c, n); });
}
extern "C" int run_rcp64(const double* x, double* got, double* want, int n) {
  return run(x, got, want, n, [=](double* a, double* b, double* c, int g) { rcp64<<<g, 256>>>(a, b, c, n); });
}
extern "C" int run_exp64(const double* x, double* got, double* want, int n, int one_minus) {
  return run(x, got, want, n, [=](double* a, double* b, double* c, int g) { exp64<<<g, 256>>>(a, b, c, n, one_minus); });
}
