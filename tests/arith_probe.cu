// Entry points for the tests of the kernels' arithmetic: each evaluates one
// device function on arrays of host memory.
#include "ba_device.cuh"
#include "ba_dfloat.cuh"

using namespace bagpu;

namespace {

// one device buffer with the inputs in front of the outputs
template <class F>
int on_device(const void* in, size_t in_bytes, void* out, size_t out_bytes, F launch) {
  char* d = nullptr;
  const size_t at = (in_bytes + 255) & ~(size_t)255;
  if (cudaMalloc(&d, at + out_bytes) != cudaSuccess) return 1;
  cudaMemcpy(d, in, in_bytes, cudaMemcpyHostToDevice);
  cudaMemset(d + at, 0, out_bytes);
  launch(d, d + at);
  const cudaError_t e = cudaMemcpy(out, d + at, out_bytes, cudaMemcpyDeviceToHost);
  cudaFree(d);
  return e == cudaSuccess && cudaGetLastError() == cudaSuccess ? 0 : 1;
}

__global__ void k_recip(const double* x, double* y, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) y[i] = recip_any(x[i]);
}

__global__ void k_sum(const dfl* ab, float* y, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) y[i] = df_sum_to_f(ab[2 * i], ab[2 * i + 1]);
}

// every binary32 significand, the low word from a hash of it: largest |b r - 1|
// of the two reciprocals (in out[0] and out[1], as the bits of a binary64)
__global__ void k_df_recip(float scale, unsigned long long* out) {
  const unsigned m = blockIdx.x * blockDim.x + threadIdx.x;
  if (m >= 1u << 23) return;
  const float hi = __int_as_float(0x3f800000u | m);
  const float lo = ldexpf((float)(int)(m * 2654435761u), -31 - 24);  // |lo| <= half an ulp of hi
  const dfl b{hi * scale, lo * scale};
  const double v = df_to_d(b);
  const dfl r[2] = {df_recip_fast(b), df_recip(b)};
  for (int i = 0; i < 2; ++i)
    atomicMax(&out[i], (unsigned long long)__double_as_longlong(fabs(fma(v, df_to_d(r[i]), -1.0))));
}

// d (3), observed (2), step (6) of n observations by one image without rotation
__global__ void k_obs_step(const float* in, float* g, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const float R[9] = {1, 0, 0, 0, 1, 0, 0, 0, 1}, intr[7] = {15625.f, 0, 0, 1e-3f, 1e-3f, 1e-3f, 1e-3f};
  const float* p = in + 11 * i;
  obs_step<float>(R, p[0], p[1], p[2], intr, p[3], p[4], 2.0f, 1.0f, p + 5, p + 8, g + 3 * i);
}

int grid(int n) { return (n + 127) / 128; }

}  // namespace

extern "C" {

int probe_recip(const double* x, double* y, int n) {
  return on_device(x, sizeof(double) * n, y, sizeof(double) * n,
                   [&](char* a, char* b) { k_recip<<<grid(n), 128>>>((double*)a, (double*)b, n); });
}

int probe_sum(const float* ab, float* y, int n) {
  return on_device(ab, 4 * sizeof(float) * n, y, sizeof(float) * n,
                   [&](char* a, char* b) { k_sum<<<grid(n), 128>>>((dfl*)a, (float*)b, n); });
}

int probe_df_recip(const float* scale, double* worst) {
  return on_device(scale, sizeof(float), worst, 2 * sizeof(double), [&](char*, char* b) {
    k_df_recip<<<grid(1 << 23), 128>>>(*scale, (unsigned long long*)b);
  });
}

int probe_obs_step(const float* in, float* g, int n) {
  return on_device(in, 11 * sizeof(float) * n, g, 3 * sizeof(float) * n,
                   [&](char* a, char* b) { k_obs_step<<<grid(n), 128>>>((float*)a, (float*)b, n); });
}

}  // extern "C"
