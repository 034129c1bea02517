// Device arithmetic of csrc/kernels.cuh and csrc/resident_blocks.cuh for the GPU
// tests: out[k] = f(in[k]), host arrays in and out.
#include "../paper_1711_10579_gb300/csrc/resident_blocks.cuh"

__global__ void k_recip(const double* in, double* out, double* div, int n) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k < n) {
    out[k] = pf::recip(in[k]);
    div[k] = 1.0 / in[k];
  }
}

__global__ void k_narrow(const double* in, float* out, int n) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k < n) out[k] = pf::narrow<float>(in[k]);
}

extern "C" int arith_recip(const double* in, double* out, double* div, int n) {
  double *d = nullptr, *r = nullptr, *q = nullptr;
  const size_t bytes = sizeof(double) * (size_t)n;
  cudaError_t e = cudaMalloc(&d, bytes);
  if (e == cudaSuccess) e = cudaMalloc(&r, bytes);
  if (e == cudaSuccess) e = cudaMalloc(&q, bytes);
  if (e == cudaSuccess) e = cudaMemcpy(d, in, bytes, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) {
    k_recip<<<(n + 255) / 256, 256>>>(d, r, q, n);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaMemcpy(out, r, bytes, cudaMemcpyDeviceToHost);
  if (e == cudaSuccess) e = cudaMemcpy(div, q, bytes, cudaMemcpyDeviceToHost);
  cudaFree(d);
  cudaFree(r);
  cudaFree(q);
  return (int)e;
}

extern "C" int arith_narrow(const double* in, float* out, int n) {
  double* d = nullptr;
  float* r = nullptr;
  cudaError_t e = cudaMalloc(&d, sizeof(double) * (size_t)n);
  if (e == cudaSuccess) e = cudaMalloc(&r, sizeof(float) * (size_t)n);
  if (e == cudaSuccess) e = cudaMemcpy(d, in, sizeof(double) * (size_t)n, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) {
    k_narrow<<<(n + 255) / 256, 256>>>(d, r, n);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaMemcpy(out, r, sizeof(float) * (size_t)n, cudaMemcpyDeviceToHost);
  cudaFree(d);
  cudaFree(r);
  return (int)e;
}
