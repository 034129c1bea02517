// Helpers shared by the resident kernels (resident.cu, feeder.cu).
#pragma once

#include "kernels.cuh"

namespace pf {

// a b + c d with the roundings written out: the kernels that inline a solve
// (alone, and in a group launch) must not contract it differently, or a
// served result would differ from the same solve alone.
__device__ __forceinline__ float dot2(float a, float b, float c, float d) {
  return __fmaf_rn(a, b, __fmul_rn(c, d));
}
__device__ __forceinline__ double dot2(double a, double b, double c, double d) {
  return __fma_rn(a, b, __dmul_rn(c, d));
}
__device__ __forceinline__ float nmac2(float v, float a, float b, float c, float d) {  // v - a b - c d
  return __fmaf_rn(-c, d, __fmaf_rn(-a, b, v));
}
__device__ __forceinline__ double nmac2(double v, double a, double b, double c, double d) {
  return __fma_rn(-c, d, __fma_rn(-a, b, v));
}

// Bus state: written by any CTA of the cluster (L2) or by this CTA alone.
template <bool CL, typename T>
__device__ __forceinline__ T ld_state(const T* p) {
  if constexpr (CL) {
    return __ldcg(p);
  } else {
    return *p;
  }
}

// The address of a shared-memory object in CTA r of the cluster.
template <bool CL, typename T>
__device__ __forceinline__ T* remote_smem(T* p, int r) {
  if constexpr (CL) {
    return cg::this_cluster().map_shared_rank(p, r);
  } else {
    return p;
  }
}

// The largest value over a cluster: every CTA's own into slot[rank] of every
// CTA; read with widest() after the next barrier.
template <bool CL>
__device__ __forceinline__ void spread(unsigned long long m, unsigned long long* red,
                                       unsigned long long* slot, int P, int crank) {
  const int tid = threadIdx.x, nwarp = blockDim.x >> 5;
  for (int off = 16; off > 0; off >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, off));
  if ((tid & 31) == 0) red[tid >> 5] = m;
  __syncthreads();
  if (tid < P) {
    unsigned long long v = 0ull;
    for (int q = 0; q < nwarp; ++q) v = max(v, red[q]);
    remote_smem<CL>(slot, tid)[crank] = v;
  }
}
__device__ __forceinline__ double widest(const unsigned long long* slot, int P) {
  unsigned long long v = 0ull;
  for (int q = 0; q < P; ++q) v = max(v, slot[q]);
  return __longlong_as_double((long long)v);
}

// The stop test of iteration it (the decisions of the other kernels).
__device__ __forceinline__ int stop_test(const DevOpts& o, int it, double nrm) {
  if (!(nrm <= 1e12)) return PF_ERR_DIVERGED;
  if (nrm <= o.tol) return PF_OK;
  return it >= o.max_iter ? (int)PF_ERR_MAXITER : kRunning;
}

__device__ __forceinline__ void put_info(pf_info* out, int st, int it, int lin, double nrm,
                                         double step) {
  if (!out) return;
  pf_info inf;
  inf.status = st;
  inf.iterations = it;
  inf.linear_iterations = lin;
  inf.fallback = 0;
  inf.mismatch = nrm;
  inf.max_step = step;
  inf.solve_us = 0.0;
  inf.q_switched = 0;
  inf.q_rounds = 1;
  *out = inf;
}

// Launch of `clusters` clusters of P CTAs (P = 1: plain CTAs).
template <class Kern>
cudaError_t configure_clusters(Kern kern, int P, int threads, size_t smem, int clusters,
                               cudaStream_t st, cudaLaunchConfig_t& cfg, cudaLaunchAttribute* attr) {
  const cudaError_t e = allow_launches((const void*)kern);
  cfg.gridDim = dim3(clusters * P);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  if (P > 1) {
    attr->id = cudaLaunchAttributeClusterDimension;
    attr->val.clusterDim.x = P;
    attr->val.clusterDim.y = 1;
    attr->val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
  }
  return e;
}

// How many such clusters the device can run at once.
template <class Kern>
int count_clusters(Kern kern, int P, int threads, size_t smem) {
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  int num = 0;
  cudaError_t e = configure_clusters(kern, P, threads, smem, 1, nullptr, cfg, attr);
  if (e == cudaSuccess)
    e = P > 1 ? cudaOccupancyMaxActiveClusters(&num, kern, &cfg)
              : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&num, kern, threads, smem);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return num;
}

}  // namespace pf
