// Resident single-phase Newton-Raphson solves (resident.h): one scenario per
// CTA or per cluster, its whole factor in shared memory.
//
// What bounds it: a solve is a chain of ~2 x 40-70 dependent levels per
// Newton step, most of them a few dozen 2x2 blocks wide.  With the factor in
// global memory (newton.cuh) a level cost two cluster barriers and two or
// three dependent L2 round trips, 1.4 us of factorisation and 2 x 1.4 us of
// sweeps; here it is one round of shared-memory reads, a few FMAs and a block
// barrier.
//
// Measured (us, persistent kernel or phase kernels -> here): single solves of
// 14 buses 276 -> 98 (a whole host call), 10,000 mixed 3,330 -> 426, 2,749 FP64
// 2,140 -> 490; batches of 2,000 x 512 mixed 2,530 -> 1,262, 14 x 9,728 428 ->
// 244, 500 x 255 mixed with reactive limits 2,070 -> 496.  Mixed grids of more
// than 32 buses come here only where the caller asks (resident_default says why).
#include "resident_blocks.cuh"

namespace pf {

namespace {

// One scenario on the CTAs of a cluster (CL) or one CTA.  w: the scenario's
// own state (B = 1).
template <typename TF, bool CL>
__device__ __forceinline__ void resident_solve(const DevSys& S, const DevWork& w, const DevOpts& o,
                                               const ResDev& R, int lin) {
  using V2 = typename Vec2<TF>::T;
  const int P = CL ? (int)cg::this_cluster().num_blocks() : 1;
  const int crank = CL ? (int)cg::this_cluster().block_rank() : 0;
  const int tid = threadIdx.x, T = blockDim.x, lane = tid & 31, warp = tid >> 5, nwarp = T >> 5;
  extern __shared__ __align__(16) unsigned char dsm[];
  TF* const A = reinterpret_cast<TF*>(dsm);
  TF* const y = A + (size_t)R.max_blk * 4;
  uint2* const ring = reinterpret_cast<uint2*>(
      dsm + (((size_t)R.max_blk * 4 * sizeof(TF) + (size_t)R.max_vec * 2 * sizeof(TF) + 15) & ~(size_t)15));
  int2* const tab = reinterpret_cast<int2*>(ring + (size_t)kResRing * T);
  __shared__ ResPart sp[2];  // this CTA's part, and the top
  __shared__ ResCta sc;
  __shared__ unsigned long long sh_norm[16], sh_step[16], sh_red[32];
  __shared__ int sh_flag;
  if (tid == 0) {
    sp[0] = R.part[crank];
    sp[1] = R.part[CL ? P : 0];
    sc = R.cta[crank];
    sh_flag = 0;
  }
  const unsigned long long t_begin = global_ns();
  __syncthreads();
  const ResPart& part = sp[0];
  const ResPart& top = sp[1];
  const bool has_top = CL && crank == 0;
  const int n_top_tab = has_top ? top.rb + top.nrb - top.rf : 0;
  for (int k = tid; k < sc.ntab; k += T) tab[k] = R.rnd[sc.tab + k];
  for (int k = tid; k < n_top_tab; k += T) tab[sc.ntab + k] = R.rnd[top.rf + k];
  TF* const Ap = A + 4 * part.blk0;
  TF* const yp = y + 2 * part.vec0;
  TF* const At = A + 4 * top.blk0;
  TF* const yt = y + 2 * top.vec0;
  const bool first = crank == 0 && tid == 0;
  const bool prof = o.prof != nullptr && blockIdx.x == 0 && tid == 0;
  unsigned long long t_last = prof ? t_begin : 0ull;
  auto tick = [&](int phase) {
    if (prof) {
      const unsigned long long t = global_ns();
      o.prof[phase] += t - t_last;
      t_last = t;
    }
  };
  // fn(row record) for this CTA's rows
  auto rows = [&](auto fn) {
    for (int g = warp; g < sc.ngrp; g += nwarp) {
      const int4 r = __ldg(R.row + (size_t)(sc.grp + g) * 32 + lane);
      if (r.x >= 0) fn(r.x & ~kResRowLevel0, r);
    }
  };
  rows([&](int i, const int4&) {
    const int oi = S.perm[i];
    setup_1ph(S, w, i, 0, w.in_p_load ? w.in_p_load[oi] : S.p_load0[i],
              w.in_q_load ? w.in_q_load[oi] : S.q_load0[i],
              w.in_p_gen ? w.in_p_gen[oi] : S.p_gen0[i]);
  });
  csync<CL>();
  tick(kProfSetup);

  int status = kRunning, passes = 0;
  double prev = 0.0;
  for (int it = 0;; ++it) {
    // ---- mismatch (Eq. 8-9), right-hand side and Jacobian (Eq. 10) ----
    bool bad = false;  // a singular first-level pivot
    for (int k = part.z0 + tid; k < part.nblk; k += T) st_blk(Ap + 4 * k, Blk<TF>{0, 0, 0, 0});
    for (int k = part.np + tid; k < part.np + part.nb; k += T)
      reinterpret_cast<V2*>(yp)[k] = mk2(TF(0), TF(0));
    if (has_top)
      for (int k = top.z0 + tid; k < top.nblk; k += T) st_blk(At + 4 * k, Blk<TF>{0, 0, 0, 0});
    const unsigned long long m = assemble<TF, CL>(S, w, R, sc, A, y, o.refine > 0, (TF*)nullptr, &bad);
    if (bad)
      for (int q = 0; q < P; ++q) *remote_smem<CL>(&sh_flag, q) = 1;
    spread<CL>(m, sh_red, sh_norm, P, crank);
    csync<CL>();
    tick(kProfMismatch);

    // ---- stop test (every thread decides alike) ----
    const double nrm = widest(sh_norm, P);
    status = stop_test(o, it, nrm);
    if (status != kRunning) {
      if (first) put_info(w.out_info, status, it, lin ? passes : 0, nrm, it > 0 ? widest(sh_step, P) : 0.0);
      break;
    }
    const bool refine = o.refine > 0 && refine_now(o, it, nrm, prev);
    prev = nrm;
    tick(kProfStop);

    // ---- factorisation with the forward sweep, backward sweep; refinement ----
    const int npass = refine ? o.refine : 0;
    bool singular = false;
    for (int pass = 0; pass <= npass; ++pass) {
      if (pass == 0) {
        run_rounds<kFactor>(tab, part.nrf, R.rec, Ap, yp, ring, &sh_flag);
      } else {
        // FP64 residual of the step so far (matrix-free), then another solve
        rows([&](int i, const int4&) { dv_row<false>(S, w, i, 0); });
        csync<CL>();
        rows([&](int i, const int4& r) {
          resid_row<false>(S, w, i, 0);
          reinterpret_cast<V2*>(y)[r.z] = mk2((TF)w.r[2 * i], (TF)w.r[2 * i + 1]);
        });
        for (int k = part.np + tid; k < part.np + part.nb; k += T)
          reinterpret_cast<V2*>(yp)[k] = mk2(TF(0), TF(0));
        __syncthreads();
        tick(kProfResidual);
        run_rounds<kForward>(tab + (part.rw - part.rf), part.nrw, R.rec, Ap, yp, ring, &sh_flag);
      }
      if constexpr (CL) {
        csync<CL>();
        if (pass == 0 && tid == 0 && crank != 0 && sh_flag) *remote_smem<CL>(&sh_flag, 0) = 1;
        if (crank == 0) {
          // the parts' Schur complements and right-hand sides, in their order
          const int g0 = pass == 0 ? 0 : R.ngat_blk;
          for (int k = g0 + tid; k < R.ngat_blk + R.ngat_vec; k += T) {
            const int4 g = __ldg(R.gat + k);
            if (k < R.ngat_blk) {
              Blk<TF> v = ld_blk(At + 4 * g.x);
              for (int q = g.y; q < g.z; ++q) {
                const int2 s = __ldg(R.gsrc + q);
                const Blk<TF> u = ld_blk(remote_smem<CL>(A, s.x) + 4 * s.y);
                v.a += u.a;
                v.b += u.b;
                v.c += u.c;
                v.d += u.d;
              }
              if (g.w && !inv2(v)) sh_flag = 1;
              st_blk(At + 4 * g.x, v);
            } else {
              V2 v = reinterpret_cast<V2*>(yt)[g.x];
              for (int q = g.y; q < g.z; ++q) {
                const int2 s = __ldg(R.gsrc + q);
                const V2 u = reinterpret_cast<const V2*>(remote_smem<CL>(y, s.x))[s.y];
                v.x += u.x;
                v.y += u.y;
              }
              reinterpret_cast<V2*>(yt)[g.x] = v;
            }
          }
          __syncthreads();
          const int2* tt = tab + sc.ntab;
          if (pass == 0)
            run_rounds<kFactor>(tt, top.nrf, R.rec, At, yt, ring, &sh_flag);
          else
            run_rounds<kForward>(tt + (top.rw - top.rf), top.nrw, R.rec, At, yt, ring, &sh_flag);
          if (pass == 0) tick(kProfFactor);
          run_rounds<kBackward>(tt + (top.rb - top.rf), top.nrb, R.rec, At, yt, ring, &sh_flag);
        }
        csync<CL>();
        if (pass == 0) singular = *remote_smem<CL>(&sh_flag, 0) != 0;
        const V2* xt = reinterpret_cast<const V2*>(remote_smem<CL>(y, 0)) + top.vec0;
        for (int k = tid; k < part.nb; k += T)
          reinterpret_cast<V2*>(yp)[part.np + k] = xt[__ldg(R.bnd + part.bnd + k)];
        __syncthreads();
      } else {
        if (pass == 0) tick(kProfFactor);
      }
      run_rounds<kBackward>(tab + (part.rb - part.rf), part.nrb, R.rec, Ap, yp, ring, &sh_flag);
      if (!CL && pass == 0) singular = sh_flag != 0;
      ++passes;
      if (npass > 0)
        rows([&](int i, const int4& r) {
          const V2 x = reinterpret_cast<const V2*>(y)[r.z];
          double2* d = reinterpret_cast<double2*>(w.dx) + i;
          *d = pass == 0 ? make_double2((double)x.x, (double)x.y)
                         : make_double2(d->x + (double)x.x, d->y + (double)x.y);
        });
      tick(kProfSolve);
      if (singular) break;
    }
    if (singular) {
      status = PF_ERR_SINGULAR;
      if (first) put_info(w.out_info, status, it, lin ? passes - 1 : 0, nrm, 0.0);
      csync<CL>();
      break;
    }

    // ---- voltage update ----
    unsigned long long ms = 0ull;
    rows([&](int i, const int4& r) {
      double dd, dm;
      if (npass > 0) {
        const double2 q = reinterpret_cast<const double2*>(w.dx)[i];
        dd = q.x;
        dm = q.y;
      } else {
        const V2 q = reinterpret_cast<const V2*>(y)[r.z];
        dd = (double)q.x;
        dm = (double)q.y;
      }
      ms = max(ms, max(abs_bits(dd), abs_bits(dm)));
      const double vm = w.vm[i] + dm, va = w.va[i] + dd;
      w.vm[i] = vm;
      w.va[i] = va;
      double sn, cs;
      sincos_tab(S.trig, va, &sn, &cs);
      if (sizeof(TF) == 8) w.U[i] = make_double2(cs, sn);
      w.V[i] = make_double2(vm * cs, vm * sn);
    });
    spread<CL>(ms, sh_red, sh_step, P, crank);
    csync<CL>();
    tick(kProfUpdate);
  }

  // ---- results in the caller's numbering ----
  rows([&](int i, const int4&) { output_row<false>(S, w, i, 0, status == PF_OK); });
  tick(kProfOutput);
  if (crank == 0) {
    __syncthreads();
    if (tid == 0 && w.out_info) w.out_info->solve_us = (double)(global_ns() - t_begin) * 1e-3;
  }
}

template <typename TF, bool CL>
__global__ void __launch_bounds__(512, 1)
    k_resident(DevSys S, DevWork w, DevOpts o, ResDev R, int lin) {
  const int gs = CL ? blockIdx.x / (int)cg::this_cluster().num_blocks() : blockIdx.x;
  resident_solve<TF, CL>(S, scenario_of(w, S.n, gs), o, R, lin);
}

// Several requests of any cases in one launch: cluster b solves desc[list.job[b]]
// and raises its done flag (as newton_group_kernel).
template <typename TF, bool CL>
__global__ void __launch_bounds__(512, 1) k_resident_group(const GroupJob* desc, GroupList list) {
  const int csize = CL ? (int)cg::this_cluster().num_blocks() : 1;
  const int crank = CL ? (int)cg::this_cluster().block_rank() : 0;
  __shared__ GroupJob job;
  __shared__ ResDev plan;
  {
    const GroupJob* src = desc + list.job[blockIdx.x / csize];
    for (int k = threadIdx.x; k < (int)(sizeof(GroupJob) / 4); k += blockDim.x)
      reinterpret_cast<unsigned*>(&job)[k] = reinterpret_cast<const unsigned*>(src)[k];
    __syncthreads();
    for (int k = threadIdx.x; k < (int)(sizeof(ResDev) / 4); k += blockDim.x)
      reinterpret_cast<unsigned*>(&plan)[k] = static_cast<const unsigned*>(job.res)[k];
  }
  __syncthreads();
  resident_solve<TF, CL>(job.S, job.w, job.o, plan, 0);
  __threadfence_system();
  csync<CL>();
  if (crank == 0 && threadIdx.x == 0) {
    __threadfence_system();
    *reinterpret_cast<volatile int*>(job.done) = 1;
  }
}

template <typename TF, bool CL>
cudaError_t launch_res(const DevSys& S, const DevWork& w, const DevOpts& o, const ResDev& R,
                       size_t smem, int B, int lin, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  const cudaError_t e = configure_clusters(k_resident<TF, CL>, R.P, R.threads, smem, B, st, cfg, attr);
  if (e != cudaSuccess) return e;
  return cudaLaunchKernelEx(&cfg, k_resident<TF, CL>, S, w, o, R, lin);
}

template <typename TF, bool CL>
cudaError_t launch_group(const GroupJob* desc, const GroupList& list, size_t smem, int P, int threads,
                         cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  const cudaError_t e =
      configure_clusters(k_resident_group<TF, CL>, P, threads, smem, list.n, st, cfg, attr);
  if (e != cudaSuccess) return e;
  return cudaLaunchKernelEx(&cfg, k_resident_group<TF, CL>, desc, list);
}

}  // namespace

cudaError_t launch_resident(bool fp32, const DevSys& S, const DevWork& w, const DevOpts& o,
                            const ResDev& R, size_t smem, int B, int lin, cudaStream_t st) {
  if (R.P > 1)
    return fp32 ? launch_res<float, true>(S, w, o, R, smem, B, lin, st)
                : launch_res<double, true>(S, w, o, R, smem, B, lin, st);
  return fp32 ? launch_res<float, false>(S, w, o, R, smem, B, lin, st)
              : launch_res<double, false>(S, w, o, R, smem, B, lin, st);
}

cudaError_t launch_resident_group(bool fp32, const GroupJob* desc, const GroupList& list, size_t smem,
                                  int P, int threads, cudaStream_t st) {
  if (list.n <= 0 || list.n > kGroupMax) return cudaErrorInvalidValue;
  if (P > 1)
    return fp32 ? launch_group<float, true>(desc, list, smem, P, threads, st)
                : launch_group<double, true>(desc, list, smem, P, threads, st);
  return fp32 ? launch_group<float, false>(desc, list, smem, P, threads, st)
              : launch_group<double, false>(desc, list, smem, P, threads, st);
}

int resident_clusters(bool fp32, int P, int threads, size_t smem) {
  if (P > 1)
    return fp32 ? count_clusters(k_resident<float, true>, P, threads, smem)
                : count_clusters(k_resident<double, true>, P, threads, smem);
  return fp32 ? count_clusters(k_resident<float, false>, P, threads, smem)
              : count_clusters(k_resident<double, false>, P, threads, smem);
}

}  // namespace pf
