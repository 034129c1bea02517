// Resident Newton-Krylov solves: restarted GMRES(m) with right ILU(0) (Sec.
// III.B), one scenario per CTA with the ILU(0) factor, the vector being
// preconditioned and the vector being orthogonalised in shared memory.
//
// What bounds it: an inner iteration is two triangular sweeps of 35-40 levels
// and 2 (k + 1) dot products and updates against the Krylov basis.  In the
// persistent kernel (newton.cuh) a sweep level cost an L2 round trip and a dot
// product two cluster barriers, 176 us per inner iteration on the 2,000-bus
// grid.  Here the sweeps run the rounds of resident.h and a warp takes a whole
// dot product (a basis vector read once, coalesced; no reduction across
// warps).  FP64 only (resident_plan says why).  Measured (ms, persistent kernel ->
// this one): 500 buses 29.4 -> 11.7, x 64 -> 12.5.
#include "resident_blocks.cuh"

namespace pf {

namespace {

using TF = double;

__global__ void __launch_bounds__(512, 1) k_resident_nk(DevSys S, DevWork w0, DevOpts o, ResDev R) {
  using V2 = double2;
  const int n = S.n, m = o.m, gs = blockIdx.x;
  const DevWork w = scenario_of(w0, n, gs);
  const size_t nnz = S.y_rowptr[n];
  TF* const JM = reinterpret_cast<TF*>(w0.jm) + (size_t)gs * nnz * 4;  // by Ybus entry
  V2* const V0 = reinterpret_cast<V2*>(w0.vb) + (size_t)gs * (m + 1) * n;
  V2* const X = reinterpret_cast<V2*>(w0.xg) + (size_t)gs * n;
  const int tid = threadIdx.x, T = blockDim.x, lane = tid & 31, warp = tid >> 5, nwarp = T >> 5;
  extern __shared__ __align__(16) unsigned char dsm[];
  TF* const A = reinterpret_cast<TF*>(dsm);
  TF* const yraw = A + (size_t)R.max_blk * 4;
  V2* const y = reinterpret_cast<V2*>(yraw);
  uint2* const ring = reinterpret_cast<uint2*>(
      dsm + (((size_t)R.max_blk * 4 * sizeof(TF) + (size_t)R.max_vec * 2 * sizeof(TF) + 15) & ~(size_t)15));
  __shared__ ResPart part;
  __shared__ ResCta sc;
  __shared__ unsigned long long sh_norm[1], sh_step[1], sh_red[32];
  __shared__ TF sh_sum[32];
  __shared__ int sh_flag, sh_kk, sh_go;
  if (tid == 0) {
    part = R.part[0];
    sc = R.cta[0];
    sh_flag = 0;
  }
  const unsigned long long t_begin = global_ns();
  __syncthreads();
  int2* const tab = reinterpret_cast<int2*>(ring + (size_t)kResRing * T);
  V2* const W = reinterpret_cast<V2*>(tab + sc.ntab + (sc.ntab & 1));
  TF* const h1 = reinterpret_cast<TF*>(W + n);
  TF* const h2 = h1 + m + 1;
  GmresState<TF> G;
  G.bind(h2 + m + 1, m, 0);
  for (int k = tid; k < sc.ntab; k += T) tab[k] = R.rnd[sc.tab + k];
  const bool prof = o.prof != nullptr && gs == 0 && tid == 0;
  unsigned long long t_last = prof ? t_begin : 0ull;
  auto tick = [&](int phase) {
    if (prof) {
      const unsigned long long t = global_ns();
      o.prof[phase] += t - t_last;
      t_last = t;
    }
  };
  auto rows = [&](auto fn) {
    for (int g = warp; g < sc.ngrp; g += nwarp) {
      const int4 r = __ldg(R.row + (size_t)(sc.grp + g) * 32 + lane);
      if (r.x >= 0) fn(r.x & ~kResRowLevel0);
    }
  };
  // sum over the CTA, the same in every thread
  auto total = [&](TF v) {
    for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    __syncthreads();
    if (lane == 0) sh_sum[warp] = v;
    __syncthreads();
    TF s = TF(0);
    for (int q = 0; q < nwarp; ++q) s += sh_sum[q];
    return s;
  };
  // row i of J u
  auto jrow = [&](int i, const V2* u) {
    V2 s = mk2(TF(0), TF(0));
#pragma unroll 2
    for (int e = S.y_rowptr[i]; e < S.y_rowptr[i + 1]; ++e) {
      const Blk<TF> b = ld_blk(JM + 4 * (size_t)e);
      const V2 q = u[S.y_col[e]];
      s.x += dot2(b.a, q.x, b.b, q.y);
      s.y += dot2(b.c, q.x, b.d, q.y);
    }
    return s;
  };
  // y <- M^-1 y by the ILU(0) sweeps
  auto precond = [&] {
    __syncthreads();
    run_rounds<kForward>(tab + (part.rw - part.rf), part.nrw, R.rec, A, yraw, ring, &sh_flag);
    run_rounds<kBackward>(tab + (part.rb - part.rf), part.nrb, R.rec, A, yraw, ring, &sh_flag);
  };
  // h_j = (V_j, W) for j <= k, a warp each, and W -= sum_j h_j V_j
  auto dots = [&](TF* h, int k) {
    for (int j = warp; j <= k; j += nwarp) {
      const V2* v = V0 + (size_t)j * n;
      TF s0 = TF(0), s1 = TF(0);
#pragma unroll 8
      for (int i = lane; i < n; i += 32) {
        const V2 a = v[i], b = W[i];
        s0 = a.x * b.x + s0;
        s1 = a.y * b.y + s1;
      }
      s0 += s1;
      for (int off = 16; off > 0; off >>= 1) s0 += __shfl_xor_sync(0xffffffffu, s0, off);
      if (lane == 0) h[j] = s0;
    }
    __syncthreads();
  };
  auto orth = [&](const TF* h, int k) {  // returns this thread's share of |W|^2
    TF s = TF(0);
    for (int i = tid; i < n; i += T) {
      V2 a = W[i];
#pragma unroll 8
      for (int j = 0; j <= k; ++j) {
        const V2 v = V0[(size_t)j * n + i];
        a.x -= h[j] * v.x;
        a.y -= h[j] * v.y;
      }
      W[i] = a;
      s += a.x * a.x + a.y * a.y;
    }
    return s;
  };

  rows([&](int i) {
    const int oi = S.perm[i];
    setup_1ph(S, w, i, 0, w.in_p_load ? w.in_p_load[oi] : S.p_load0[i],
              w.in_q_load ? w.in_q_load[oi] : S.q_load0[i],
              w.in_p_gen ? w.in_p_gen[oi] : S.p_gen0[i]);
  });
  __syncthreads();
  tick(kProfSetup);

  int status = kRunning, lin = 0;
  for (int it = 0;; ++it) {
    bool bad = false;
    const unsigned long long mx = assemble<TF, false>(S, w, R, sc, A, yraw, true, JM, &bad);
    if (bad) sh_flag = 1;
    spread<false>(mx, sh_red, sh_norm, 1, 0);
    __syncthreads();
    tick(kProfMismatch);
    const double nrm = widest(sh_norm, 1);
    status = stop_test(o, it, nrm);
    if (status != kRunning) {
      if (tid == 0) put_info(w.out_info, status, it, lin, nrm, it > 0 ? widest(sh_step, 1) : 0.0);
      break;
    }
    tick(kProfStop);
    // ILU(0); the vector items of the same rounds work on y, which is free here
    run_rounds<kFactor>(tab, part.nrf, R.rec, A, yraw, ring, &sh_flag);
    __syncthreads();
    tick(kProfFactor);
    if (sh_flag) {
      status = PF_ERR_SINGULAR;
      if (tid == 0) put_info(w.out_info, status, it, lin, nrm, 0.0);
      break;
    }

    // ---- GMRES(m) on J dx = F to |r| <= eta |F| ----
    auto rhs = [&](int i) {
      const double2 f = reinterpret_cast<const double2*>(w.F)[i];
      return mk2((TF)f.x, (TF)f.y);
    };
    TF s = TF(0);
    for (int i = tid; i < n; i += T) {
      const V2 f = rhs(i);
      s += f.x * f.x + f.y * f.y;
      X[i] = mk2(TF(0), TF(0));
    }
    const TF bnorm = sqrt(total(s));
    const TF eta = (TF)fmin(0.1, fmax(o.rtol, nrm));
    int step = 0;
    for (int restart = 0;; ++restart) {
      // r = F - J x into V_0
      s = TF(0);
      for (int i = tid; i < n; i += T) {
        V2 r = rhs(i);
        if (restart > 0) {
          const V2 q = jrow(i, X);
          r.x -= q.x;
          r.y -= q.y;
        }
        V0[i] = r;
        s += r.x * r.x + r.y * r.y;
      }
      const TF beta = sqrt(total(s));
      if (!(beta > eta * bnorm) || step >= o.max_lin) break;
      const TF inv = TF(1) / beta;
      for (int i = tid; i < n; i += T) V0[i] = y[i] = mk2(V0[i].x * inv, V0[i].y * inv);
      if (tid == 0) {
        G.g[0] = beta;
        sh_kk = 0;
      }
      for (int k = 0; k < m; ++k) {
        precond();  // y = M^-1 v_k
        for (int i = tid; i < n; i += T) W[i] = jrow(i, y);
        __syncthreads();
        // classical Gram-Schmidt, twice
        dots(h1, k);
        orth(h1, k);
        __syncthreads();
        dots(h2, k);
        const TF hk1 = sqrt(total(orth(h2, k)));
        ++lin;
        ++step;
        if (tid == 0) {  // Hessenberg column k: the earlier rotations and a new one
          TF* Hk = G.H + (size_t)k * (m + 1);
          for (int j = 0; j <= k; ++j) Hk[j] = h1[j] + h2[j];
          for (int j = 0; j < k; ++j) {
            const TF a0 = Hk[j], a1 = Hk[j + 1];
            Hk[j] = G.cs[j] * a0 + G.sn[j] * a1;
            Hk[j + 1] = -G.sn[j] * a0 + G.cs[j] * a1;
          }
          const TF den = sqrt(Hk[k] * Hk[k] + hk1 * hk1);
          bool stop = !(den > TF(0));  // breakdown with a zero column: keep the first k steps
          if (!stop) {
            G.cs[k] = Hk[k] / den;
            G.sn[k] = hk1 / den;
            Hk[k] = den;
            Hk[k + 1] = TF(0);
            G.g[k + 1] = -G.sn[k] * G.g[k];
            G.g[k] = G.cs[k] * G.g[k];
            sh_kk = k + 1;
            stop = fabs(G.g[k + 1]) <= eta * bnorm;
          }
          sh_go = !stop && step < o.max_lin && hk1 > TF(0);
        }
        __syncthreads();
        if (!sh_go) break;
        if (k + 1 < m) {
          const TF ih = TF(1) / hk1;
          V2* v = V0 + (size_t)(k + 1) * n;
          for (int i = tid; i < n; i += T) v[i] = y[i] = mk2(W[i].x * ih, W[i].y * ih);
        }
      }
      // x += M^-1 (V c), R c = g
      const int kk = sh_kk;
      if (tid == 0)
        for (int j = kk - 1; j >= 0; --j) {
          TF v = G.g[j];
          for (int l = j + 1; l < kk; ++l) v -= G.H[j + (size_t)l * (m + 1)] * G.y[l];
          G.y[j] = v / G.H[j + (size_t)j * (m + 1)];
        }
      __syncthreads();
      for (int i = tid; i < n; i += T) {
        V2 v = mk2(TF(0), TF(0));
#pragma unroll 8
        for (int j = 0; j < kk; ++j) {
          const V2 q = V0[(size_t)j * n + i];
          v.x += G.y[j] * q.x;
          v.y += G.y[j] * q.y;
        }
        y[i] = v;
      }
      precond();
      for (int i = tid; i < n; i += T) X[i] = mk2(X[i].x + y[i].x, X[i].y + y[i].y);
      __syncthreads();
    }
    tick(kProfSolve);

    // ---- voltage update ----
    __syncthreads();
    unsigned long long ms = 0ull;
    rows([&](int i) {
      const V2 q = X[i];
      const double dd = (double)q.x, dm = (double)q.y;
      ms = max(ms, max(abs_bits(dd), abs_bits(dm)));
      const double vm = w.vm[i] + dm, va = w.va[i] + dd;
      w.vm[i] = vm;
      w.va[i] = va;
      double sn, cs;
      sincos_tab(S.trig, va, &sn, &cs);
      w.U[i] = make_double2(cs, sn);
      w.V[i] = make_double2(vm * cs, vm * sn);
    });
    spread<false>(ms, sh_red, sh_step, 1, 0);
    __syncthreads();
    tick(kProfUpdate);
  }

  rows([&](int i) { output_row<false>(S, w, i, 0, status == PF_OK); });
  tick(kProfOutput);
  __syncthreads();
  if (tid == 0 && w.out_info) w.out_info->solve_us = (double)(global_ns() - t_begin) * 1e-3;
}

}  // namespace

// The plan's shared memory, the orthogonalised vector, two columns of
// coefficients and the Hessenberg state.
size_t resident_nk_smem(size_t plan_smem, int n, int m) {
  return plan_smem + 32 + ((size_t)2 * n + 2 * (m + 1) + (size_t)(m + 1) * m + 4 * m + 1) * sizeof(TF);
}

cudaError_t launch_resident_nk(const DevSys& S, const DevWork& w, const DevOpts& o, const ResDev& R,
                               size_t smem, int B, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  const cudaError_t e = configure_clusters(k_resident_nk, 1, R.threads, smem, B, st, cfg, attr);
  if (e != cudaSuccess) return e;
  return cudaLaunchKernelEx(&cfg, k_resident_nk, S, w, o, R);
}

}  // namespace pf
