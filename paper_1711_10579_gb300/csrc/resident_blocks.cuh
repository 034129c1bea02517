// Device code shared by the single-phase resident kernels (resident.cu,
// resident_nk.cu): 2x2 blocks, the rounds, and the mismatch with the Jacobian.
#pragma once

#include "resident.cuh"
#include "resident.h"

namespace pf {

// 8-byte asynchronous copy global -> shared.
__device__ __forceinline__ void cp8(void* smem, const void* gmem) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(s), "l"(gmem) : "memory");
}

template <typename TF>
struct Blk {
  TF a, b, c, d;  // [a b; c d]
};
template <typename TF>
struct Vec2;
template <>
struct Vec2<float> {
  using T = float2;
};
template <>
struct Vec2<double> {
  using T = double2;
};

__device__ __forceinline__ Blk<float> ld_blk(const float* p) {
  const float4 v = *reinterpret_cast<const float4*>(p);
  return {v.x, v.y, v.z, v.w};
}
__device__ __forceinline__ Blk<double> ld_blk(const double* p) {
  const double2 v = reinterpret_cast<const double2*>(p)[0], u = reinterpret_cast<const double2*>(p)[1];
  return {v.x, v.y, u.x, u.y};
}
__device__ __forceinline__ void st_blk(float* p, const Blk<float>& v) {
  *reinterpret_cast<float4*>(p) = make_float4(v.a, v.b, v.c, v.d);
}
__device__ __forceinline__ void st_blk(double* p, const Blk<double>& v) {
  reinterpret_cast<double2*>(p)[0] = make_double2(v.a, v.b);
  reinterpret_cast<double2*>(p)[1] = make_double2(v.c, v.d);
}
__device__ __forceinline__ float2 mk2(float x, float y) { return make_float2(x, y); }
__device__ __forceinline__ double2 mk2(double x, double y) { return make_double2(x, y); }

// Inverse in closed form; false for a zero or non-finite determinant or
// inverse (the rule of the batched factorisation).  A determinant has the square
// of the entries' range: FP32 plans are made for grids in ordinary units only
// (upload_resident); elimination with row exchanges, which needs no such rule,
// costs 14 buses x 9,728 3%.
template <typename TF>
__device__ __forceinline__ bool inv2(Blk<TF>& m) {
  const TF det = dot2(m.a, m.d, -m.b, m.c);
  const TF r = recip(det);
  const Blk<TF> v{m.d * r, -m.b * r, -m.c * r, m.a * r};
  m = v;
  return det != TF(0) && isfinite(v.a) && isfinite(v.b) && isfinite(v.c) && isfinite(v.d);
}

enum { kFactor = 0, kForward = 1, kBackward = 2 };

// The rounds tab[0 .. nr) of one part (blocks A, vector y).  A thread's items
// of the next kResRing rounds are in flight by cp.async, so a round waits
// for no global load.  Ends with a block barrier (nr > 0).
template <int MODE>
__device__ __noinline__ void run_rounds(const int2* tab, int nr, const uint2* __restrict__ rec,
                                        float* A, float* y, uint2* ring, int* flag) {
  using TF = float;
  using V2 = float2;
  constexpr int D = kResRing;
  const int t = threadIdx.x, T = blockDim.x;
  V2* yv = reinterpret_cast<V2*>(y);
#pragma unroll
  for (int d = 0; d < D; ++d) {
    if (d < nr) {
      const int2 q = tab[d];
      if (t < (q.y & 0xffff)) cp8(ring + d * T + t, rec + q.x + t);
    }
    cp_commit();
  }
  for (int r = 0; r < nr; ++r) {
    const int2 q = tab[r];
    cp_wait<D - 1>();
    uint2* mine = ring + (r & (D - 1)) * T + t;
    if (t < (q.y & 0xffff)) {
      const uint2 it = *mine;
      const int x = it.x & 0xffff;
      if (x != kResNone) {
        const int b = it.x >> 16, c = it.y & 0xffff, k = (it.y >> 16) & (kResMaxRows - 1);
        if constexpr (MODE == kBackward) {
          V2 v = yv[x];
          if (b != kResNone) {
            const Blk<TF> B = ld_blk(A + 4 * b);
            const V2 u = yv[c];
            v.x = nmac2(v.x, B.a, u.x, B.b, u.y);
            v.y = nmac2(v.y, B.c, u.x, B.d, u.y);
          }
          if (it.y & kResFinal) {
            const Blk<TF> Di = ld_blk(A + 4 * x);
            v = mk2(dot2(Di.a, v.x, Di.b, v.y), dot2(Di.c, v.x, Di.d, v.y));
          }
          yv[x] = v;
        } else {
          const Blk<TF> B = ld_blk(A + 4 * b), Di = ld_blk(A + 4 * k);
          if (MODE == kForward || (it.y & kResVec)) {
            const V2 u = yv[k];
            V2 v = yv[x];
            const TF m0 = dot2(Di.a, u.x, Di.b, u.y), m1 = dot2(Di.c, u.x, Di.d, u.y);
            v.x = nmac2(v.x, B.a, m0, B.b, m1);
            v.y = nmac2(v.y, B.c, m0, B.d, m1);
            yv[x] = v;
          } else {
            const Blk<TF> U = ld_blk(A + 4 * c);
            Blk<TF> v = ld_blk(A + 4 * x);
            const Blk<TF> m{dot2(Di.a, U.a, Di.b, U.c), dot2(Di.a, U.b, Di.b, U.d),
                            dot2(Di.c, U.a, Di.d, U.c), dot2(Di.c, U.b, Di.d, U.d)};
            v.a = nmac2(v.a, B.a, m.a, B.b, m.c);
            v.b = nmac2(v.b, B.a, m.b, B.b, m.d);
            v.c = nmac2(v.c, B.c, m.a, B.d, m.c);
            v.d = nmac2(v.d, B.c, m.b, B.d, m.d);
            if (it.y & kResFinal) {
              if (!inv2(v)) *flag = 1;
            }
            st_blk(A + 4 * x, v);
          }
        }
      }
    }
    if (r + D < nr) {
      const int2 f = tab[r + D];
      if (t < (f.y & 0xffff)) cp8(mine, rec + f.x + t);
    }
    cp_commit();
    if (q.y < 0) __syncthreads();
  }
}

// FP64: two threads an item, a row each.  A warp's FP64 instruction takes 64
// cycles of its sub-partition whether one lane is active or all, so a level of
// few items waits for the instructions of one lane: 8 instead of 16 for an
// update (2,749 buses: factorisations 402 -> 323 us, the solve 590 -> 509 us).
template <int MODE>
__device__ __noinline__ void run_rounds(const int2* tab, int nr, const uint2* __restrict__ rec,
                                        double* A, double* y, uint2* ring, int* flag) {
  constexpr int D = kResRing;
  const int t = threadIdx.x, T = blockDim.x, slot = t >> 1, h = t & 1;  // h: the row of the block
  auto fetch = [&](int r) {
    if (r < nr) {
      const int2 q = tab[r];
      if (slot < (q.y & 0xffff)) cp8(ring + (r & (D - 1)) * T + t, rec + q.x + slot);
    }
    cp_commit();
  };
  auto row = [&](int blk, int r) { return reinterpret_cast<const double2*>(A)[2 * blk + r]; };
  for (int r = 0; r < D; ++r) fetch(r);
  for (int r = 0; r < nr; ++r) {
    const int2 q = tab[r];
    cp_wait<D - 1>();
    const uint2 it = slot < (q.y & 0xffff) ? ring[(r & (D - 1)) * T + t] : make_uint2(kResNone, 0);
    const int x = it.x & 0xffff, b = it.x >> 16, c = it.y & 0xffff, k = (it.y >> 16) & (kResMaxRows - 1);
    const bool on = x != kResNone;
    if constexpr (MODE == kBackward) {
      double v = 0.0;
      if (on) {
        v = y[2 * x + h];
        if (b != kResNone) {
          const double2 B = row(b, h);
          v = nmac2(v, B.x, y[2 * c], B.y, y[2 * c + 1]);
        }
      }
      const double w = __shfl_xor_sync(0xffffffffu, v, 1);  // the pair's other row
      if (on) {
        if (it.y & kResFinal) {
          const double2 Q = row(x, h);
          v = dot2(Q.x, h ? w : v, Q.y, h ? v : w);
        }
        y[2 * x + h] = v;
      }
    } else {
      double2 v = make_double2(0, 0);
      const bool vec = MODE == kForward || (it.y & kResVec);
      if (on) {
        const double2 B = row(b, h), k0 = row(k, 0), k1 = row(k, 1);
        // the row of A_b A_k^-1
        const double m0 = dot2(B.x, k0.x, B.y, k1.x), m1 = dot2(B.x, k0.y, B.y, k1.y);
        if (vec) {
          y[2 * x + h] = nmac2(y[2 * x + h], m0, y[2 * k], m1, y[2 * k + 1]);
        } else {
          const double2 u0 = row(c, 0), u1 = row(c, 1);
          v = row(x, h);
          v.x = nmac2(v.x, m0, u0.x, m1, u1.x);
          v.y = nmac2(v.y, m0, u0.y, m1, u1.y);
        }
      }
      if constexpr (MODE == kFactor) {
        const double2 w = make_double2(__shfl_xor_sync(0xffffffffu, v.x, 1),
                                       __shfl_xor_sync(0xffffffffu, v.y, 1));
        if (on && !vec) {
          if (it.y & kResFinal) {
            const double2 r0 = h ? w : v, r1 = h ? v : w;  // [a b], [c d]
            const double det = dot2(r0.x, r1.y, -r0.y, r1.x), rd = recip(det);
            v = h ? make_double2(-r1.x * rd, r0.x * rd) : make_double2(r1.y * rd, -r0.y * rd);
            if (det == 0.0 || !isfinite(v.x) || !isfinite(v.y)) *flag = 1;
          }
          reinterpret_cast<double2*>(A)[2 * x + h] = v;
        }
      }
    }
    fetch(r + D);
    if (q.y < 0) __syncthreads();
  }
}

// Off-diagonal Jacobian block (Eq. 10) of entry (i, j) of types ti, tj.
template <bool CL>
__device__ __forceinline__ Blk<float> jac_block(const DevWork& w, int i, int j, int ti, int tj,
                                                float2 y) {
  const double2 Vi = ld_state<CL>(w.V + i), Vj = ld_state<CL>(w.V + j);
  Blk<float> o{0.f, 0.f, 0.f, 0.f};
  if (ti == PF_SLACK || tj == PF_SLACK) return o;
  const float vix = to_f32_trunc(Vi.x), viy = to_f32_trunc(Vi.y);
  const float vjx = to_f32_trunc(Vj.x), vjy = to_f32_trunc(Vj.y);
  const float yvx = dot2(y.x, vjx, -y.y, vjy), yvy = dot2(y.x, vjy, y.y, vjx);
  const float cx = dot2(vix, yvx, viy, yvy), cy = dot2(viy, yvx, -vix, yvy);
  o.a = cy;
  o.c = -cx;
  if (tj >= PF_PQ) {
    const float rv = rsqrtf(dot2(vjx, vjx, vjy, vjy));
    o.b = cx * rv;
    o.d = cy * rv;
  }
  if (ti == PF_PV) o.c = o.d = 0.f;
  return o;
}
template <bool CL>
__device__ __forceinline__ Blk<double> jac_block(const DevWork& w, int i, int j, int ti, int tj,
                                                 double2 y) {
  const double2 Vi = ld_state<CL>(w.V + i), Uj = ld_state<CL>(w.U + j);
  const double vmj = ld_state<CL>(w.vm + j);
  Blk<double> o{0.0, 0.0, 0.0, 0.0};
  if (ti == PF_SLACK || tj == PF_SLACK) return o;
  const double yux = dot2(y.x, Uj.x, -y.y, Uj.y), yuy = dot2(y.x, Uj.y, y.y, Uj.x);
  const double cx = dot2(Vi.x, yux, Vi.y, yuy), cy = dot2(Vi.y, yux, -Vi.x, yuy);
  o.a = vmj * cy;
  o.c = -vmj * cx;
  if (tj >= PF_PQ) {
    o.b = cx;
    o.d = cy;
  }
  if (ti == PF_PV) o.c = o.d = 0.0;
  return o;
}

// Diagonal Jacobian block of row i: V and I of the row, its loads, the Ybus
// diagonal.
__device__ __forceinline__ Blk<float> diag_block(const DevSys& S, int i, int t, double2 Vi, double2,
                                                 double vm, double2 I, double pl, double ql,
                                                 float2 y) {
  if (t == PF_SLACK) return {1.f, 0.f, 0.f, 1.f};
  const float vix = to_f32_trunc(Vi.x), viy = to_f32_trunc(Vi.y);
  const float Ix = to_f32_trunc(I.x), Iy = to_f32_trunc(I.y);
  const float rvi = rsqrtf(dot2(vix, vix, viy, viy));
  const float uix = vix * rvi, uiy = viy * rvi;
  const float yvx = dot2(y.x, vix, -y.y, viy), yvy = dot2(y.x, viy, y.y, vix);
  const float scx = dot2(vix, Ix, viy, Iy), scy = dot2(viy, Ix, -vix, Iy);
  const float dx = dot2(vix, yvx, viy, yvy), dy = dot2(viy, yvx, -vix, yvy);
  const float ax = Ix + yvx, ay = Iy + yvy;
  const float ex = dot2(uix, ax, uiy, ay), ey = dot2(uiy, ax, -uix, ay);
  const float dshape = fmaf(2.f * S.zip32[3 * i + 2], to_f32_trunc(vm), S.zip32[3 * i + 1]);
  Blk<float> o{-(scy - dy), fmaf(to_f32_trunc(pl), dshape, ex), scx - dx,
               fmaf(to_f32_trunc(ql), dshape, ey)};
  if (t == PF_PV) {
    o.b = o.c = 0.f;
    o.d = 1.f;
  }
  return o;
}
__device__ __forceinline__ Blk<double> diag_block(const DevSys& S, int i, int t, double2 Vi,
                                                  double2 Ui, double vm, double2 I,
                                                  double pl, double ql, double2 y) {
  if (t == PF_SLACK) return {1.0, 0.0, 0.0, 1.0};
  // dS/d delta = j V conj(I - Y_ii V), dS/d|V| = U conj(I + Y_ii V) and the
  // load's slope
  const double yvx = dot2(y.x, Vi.x, -y.y, Vi.y), yvy = dot2(y.x, Vi.y, y.y, Vi.x);
  const double ox = I.x - yvx, oy = I.y - yvy, ax = I.x + yvx, ay = I.y + yvy;
  Blk<double> o{dot2(Vi.x, oy, -Vi.y, ox), dot2(Ui.x, ax, Ui.y, ay), dot2(Vi.x, ox, Vi.y, oy),
                dot2(Ui.y, ax, -Ui.x, ay)};
  const double zi = S.zip[3 * i + 1], zz = S.zip[3 * i + 2];
  if (nonzero(zi, zz)) {
    const double dshape = fma(2.0 * zz, vm, zi);
    o.b = fma(pl, dshape, o.b);
    o.d = fma(ql, dshape, o.d);
  }
  if (t == PF_PV) {
    o.b = o.c = 0.0;
    o.d = 1.0;
  }
  return o;
}

// FP64 -> TF, to the nearest by integer instructions (ties away from zero;
// infinities become NaN: their scenario has diverged).
template <typename TF>
__device__ __forceinline__ TF narrow(double v) {
  if constexpr (sizeof(TF) == 8) {
    return v;
  } else {
    return to_f32_trunc(__longlong_as_double(__double_as_longlong(v) + (1ll << 28)));
  }
}

// The mismatch of Eq. 8-9 of this CTA's rows (into the right-hand side y and,
// keep_f, w.F), their largest (returned, as bits) and the Jacobian blocks of
// Eq. 10 of its entries (into A and, where jm is given, jm by Ybus entry); the
// diagonal blocks of the first level are inverted (bad: one is singular).
template <typename TF, bool CL>
__device__ __forceinline__ unsigned long long assemble(const DevSys& S, const DevWork& w,
                                                       const ResDev& R, const ResCta& sc, TF* A, TF* y,
                                                       bool keep_f, TF* jm, bool* bad) {
  using V2 = typename Vec2<TF>::T;
  const int tid = threadIdx.x, T = blockDim.x, lane = tid & 31, warp = tid >> 5, nwarp = T >> 5;
  for (int e = tid; e < sc.njac; e += T) {
    const int4 r = __ldg(R.jac + sc.jac + e);
    const V2 yv = __ldg(reinterpret_cast<const V2*>(R.jac_y) + sc.jac + e);
    const int ti = w.bt ? w.bt[r.y] : (r.w & 3), tj = w.bt ? w.bt[r.z] : ((r.w >> 2) & 3);
    const Blk<TF> v = jac_block<CL>(w, r.y, r.z, ti, tj, yv);
    st_blk(A + 4 * r.x, v);
    if (jm) st_blk(jm + 4 * (size_t)(r.w >> 4), v);
  }
  unsigned long long m = 0ull;
  for (int g = warp; g < sc.ngrp; g += nwarp) {
    const ResGroup G = R.grp[sc.grp + g];
    const size_t rl = (size_t)(sc.grp + g) * 32 + lane;
    const int4 r = __ldg(R.row + rl);
    const bool on = r.x >= 0;
    const int i = on ? (r.x & ~kResRowLevel0) : 0;
    const double2 Vi = ld_state<CL>(w.V + i);
    const double vmi = ld_state<CL>(w.vm + i);
    const double pl = w.spec[3 * (size_t)i], ql = w.spec[3 * (size_t)i + 1],
                 pg = w.spec[3 * (size_t)i + 2];
    const double zp = S.zip[3 * i], zi = S.zip[3 * i + 1], zz = S.zip[3 * i + 2];
    const int t = w.bt ? w.bt[i] : S.btype[i];
    double2 I = make_double2(0.0, 0.0), yd = make_double2(0.0, 0.0);
#pragma unroll 4
    for (int e = 0; e < G.width; ++e) {
      const size_t q = (size_t)G.ell + 32 * e + lane;
      const int j = __ldg(R.ell_col + q);
      const double2 yv = __ldg(R.ell_y + q), v = ld_state<CL>(w.V + j);
      if (sizeof(TF) == 8 && e == 0) yd = yv;
      I.x = fma(yv.x, v.x, I.x);
      I.x = fma(-yv.y, v.y, I.x);
      I.y = fma(yv.x, v.y, I.y);
      I.y = fma(yv.y, v.x, I.y);
    }
    if (!on) continue;
    double shape = zp;
    if (nonzero(zi, zz)) shape = load_shape(zz, zi, zp, vmi);
    const double qgen = (t == kPQLimit) ? w.qsw[i] : S.q_gen[i];
    double f0 = fma(-Vi.x, I.x, fma(-Vi.y, I.y, fma(-pl, shape, pg)));
    double f1 = fma(-Vi.y, I.x, fma(Vi.x, I.y, fma(-ql, shape, qgen)));
    f0 = t != PF_SLACK ? f0 : 0.0;
    f1 = t >= PF_PQ ? f1 : 0.0;
    if (keep_f) reinterpret_cast<double2*>(w.F)[i] = make_double2(f0, f1);
    reinterpret_cast<V2*>(y)[r.z] = mk2(narrow<TF>(f0), narrow<TF>(f1));
    m = max(m, max(abs_bits(f0), abs_bits(f1)));
    Blk<TF> D;
    if constexpr (sizeof(TF) == 4) {
      D = diag_block(S, i, t, Vi, Vi, vmi, I, pl, ql, __ldg(R.diag32 + rl));
    } else {
      D = diag_block(S, i, t, Vi, ld_state<CL>(w.U + i), vmi, I, pl, ql, yd);
    }
    if (jm) st_blk(jm + 4 * (size_t)r.w, D);
    if ((r.x & kResRowLevel0) && !inv2(D)) *bad = true;
    st_blk(A + 4 * r.y, D);
  }
  return m;
}

// Scenario gs of a state laid out [scenario][row].
__device__ __forceinline__ DevWork scenario_of(DevWork w, int n, int gs) {
  const size_t r = (size_t)gs * n;
  w.B = 1;
  if (w.in_p_load) w.in_p_load += r;
  if (w.in_q_load) w.in_q_load += r;
  if (w.in_p_gen) w.in_p_gen += r;
  if (w.in_vm) w.in_vm += r;
  if (w.in_va) w.in_va += r;
  if (w.out_vm) w.out_vm += r;
  if (w.out_va) w.out_va += r;
  if (w.out_info) w.out_info += gs;
  w.spec += 3 * r;
  w.vm += r;
  w.va += r;
  w.V += r;
  if (w.U) w.U += r;
  w.dV += r;
  w.F += 2 * r;
  w.dx += 2 * r;
  w.r += 2 * r;
  if (w.bt) {
    w.bt += r;
    w.qsw += r;
  }
  return w;
}

}  // namespace pf
