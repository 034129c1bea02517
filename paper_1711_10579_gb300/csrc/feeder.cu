// Resident Newton solves of radial three-phase feeders (feeder.h): one
// scenario per CTA or per cluster, its 6x6 diagonal blocks in shared memory.
//
// What bounds it: the chain of tree levels (about as many as the feeder is
// deep) and, in FP64, the FP64 pipe (a 6x6 elimination is ~150 instructions
// of 64 cycles per warp).  The persistent kernel (newton.cuh) gave a block to
// one thread, about 1,000 FP64 instructions in a row, and paid cluster
// barriers and L2 round trips on every level of the factorisation and both
// sweeps.  Here 8 lanes share a node, one column of [S + Y | S | y] each: the
// column to eliminate is broadcast by shuffles, the pivot is chosen by every
// lane alike, and a level ends with a block barrier.
//
// Measured (us, persistent kernel -> here): 8,000 nodes FP64 8,720 -> 1,810,
// 1,000 nodes mixed 1,450 -> 390; batches of 1,000 nodes x 61 mixed 2,410 ->
// 530, x 250 FP64 5,830 -> 4,970.  Splitting a column's rows over two lanes
// (half the FP64 instructions of an elimination, twice the warps) was no
// faster alone and 1.7 times slower in batches; Gauss-Jordan with a full pivot
// search and a division per pivot was 20% slower.
#include "feeder.h"
#include "resident.cuh"

namespace pf {

namespace {

enum { kElim = 0, kForward = 1, kBackward = 2 };

__device__ __forceinline__ float fmar(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double fmar(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ float mulr(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mulr(double a, double b) { return __dmul_rn(a, b); }
// |v| to a few digits as an ordered integer (compares stay off the FP64 pipe)
// and its step for a factor of two.
__device__ __forceinline__ int mag(float v) { return __float_as_int(v) & 0x7fffffff; }
__device__ __forceinline__ int mag(double v) { return __double2hiint(v) & 0x7fffffff; }
template <typename TF>
struct Mag {
  static constexpr int two = sizeof(TF) == 4 ? 1 << 23 : 1 << 20;
  static constexpr int inf = sizeof(TF) == 4 ? 0x7f800000 : 0x7ff00000;
};

// d += Y g for a branch admittance (complex 3x3 in the form of Eq. 21: rows
// Im, Re of the current, columns Re, Im of the voltage).
template <typename TF>
__device__ __forceinline__ void branch_madd(const TF* br, const TF (&g)[6], TF (&d)[6]) {
#pragma unroll
  for (int a = 0; a < 3; ++a)
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const TF re = br[3 * a + c], im = br[9 + 3 * a + c];
      d[a] = fmar(re, g[3 + c], fmar(im, g[c], d[a]));
      d[3 + a] = fmar(-im, g[3 + c], fmar(re, g[c], d[3 + a]));
    }
}

// D X = [b e] for the 6x6 block D (column j in d of lane j < 6) by LU: the
// column to eliminate is broadcast by shuffles and every lane updates its own
// columns; b and (INV) e end as the solution.  A diagonal entry within a
// factor of two of its column's largest is taken as the pivot; the rows are
// exchanged for the largest otherwise.  False for a zero or non-finite pivot.
template <bool INV, typename TF>
__device__ __forceinline__ bool eliminate(TF (&d)[6], TF (&b)[6], TF (&e)[6], unsigned gmask) {
  bool ok = true;
  TF U[6][6];  // [r][c], r < c: the scaled pivot rows' entries of later columns
#pragma unroll
  for (int c = 0; c < 6; ++c) {
    TF col[6];
#pragma unroll
    for (int r = 0; r < 6; ++r) {
      col[r] = __shfl_sync(gmask, d[r], c, kFeedLanes);
      if (r < c) U[r][c] = col[r];
    }
    int most = 0;
#pragma unroll
    for (int r = c + 1; r < 6; ++r) most = max(most, mag(col[r]));
    if (mag(col[c]) + Mag<TF>::two < most) {  // (the group's lanes alike)
      bool found = false;
#pragma unroll
      for (int r = c + 1; r < 6; ++r) {
        if (found || mag(col[r]) != most) continue;
        found = true;
        auto swap = [](TF& x, TF& y) {
          const TF t = x;
          x = y;
          y = t;
        };
        swap(d[c], d[r]);
        swap(b[c], b[r]);
        if (INV) swap(e[c], e[r]);
        swap(col[c], col[r]);
      }
    }
    ok = ok && col[c] != TF(0) && mag(col[c]) < Mag<TF>::inf;
    const TF rv = recip(col[c]);
    if (c < 5) d[c] = mulr(d[c], rv);
    b[c] = mulr(b[c], rv);
    if (INV) e[c] = mulr(e[c], rv);
#pragma unroll
    for (int r = c + 1; r < 6; ++r) {
      d[r] = fmar(-col[r], d[c], d[r]);
      b[r] = fmar(-col[r], b[c], b[r]);
      if (INV) e[r] = fmar(-col[r], e[c], e[r]);
    }
  }
#pragma unroll
  for (int c = 5; c > 0; --c)
#pragma unroll
    for (int r = 0; r < c; ++r) {
      b[r] = fmar(-U[r][c], b[c], b[r]);
      if (INV) e[r] = fmar(-U[r][c], e[c], e[r]);
    }
  return ok;
}

// The rounds tab[0 .. nr) of one part (offsets into rec).  Group g of lanes
// executes record tab[r].x + g of round r; the branch blocks of its next
// kFeedRing rounds are in flight by cp.async.
template <int MODE, typename TF, bool CL>
__device__ __noinline__ void run_feed(const int2* tab, int nr, const uint2* rec, TF* base,
                                      const TF* __restrict__ branch, TF* ring, int* flag) {
  constexpr int NV = FeedShape<TF>::node, NB = FeedShape<TF>::branch, D = kFeedRing;
  constexpr int kPieces = NB * (int)sizeof(TF) / 16;
  constexpr bool INV = sizeof(TF) == 4;  // refinement passes need D^-1
  // consecutive groups are in different warps: the few nodes of a narrow level
  // neither share a warp (their operations differ) nor a sub-partition
  const int lane = threadIdx.x & 31, j = lane & 7;
  const int g = (lane >> 3) * (int)(blockDim.x >> 5) + (int)(threadIdx.x >> 5);
  const unsigned gmask = 0xffu << (lane & 24);
  const int crank = CL ? (int)cg::this_cluster().block_rank() : 0;
  TF* const mine = ring + (size_t)g * D * NB;
  auto fetch = [&](int r) {  // the branch block of round r's operation
    if (r < nr) {
      const int2 q = tab[r];
      if (g < (q.y & 0xffff)) {
        const uint2 it = rec[q.x + g];
        if (it.x != kFeedNone) {
          const char* src = reinterpret_cast<const char*>(branch + (size_t)(it.y & (kFeedMaxNodes - 1)) * NB);
          char* dst = reinterpret_cast<char*>(mine + (r & (D - 1)) * NB);
          for (int k = j; k < kPieces; k += kFeedLanes) cp16(dst + 16 * k, src + 16 * k);
        }
      }
    }
    cp_commit();
  };
  if constexpr (MODE != kBackward)
    for (int r = 0; r < D; ++r) fetch(r);
  TF d[6], v = TF(0);
#pragma unroll
  for (int r = 0; r < 6; ++r) d[r] = TF(0);
  for (int r = 0; r < nr; ++r) {
    const int2 q = tab[r];
    const uint2 it = g < (q.y & 0xffff) ? rec[q.x + g] : make_uint2(kFeedNone, 0);
    if constexpr (MODE != kBackward) {
      cp_wait<D - 1>();
      __syncwarp(gmask);
    }
    if (it.x != kFeedNone) {
      TF* const me = base + (size_t)(it.x & 0xffff) * NV;
      const int other = it.x >> 16, rank = (it.y >> kFeedRankShift) & 15;
      const TF* const br = mine + (r & (D - 1)) * NB;
      if constexpr (MODE == kBackward) {
        // x_k = w_k + x_p - H_k x_p
        TF x[6];
        if (!CL || rank == crank) {
          const TF* src = base + (size_t)other * NV + 36;
#pragma unroll
          for (int c = 0; c < 6; ++c) x[c] = src[c];
        } else {
          const TF* src = remote_smem<CL>(base, rank) + (size_t)other * NV + 36;
#pragma unroll
          for (int c = 0; c < 6; ++c) x[c] = src[c];
        }
        if (j < 6) {
          TF xj = x[0];
#pragma unroll
          for (int c = 1; c < 6; ++c) xj = c == j ? x[c] : xj;
          TF s0 = xj, s1 = me[36 + j];
#pragma unroll
          for (int c = 0; c < 3; ++c) {
            s0 = fmar(-me[6 * c + j], x[c], s0);
            s1 = fmar(-me[6 * (3 + c) + j], x[3 + c], s1);
          }
          me[36 + j] = s0 + s1;
        }
      } else if constexpr (MODE == kElim) {
        if (it.y & kFeedFirst) {
#pragma unroll
          for (int k = 0; k < 6; ++k) d[k] = j < 7 ? me[6 * j + k] : TF(0);  // lane 6: y
        }
        if (!(it.y & kFeedFactor)) {
          TF x[6];
          const int jj = j < 7 ? j : 0;
          if (!CL || rank == crank) {
            const TF* src = base + (size_t)other * NV + 6 * jj;
#pragma unroll
            for (int k = 0; k < 6; ++k) x[k] = src[k];
          } else {
            const TF* src = remote_smem<CL>(base, rank) + (size_t)other * NV + 6 * jj;
#pragma unroll
            for (int k = 0; k < 6; ++k) x[k] = src[k];
          }
          branch_madd(br, x, d);
        } else {
          // H = (S + Y)^-1 S and w = (S + Y)^-1 y, Y to the parent
          TF b[6], e[6];
#pragma unroll
          for (int k = 0; k < 6; ++k) b[k] = d[k];
          if (!(it.y & kFeedRoot) && j < 6) {
#pragma unroll
            for (int a = 0; a < 3; ++a) {
              d[a] += j < 3 ? br[9 + 3 * a + j] : br[3 * a + j - 3];
              d[3 + a] += j < 3 ? br[3 * a + j] : -br[9 + 3 * a + j - 3];
            }
          }
#pragma unroll
          for (int k = 0; k < 6; ++k) e[k] = k == j ? TF(1) : TF(0);
          if (!eliminate<INV>(d, b, e, gmask)) *flag = 1;
          if (j < 7) {
#pragma unroll
            for (int k = 0; k < 6; ++k) me[6 * j + k] = b[k];
          }
          if (INV && j < 6) {
#pragma unroll
            for (int k = 0; k < 6; ++k) me[42 + 6 * j + k] = e[k];
          }
        }
      } else if constexpr (INV) {
        // forward sweep alone (FP32): lane j < 6 holds row j
        if (it.y & kFeedFirst) v = j < 6 ? me[36 + j] : TF(0);
        if (!(it.y & kFeedFactor)) {
          const TF* src = (!CL || rank == crank ? base : remote_smem<CL>(base, rank)) + (size_t)other * NV + 36;
          const int a = j < 3 ? j : (j < 6 ? j - 3 : 0);
#pragma unroll
          for (int c = 0; c < 3; ++c) {
            const TF re = br[3 * a + c], im = br[9 + 3 * a + c];
            v = j < 3 ? fmar(re, src[3 + c], fmar(im, src[c], v)) : fmar(-im, src[3 + c], fmar(re, src[c], v));
          }
        } else {
          TF s = TF(0);
#pragma unroll
          for (int c = 0; c < 6; ++c) {
            const TF yc = __shfl_sync(gmask, v, c, kFeedLanes);
            if (j < 6) s = fmar(me[42 + 6 * c + j], yc, s);
          }
          if (j < 6) me[36 + j] = s;
        }
      }
    }
    if constexpr (MODE != kBackward) {
      __syncwarp(gmask);  // the group has read its branch block
      fetch(r + D);
    }
    if (q.y < 0) __syncthreads();
  }
}

// Load current of a phase, I = conj(S(m)) V / m^2 (Eq. 17 with the ZIP load
// of Eq. 14-15, m = |V|), and its derivatives: with conj(S) = k (zp + zi m +
// zz m^2), k = (-pl, ql), I = k s V for s = zp/m^2 + zi/m + zz, and dI = k (s
// dV + V t (Vr dVr + Vi dVi)), t = (ds/dm)/m = -(2 zp + zi m) / m^4.
__device__ __forceinline__ void load_current(double2 V, double pl, double ql, double zp, double zi,
                                             double zz, double2& I, double2& dr, double2& di) {
  const double m2 = dot2(V.x, V.x, V.y, V.y);
  const double m = sqrt(m2), r = 1.0 / m2, q = __dmul_rn(zi, m);
  const double s = __fma_rn(zp + q, r, zz);
  const double t = __dmul_rn(__dmul_rn(-__fma_rn(2.0, zp, q), r), r);
  const double tx = __dmul_rn(t, V.x), ty = __dmul_rn(t, V.y), xy = __dmul_rn(tx, V.y);
  const double sx = __dmul_rn(s, V.x), sy = __dmul_rn(s, V.y);
  const double ux = __fma_rn(tx, V.x, s), uy = __fma_rn(ty, V.y, s);
  I = make_double2(dot2(-pl, sx, -ql, sy), dot2(-pl, sy, ql, sx));
  dr = make_double2(dot2(-pl, ux, -ql, xy), dot2(-pl, xy, ql, ux));
  di = make_double2(dot2(-pl, xy, -ql, uy), dot2(-pl, uy, ql, xy));
}

template <typename TF, bool CL>
__device__ __forceinline__ void feeder_solve(const DevSys& S, const DevWork& w, const DevOpts& o,
                                             const FeedDev& R, int lin) {
  constexpr int NV = FeedShape<TF>::node, NB = FeedShape<TF>::branch;
  const int P = CL ? (int)cg::this_cluster().num_blocks() : 1;
  const int crank = CL ? (int)cg::this_cluster().block_rank() : 0;
  const int tid = threadIdx.x, T = blockDim.x, lane = tid & 31, warp = tid >> 5, nwarp = T >> 5;
  extern __shared__ __align__(16) unsigned char dsm[];
  TF* const base = reinterpret_cast<TF*>(dsm);
  TF* const ring = reinterpret_cast<TF*>(
      dsm + (((size_t)R.max_slots * NV * sizeof(TF) + 15) & ~(size_t)15));
  uint2* const rec =
      reinterpret_cast<uint2*>(ring + (size_t)(T / kFeedLanes) * kFeedRing * NB);
  int2* const tab = reinterpret_cast<int2*>(rec + R.max_rec);
  __shared__ FeedPart sp[2];  // this CTA's part, and the top
  __shared__ FeedCta sc;
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
  const FeedPart& part = sp[0];
  const FeedPart& top = sp[1];
  const bool has_top = CL && crank == 0;
  // records and rounds of the part and the top, with offsets into rec
  const int nrnd = part.nrf + part.nrb;
  int nrec = 0;
  for (int p = 0; p < (has_top ? 2 : 1); ++p) {
    const FeedPart& Q = sp[p];
    const int nr = Q.nrf + Q.nrb, at = p ? nrnd : 0;
    if (nr == 0) continue;
    const int r0 = R.rnd[Q.rf].x;
    const int2 last = R.rnd[Q.rf + nr - 1];
    const int cnt = last.x + (last.y & 0xffff) - r0;
    for (int k = tid; k < nr; k += T) {
      const int2 q = R.rnd[Q.rf + k];
      tab[at + k] = make_int2(q.x - r0 + nrec, q.y);
    }
    for (int k = tid; k < cnt; k += T) rec[nrec + k] = R.rec[r0 + k];
    nrec += cnt;
  }
  const TF* const branch = reinterpret_cast<const TF*>(R.branch);
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
  auto nodes = [&](auto fn) {  // fn(node, its values in shared memory)
    for (int k = tid; k < sc.nown; k += T) {
      const int2 q = __ldg(R.node + sc.own + k);
      fn(q.x, base + (size_t)q.y * NV);
    }
  };
  nodes([&](int i, TF*) { setup_row<true>(S, w, i, 0); });
  csync<CL>();
  tick(kProfSetup);

  int status = kRunning, passes = 0;
  double prev = 0.0;
  for (int it = 0;; ++it) {
    // ---- current mismatch (Eq. 12-19) and diagonal blocks (Eq. 21-23) ----
    unsigned long long m = 0ull;
    for (int gq = warp; gq < sc.ngrp; gq += nwarp) {
      const FeedGroup G = R.grp[sc.grp + gq];
      const int2 id = __ldg(R.item + (size_t)(sc.grp + gq) * 32 + lane);
      const bool on = id.x >= 0, fr = on && (id.x >> 30);
      const int k = on ? (id.x & (kFeedMaxNodes - 1)) : 0, a = on ? (id.x >> 28) & 3 : 0;
      double2 I = make_double2(0.0, 0.0);
#pragma unroll 2
      for (int e = 0; e < G.width; ++e) {
        const size_t q = (size_t)G.ell + 32 * e + lane;
        const int c = __ldg(R.ell_col + q);
        const double2* yv = R.ell_y + 3 * ((size_t)G.ell + 32 * e) + lane;
#pragma unroll
        for (int b = 0; b < 3; ++b) {
          const double2 yb = __ldg(yv + 32 * b), v = ld_state<CL>(w.V + 3 * (size_t)c + b);
          I.x = fma(yb.x, v.x, I.x);
          I.x = fma(-yb.y, v.y, I.x);
          I.y = fma(yb.x, v.y, I.y);
          I.y = fma(yb.y, v.x, I.y);
        }
      }
      if (!on) continue;
      TF* const me = base + (size_t)id.y * NV;
      double2 dI = make_double2(0.0, 0.0), dr = dI, di = dI;
      if (fr) {
        const double2 V = ld_state<CL>(w.V + 3 * (size_t)k + a);
        const double pl = w.spec[(size_t)k * 6 + a], ql = w.spec[(size_t)k * 6 + 3 + a];
        double2 Isp;
        load_current(V, pl, ql, S.zip[3 * k], S.zip[3 * k + 1], S.zip[3 * k + 2], Isp, dr, di);
        dI = csub(Isp, I);
        const double sx = dot2(V.x, dI.x, V.y, dI.y), sy = dot2(V.y, dI.x, -V.x, dI.y);
        m = max(m, max(abs_bits(sx), abs_bits(sy)));
      }
      me[36 + a] = (TF)dI.y;
      me[39 + a] = (TF)dI.x;
      // rows a and 3 + a of S: what the branches do not carry to a parent or a
      // child, less the load's slope
      const TF* yd = reinterpret_cast<const TF*>(R.ydiag) + ((size_t)k * 3 + a) * 6;
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        TF re = TF(0), im = TF(0);
        if (fr) {
          re = __ldg(yd + 2 * c);
          im = __ldg(yd + 2 * c + 1);
        }
        const bool own = c == a;
        me[6 * c + a] = own ? (fr ? im - (TF)dr.y : TF(1)) : im;
        me[6 * (3 + c) + a] = own && fr ? re - (TF)di.y : re;
        me[6 * c + 3 + a] = own && fr ? re - (TF)dr.x : re;
        me[6 * (3 + c) + 3 + a] = own ? (fr ? -im - (TF)di.x : TF(1)) : -im;
      }
      if (o.refine > 0) {
        w.F[(size_t)k * 6 + a] = dI.y;
        w.F[(size_t)k * 6 + 3 + a] = dI.x;
        w.abcd[(size_t)k * 12 + a] = dr.y;
        w.abcd[(size_t)k * 12 + 3 + a] = di.y;
        w.abcd[(size_t)k * 12 + 6 + a] = dr.x;
        w.abcd[(size_t)k * 12 + 9 + a] = di.x;
      }
    }
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

    // ---- elimination towards the root, substitution back; refinement ----
    const int npass = refine ? o.refine : 0;
    bool singular = false;
    for (int pass = 0; pass <= npass; ++pass) {
      if (pass == 0) {
        run_feed<kElim, TF, CL>(tab, part.nrf, rec, base, branch, ring, &sh_flag);
      } else {
        nodes([&](int i, TF*) { dv_row<true>(S, w, i, 0); });
        csync<CL>();
        nodes([&](int i, TF* me) {
          resid_row<true>(S, w, i, 0);
          for (int c = 0; c < 6; ++c) me[36 + c] = (TF)w.r[(size_t)i * 6 + c];
        });
        __syncthreads();
        tick(kProfResidual);
        run_feed<kForward, TF, CL>(tab, part.nrf, rec, base, branch, ring, &sh_flag);
      }
      if constexpr (CL) {
        csync<CL>();
        if (pass == 0 && tid == 0 && crank != 0 && sh_flag) *remote_smem<CL>(&sh_flag, 0) = 1;
        if (crank == 0) {
          if (pass == 0)
            run_feed<kElim, TF, CL>(tab + nrnd, top.nrf, rec, base, branch, ring, &sh_flag);
          else
            run_feed<kForward, TF, CL>(tab + nrnd, top.nrf, rec, base, branch, ring, &sh_flag);
          if (pass == 0) tick(kProfFactor);
          run_feed<kBackward, TF, CL>(tab + nrnd + top.nrf, top.nrb, rec, base, branch, ring, &sh_flag);
        }
        csync<CL>();
        if (pass == 0) singular = *remote_smem<CL>(&sh_flag, 0) != 0;
      } else {
        if (pass == 0) tick(kProfFactor);
      }
      run_feed<kBackward, TF, CL>(tab + part.nrf, part.nrb, rec, base, branch, ring, &sh_flag);
      if (!CL && pass == 0) singular = sh_flag != 0;
      ++passes;
      if (npass > 0)
        nodes([&](int i, TF* me) {
          for (int c = 0; c < 6; ++c) {
            double* d = w.dx + (size_t)i * 6 + c;
            *d = pass == 0 ? (double)me[36 + c] : *d + (double)me[36 + c];
          }
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
    nodes([&](int i, TF* me) {
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        const double dr = npass > 0 ? w.dx[(size_t)i * 6 + a] : (double)me[36 + a];
        const double di = npass > 0 ? w.dx[(size_t)i * 6 + 3 + a] : (double)me[39 + a];
        ms = max(ms, max(abs_bits(dr), abs_bits(di)));
        const double2 v = w.V[(size_t)i * 3 + a];
        w.V[(size_t)i * 3 + a] = make_double2(v.x + dr, v.y + di);
      }
    });
    spread<CL>(ms, sh_red, sh_step, P, crank);
    csync<CL>();
    tick(kProfUpdate);
  }

  // ---- results in the caller's numbering ----
  nodes([&](int i, TF*) { output_row<true>(S, w, i, 0, status == PF_OK); });
  tick(kProfOutput);
  if (crank == 0) {
    __syncthreads();
    if (tid == 0 && w.out_info) w.out_info->solve_us = (double)(global_ns() - t_begin) * 1e-3;
  }
}

// Scenario gs of a state laid out [scenario][node].
__device__ __forceinline__ DevWork feeder_scenario(DevWork w, int n, int gs) {
  const size_t r = (size_t)gs * n;
  w.B = 1;
  if (w.in_p_load) w.in_p_load += 3 * r;
  if (w.in_q_load) w.in_q_load += 3 * r;
  if (w.in_vm) w.in_vm += 3 * r;
  if (w.in_va) w.in_va += 3 * r;
  if (w.out_vm) w.out_vm += 3 * r;
  if (w.out_va) w.out_va += 3 * r;
  if (w.out_info) w.out_info += gs;
  w.spec += 6 * r;
  w.V += 3 * r;
  w.dV += 3 * r;
  w.abcd += 12 * r;
  w.F += 6 * r;
  w.dx += 6 * r;
  w.r += 6 * r;
  w.qg += 3 * r;
  if (w.bt) w.bt += r;
  return w;
}

template <typename TF, bool CL>
__global__ void __launch_bounds__(256)
    k_feeder(DevSys S, DevWork w, DevOpts o, FeedDev R, int lin) {
  const int gs = CL ? blockIdx.x / (int)cg::this_cluster().num_blocks() : blockIdx.x;
  feeder_solve<TF, CL>(S, feeder_scenario(w, S.n, gs), o, R, lin);
}

// Several requests in one launch (as k_resident_group).
template <typename TF, bool CL>
__global__ void __launch_bounds__(256) k_feeder_group(const GroupJob* desc, GroupList list) {
  const int csize = CL ? (int)cg::this_cluster().num_blocks() : 1;
  const int crank = CL ? (int)cg::this_cluster().block_rank() : 0;
  __shared__ GroupJob job;
  __shared__ FeedDev plan;
  {
    const GroupJob* src = desc + list.job[blockIdx.x / csize];
    for (int k = threadIdx.x; k < (int)(sizeof(GroupJob) / 4); k += blockDim.x)
      reinterpret_cast<unsigned*>(&job)[k] = reinterpret_cast<const unsigned*>(src)[k];
    __syncthreads();
    for (int k = threadIdx.x; k < (int)(sizeof(FeedDev) / 4); k += blockDim.x)
      reinterpret_cast<unsigned*>(&plan)[k] = static_cast<const unsigned*>(job.res)[k];
  }
  __syncthreads();
  feeder_solve<TF, CL>(job.S, job.w, job.o, plan, 0);
  __threadfence_system();
  csync<CL>();
  if (crank == 0 && threadIdx.x == 0) {
    __threadfence_system();
    *reinterpret_cast<volatile int*>(job.done) = 1;
  }
}

template <typename TF, bool CL>
cudaError_t launch_feed(const DevSys& S, const DevWork& w, const DevOpts& o, const FeedDev& R,
                        size_t smem, int B, int lin, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  const cudaError_t e = configure_clusters(k_feeder<TF, CL>, R.P, R.threads, smem, B, st, cfg, attr);
  if (e != cudaSuccess) return e;
  return cudaLaunchKernelEx(&cfg, k_feeder<TF, CL>, S, w, o, R, lin);
}

template <typename TF, bool CL>
cudaError_t launch_group(const GroupJob* desc, const GroupList& list, size_t smem, int P, int threads,
                         cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  const cudaError_t e =
      configure_clusters(k_feeder_group<TF, CL>, P, threads, smem, list.n, st, cfg, attr);
  if (e != cudaSuccess) return e;
  return cudaLaunchKernelEx(&cfg, k_feeder_group<TF, CL>, desc, list);
}

}  // namespace

cudaError_t launch_feeder(bool fp32, const DevSys& S, const DevWork& w, const DevOpts& o,
                          const FeedDev& R, size_t smem, int B, int lin, cudaStream_t st) {
  if (R.P > 1)
    return fp32 ? launch_feed<float, true>(S, w, o, R, smem, B, lin, st)
                : launch_feed<double, true>(S, w, o, R, smem, B, lin, st);
  return fp32 ? launch_feed<float, false>(S, w, o, R, smem, B, lin, st)
              : launch_feed<double, false>(S, w, o, R, smem, B, lin, st);
}

cudaError_t launch_feeder_group(bool fp32, const GroupJob* desc, const GroupList& list, size_t smem,
                                int P, int threads, cudaStream_t st) {
  if (list.n <= 0 || list.n > kGroupMax) return cudaErrorInvalidValue;
  if (P > 1)
    return fp32 ? launch_group<float, true>(desc, list, smem, P, threads, st)
                : launch_group<double, true>(desc, list, smem, P, threads, st);
  return fp32 ? launch_group<float, false>(desc, list, smem, P, threads, st)
              : launch_group<double, false>(desc, list, smem, P, threads, st);
}

int feeder_clusters(bool fp32, int P, int threads, size_t smem) {
  if (P > 1)
    return fp32 ? count_clusters(k_feeder<float, true>, P, threads, smem)
                : count_clusters(k_feeder<double, true>, P, threads, smem);
  return fp32 ? count_clusters(k_feeder<float, false>, P, threads, smem)
              : count_clusters(k_feeder<double, false>, P, threads, smem);
}

}  // namespace pf
