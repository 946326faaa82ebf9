// adjoint_fx.cuh -- the KEP flux's transposed volume integral in fixed point.
//
// The pair terms of the adjoint (45 FP64 operations each, 540 of the element
// kernel's 1124 FP64 instructions per node) run on the integer pipes in the
// arithmetic of volume_fx.cuh: the state and the cotangents lam~ = -lam / J are
// 62-bit integers in units of the element, one for the density's cotangent, one
// for the momentum's and one for the energy's.  In the terms that add them, mu0 +
// (mu_m . S_u + mu_4 S_h) / 2, each is shifted to the coarsest of the three
// units.  Cotangents are of either sign and any size, so the terms lie further
// below their bounds than the forward fluxes do; a line's sums therefore keep
// 28 more bits (the full product of the last factors), the sum of the three is
// normalised in each lane before it is multiplied, and the directions' sums are
// added in FP64: the error against the extended-precision oracle's J^T lam
// stays at FP64's.  Elements out of range (non-finite values; a value's or a
// cotangent's largest magnitude beyond 2^200 or below 2^-200 without being zero;
// density or enthalpy differing by more than a factor 4 over the nodes: the gradients
// at the light ones are divided by their own density) are summed in FP64.
#pragma once
#include "adjoint.cuh"
#include "volume_fx.cuh"

namespace dg {

enum { AX_RHO, AX_U, AX_H, AX_L0, AX_LM, AX_LE, AX_NRHO, AX_NH, AX_V, AX_W, AX_LM1, AX_LM2, AX_NUM };
struct AdjFxPlan {
  int ok;
  int bR, bU, bH, bL0, bLM, bLE;  // biased exponent bounds for fx_of
  int s0, s1, s2;                 // right shifts of mu0, mu_m . S_u, mu_4 S_h to their common unit
  int eg[4];                      // the units of the sums rho, u, p, h
};
// Stretched elements (FxMetric): what differs by component c of u, Ja and the
// momentum's cotangent (s1, eg[1] and bU, bLM of AdjFxPlan are not used); as FxRows
struct AdjFxRows {
  int bU[3], bLM[3];
  int t[3], s1[3], sz[3];         // right shifts of S_u S_a, mu_c S_u and mu_c S_a to their sums' units
  int yt[3], yq[3];               // and of tt S_a and (S_u . S_a / 2) mu_c to that of the velocity's term
  long long ht[3], h1[3], hz[3], hyt[3], hyq[3];  // half of what they drop
  int eg[3];                      // the units of the sums u
};

// ex: the largest fx_mag of each value (AX_NRHO, AX_NH: of 0x7fffffff - fx_mag); mt: the element's metrics; eW:
// lam~ / w is in units 2^eW times lam~'s.  Bounds in units of 2^60, times Q for the
// pair terms: the sum of the three parts 3 (half of 6, by the extra shift), rho
// and u 1.1, p 1.5, h 0.75; a line's sum of |Q| is below 3.7.
template <bool GEN>
__device__ __forceinline__ AdjFxPlan adj_fx_plan(const int* ex, const FxMetric& mt, int eW, AdjFxRows* rows) {
  AdjFxPlan f;
  const bool st = GEN && mt.kind == FX_STRETCHED;
  const int xU[3] = {ex[AX_U], ex[AX_V], ex[AX_W]}, xM[3] = {ex[AX_LM], ex[AX_LM1], ex[AX_LM2]};
  int eX[AX_NRHO];
  bool zero[AX_NRHO];
  bool ok = true;
#pragma unroll
  for (int x = 0; x < AX_NRHO; ++x) {
    int mag = ex[x];
    if (GEN && x == AX_U) mag = max(mag, max(xU[1], xU[2]));
    if (GEN && x == AX_LM) mag = max(mag, max(xM[1], xM[2]));
    const int e = (mag >> 20) - 1022;
    eX[x] = max(e, -200);  // (zeros in that unit)
    ok = ok && e < 200 && (e > -200 || mag == 0);
    zero[x] = mag == 0;
  }
  const int eA = (max(mt.col[0], max(mt.col[1], mt.col[2])) >> 20) - 1022;
  f.bR = eX[AX_RHO] + 1022; f.bU = eX[AX_U] + 1022; f.bH = eX[AX_H] + 1022;
  f.bL0 = eX[AX_L0] + 1022; f.bLM = eX[AX_LM] + 1022; f.bLE = eX[AX_LE] + 1022;
  // units of the three parts of mu0 + (mu_m . S_u + mu_4 S_h) / 2 (a part that is zero
  // must not raise the others' unit)
  auto unit = [](bool zero, int e) { return zero ? -2000 : e; };
  const int e0 = unit(zero[AX_L0], eX[AX_L0] + eW - 60),
            e2 = unit(zero[AX_LE] || zero[AX_H], eX[AX_LE] + eX[AX_H] + eW - 59);
  int e1 = unit(zero[AX_LM] || zero[AX_U], eX[AX_LM] + eX[AX_U] + eW - 59);
  // stretched: exponents of u_c, mu_c (no further than 2^-40 below the largest) and Ja_c
  int eC[3], eM[3], aC[3], E = eX[AX_U] + eA, Z = -3000;  // E, Z: of S_u . S_a and mu . S_a
  if (st) {
    e1 = -2000;
    E = -3000;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      eC[c] = max((xU[c] >> 20) - 1022, eX[AX_U] - 40);
      eM[c] = max((xM[c] >> 20) - 1022, eX[AX_LM] - 40);
      aC[c] = (mt.col[c] >> 20) - 1022;
      ok = ok && abs(aC[c]) < 200;
      E = max(E, eC[c] + aC[c]);
      Z = max(Z, eM[c] + aC[c]);
      e1 = max(e1, unit(zero[AX_LM] || zero[AX_U], eM[c] + eC[c] + eW - 59));
    }
  }
  const int et = max(e0, max(e1, e2)) + 1;
  if (st) {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      auto shift = [](int x) { return min(max(x, 0), 62); };
      auto half = [](int k) { return (1LL << k) >> 1; };
      rows->bU[c] = eC[c] + 1022;
      rows->bLM[c] = eM[c] + 1022;
      rows->t[c] = shift(E - eC[c] - aC[c]);
      rows->s1[c] = shift(et - (eM[c] + eC[c] + eW - 59));
      rows->sz[c] = shift(Z - eM[c] - aC[c]);
      const int ut = et + aC[c] + 3, uq = unit(zero[AX_LM], E + eM[c] + eW - 56), G = max(ut, uq);
      rows->yt[c] = shift(G - ut);
      rows->yq[c] = shift(G - uq);
      rows->eg[c] = G + eX[AX_RHO] - 1;
      rows->ht[c] = half(rows->t[c]);
      rows->h1[c] = half(rows->s1[c]);
      rows->hz[c] = half(rows->sz[c]);
      rows->hyt[c] = half(rows->yt[c]);
      rows->hyq[c] = half(rows->yq[c]);
    }
  }
  f.s0 = min(et - e0, 63); f.s1 = min(et - e1, 63); f.s2 = min(et - e2, 63);
  f.eg[0] = et + E + 3;
  f.eg[1] = et + eX[AX_RHO] + eA + 2;
  f.eg[2] = (st ? Z : eX[AX_LM] + eA) + eW - 58;
  f.eg[3] = E + eX[AX_LE] + eW + eX[AX_RHO] - 57;
  const bool even = (ex[AX_RHO] >> 20) - ((0x7fffffff - ex[AX_NRHO]) >> 20) <= 1 &&
                    (ex[AX_H] >> 20) - ((0x7fffffff - ex[AX_NH]) >> 20) <= 1;
  f.ok = ok && even && abs(eA) < 200 && mt.kind < FX_GRADED;
  return f;
}

// a product in units of 2^62 of the factors' units and its next 32 bits (lo in
// units of 2^-31: the sum of lo's may carry)
struct Fx96 {
  long long hi;
  unsigned lo;
};
__device__ __forceinline__ Fx96 fx_mul96(Fx a, Fx b) {
  const long long ll = mulw(a.l, b.l);
  const long long x = madw((int)(ll >> 32), 2, madw(a.l, b.h, mulw(a.h, b.l)));
  return Fx96{madw((int)(x >> 32), 2, mulw(a.h, b.h)), (unsigned)x};
}

template <int N>
struct AdjFxShape {
  static constexpr int n = N + 1, n2 = n * n, n3 = n2 * n;
  // 8-byte values per node: 6 node values (fixed point 5), 5 cotangents, 5 of
  // them over w, 3 metrics of the pass's direction, 6 sums
  static constexpr int SMEM = (25 * n3 + n2 + 2 * n) * 8;
  // lam~ / w is kept in units 2^(eW + 1 - LSH) times lam~'s: at N = 8 the largest
  // 1 / w, 36, leaves almost a bit of 2^eW = 64 unused
  static constexpr int LSH = N == 8 ? 2 : 1;
};

// The three direction passes: sQ [5][n3] (rho, u, v, w, h), sL [5][n3], sLt
// [5][n3] scratch, sA [3][n3] scratch, sG [6][n3] the sums of (rho, u, v, w, p', h),
// in FP64.
// Lanes, pairs and shuffles as in volume_passes_fx; a pair's terms are the same
// for its two nodes.  ST: a stretched element, with its rows r (read from shared
// memory as in volume_passes_fx).
template <int N, bool ST>
__device__ __forceinline__ void adj_passes_fx(const Fx* sQ, const Fx* sL, Fx* sLt, Fx* sA, double* sG, const Fx* sT,
                                              const long long* sW, const MeshDev<double>& m, size_t S, size_t e0, int e,
                                              const AdjFxPlan& f, const volatile AdjFxRows& r, int t) {
  using Sh = VolShape<N>;
  constexpr int n = Sh::n, n2 = Sh::n2, n3 = Sh::n3, LPW = Sh::LPW;
  const int warp = t >> 5, lane = t & 31;
  const int seg = lane / n, pos = lane - seg * n;
  const int L0 = warp * LPW + seg;
  const bool active = (seg < LPW) && (L0 < n2);
  const int L = active ? L0 : 0;
  const int base = seg * n;
  const int la = L % n, lb = L / n;
#pragma unroll 1
  for (int dir = 0; dir < 3; ++dir) {
    const int me = dir == 0 ? pos + n * L : (dir == 1 ? la + n * pos + n2 * lb : L + n2 * pos);
    const int ms = vslot<N, double>(me);
    Fx q[5], a[3], l[5];
    {
      // lam~ / w
      const Fx wi = fx_split<0>(sW[pos]);
#pragma unroll
      for (int v = 0; v < 5; ++v) {
        l[v] = fx_split<0>(fx_mul_shl(sL[v * n3 + ms], wi, AdjFxShape<N>::LSH));
        if (active) sLt[v * n3 + ms] = l[v];
      }
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const size_t x = (size_t)(dir * 3 + c) * S + e0 + me;
        a[c] = N == 7 || m.JaX ? m.JaX[x] : metric_fx(m.Ja[x], m.JaX_max[e], c);
        if (active) sA[c * n3 + ms] = a[c];
      }
    }
#pragma unroll
    for (int v = 0; v < 5; ++v) q[v] = sQ[v * n3 + ms];
    __syncthreads();
    long long acc[6] = {0, 0, 0, 0, 0, 0};
    unsigned low[6] = {0, 0, 0, 0, 0, 0};  // their next 28 bits, units of 2^-27
#pragma unroll
    for (int d = 1; d <= n / 2; ++d) {
      const int pm = pos + d < n ? pos + d : pos + d - n;
      const int sm = __shfl_sync(0xffffffffu, ms, base + pm);
      const Fx Q = sT[pos * n + pm];
      auto dif = [&](int v) {
        const Fx x = sLt[v * n3 + sm];
        return Fx{l[v].h - x.h, l[v].l - x.l};
      };
      const Fx Sa0 = a[0] + sA[sm], Sa1 = a[1] + sA[n3 + sm], Sa2 = a[2] + sA[2 * n3 + sm];
      const Fx Su = q[1] + sQ[n3 + sm], Sv = q[2] + sQ[2 * n3 + sm], Sw = q[3] + sQ[3 * n3 + sm];
      const Fx m1 = dif(1), m2 = dif(2), m3 = dif(3), m4 = dif(4);
      long long qv, mu;  // S_u . S_a; mu_m . S_u in the unit of tt
      if constexpr (ST) {
        qv = (FxSum(Su, Sa0, r.ht[0]).get() >> r.t[0]) + (FxSum(Sv, Sa1, r.ht[1]).get() >> r.t[1]) +
             (FxSum(Sw, Sa2, r.ht[2]).get() >> r.t[2]);
        mu = (FxSum(m1, Su, r.h1[0]).get() >> r.s1[0]) + (FxSum(m2, Sv, r.h1[1]).get() >> r.s1[1]) +
             (FxSum(m3, Sw, r.h1[2]).get() >> r.s1[2]);
      } else {
        FxSum k(Su, Sa0);
        k.add(Sv, Sa1);
        k.fold();
        k.add(Sw, Sa2);
        qv = k.get();
        FxSum x(m1, Su);  // (differences have limbs as large as sums: one term is up to 4.3 2^60)
        x.fold();
        x.add(m2, Sv);
        x.fold();
        x.add(m3, Sw);
        mu = x.get() >> f.s1;
      }
      const Fx m0 = dif(0);
      const long long tt =
          ((((long long)m0.h << 31) + m0.l) >> f.s0) + mu + (fx_mul(m4, q[4] + sQ[4 * n3 + sm]) >> f.s2);
      const Fx Qv = fx_split<1>(qv);
      const long long sq = fx_mul(q[0] + sQ[sm], Q);  // S_rho Q
      // tt (and S_u . S_a / 2 beside it) shifted up in this lane as far as both
      // have room, S_rho Q down by as much
      auto room = [](long long r) { return __clzll(r ^ (r >> 63)) - 3; };
      const int s1 = ST ? 0 : f.s1;
      const int up = max(0, min(min(room(tt), room(qv) + s1), 20));
      const Fx Tn = fx_split<0>(tt << up);
      const Fx Qs = fx_split<0>(up > s1 ? qv << (up - s1) : qv >> (s1 - up));
      const Fx Sr = fx_split<1>(sq), Sn = fx_split<1>(sq >> up);
      Fx96 F[6];
      F[0] = fx_mul96(fx_split<0>(tt), fx_split<0>(fx_mul(Qv, Q)));
      auto vel = [&](Fx Sa, Fx mk, int c) {
        if constexpr (ST) {
          return fx_mul96(Sn, fx_split<1>((FxSum(Tn, Sa, r.hyt[c]).get() >> r.yt[c]) +
                                          (FxSum(Qs, mk, r.hyq[c]).get() >> r.yq[c])));
        } else {
          FxSum y(Tn, Sa);
          y.add(Qs, mk);
          return fx_mul96(Sn, fx_split<1>(y.get()));
        }
      };
      F[1] = vel(Sa0, m1, 0);
      F[2] = vel(Sa1, m2, 1);
      F[3] = vel(Sa2, m3, 2);
      long long zz;  // mu_m . S_a
      if constexpr (ST) {
        zz = (FxSum(m1, Sa0, r.hz[0]).get() >> r.sz[0]) + (FxSum(m2, Sa1, r.hz[1]).get() >> r.sz[1]) +
             (FxSum(m3, Sa2, r.hz[2]).get() >> r.sz[2]);
      } else {
        FxSum z(m1, Sa0);
        z.add(m2, Sa1);
        z.fold();
        z.add(m3, Sa2);
        zz = z.get();
      }
      F[4] = fx_mul96(fx_split<1>(zz), Q);
      F[5] = fx_mul96(Sr, fx_split<0>(fx_mul(Qv, m4)));
#pragma unroll
      for (int v = 0; v < 6; ++v) {
        F[v].lo >>= 4;
        acc[v] += F[v].hi;
        low[v] += F[v].lo;
      }
      if (2 * d != n) {
        const int src = base + (pos - d >= 0 ? pos - d : pos - d + n);
#pragma unroll
        for (int v = 0; v < 6; ++v) {
          acc[v] += __shfl_sync(0xffffffffu, F[v].hi, src);
          low[v] += __shfl_sync(0xffffffffu, F[v].lo, src);
        }
      }
    }
    if (active) {
#pragma unroll
      for (int v = 0; v < 6; ++v) {
        // to FP64, with as many of the low bits as there is room for
        const long long s = acc[v] + (low[v] >> 27);
        const int k = min(max(__clzll(s ^ (s >> 63)) - 2, 0), 27);
        const long long w = (s << k) + ((low[v] & 0x7ffffffu) >> (27 - k));
        const int eg = ST && v > 0 && v < 4 ? r.eg[v - 1] : f.eg[v == 0 ? 0 : (v < 4 ? 1 : v - 2)];
        const double x = fx_double(w, eg - k);
        sG[v * n3 + ms] = dir == 0 ? x : x + sG[v * n3 + ms];
      }
    }
    __syncthreads();
  }
}

// an element summed in FP64 (adj_fx_plan); rare, so kept out of line
template <int N>
__device__ __noinline__ void adj_volume_fp64(double* smem, const MeshDev<double>& m, const PhysDev& ph,
                                             const Tables<N>& tab, int e, int t) {
  constexpr int n = N + 1, n2 = n * n, n3 = n2 * n, T = VolShape<N>::THREADS;
  double *sQ = smem, *sL = sQ + 6 * n3, *sLt = sL + 5 * n3, *sA = sLt + 5 * n3, *sG = sA + 3 * n3, *sDVS = sG + 6 * n3,
         *siw = sDVS + n2;
  for (int x = t; x < n2; x += T) sDVS[x] = 8.0 * tab.DVS8[x] / tab.iw[x / n];
  if (t < n) siw[t] = tab.iw[t];
  __syncthreads();
  adj_pairs_fp64<N, false>(sQ, sL, sLt, sG, sDVS, siw, ph, t, [&](int dir, int me, bool active) {
#pragma unroll
    for (int c = 0; c < 3; ++c)
      if (active) sA[c * n3 + me] = m.Ja[(size_t)(dir * 3 + c) * ((size_t)m.K * n3) + (size_t)e * n3 + me];
    return (const double*)sA;
  });
}

// k_adj_volume: one CTA per element; gV = the volume integral's and the body
// force's part of gU (through the primitives).  Measured at N = 7, 10^3
// elements: the element kernel with the pairs in FP64 1181 us (FP64 pipe 86 %
// busy); 497 us without them and 231 us here (issue 51 %, integer pipes 39 %,
// FP64 pipe 30 %, of which the recovery of the primitives and its transpose).
// GEN: for meshes with stretched elements.
template <int N, bool GEN>
__global__ void __launch_bounds__(VolShape<N>::THREADS, (resident_ctas(VolShape<N>::THREADS, AdjFxShape<N>::SMEM, 1024)))
k_adj_volume(const double* __restrict__ U, const double* __restrict__ lam, const MeshDev<double> m, const PhysDev ph,
             const Tables<N> tab, const FxTab<N> ft, double* __restrict__ gV) {
  constexpr int n = N + 1, n2 = n * n, n3 = n2 * n, T = VolShape<N>::THREADS;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ int sEx[AX_NUM];
  __shared__ AdjFxPlan sF;
  __shared__ AdjFxRows sRows;
  Fx* sQ = reinterpret_cast<Fx*>(smem_raw);
  Fx* sL = sQ + 6 * n3;
  Fx* sLt = sL + 5 * n3;
  Fx* sA = sLt + 5 * n3;
  double* sG = reinterpret_cast<double*>(sA + 3 * n3);
  Fx* sT = reinterpret_cast<Fx*>(sG + 6 * n3);
  long long* sW = reinterpret_cast<long long*>(sT + n2);
  const int e = blockIdx.x, t = threadIdx.x;
  const size_t S = (size_t)m.K * n3, e0 = (size_t)e * n3, g = e0 + t;
  Prim<double> q{0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
  double l[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
  if (t < n3) {
    q = primitive<double>(U[g], U[S + g], U[2 * S + g], U[3 * S + g], U[4 * S + g], ph);
    const double iJ = m.invJ[g];
#pragma unroll
    for (int v = 0; v < 5; ++v) l[v] = -lam[v * S + g] * iJ;
  }
  if (t < AX_NUM) sEx[t] = 0;
  for (int x = t; x < n2; x += T) sT[x] = ft.Q[x];
  if (t < n) sW[t] = ft.iw[t];
  __syncthreads();
  {
    const bool in = t < n3;
    const int mu = max(max(fx_mag(q.u), fx_mag(q.v)), fx_mag(q.w)), ml = max(max(fx_mag(l[1]), fx_mag(l[2])), fx_mag(l[3]));
    const int ex[AX_NUM] = {fx_mag(q.rho), GEN ? fx_mag(q.u) : mu, fx_mag(q.h), fx_mag(l[0]), GEN ? fx_mag(l[1]) : ml,
                            fx_mag(l[4]), in ? 0x7fffffff - fx_mag(q.rho) : 0, in ? 0x7fffffff - fx_mag(q.h) : 0,
                            fx_mag(q.v), fx_mag(q.w), fx_mag(l[2]), fx_mag(l[3])};
#pragma unroll
    for (int x = 0; x < (GEN ? AX_NUM : AX_V); ++x) {
      const int mx = __reduce_max_sync(0xffffffffu, ex[x]);
      if ((t & 31) == 0) atomicMax(&sEx[x], mx);
    }
  }
  __syncthreads();
  if (t == 0) sF = adj_fx_plan<GEN>(sEx, m.JaX_max[e], ft.eW + 1 - AdjFxShape<N>::LSH, &sRows);
  __syncthreads();
  const AdjFxPlan f = sF;
  const bool st = GEN && m.JaX_max[e].kind == FX_STRETCHED;
  // node slots: swizzled in fixed point (vslot), natural in FP64
  if (t < n3) {
    const int ts = f.ok ? vslot<N, double>(t) : t;
    const double x[6] = {q.rho, q.u, q.v, q.w, f.ok ? q.h : q.p, q.h};
#pragma unroll
    for (int v = 0; v < 6; ++v) {
      if (!f.ok) reinterpret_cast<double*>(sQ)[v * n3 + ts] = x[v];
      else if (v < 5) sQ[v * n3 + ts] = fx_of(x[v], v == 0 ? f.bR : (v < 4 ? (st ? sRows.bU[v - 1] : f.bU) : f.bH));
    }
#pragma unroll
    for (int v = 0; v < 5; ++v) {
      if (!f.ok) reinterpret_cast<double*>(sL)[v * n3 + ts] = l[v];
      else sL[v * n3 + ts] = fx_of(l[v], v == 0 ? f.bL0 : (v < 4 ? (st ? sRows.bLM[v - 1] : f.bLM) : f.bLE));
    }
  }
  if (f.ok) {
    __syncthreads();
    if (st) adj_passes_fx<N, GEN>(sQ, sL, sLt, sA, sG, sT, sW, m, S, e0, e, f, sRows, t);
    else adj_passes_fx<N, false>(sQ, sL, sLt, sA, sG, sT, sW, m, S, e0, e, f, sRows, t);
  } else {
    adj_volume_fp64<N>(reinterpret_cast<double*>(smem_raw), m, ph, tab, e, t);
  }
  if (t >= n3) return;
  double gQ[6], Uo[5], out[5] = {0, 0, 0, 0, 0};
  const int ts = f.ok ? vslot<N, double>(t) : t;
#pragma unroll
  for (int v = 0; v < 6; ++v) gQ[v] = sG[v * n3 + ts];
#pragma unroll
  for (int v = 0; v < 5; ++v) Uo[v] = U[v * S + g];
  prim_vjp(Uo, ph, gQ, out);
  source_vjp(Uo, ph, lam[4 * S + g], out);
#pragma unroll
  for (int v = 0; v < 5; ++v) gV[v * S + g] = out[v];
}

}  // namespace dg
