// volume_fx.cuh -- the FP64 form's split-form volume term in fixed point.
//
// GB300 issues 2 FP64 operations per clock and SM, but 64 32 x 32 -> 64 bit
// integer multiply-adds and 128 integer additions, so the two-point fluxes of
// an element (some 320 of its 353 FP64 instructions per node) run on the
// integer pipes instead: every quantity of a pair flux is a 62-bit integer in
// units of a power of two fixed per element, products are formed from 31-bit
// limbs by mad.wide.s32, and the sums over a line are exact.
//
// Rounding.  The element's largest |rho|, |u_c|, |h|, |Ja| land between 2^59
// and 2^60 (2^58 and 2^59 for Ja) units; a product keeps 57 to 60 bits below
// its largest value and is rounded to the nearest unit.  FP64 rounds the same
// product to 53 bits of its own value, in every operation, the additions
// among them; so the fixed-point sums are the more exact ones wherever a
// node's fluxes are not far below the element's largest (against the
// extended-precision oracle the operator's error fell by 5 to 30 % on meshes
// of degree 2 to 8; with densities 20 apart within an element it tripled).
// An element in which they may be is summed in FP64 as before (fx_plan:
// non-finite values, density or enthalpy differing by more than a factor 8
// over its nodes, or a Mach number so small that the common unit of the
// momentum flux would cost the velocity bits).
#pragma once
#include <cuda_runtime.h>

#include "kernels.cuh"

namespace dg {

// Fx (kernels.cuh): h 2^31 + l, |l| <= 2^31; normalised numbers have
// |l| <= 2^30, so that the sum of two needs no carry
__device__ __forceinline__ long long mulw(int a, int b) { return (long long)a * (long long)b; }
__device__ __forceinline__ long long madw(int a, int b, long long c) {
  long long r;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
  return r;
}
__device__ __forceinline__ Fx operator+(Fx a, Fx b) { return Fx{a.h + b.h, a.l + b.l}; }

// A sum of products in units of 2^62 of the factors' units: hh collects the
// high limbs' products, x the cross products (units of 2^31; they start at
// 2^31, half a unit of what is kept).  The low limbs' products, below half a
// unit, are left out.
struct FxSum {
  long long hh, x;
  __device__ __forceinline__ FxSum(Fx a, Fx b) {
    x = madw(a.l, b.h, madw(a.h, b.l, 1LL << 31));
    hh = mulw(a.h, b.h);
  }
  __device__ __forceinline__ void add(Fx a, Fx b) {
    x = madw(a.l, b.h, madw(a.h, b.l, x));
    hh = madw(a.h, b.h, hh);
  }
  // hh + x / 2^31: the high word of x counts twice
  __device__ __forceinline__ long long get() const { return madw((int)(x >> 32), 2, hh); }
};
__device__ __forceinline__ long long fx_mul(Fx a, Fx b) { return FxSum(a, b).get(); }

// limbs of r 2^k
template <int k>
__device__ __forceinline__ Fx fx_split(long long r) {
  return Fx{(int)(r >> (31 - k)), (int)(((unsigned)r << k) & 0x7fffffffu)};
}

__device__ __forceinline__ int fx_biased_exp(double x) { return (__double2hiint(x) >> 20) & 0x7ff; }

// x 2^(60 - eb + 1022), |x| < 2^(eb - 1022), truncated, in normalised limbs
__device__ __forceinline__ Fx fx_of(double x, int eb) {
  const int hi = __double2hiint(x);
  const unsigned long long m =
      ((unsigned long long)((hi & 0xfffff) | 0x100000) << 32 | (unsigned)__double2loint(x)) << 7;
  const int rs = min(eb - ((hi >> 20) & 0x7ff), 63);
  const long long s = hi >> 31;
  const long long v = ((long long)(m >> rs) ^ s) - s;
  const long long c = v + (1LL << 30);
  return Fx{(int)(c >> 31), ((int)c & 0x7fffffff) - (1 << 30)};
}

// the double nearest to r 2^e (results in the normal range)
__device__ __forceinline__ double fx_double(long long r, int e) {
  const long long s = r >> 63;
  const unsigned long long a = (unsigned long long)((r ^ s) - s);
  const int lz = __clzll((long long)a);
  const unsigned long long m = a << (lz & 63);
  // 53 bits, rounded half up; a carry moves into the exponent
  unsigned long long b = (m >> 11) + ((m >> 10) & 1);
  b += (unsigned long long)(unsigned)(e + 63 - lz + 1022) << 52;
  b |= (unsigned long long)s << 63;
  return a ? __longlong_as_double((long long)b) : 0.0;
}

// Line tables: Q_im = w_i D_im in units of 2^-61 (antisymmetric off the
// diagonal, where the split form's DVS = 2 D - B / w is 2 D and has zeros at
// the corners), and 1 / w_i in units of 2^(eW - 61)
template <int N>
struct FxTab {
  Fx Q[(N + 1) * (N + 1)];
  Fx iw[N + 1];
  int eW;
};

// the element's units, from the largest (and, of rho and h, smallest) biased
// exponents of its nodes
enum { FX_RHO, FX_U, FX_P, FX_H, FX_NRHO, FX_NH, FX_NUM };
struct FxPlan {
  int ok;              // 0: the element is summed in FP64
  int bR, bU, bP, bH;  // biased exponent bounds of rho, u, p', h (fx_of)
  int kp;              // the momentum flux's unit is 2^kp times that of m u
  int e0, em, ee;      // the sums' units: mass, momentum, energy rows
};

// ex: FX_RHO.. the maxima, FX_NRHO, FX_NH the maxima of 2047 - exponent; bA:
// exponent bound of the metrics; eW of the table
__device__ __forceinline__ FxPlan fx_plan(const int* ex, int bA, int eW) {
  FxPlan f;
  f.bR = ex[FX_RHO]; f.bH = ex[FX_H];
  const int eR = f.bR - 1022, eH = f.bH - 1022, eA = bA - 1022, eP = ex[FX_P] - 1022;
  // p' is summed with rho u u: below 2^(eR + 2 eU - 1) in the unit of m u; a
  // larger p' (low Mach numbers, no reference pressure) raises that unit by
  // 2^kp, and beyond kp = 40 the velocity's
  const int eUt = ex[FX_U] - 1022;
  int eU = max(eUt, -200);
  eU = max(eU, (eP - eR + 1 - 40 + 1) >> 1);
  f.bU = eU + 1022;
  f.kp = max(0, eP - (eR + 2 * eU - 1));
  f.bP = eR + 2 * eU - 1 + f.kp + 1022;
  const int base = eA + eW - 57;
  f.e0 = eR + eU + base;
  f.em = eR + 2 * eU + base + f.kp;
  f.ee = eR + eU + eH + base;
  const bool finite = ex[FX_RHO] < 0x7ff && ex[FX_U] < 0x7ff && ex[FX_P] < 0x7ff && ex[FX_H] < 0x7ff;
  const bool range = abs(eR) < 200 && abs(eH) < 200 && abs(eA) < 200 && eU < 200 && eP < 200;
  const bool even = f.bR - (2047 - ex[FX_NRHO]) <= 2 && f.bH - (2047 - ex[FX_NH]) <= 2;
  f.ok = finite && range && even && (eU - eUt <= 5 || ex[FX_U] == 0);
  return f;
}

// The metrics Ja of every element in its own unit: limbs [9][K n3] and the
// exponent bounds [K] (|Ja| < 2^(bA - 1023): one bit below fx_of's bound, so
// that a pair's sum of three products S_u . S_a has room).  One block per
// element, once per mesh.
static __global__ void k_metric_fx(int n3, long long S, const double* __restrict__ Ja, Fx* __restrict__ JaX,
                                   int* __restrict__ bA) {
  __shared__ int mx;
  if (threadIdx.x == 0) mx = 0;
  __syncthreads();
  const size_t e0 = (size_t)blockIdx.x * n3;
  int b = 0;
  for (int t = threadIdx.x; t < n3; t += blockDim.x)
    for (int c = 0; c < 9; ++c) b = max(b, fx_biased_exp(Ja[c * S + e0 + t]));
  atomicMax(&mx, b);
  __syncthreads();
  const int eb = max(mx, 100) + 1;
  for (int t = threadIdx.x; t < n3; t += blockDim.x)
    for (int c = 0; c < 9; ++c) JaX[c * S + e0 + t] = fx_of(Ja[c * S + e0 + t], eb);
  if (threadIdx.x == 0) bA[blockIdx.x] = eb - 1;
}


template <int N>
struct VolFxShape {
  using Sh = VolShape<N>;
  static constexpr int n = Sh::n, n2 = Sh::n2, n3 = Sh::n3;
  // bytes: 7 node values, 9 metrics, 5 sums per node (8 bytes each; six node
  // values in fixed point, seven in FP64), the line tables (fixed point: Q and
  // 1 / w; FP64: three coefficient tables)
  static constexpr int SMEM = (21 * n3 + 3 * n2) * 8;
};

// The three direction passes in fixed point: sQ [6][n3] (rho, u, v, w, p', h),
// sA [9][n3], sR [5][n3] the sums in units 2^em, sT [n2] Q and sW [n] 1 / w.
// A line's n nodes are on n consecutive lanes; a lane forms the pairs with the
// nodes at cyclic distance 1 .. n/2 and hands their flux to the partner by
// shuffle, where it is subtracted (Q is antisymmetric); a pair at distance n/2
// is formed by both of its lanes.
template <int N>
__device__ __forceinline__ void volume_passes_fx(const Fx* sQ, const Fx* sA, long long* sR, const Fx* sT, const Fx* sW,
                                                 int kp, int t) {
  using Sh = VolShape<N>;
  constexpr int n = Sh::n, n2 = Sh::n2, n3 = Sh::n3, LPW = Sh::LPW;
  const int warp = t >> 5, lane = t & 31;
  const int seg = lane / n, pos = lane - seg * n;
  const int L0 = warp * LPW + seg;
  const bool active = (seg < LPW) && (L0 < n2);
  const int L = active ? L0 : 0;
  const int base = seg * n;
  const int la = L % n, lb = L / n;
  const Fx wi = sW[pos];
#pragma unroll 1
  for (int dir = 0; dir < 3; ++dir) {
    auto slot_at = [&](int q) {
      return vslot<N, double>(dir == 0 ? q + n * L : (dir == 1 ? la + n * q + n2 * lb : L + n2 * q));
    };
    const int ms = slot_at(pos);
    const Fx* sD = sA + dir * 3 * n3;
    Fx q[6], a[3];
#pragma unroll
    for (int v = 0; v < 6; ++v) q[v] = sQ[v * n3 + ms];
#pragma unroll
    for (int c = 0; c < 3; ++c) a[c] = sD[c * n3 + ms];
    long long acc[5] = {0, 0, 0, 0, 0};
#pragma unroll
    for (int d = 1; d <= n / 2; ++d) {
      const int pm = pos + d < n ? pos + d : pos + d - n;
      const int sm = slot_at(pm);
      const Fx Q = sT[pos * n + pm];
      const Fx Sa0 = a[0] + sD[sm], Sa1 = a[1] + sD[n3 + sm], Sa2 = a[2] + sD[2 * n3 + sm];
      const Fx Su = q[1] + sQ[n3 + sm], Sv = q[2] + sQ[2 * n3 + sm], Sw = q[3] + sQ[3 * n3 + sm];
      FxSum s(Su, Sa0);
      s.add(Sv, Sa1);
      s.add(Sw, Sa2);
      const Fx ua = fx_split<1>(s.get());                              // 4 {u}.{a}
      const Fx rq = fx_split<1>(fx_mul(q[0] + sQ[sm], Q));             // 2 Q {rho}
      const Fx pq = fx_split<0>(fx_mul(q[4] + sQ[4 * n3 + sm], Q));    // 2 Q {p'}
      const long long m = fx_mul(rq, ua);                              // 8 Q {rho}{u}.{a}
      const Fx mu = fx_split<1>(m >> kp), mh = fx_split<1>(m);
      long long F[5];
      F[0] = m;
      auto momentum = [&](Fx S, Fx Sa) {
        FxSum f(mu, S);
        f.add(pq, Sa);
        return f.get();
      };
      F[1] = momentum(Su, Sa0);
      F[2] = momentum(Sv, Sa1);
      F[3] = momentum(Sw, Sa2);
      F[4] = fx_mul(mh, q[5] + sQ[5 * n3 + sm]);
#pragma unroll
      for (int v = 0; v < 5; ++v) acc[v] += F[v];
      if (2 * d != n) {
        const int src = base + (pos - d >= 0 ? pos - d : pos - d + n);
#pragma unroll
        for (int v = 0; v < 5; ++v) acc[v] -= __shfl_sync(0xffffffffu, F[v], src);
      }
    }
    if (active) {
#pragma unroll
      for (int v = 0; v < 5; ++v) {
        const long long r = fx_mul(fx_split<0>(acc[v]), wi);
        sR[v * n3 + ms] = dir == 0 ? r : r + sR[v * n3 + ms];
      }
    }
    __syncthreads();
  }
}

// an element summed in FP64 (fx_plan); rare, so kept out of line
template <int N>
__device__ __noinline__ void volume_passes_fp64(double* smem, const MeshDev<double>& m, const PhysDev& ph,
                                                const Tables<N>& tab, const double* __restrict__ Rv, int e, int t) {
  constexpr int n3 = VolShape<N>::n3, n2 = VolShape<N>::n2, T = VolShape<N>::THREADS;
  double *sQ = smem, *sA = sQ + 7 * n3, *sR = sA + 9 * n3, *sC8 = sR + 5 * n3, *sC16 = sC8 + n2, *sC1 = sC16 + n2;
  for (int x = t; x < n2; x += T) {
    sC8[x] = tab.DVS8[x];
    sC16[x] = 0.5 * tab.DVS8[x];
    sC1[x] = 8.0 * tab.DVS8[x];
  }
  if (t < n3) {
    const int ts = vslot<N, double>(t);
#pragma unroll
    for (int c = 0; c < 9; ++c) sA[c * n3 + ts] = m.Ja[(size_t)c * ((size_t)m.K * n3) + (size_t)e * n3 + t];
  }
  __syncthreads();
  volume_passes<N, double, false, false>(VolSmem<double>{sQ, sA, sR, sC8, sC16, sC1}, m, ph, Rv, e, t);
}

// k_volume of the FP64 form with the KEP fluxes: one CTA per element, the
// passes in fixed point (Kennedy-Gruber's flux and elements out of fx_plan's
// range: in FP64), the epilogue in FP64.  Measured at N = 7, 32^3 elements:
// 10.08 ms with FP64 pair fluxes (FP64 pipe 90 % busy), 3.07 ms in fixed point
// (issue 52 %, integer pipes 37 %, FP64 pipe 30 %).
template <int N, int MODE>
__global__ void __launch_bounds__(VolShape<N>::THREADS, (vol_min_blocks<N, double, false>()))
k_volume_fx(const double* __restrict__ Uin, const MeshDev<double> m, const PhysDev ph, const Tables<N> tab,
            const FxTab<N> ft, const double* __restrict__ Rv, const double* __restrict__ Fs, double* __restrict__ Out,
            double* __restrict__ dU, double* __restrict__ Uout, const StageArgs st, int* __restrict__ status) {
  using Sh = VolShape<N>;
  constexpr int n = Sh::n, n2 = Sh::n2, n3 = Sh::n3, T = Sh::THREADS;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ int sEx[FX_NUM];
  Fx* sQ = reinterpret_cast<Fx*>(smem_raw);
  Fx* sA = sQ + 7 * n3;
  long long* sR = reinterpret_cast<long long*>(sA + 9 * n3);
  Fx* sT = reinterpret_cast<Fx*>(sR + 5 * n3);
  Fx* sW = sT + n2;
  const int e = blockIdx.x, t = threadIdx.x;
  const size_t S = (size_t)m.K * n3;
  const size_t g = (size_t)e * n3 + t;
  Prim<double> q{1.0, 0.0, 0.0, 0.0, 0.0, 1.0};
  if (t < n3) {
    q = m.W64 ? load_prim64(m.W64, S, g) : primitive<double>(Uin[g], Uin[S + g], Uin[2 * S + g], Uin[3 * S + g], Uin[4 * S + g], ph);
    const int ts = vslot<N, double>(t);
#pragma unroll
    for (int c = 0; c < 9; ++c) sA[c * n3 + ts] = m.JaX[(size_t)c * S + g];
  }
  if (t < FX_NUM) sEx[t] = 0;
  for (int x = t; x < n2; x += T) sT[x] = ft.Q[x];
  if (t < n) sW[t] = ft.iw[t];
  const int eA = m.JaX_exp[e];
  __syncthreads();
  {
    const int bR = fx_biased_exp(q.rho), bH = fx_biased_exp(q.h);
    int ex[FX_NUM];
    ex[FX_RHO] = bR;
    ex[FX_U] = max(max(fx_biased_exp(q.u), fx_biased_exp(q.v)), fx_biased_exp(q.w));
    ex[FX_P] = fx_biased_exp(q.p);
    ex[FX_H] = bH;
    ex[FX_NRHO] = 2047 - bR;
    ex[FX_NH] = 2047 - bH;
    if (t >= n3) {
#pragma unroll
      for (int x = 0; x < FX_NUM; ++x) ex[x] = 0;
    }
#pragma unroll
    for (int x = 0; x < FX_NUM; ++x) {
      const int mx = __reduce_max_sync(0xffffffffu, ex[x]);
      if ((t & 31) == 0) atomicMax(&sEx[x], mx);
    }
  }
  __syncthreads();
  const FxPlan f = fx_plan(sEx, eA, ft.eW);
  const bool fx = f.ok && ph.vol_flux == 0;
  if (t < n3) {
    const int ts = vslot<N, double>(t);
    if (fx) {
      sQ[ts] = fx_of(q.rho, f.bR);
      sQ[n3 + ts] = fx_of(q.u, f.bU);
      sQ[2 * n3 + ts] = fx_of(q.v, f.bU);
      sQ[3 * n3 + ts] = fx_of(q.w, f.bU);
      sQ[4 * n3 + ts] = fx_of(q.p, f.bP);
      sQ[5 * n3 + ts] = fx_of(q.h, f.bH);
    } else {
      double* d = reinterpret_cast<double*>(smem_raw) + ts;
      d[0] = q.rho; d[n3] = q.u; d[2 * n3] = q.v; d[3 * n3] = q.w; d[4 * n3] = 4.0 * q.p;
      d[5 * n3] = q.h;
      if (ph.vol_flux == 1) {
        const double pf = q.p + ph.p_ref;
        d[5 * n3] = q.h - pf / q.rho;
        d[6 * n3] = 2.0 * pf;
      }
    }
  }
  if (fx) {
    __syncthreads();
    volume_passes_fx<N>(sQ, sA, sR, sT, sW, f.kp, t);
  } else {
    volume_passes_fp64<N>(reinterpret_cast<double*>(smem_raw), m, ph, tab, Rv, e, t);
  }
  volume_epilogue<N, double, MODE>(
      Uin, m, ph, tab, Fs, Out, dU, Uout, st, status, e, t, [&](int nd, size_t gn, double acc[5]) {
        const int ts = vslot<N, double>(nd);
        if (fx) {
          const int eu[5] = {f.e0, f.em, f.em, f.em, f.ee};
#pragma unroll
          for (int v = 0; v < 5; ++v) acc[v] = fx_double(sR[v * n3 + ts], eu[v]);
          if (ph.viscous) {
#pragma unroll
            for (int v = 1; v < 5; ++v) acc[v] += Rv[(size_t)(v - 1) * S + gn];
          }
        } else {
          const double* d = reinterpret_cast<const double*>(sR);
#pragma unroll
          for (int v = 0; v < 5; ++v) acc[v] = d[v * n3 + ts];
        }
      });
}

}  // namespace dg
