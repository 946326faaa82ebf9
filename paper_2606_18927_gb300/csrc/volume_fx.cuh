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
// node's fluxes are not far below the element's largest.  Against the
// extended-precision oracle the mass row's error (2-norm) is 0.4 to 0.7 of FP64's on
// straight boxes of degree 3 to 7 with sides 1 : 1 to 1 : 1000, the energy row's 0.5
// to 0.8, the momentum rows' 0.9 to 1.1; the whole operator's fell by up to 30 % on
// curved meshes of degree 2 to 8.  Stretched elements have units of their own for
// every component of u and column of Ja (FxMetric, FxRows).
// An element whose fluxes may be far below its largest is summed in FP64 as before
// (fx_plan: non-finite values; density or enthalpy differing by more than a factor 4
// over its nodes, with the entropy-conserving flux density or internal energy
// by more than an eighth, where its logarithmic means' series end; a Mach number so
// small that the common unit of the momentum flux would cost the velocity bits; a
// column of Ja that falls below an eighth of its largest).
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
// Bounds of x: limbs are |l| <= 2^31 and |h| <= 2^(b - 31) for values below 2^b, so
// a pair's S_u S_a (b = 61, 60) adds up to 3 2^60, its two momentum terms together
// 7 2^60 (|Q| < 1).  Sums of more stay below 2^63 = 8 2^60 by fold() between the
// terms: two products S_u S_a fit, a third does not.
struct FxSum {
  long long hh, x;
  __device__ __forceinline__ FxSum(Fx a, Fx b) {
    x = madw(a.l, b.h, madw(a.h, b.l, 1LL << 31));
    hh = mulw(a.h, b.h);
  }
  // with half added to the sum: half = 2^(k - 1) for a sum that is shifted by k
  __device__ __forceinline__ FxSum(Fx a, Fx b, long long half) {
    x = madw(a.l, b.h, madw(a.h, b.l, 1LL << 31));
    hh = madw(a.h, b.h, half);
  }
  __device__ __forceinline__ void add(Fx a, Fx b) {
    x = madw(a.l, b.h, madw(a.h, b.l, x));
    hh = madw(a.h, b.h, hh);
  }
  // x's high word (it counts twice) into hh; the sum's bits stay the same
  __device__ __forceinline__ void fold() {
    hh = madw((int)(x >> 32), 2, hh);
    x = (long long)(unsigned)x;
  }
  // hh + x / 2^31: the high word of x counts twice
  __device__ __forceinline__ long long get() const { return madw((int)(x >> 32), 2, hh); }
};
__device__ __forceinline__ long long fx_mul(Fx a, Fx b) { return FxSum(a, b).get(); }
// a b 2^k in the same units, to the nearest 2^-k'th below
__device__ __forceinline__ long long fx_mul_shl(Fx a, Fx b, int k) {
  return (mulw(a.h, b.h) << k) + (madw(a.l, b.h, mulw(a.h, b.l)) >> (31 - k));
}

// limbs of r 2^k
template <int k>
__device__ __forceinline__ Fx fx_split(long long r) {
  return Fx{(int)(r >> (31 - k)), (int)(((unsigned)r << k) & 0x7fffffffu)};
}

__device__ __forceinline__ int fx_biased_exp(double x) { return (__double2hiint(x) >> 20) & 0x7ff; }
// |x| ordered as integers (the high words), and the factor by which the largest
// lies below its power of two (rounded up)
__device__ __forceinline__ int fx_mag(double x) { return __double2hiint(x) & 0x7fffffff; }
__device__ __forceinline__ float fx_mant(int mag) { return (float)((mag & 0xfffff) + 0x100001) * (1.0f / 2097152.0f); }

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
// the corners), 1 / w_i in units of 2^(eW - 61), and the bits hd_i by which
// 1 / w_i is below 2^eW: a node's sums are kept in units finer by the least of
// its three positions' (in one unit for all nodes the interior ones, where
// 1 / w is a tenth of its end value, would lose those bits)
template <int N>
struct FxTab {
  Fx Q[(N + 1) * (N + 1)];
  long long iw[N + 1];
  int hd[N + 1];
  int eW;
};

// Logarithmic means in fixed point (the entropy-conserving flux; see
// logmean_G): with t = (a - b)^2 / (4 a b) < 2^-8 (a and b within an eighth of
// each other), T = 256 t in units of 2^-61, the series
//   1 - t (c1 - t (c2 - t (c3 - t (c4 - t (c5 - t c6)))))
// to 2^-61 (truncation below 2^-56 at t = 2^-8).  c3 .. c6 in units of 2^-30 by
// the high limb alone, c1 and c2 in units of 2^-61.
struct FxSeries {
  long long c1, c2;
  int c3, c4, c5, c6;
};
constexpr int fx_q30(double x) { return (int)(x * 1073741824.0 + 0.5); }
// G = tanh(s) / s, Q = 2 s / sinh(2 s) (s = asinh sqrt t), R = 1 / (1 + t)
constexpr FxSeries FX_G{(1LL << 61) / 3, (1LL << 61) / 45 * 11, fx_q30(191.0 / 945.0), fx_q30(2497.0 / 14175.0),
                        fx_q30(14797.0 / 93555.0), fx_q30(92427157.0 / 638512875.0)};
constexpr FxSeries FX_Q{(1LL << 61) / 3 * 2, (1LL << 61) / 15 * 8, fx_q30(16.0 / 35.0), fx_q30(128.0 / 315.0),
                        fx_q30(256.0 / 693.0), fx_q30(1024.0 / 3003.0)};
constexpr FxSeries FX_R{1LL << 61, 1LL << 61, 1 << 30, 1 << 30, 1 << 30, 1 << 30};

__device__ __forceinline__ Fx fx_series(Fx T, const FxSeries c) {
  auto low = [&](int cc, int s) { return cc - ((int)(mulw(T.h, s) >> 32) >> 6); };
  const int s3 = low(c.c3, low(c.c4, low(c.c5, c.c6)));
  const Fx s2 = fx_split<0>(c.c2 - (mulw(T.h, s3) >> 7));
  const Fx s1 = fx_split<0>(c.c1 - (fx_mul(T, s2) >> 7));
  return fx_split<0>((1LL << 61) - (fx_mul(T, s1) >> 7));
}

// 256 t in units of 2^-61 from d = a - b (|d| < 2^57) and the nodes' 1 / (2 a),
// 1 / (2 b); sh = 7 + 2 (e_a + e_i), the exponents of the units of a and 1 / 2a
__device__ __forceinline__ Fx fx_mean_arg(Fx a, Fx b, Fx ia, Fx ib, int sh) {
  const int h = a.h - b.h, l = a.l - b.l;
  const Fx d{h * 8 + (l >> 28), (l & 0x0fffffff) << 3};  // 8 (a - b)
  const long long t = fx_mul(fx_split<0>(fx_mul(d, d)), fx_split<2>(fx_mul(ia, ib)));
  return fx_split<0>(t << sh);
}

// The element's units, from its nodes' largest magnitudes.  Node values: rho,
// u, p' and h; Kennedy-Gruber: e = E / rho for h, and 2 p; entropy-conserving
// flux: rho, u, p', e = p / ((gamma - 1) rho),
// b = 1 / (2 e) and 1 / (2 rho), with b p' in the place of p'.
enum { FX_KEP, FX_KG, FX_EC };  // the volume flux, as PhysDev::vol_flux
enum { FX_RHO, FX_U, FX_P, FX_H, FX_NRHO, FX_NH, FX_B, FX_IR, FX_V, FX_W, FX_NUM };
struct FxPlan {
  int ok;              // 0: the element is summed in FP64
  int bR, bU, bP, bH;  // biased exponent bounds of rho, u, p' (EC: b p'), h (EC: e) for fx_of
  int bB, bI;          // EC: of b and 1 / (2 rho)
  int kp;              // the momentum flux's unit is 2^kp times that of m u
  int e0, em, ee;      // the sums' units: mass, momentum, energy rows
  int k0, km, ke;      // bits that the sums' bounds leave free: kept when 1 / w is applied
  int sr, sb;          // EC: shifts of fx_mean_arg for rho and b
  int bZ;              // Kennedy-Gruber: of 2 p
  int kt, kd, kz;      // EC: right shifts of e Q, u.u and 4 p~' to the energy bracket's units
  long long pref;      // EC: 4 p_ref in the bracket's unit
};
// Stretched elements: what differs by component c of u, Ja and the momentum
// (FxPlan's bU, kp, em, km and kd are not used).  The passes read it from shared
// memory pair by pair (volatile): in registers it spilled (N = 7, sides 1 : 8,
// 12^3 elements: volume kernel 227 us, so 181; 160 for even elements).
struct FxRows {
  int bU[3];                      // biased exponent bounds of u_c
  int t[3], s1[3], s2[3], kd[3];  // right shifts of S_u S_a, m u_c, p Ja_c and (EC) u_c u_c to the common units
  long long ht[3], h1[3], h2[3];  // half of what the first three drop
  int em[3], km[3];
};

// An element's metrics (k_metric_fx): the largest |Ja^d_c| of each column c over
// nodes and directions (as fx_mag), and its kind.  FX_EVEN: the columns are within
// a factor 2 of each other, and the metrics and the velocities have one unit each.
// FX_STRETCHED: a side is short against another.  The flux S_u . S_a then adds
// products of large velocities with small metrics and of small velocities with
// large ones: in common units both lose as many bits as the sides' ratio has (the
// mass row's error was 3 times FP64's at ratio 10, 280 times at 1000), so every
// column and every velocity component has its own, and the products are shifted
// to the largest one's.  FX_GRADED: some column is below an eighth of its largest at
// some node (thin at one end); its lines there would lose as much: summed in FP64.
// FX_THIN: below a 64th.
enum { FX_EVEN, FX_STRETCHED, FX_GRADED, FX_THIN };
struct FxMetric {
  int col[3], kind;
};

// ex: the largest fx_mag of each value (FX_NRHO, FX_NH: of 0x7fffffff - fx_mag);
// mt: the element's metrics; eW of the line table; rows: for stretched elements
// (GEN: the mesh has some)
template <int VF, bool GEN>
__device__ __forceinline__ FxPlan fx_plan(const int* ex, const FxMetric& mt, int eW, double p_ref, double gm1,
                                          FxRows* rows) {
  constexpr bool EC = VF == FX_EC;
  FxPlan f;
  const bool st = GEN && mt.kind == FX_STRETCHED;
  const int mA = max(mt.col[0], max(mt.col[1], mt.col[2]));
  const int xU = GEN ? max(ex[FX_U], max(ex[FX_V], ex[FX_W])) : ex[FX_U];
  f.bR = ex[FX_RHO] >> 20;
  f.bH = ex[FX_H] >> 20;
  const int eR = f.bR - 1022, eA = (mA >> 20) - 1022, eP = (ex[FX_P] >> 20) - 1022;
  int eH = f.bH - 1022;
  // p' is summed with rho u u: below 2^(eR + 2 eU - 1) in the unit of m u; a
  // larger p' (low Mach numbers, no reference pressure) raises that unit by
  // 2^kp, and beyond kp = 40 the velocity's
  const int eUt = (xU >> 20) - 1022;
  int eU = max(eUt, -200);
  if (!st) eU = max(eU, (eP - eR + 1 - 40 + 1) >> 1);
  f.bU = eU + 1022;
  f.kp = max(0, eP - (eR + 2 * eU - 1));
  int ePt = eR + 2 * eU - 1 + f.kp, E = eU + eA;  // E: of S_u . S_a
  // what the largest values leave of the bounds (all below 1)
  const float mr = fx_mant(ex[FX_RHO]), mh = fx_mant(ex[FX_H]), ma = fx_mant(mA);
  const float mu = ldexpf(fx_mant(xU), max(eUt - eU, -60));
  float mass = mr * mu * ma;
  bool range = abs(eR) < 200 && abs(eH) < 200 && abs(eA) < 200 && eU < 200 && eP < 200;
  int eC[3], aC[3];  // stretched: exponents of u_c (no further than 2^-40 below the largest) and of Ja_c
  float uC[3] = {0.0f, 0.0f, 0.0f};
  if (st) {
    const int x[3] = {ex[FX_U], ex[FX_V], ex[FX_W]};
    E = -1000;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const int e = (x[c] >> 20) - 1022;
      eC[c] = max(e, eU - 40);
      aC[c] = (mt.col[c] >> 20) - 1022;
      uC[c] = ldexpf(fx_mant(x[c]), max(e - eC[c], -60));
      E = max(E, eC[c] + aC[c]);
      range = range && abs(aC[c]) < 200;
    }
    // p' in its own unit, but no finer than the least row m u_c needs
    mass = 0.0f;
    ePt = 1000;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const int t = min(E - eC[c] - aC[c], 62);
      rows->bU[c] = eC[c] + 1022;
      rows->t[c] = t;
      rows->ht[c] = (1LL << t) >> 1;
      mass += ldexpf(uC[c] * fx_mant(mt.col[c]), -t);
      ePt = min(ePt, eR + E + eC[c] - 1 - aC[c]);
    }
    mass *= mr * (1.0f / 3.0f);
    ePt = max(ePt, eP);
  }
  f.bP = ePt + 1022;
  const bool finite = f.bR < 0x7ff && (xU >> 20) < 0x7ff && (ex[FX_P] >> 20) < 0x7ff && f.bH < 0x7ff;
  const float mp = ldexpf(fx_mant(ex[FX_P]), max(eP - ePt, -60));
  float energy = mass * mh;
  bool even;
  if constexpr (EC) {
    // rho and e within an eighth over the element (t < 2^-8)
    auto near = [](int mx, int nmn) {
      const double hi = __hiloint2double(mx + 1, 0), lo = __hiloint2double(0x7fffffff - nmn, 0);
      return hi - lo < 0.125 * lo;
    };
    even = near(ex[FX_RHO], ex[FX_NRHO]) && near(ex[FX_H], ex[FX_NH]);
    f.bB = ex[FX_B] >> 20; f.bI = ex[FX_IR] >> 20;
    f.sr = 7 + 2 * (eR + f.bI - 1022);
    f.sb = 7 + 2 * (eH + f.bB - 1022);
    // b p' in the unit that makes (b p' sums) (e sums) / (1 + t) that of p'
    f.bP = ePt - eH + 1 + 1022;
    const int e1 = eH - 59, e2 = 2 * eU - 58, eY = max(e1, e2);  // units of e Q and u.u
    f.kt = min(eY - e1, 63);
    f.kd = min(eY - e2, 63);
    if (st) {
#pragma unroll
      for (int c = 0; c < 3; ++c) rows->kd[c] = min(eY - (2 * eC[c] - 58), 63);
    }
    energy = mass * fminf(1.0f, (ldexpf(mh, -f.kt) + ldexpf(mu * mu, -f.kd)) * 0.58f);
    const int eZ = eR + eY + 2;  // of rho (e Q + u.u)
    f.kz = eZ - (ePt - 60) - 1;
    even = even && f.kz >= 0 && f.kz < 64 && f.sr >= 7 && f.sr <= 9 && f.sb >= 7 && f.sb <= 9 &&
           fx_biased_exp(p_ref) + 2 - 1022 <= eZ + 59 && gm1 < 0.7;
    f.pref = __double2ll_rn(4.0 * p_ref * __hiloint2double((1023 - eZ) << 20, 0));
    eH = eY + 60;
  } else {
    // (magnitudes within a factor 4, by exponents: there no row's error is more than 3 %
    // above FP64's; within 8 the momentum rows' was up to 16 %, the energy row's 10 %)
    even = f.bR - ((0x7fffffff - ex[FX_NRHO]) >> 20) <= 1 && f.bH - ((0x7fffffff - ex[FX_NH]) >> 20) <= 1;
    f.bB = f.bI = f.sr = f.sb = f.kt = f.kd = f.kz = 0;
    f.pref = 0;
    if constexpr (VF == FX_KG) {
      // 2 p (below 2 (gamma - 1) rho e) in the unit of rho e
      f.bZ = eR + eH + 2 + 1022;
      even = even && gm1 < 0.7 && (ex[FX_B] >> 20) <= f.bZ;
    }
  }
  auto free_bits = [](float x) { return max(0, min(6, -1 - ilogbf(fmaxf(x, 1e-6f)))); };
  f.k0 = free_bits(mass);
  f.km = free_bits((ldexpf(mass * mu, -f.kp) + 0.34f * mp * ma) * 0.76f);
  f.ke = free_bits(energy);
  f.e0 = eR + E + eW - 57 - f.k0;
  f.em = eR + eU + E + eW - 57 + f.kp - f.km;
  f.ee = eR + E + eH + eW - 57 - f.ke;
  if constexpr (GEN) {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      if (st) {
        // units of m u_c and p Ja_c; the sums are in the coarser one
        const int u1 = eR + E + eC[c] - 55, u2 = ePt + aC[c] - 54, T = max(u1, u2);
        const int s1 = min(T - u1, 62), s2 = min(T - u2, 62);
        rows->s1[c] = s1;
        rows->s2[c] = s2;
        rows->h1[c] = (1LL << s1) >> 1;
        rows->h2[c] = (1LL << s2) >> 1;
        rows->km[c] = free_bits((ldexpf(mass * uC[c], -s1) + 0.34f * ldexpf(mp * fx_mant(mt.col[c]), -s2)) * 0.76f);
        rows->em[c] = T + eW - 2 - rows->km[c];
      } else {
        rows->bU[c] = f.bU;
        rows->em[c] = f.em;
      }
    }
  }
  f.ok = finite && range && even && mt.kind < FX_GRADED && (eU - eUt <= 5 || xU >> 20 == 0);
  return f;
}

// A metric Ja^d_c in the element's unit, one bit below fx_of's bound, so that a
// pair's sum of three products S_u . S_a has room
__device__ __forceinline__ Fx metric_fx(double a, const FxMetric& mt, int c) { return fx_of(a, (mt.col[c] >> 20) + 1); }

// The elements' FxMetric [K], and with JaX the metrics in their units, limbs
// [9][K n3].  One block per element, once per mesh; *kinds collects the kinds.
static __global__ void k_metric_fx(int n3, long long S, const double* __restrict__ Ja, Fx* __restrict__ JaX,
                                   FxMetric* __restrict__ mt, int* __restrict__ kinds) {
  __shared__ int mx[3], graded, thin;
  __shared__ FxMetric my;
  if (threadIdx.x < 3) mx[threadIdx.x] = 100 << 20;
  if (threadIdx.x == 3) graded = thin = 0;
  __syncthreads();
  const size_t e0 = (size_t)blockIdx.x * n3;
  auto column = [&](int t, int c) {
    int b = 0;
    for (int d = 0; d < 3; ++d) b = max(b, fx_mag(Ja[(d * 3 + c) * S + e0 + t]));
    return b;
  };
  for (int c = 0; c < 3; ++c) {
    int b = 0;
    for (int t = threadIdx.x; t < n3; t += blockDim.x) b = max(b, column(t, c));
    atomicMax(&mx[c], b);
  }
  __syncthreads();
  const int most = max(mx[0], max(mx[1], mx[2])), least = min(mx[0], min(mx[1], mx[2]));
  const bool even = most - least <= 1 << 20;
  for (int t = threadIdx.x; t < n3; t += blockDim.x)
    for (int c = 0; c < 3; ++c) {
      const int below = mx[c] - column(t, c);
      if (below > 3 << 20) graded = 1;
      if (below > 6 << 20) thin = 1;
    }
  __syncthreads();
  if (threadIdx.x == 0) {
    const int kind = thin ? FX_THIN : (graded ? FX_GRADED : (even ? FX_EVEN : FX_STRETCHED));
    my = FxMetric{{even ? most : mx[0], even ? most : mx[1], even ? most : mx[2]}, kind};
    mt[blockIdx.x] = my;
    if (kind != FX_EVEN) atomicOr(kinds, 1 << kind);
  }
  __syncthreads();
  if (JaX)
    for (int t = threadIdx.x; t < n3; t += blockDim.x)
      for (int x = 0; x < 9; ++x) JaX[x * S + e0 + t] = metric_fx(Ja[x * S + e0 + t], my, x % 3);
}

template <int N, int VF>
struct VolFxShape {
  using Sh = VolShape<N>;
  static constexpr int n = Sh::n, n2 = Sh::n2, n3 = Sh::n3;
  // 8-byte values per node: 6 node values in fixed point (EC: 8), 7 in FP64
  // (EC: 9), 9 metrics, 5 sums; the line tables (fixed point: Q and 1 / w;
  // FP64: three coefficient tables)
  static constexpr int QS = VF == FX_EC ? 9 : 7;
  static constexpr int SMEM = ((QS + 14) * n3 + 3 * n2) * 8;
};

// The three direction passes in fixed point: sQ [6][n3] (rho, u, v, w, p', h;
// Kennedy-Gruber [7][n3]: e for h, and 2 p; EC [8][n3]: rho, u, v, w, b p', e, b, 1 / (2 rho)), sA [9][n3], sR [5][n3] the
// sums in the plan's units, sT [n2] Q, sW [n] 1 / w and sH [n] hd.  A line's n nodes are on
// n consecutive lanes; a lane forms the pairs with the nodes at cyclic distance
// 1 .. n/2 and hands their flux to the partner by shuffle, where it is
// subtracted (Q is antisymmetric); a pair at distance n/2 is formed by both of
// its lanes.  ST: a stretched element, with its rows r.
template <int N, int VF, bool ST>
__device__ __forceinline__ void volume_passes_fx(const Fx* sQ, const Fx* sA, long long* sR, const Fx* sT,
                                                 const long long* sW, const int* sH, const FxPlan& f,
                                                 const volatile FxRows& r, int t) {
  using Sh = VolShape<N>;
  constexpr int n = Sh::n, n2 = Sh::n2, n3 = Sh::n3, LPW = Sh::LPW, NQ = VF == FX_EC ? 8 : 6 + VF;
  const int warp = t >> 5, lane = t & 31;
  const int seg = lane / n, pos = lane - seg * n;
  const int L0 = warp * LPW + seg;
  const bool active = (seg < LPW) && (L0 < n2);
  const int L = active ? L0 : 0;
  const int base = seg * n;
  const int la = L % n, lb = L / n;
#pragma unroll 1
  for (int dir = 0; dir < 3; ++dir) {
    const int ms = vslot<N, double>(dir == 0 ? pos + n * L : (dir == 1 ? la + n * pos + n2 * lb : L + n2 * pos));
    const Fx* sD = sA + dir * 3 * n3;
    Fx q[NQ], a[3];
#pragma unroll
    for (int v = 0; v < NQ; ++v) q[v] = sQ[v * n3 + ms];
#pragma unroll
    for (int c = 0; c < 3; ++c) a[c] = sD[c * n3 + ms];
    long long acc[5] = {0, 0, 0, 0, 0};
#pragma unroll
    for (int d = 1; d <= n / 2; ++d) {
      const int pm = pos + d < n ? pos + d : pos + d - n;
      const int sm = __shfl_sync(0xffffffffu, ms, base + pm);  // the partner's slot, from its lane
      const Fx Q = sT[pos * n + pm];
      const Fx Sa0 = a[0] + sD[sm], Sa1 = a[1] + sD[n3 + sm], Sa2 = a[2] + sD[2 * n3 + sm];
      const Fx mv1 = sQ[n3 + sm], mv2 = sQ[2 * n3 + sm], mv3 = sQ[3 * n3 + sm];
      const Fx Su = q[1] + mv1, Sv = q[2] + mv2, Sw = q[3] + mv3;
      Fx ua;  // 4 {u}.{a}
      if constexpr (ST) {
        ua = fx_split<1>((FxSum(Su, Sa0, r.ht[0]).get() >> r.t[0]) + (FxSum(Sv, Sa1, r.ht[1]).get() >> r.t[1]) +
                         (FxSum(Sw, Sa2, r.ht[2]).get() >> r.t[2]));
      } else {
        FxSum s(Su, Sa0);
        s.add(Sv, Sa1);
        s.fold();
        s.add(Sw, Sa2);
        ua = fx_split<1>(s.get());
      }
      long long F[5];
      Fx pq;  // 2 Q {p'} (EC: 2 Q (p~ - p_ref))
      if constexpr (VF == FX_KEP) {
        const Fx rq = fx_split<1>(fx_mul(q[0] + sQ[sm], Q));        // 2 Q {rho}
        pq = fx_split<0>(fx_mul(q[4] + sQ[4 * n3 + sm], Q));
        F[0] = fx_mul(rq, ua);                                      // 8 Q {rho}{u}.{a}
        F[4] = fx_mul(fx_split<1>(F[0]), q[5] + sQ[5 * n3 + sm]);   // times 2 {h}
      } else if constexpr (VF == FX_KG) {
        const Fx uq = fx_split<1>(fx_mul(ua, Q)), Sr = q[0] + sQ[sm], Sp = q[6] + sQ[6 * n3 + sm];
        pq = fx_split<0>(fx_mul(q[4] + sQ[4 * n3 + sm], Q));
        F[0] = fx_mul(Sr, uq);
        // 16 F_E = 4 {u}.{a} [S_rho S_e + 4 {p}]
        const long long Z = fx_mul(Sr, q[5] + sQ[5 * n3 + sm]) + (((long long)Sp.h << 31) + Sp.l);
        F[4] = fx_mul(uq, fx_split<1>(Z));
      } else {
        const Fx uq = fx_split<1>(fx_mul(ua, Q));
        const Fx rm = sQ[sm];
        // ln-mean of rho: (S_rho / 2) G(t)
        const Fx Sr = fx_split<1>(fx_mul(q[0] + rm, fx_series(fx_mean_arg(q[0], rm, q[7], sQ[7 * n3 + sm], f.sr), FX_G)));
        const Fx em = sQ[5 * n3 + sm];
        const Fx Se = q[5] + em;
        const Fx tb = fx_mean_arg(q[6], sQ[6 * n3 + sm], q[5], em, f.sb);
        // 2 (p~ - p_ref) = (b p' sums) (e sums) / (1 + t)
        const long long pt = fx_mul_shl(q[4] + sQ[4 * n3 + sm], fx_split<1>(fx_mul(Se, fx_series(tb, FX_R))), 3);
        pq = fx_split<0>(fx_mul(fx_split<0>(pt), Q));
        F[0] = fx_mul(Sr, uq);  // 8 Q F_rho
        // 16 F_E = 4 {u}.{a} [S_rho G (S_e Q(t) + u_A.u_B) + 4 (p~ - p_ref) + 4 p_ref]
        long long uu;
        if constexpr (ST) {
          uu = (fx_mul(q[1], mv1) >> r.kd[0]) + (fx_mul(q[2], mv2) >> r.kd[1]) + (fx_mul(q[3], mv3) >> r.kd[2]);
        } else {
          FxSum k(q[1], mv1);
          k.add(q[2], mv2);
          k.add(q[3], mv3);
          uu = k.get() >> f.kd;
        }
        const long long Y = (fx_mul(Se, fx_series(tb, FX_Q)) >> f.kt) + uu;
        const long long Z = fx_mul(Sr, fx_split<0>(Y)) + (pt >> f.kz) + f.pref;
        F[4] = fx_mul(uq, fx_split<1>(Z));
      }
      const Fx mu = fx_split<1>(ST ? F[0] : F[0] >> f.kp);
      auto momentum = [&](Fx S, Fx Sa, int c) {
        if constexpr (ST) {
          return (FxSum(mu, S, r.h1[c]).get() >> r.s1[c]) + (FxSum(pq, Sa, r.h2[c]).get() >> r.s2[c]);
        } else {
          FxSum x(mu, S);
          x.add(pq, Sa);
          return x.get();
        }
      };
      F[1] = momentum(Su, Sa0, 0);
      F[2] = momentum(Sv, Sa1, 1);
      F[3] = momentum(Sw, Sa2, 2);
#pragma unroll
      for (int v = 0; v < 5; ++v) acc[v] += F[v];
      if (2 * d != n) {
        const int src = base + (pos - d >= 0 ? pos - d : pos - d + n);
#pragma unroll
        for (int v = 0; v < 5; ++v) acc[v] -= __shfl_sync(0xffffffffu, F[v], src);
      }
    }
    if (active) {
      const Fx wi = fx_split<0>(sW[pos] << min(sH[pos], min(sH[la], sH[lb])));
#pragma unroll
      for (int v = 0; v < 5; ++v) {
        const int k = v == 0 ? f.k0 : (v == 4 ? f.ke : (ST ? r.km[v - 1] : f.km));
        const long long x = fx_mul_shl(fx_split<0>(acc[v]), wi, k);
        sR[v * n3 + ms] = dir == 0 ? x : x + sR[v * n3 + ms];
      }
    }
    __syncthreads();
  }
}

// the double nearest to the sum of two fixed-point metrics in units of 2^e
__device__ __forceinline__ double metric_sum(Fx a, Fx b, int e) {
  return fx_double(((long long)(a.h + b.h) << 31) + (a.l + b.l), e);
}

// An element summed in FP64 (fx_plan); rare, so kept out of line.  The FP64 pipe
// bounds it (30 operations a pair; KEP flux, N = 7, 12^3 elements all of them: 601 us
// with the metrics' sums added on it), so these three are formed from the staged
// fixed-point metrics on the integer pipes (545; 539 when such meshes kept the
// pairs' sums in memory, 252 bytes a node).  Ja read again in FP64 (FXM false) where a
// column falls so far below its largest that its limbs hold less than FP64's 53 bits.
template <int N, int VF, bool FXM>
__device__ __noinline__ void volume_passes_fp64(double* smem, const MeshDev<double>& m, const PhysDev& ph,
                                                const Tables<N>& tab, const double* __restrict__ Rv, int e, int t) {
  constexpr int n3 = VolShape<N>::n3, n2 = VolShape<N>::n2, T = VolShape<N>::THREADS;
  double *sQ = smem, *sA = sQ + VolFxShape<N, VF>::QS * n3, *sR = sA + 9 * n3, *sC8 = sR + 5 * n3, *sC16 = sC8 + n2, *sC1 = sC16 + n2;
  for (int x = t; x < n2; x += T) {
    sC8[x] = tab.DVS8[x];
    sC16[x] = 0.5 * tab.DVS8[x];
    sC1[x] = 8.0 * tab.DVS8[x];
  }
  if constexpr (!FXM) {
    if (t < n3) {
      const int ts = vslot<N, double>(t);
#pragma unroll
      for (int c = 0; c < 9; ++c) sA[c * n3 + ts] = m.Ja[(size_t)c * ((size_t)m.K * n3) + (size_t)e * n3 + t];
    }
    __syncthreads();
    volume_passes<N, double, VF == FX_EC>(VolSmem<double>{sQ, sA, sR, sC8, sC16, sC1}, m, ph, Rv, e, t);
  } else {
    const FxMetric& mt = m.JaX_max[e];
    VolSmem<double, Fx> sm{sQ, reinterpret_cast<Fx*>(sA), sR, sC8, sC16, sC1};
#pragma unroll
    for (int c = 0; c < 3; ++c) sm.eA[c] = (mt.col[c] >> 20) - 1022 - 59;
    __syncthreads();
    volume_passes<N, double, VF == FX_EC, Fx>(sm, m, ph, Rv, e, t);
  }
}

// k_volume of the FP64 form: one CTA per element, the passes in fixed point
// (elements out of fx_plan's range: in FP64), the epilogue in FP64.  Measured at N = 7,
// 32^3 elements: KEP flux 10.08 ms with FP64 pair fluxes (FP64 pipe 90 % busy), 3.04 ms
// in fixed point (16^3: issue 55 %, integer pipes 41 and 21 %, FP64 pipe 45 %).
// GEN: for meshes with stretched elements (their passes beside the others').
template <int N, int MODE, int VF, bool GEN>
__global__ void __launch_bounds__(VolShape<N>::THREADS, (resident_ctas(VolShape<N>::THREADS, VolFxShape<N, VF>::SMEM, 1024)))
k_volume_fx(const double* __restrict__ Uin, const MeshDev<double> m, const PhysDev ph, const Tables<N> tab,
            const FxTab<N> ft, const double* __restrict__ Rv, const double* __restrict__ Fs, double* __restrict__ Out,
            double* __restrict__ dU, double* __restrict__ Uout, const StageArgs st, int* __restrict__ status) {
  using Sh = VolShape<N>;
  constexpr int n = Sh::n, n2 = Sh::n2, n3 = Sh::n3, T = Sh::THREADS, QS = VolFxShape<N, VF>::QS;
  constexpr bool EC = VF == FX_EC;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ int sEx[FX_NUM];
  __shared__ FxPlan sF;
  __shared__ FxRows sRows;
  Fx* sQ = reinterpret_cast<Fx*>(smem_raw);
  Fx* sA = sQ + QS * n3;
  long long* sR = reinterpret_cast<long long*>(sA + 9 * n3);
  Fx* sT = reinterpret_cast<Fx*>(sR + 5 * n3);
  long long* sW = reinterpret_cast<long long*>(sT + n2);
  int* sH = reinterpret_cast<int*>(sW + n);
  const int e = blockIdx.x, t = threadIdx.x;
  const size_t S = (size_t)m.K * n3;
  const size_t g = (size_t)e * n3 + t;
  Prim<double> q{1.0, 0.0, 0.0, 0.0, 0.0, 1.0};
  // EC: e = p / ((gamma - 1) rho), 1 / (2 e), 1 / (2 rho); Kennedy-Gruber: E / rho, 2 p
  double en = 1.0, be = 0.5, irh = 0.5;
  if (t < n3) {
    q = m.W64 ? load_prim64(m.W64, S, g) : primitive<double>(Uin[g], Uin[S + g], Uin[2 * S + g], Uin[3 * S + g], Uin[4 * S + g], ph);
    const int ts = vslot<N, double>(t);
#pragma unroll
    for (int c = 0; c < 9; ++c)
      sA[c * n3 + ts] = N == 7 || m.JaX ? m.JaX[(size_t)c * S + g] : metric_fx(m.Ja[(size_t)c * S + g], m.JaX_max[e], c % 3);
    if constexpr (EC) {
      const double ir = rcp_pos(q.rho);
      // (the quotient's remainder added back: half an ulp instead of two)
      const double pf = q.p + ph.p_ref, a = ph.rgm1 * pf;
      en = a * ir;
      en = fma(fma(-en, q.rho, a) + fma(ph.rgm1, pf, -a), ir, en);
      be = 0.5 * rcp_pos(en);
      irh = 0.5 * ir;
    }
    if constexpr (VF == FX_KG) {
      const double ir = rcp_pos(q.rho);
      be = q.p + ph.p_ref;  // p
      const double pr = be * ir;
      en = q.h - fma(fma(-pr, q.rho, be), ir, pr);  // e = h - p / rho
      be *= 2.0;
    }
  }
  if (t < FX_NUM) sEx[t] = 0;
  for (int x = t; x < n2; x += T) sT[x] = ft.Q[x];
  if (t < n) { sW[t] = ft.iw[t]; sH[t] = ft.hd[t]; }
  __syncthreads();
  {
    // (EC: rho and e are positive, else the element is out of range)
    const bool pos = !EC || (q.rho > 0.0 && en > 0.0);
    int ex[FX_NUM];
    ex[FX_RHO] = pos ? fx_mag(q.rho) : 0x7ff00000;
    ex[FX_H] = fx_mag(VF == FX_KEP ? q.h : en);
    ex[FX_NRHO] = 0x7fffffff - fx_mag(q.rho);
    ex[FX_NH] = 0x7fffffff - ex[FX_H];
    ex[FX_U] = GEN ? fx_mag(q.u) : max(max(fx_mag(q.u), fx_mag(q.v)), fx_mag(q.w));
    ex[FX_V] = fx_mag(q.v);
    ex[FX_W] = fx_mag(q.w);
    ex[FX_P] = fx_mag(q.p);
    ex[FX_B] = fx_mag(be);
    ex[FX_IR] = fx_mag(irh);
    if (t >= n3) {
#pragma unroll
      for (int x = 0; x < FX_NUM; ++x) ex[x] = 0;
    }
#pragma unroll
    for (int x = 0; x < FX_NUM; ++x) {
      if (x >= FX_V ? !GEN : x >= (EC ? FX_V : FX_B + VF)) continue;
      const int mx = __reduce_max_sync(0xffffffffu, ex[x]);
      if ((t & 31) == 0) atomicMax(&sEx[x], mx);
    }
  }
  __syncthreads();
  if (t == 0) sF = fx_plan<VF, GEN>(sEx, m.JaX_max[e], ft.eW, ph.p_ref, ph.gm1, &sRows);
  __syncthreads();
  const FxPlan f = sF;
  const bool fx = f.ok != 0;
  if (t < n3) {
    const int ts = vslot<N, double>(t);
    if (fx) {
      sQ[ts] = fx_of(q.rho, f.bR);
      sQ[n3 + ts] = fx_of(q.u, GEN ? sRows.bU[0] : f.bU);
      sQ[2 * n3 + ts] = fx_of(q.v, GEN ? sRows.bU[1] : f.bU);
      sQ[3 * n3 + ts] = fx_of(q.w, GEN ? sRows.bU[2] : f.bU);
      if constexpr (EC) {
        sQ[4 * n3 + ts] = fx_of(be * q.p, f.bP);
        sQ[5 * n3 + ts] = fx_of(en, f.bH);
        sQ[6 * n3 + ts] = fx_of(be, f.bB);
        sQ[7 * n3 + ts] = fx_of(irh, f.bI);
      } else {
        sQ[4 * n3 + ts] = fx_of(q.p, f.bP);
        sQ[5 * n3 + ts] = fx_of(VF == FX_KEP ? q.h : en, f.bH);
        if constexpr (VF == FX_KG) sQ[6 * n3 + ts] = fx_of(be, f.bZ);
      }
    } else {
      // as stage_node, from this kernel's own e and reciprocals
      double* d = reinterpret_cast<double*>(smem_raw) + ts;
      d[0] = q.rho; d[n3] = q.u; d[2 * n3] = q.v; d[3 * n3] = q.w;
      d[4 * n3] = 4.0 * q.p;
      if constexpr (EC) {
        const double beta = be * ph.rgm1;
        d[4 * n3] = 8.0 * beta * q.p;
        d[5 * n3] = beta;
        d[6 * n3] = q.u * q.u + q.v * q.v + q.w * q.w;
        d[7 * n3] = en * ph.gm1;  // 1 / (2 beta)
        d[8 * n3] = irh;
      } else {
        d[5 * n3] = VF == FX_KG ? en : q.h;
        if constexpr (VF == FX_KG) d[6 * n3] = be;
      }
    }
  }
  if (fx) {
    __syncthreads();
    if (GEN && m.JaX_max[e].kind == FX_STRETCHED) volume_passes_fx<N, VF, GEN>(sQ, sA, sR, sT, sW, sH, f, sRows, t);
    else volume_passes_fx<N, VF, false>(sQ, sA, sR, sT, sW, sH, f, sRows, t);
  } else {
    double* smem = reinterpret_cast<double*>(smem_raw);
    if (GEN && m.JaX_max[e].kind == FX_THIN) volume_passes_fp64<N, VF, !GEN>(smem, m, ph, tab, Rv, e, t);
    else volume_passes_fp64<N, VF, true>(smem, m, ph, tab, Rv, e, t);
  }
  volume_epilogue<N, double, MODE>(
      Uin, m, ph, tab, Fs, Out, dU, Uout, st, status, e, t, [&](int nd, size_t gn, double acc[5]) {
        const int ts = vslot<N, double>(nd);
        if (fx) {
          const int k = min(sH[nd % n], min(sH[nd / n % n], sH[nd / n2]));
          const int eu[5] = {f.e0 - k, (GEN ? sRows.em[0] : f.em) - k, (GEN ? sRows.em[1] : f.em) - k,
                             (GEN ? sRows.em[2] : f.em) - k, f.ee - k};
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
