// rk4_split.cuh -- the FP64 RK4 step with most of its arithmetic on the FP32 pipe.
//
// GB300 issues FP64 at 1/64 of its FP32 lane rate, so the 49 DFMA of a step
// (rk4_device.cuh) bound every FP64 kernel while the FP32 pipe idles.  This form keeps in FP64
// what decides the accuracy -- the state, the first slope and the final update -- and computes
// the later stages' differences from the first slope in float pairs (an unevaluated sum h + l
// of two floats, about 48 bits), with the error-free transformations of Knuth (two-sum) and
// Dekker / Ogita, Rump and Oishi (two-product by FMA).
//
//   K1 = f(y)                                   FP64, as slope() computes it
//   d2 = K1, d3 = K2 = K1 + D2, d4 = 2 (K1 + D3)     stage increments over tau = dt / 2:
//                                                u_j = y + tau d_j      (Eq. (4))
//   Dj = f(y + tau d_j) - f(y)                  float pairs, by the exact difference formula
//        x: kappa tau lap(dx) - tau (dy + dz)   y: tau dx + a tau dy
//        z: z tau dx + tau dz ((x - c) + tau dx)    (f's only product: Eq. (6))
//        harmonic q: tau dp   p: kappa tau lap(dq) - w2 tau dq
//   y <- y + (tau / 3) (6 K1 + 2 D2 + 2 D3 + D4)     FP64, one rounding      (Eq. (5))
//
// Why this loses nothing: a pair's relative error is about 2^-49, D is dt |J| times K1, and D
// enters the state times dt; with dt |J| at most about 1/4 (split_allowed bounds the coefficients,
// split_in_range the state: the Roessler chain's J holds x - c and z) that stays below the rounding of
// the state, and the state is rounded once per component and step where the FP64 form rounds it four
// times.  Error against long double in units of the FP64 form's (2-norms per component):
//   dt = 0.01, kappa = 1 and 2, uniform[-1, 1) and 1 .. 1000 steps         0.48 .. 0.57
//   on the attractor (c = 5.7 .. 12.5, dt c up to 1/8)                      0.50
//   one step, uniform states, dt = 1e-4 .. 1/16, at the edge of both rules  x, y 0.5 .. 0.75, z up to 0.97
// Where a step changes a component by more than its own size (a Roessler chain's z below 12 dt b, the
// momenta of a harmonic chain at rest) the error of that step is up to 3 (1.25) times the FP64 form's:
// the stages share the first slope's rounding, and a difference is no longer small.  Beyond the rules
// (uniform states, dt = 0.01, one step) z lost a factor of 1.6 at |x|, |z| = 40 and 24 at 160.
//
// Every function is written over a lane type T: float (one site) or f32x2 (two sites in one
// packed instruction), which round alike, so kernels with any number of sites per thread and
// the one-stage-per-launch kernel agree bit for bit.
//
// Range: a pair needs the exponent room of FP32.  Tiles whose values leave it (split_in_range)
// are advanced in the FP64 form instead (tile_item returns false and the caller runs it again).  Zeros are
// in range, but a front that runs into a chain at rest decays through every magnitude: where FP64 has 1e-60 a
// difference underflows to an exact zero, and one of 1e-46 comes out of FP32's subnormals.  Values that
// stay below 2^-70 send the tile to the FP64 form; zeros do (split_tile_bits) when the tile starts with two
// neighbouring sites all zero beside one that is not, or stores a component as zero at one site and holds
// it nonzero at another.  What is left is exact: a component that is zero throughout a tile before and after
// has a slope of zero (a wrong zero slope elsewhere shows in the same site's other components).
// A tile of NaN alone, what a chain that has blown up consists of, stays: its first slope and so
// its result are NaN in either form.
#pragma once
#include "rk4_device.cuh"
#include "rk4_internal.h"

namespace rk4d {

typedef unsigned long long f32x2;

__device__ __forceinline__ f32x2 pack2(float a, float b) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ float lane0(f32x2 v) {
  float a, b;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
  (void)b;
  return a;
}
__device__ __forceinline__ float lane1(f32x2 v) {
  float a, b;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
  (void)a;
  return b;
}
__device__ __forceinline__ float vadd(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float vsub(float a, float b) { return __fsub_rn(a, b); }
// Products as FMAs with a zero addend (a zero product comes out as +0): ptxas was seen to contract
// a packed mul.rn and a later add.rn into one FMA (CUDA 13.0; the packed and the scalar forms of
// a sum after a product then differed), which an FMA rules out at the same cost.
__device__ __forceinline__ float vmul(float a, float b) { return __fmaf_rn(a, b, 0.f); }
__device__ __forceinline__ float vfma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ f32x2 vadd(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f32x2 vsub(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f32x2 vmul(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(0ull));
  return r;
}
__device__ __forceinline__ f32x2 vfma(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
template <typename T> __device__ __forceinline__ T vset(float a);
template <> __device__ __forceinline__ float vset<float>(float a) { return a; }
template <> __device__ __forceinline__ f32x2 vset<f32x2>(float a) { return pack2(a, a); }

template <typename T> struct FPair {
  T h, l;
};

// a + b = s + e exactly (Knuth).
template <typename T> __device__ __forceinline__ void two_sum(T a, T b, T &s, T &e) {
  s = vadd(a, b);
  const T bb = vsub(s, a);
  e = vadd(vsub(a, vsub(s, bb)), vsub(b, bb));
}
// a - b = s + e exactly.
template <typename T> __device__ __forceinline__ void two_diff(T a, T b, T &s, T &e) {
  s = vsub(a, b);
  const T bb = vsub(s, a);
  e = vsub(vsub(a, vsub(s, bb)), vadd(b, bb));
}
// a + m b = s + e exactly, for m = 2 or -2.
template <typename T> __device__ __forceinline__ void two_sum_m(T a, T m, T b, T &s, T &e) {
  s = vfma(m, b, a);
  const T nb = vsub(a, s);
  e = vadd(vsub(a, vadd(s, nb)), vfma(m, b, nb));
}
// c v = e - np for a coefficient c (nch = -c.h) and a pair v.
template <typename T> __device__ __forceinline__ void mul_coef(const FPair<T> &c, T nch, const FPair<T> &v, T &np, T &e) {
  np = vmul(nch, v.h);
  e = vfma(c.h, v.h, np);
  e = vfma(c.h, v.l, e);
  e = vfma(c.l, v.h, e);
}
// The pair with its tail at most half a unit of its head (|h| >= |l| up to the head's cancellation).
template <typename T> __device__ __forceinline__ FPair<T> pair_norm(const FPair<T> &v) {
  const T s = vadd(v.h, v.l);
  return {s, vsub(v.l, vsub(s, v.h))};
}
// a - n as a pair.
template <typename T> __device__ __forceinline__ FPair<T> pair_sub(const FPair<T> &a, const FPair<T> &n) {
  FPair<T> r;
  T e;
  two_diff(a.h, n.h, r.h, e);
  r.l = vsub(vadd(e, a.l), n.l);
  return r;
}

// ---- FP64 <-> pair by integer operations (the F2F conversions issue on the FP64 pipe) --------

// A double as head (rounded to 24 bits, ties away from zero), the tail's integer significand m (28
// bits and sign) and the power of two p of the double itself: the value is h + m 2^-52 p.  Zero
// gives h = p = 0, magnitudes below 2^-126 at most a few denormals.  (A truncated head would save
// four integer operations; its one-signed tails, up to twice as large, doubled the error of the
// later slopes' differences.)
__device__ __forceinline__ void split_bits(double y, float &h, float &m, float &p) {
  const int hi = __double2hiint(y);
  const unsigned lo = (unsigned)__double2loint(y);
  const unsigned sign = (unsigned)hi & 0x80000000u;
  const unsigned a = (unsigned)max((hi & 0x7fffffff) - 0x38000000, 0);  // exponent bias 1023 -> 127
  const unsigned rl = lo + 0x10000000u, rh = a + (rl < lo ? 1u : 0u);
  h = __uint_as_float(__funnelshift_l(rl, rh, 3) | sign);
  m = __int2float_rn((int)(lo << 3) >> 3);
  p = __uint_as_float(((a << 3) & 0x7f800000u) | sign);
}
__device__ __forceinline__ FPair<float> split1(double y) {
  float h, m, p;
  split_bits(y, h, m, p);
  return {h, vmul(vmul(m, 0x1p-52f), p)};
}
template <typename T> struct Lanes;
template <> struct Lanes<float> {
  static constexpr int n = 1;
  static __device__ __forceinline__ FPair<float> split(const double *y, int) { return split1(y[0]); }
};
template <> struct Lanes<f32x2> {
  static constexpr int n = 2;
  // the pair of y[0] and y[stride]
  static __device__ __forceinline__ FPair<f32x2> split(const double *y, int stride) {
    float h0, m0, p0, h1, m1, p1;
    split_bits(y[0], h0, m0, p0);
    split_bits(y[stride], h1, m1, p1);
    return {pack2(h0, h1), vmul(vmul(pack2(m0, m1), vset<f32x2>(0x1p-52f)), pack2(p0, p1))};
  }
};

// h + m 2^-52 p as a double, for a normalised pair whose tail is given as m = l 2^52 / p rounded
// to an integer (p: h's power of two): the head's bits rebiased, plus m in units of the double's
// last place.  A negative m below a power of two borrows into the binade whose last place is
// half as large, hence the doubling.
__device__ __forceinline__ double join_bits(float h, int m) {
  const unsigned b = __float_as_uint(h);
  if (((b << 9) == 0u) && m < 0) m += m;
  unsigned hh = ((unsigned)((int)b >> 3) & 0x8fffffffu) + 0x38000000u;
  unsigned hl = b << 29;
  const bool zero = (b & 0x7fffffffu) == 0u;
  asm("add.cc.u32 %0, %0, %2;\n\taddc.u32 %1, %1, %3;" : "+r"(hl), "+r"(hh) : "r"(m), "r"(m >> 31));
  return __hiloint2double(zero ? 0 : (int)hh, zero ? 0 : (int)hl);
}
// 1 / p for h's power of two p (with h's sign).
__device__ __forceinline__ float inv_pow2(float h) {
  return __uint_as_float(0x7F000000u - (__float_as_uint(h) & 0xff800000u));
}
// The doubles nearest the pair's lanes.
__device__ __forceinline__ void join(FPair<float> v, double *out, int) {
  const float s = vadd(v.h, v.l);
  const float l = vsub(v.l, vsub(s, v.h));
  out[0] = join_bits(s, __float2int_rn(vmul(vmul(l, 0x1p52f), inv_pow2(s))));
}
__device__ __forceinline__ void join(FPair<f32x2> v, double *out, int stride) {
  const f32x2 s = vadd(v.h, v.l);
  const f32x2 l = vsub(v.l, vsub(s, v.h));
  const float s0 = lane0(s), s1 = lane1(s);
  const f32x2 m = vmul(vmul(l, vset<f32x2>(0x1p52f)), pack2(inv_pow2(s0), inv_pow2(s1)));
  out[0] = join_bits(s0, __float2int_rn(lane0(m)));
  out[stride] = join_bits(s1, __float2int_rn(lane1(m)));
}

// ---- range ----------------------------------------------------------------------------------

// Whether component d of a site's state is zero or of a magnitude the differences' pairs are good
// for: at least 2^-70, whose products keep their relative precision through a step, and at most what
// keeps dt |J| where their errors stay below the state's rounding.  The Roessler chain's J holds x - c
// and z: dt |x - c| <= 1/4, dt |y| and dt |z| <= 0.3 (c: the site's own).  The harmonic chain is linear,
// and its limit, 2^40, only leaves room in FP32's exponents.  NaN and infinity are out of range.
// split_holds: the same without zero.  Integer operations on the high words: with |x - c| in FP64 the two
// subtractions per site and launch cost 9 % at k = 1 (2^22 sites, 256 x 4 x 1, 8 steps: 1144 -> 1246 us).  own_c: a
// heterogeneous chain's c of the site (then by the FP32 heads), else NULL.
__device__ __forceinline__ bool is_zero(double v) {
  return (((unsigned)__double2hiint(v) & 0x7fffffffu) | (unsigned)__double2loint(v)) == 0u;
}
__device__ __forceinline__ float truncated_head(double v) {  // of a magnitude in FP32's range, or 0
  const int hi = __double2hiint(v);
  const unsigned a = (unsigned)max((hi & 0x7fffffff) - 0x38000000, 0);
  return __uint_as_float(__funnelshift_l((unsigned)__double2loint(v), a, 3) | ((unsigned)hi & 0x80000000u));
}
template <int MODEL>
__device__ __forceinline__ bool split_holds(double v, int d, const double *own_c, const SplitCoef &s) {
  constexpr unsigned lo = (1023u - 70u) << 20;
  const int hi = __double2hiint(v);
  const unsigned a = (unsigned)hi & 0x7fffffffu;
  if (MODEL == ROESSLER && d == 0) {
    if (own_c) return (a >= lo) & (a <= s.most_x) & (fabsf(__fsub_rn(truncated_head(v), truncated_head(*own_c))) <= s.far);
    return (a >= lo) & (a <= (hi < 0 ? s.least_x : s.most_x));
  }
  return (a >= lo) & (a <= s.big);
}
template <int MODEL>
__device__ __forceinline__ bool split_in_range(double v, int d, const double *own_c, const SplitCoef &s) {
  return is_zero(v) || split_holds<MODEL>(v, d, own_c, s);
}
__device__ __forceinline__ bool is_nan(double v) {
  const unsigned a = (unsigned)__double2hiint(v) & 0x7fffffffu;
  return a > 0x7ff00000u || (a == 0x7ff00000u && __double2loint(v) != 0);
}
// The same for a site's own parameter of a heterogeneous chain: zero, or at least 2^-60 and with
// the high word at most `most` (that of the largest value split_allowed takes).
__device__ __forceinline__ bool split_param_in_range(double v, unsigned most) {
  constexpr unsigned lo = (1023u - 60u) << 20;
  const unsigned a = (unsigned)__double2hiint(v) & 0x7fffffffu;
  return ((a >= lo) & (a <= most)) | ((a | (unsigned)__double2loint(v)) == 0u);
}

// ---- coefficients -----------------------------------------------------------------------------

// c tau as a pair, c a double (host and device compute the same bits).
__device__ __forceinline__ FPair<float> times_tau(double c, const SplitCoef &s) {
  const FPair<float> v = split1(c);
  float np, e;
  mul_coef<float>({s.tauh, s.taul}, -s.tauh, v, np, e);
  return {-np, e};
}
__device__ __forceinline__ void split_set_kappa(SplitCoef &s, double kappa) {
  const FPair<float> k = times_tau(kappa, s);
  s.kth = k.h;
  s.ktl = k.l;
}
// The pair coefficients of a stage in lane type T.  at: Roessler a tau; harmonic w2 tau.
template <typename T> struct StageCoef {
  FPair<T> kt, at, tau, k2;  // k2: kappa2 tau (coupling range 2)
};
template <typename T> __device__ __forceinline__ StageCoef<T> stage_coef(const SplitCoef &s) {
  return {{vset<T>(s.kth), vset<T>(s.ktl)},
          {vset<T>(s.ath), vset<T>(s.atl)},
          {vset<T>(s.tauh), vset<T>(s.taul)},
          {vset<T>(s.k2h), vset<T>(s.k2l)}};
}

// ---- one stage ----------------------------------------------------------------------------------

// The base point's part of the z difference: z and x - c at the step's start.
template <typename T> struct SplitBase {
  FPair<T> z, t;
};
template <typename T> __device__ __forceinline__ FPair<T> x_minus_c(const FPair<T> &x, const FPair<T> &c) {
  FPair<T> r;
  T e;
  two_diff(x.h, c.h, r.h, e);
  r.l = vsub(vadd(e, x.l), c.l);
  return r;
}

// lap(dx) as (g, lo).
template <typename T>
__device__ __forceinline__ FPair<T> pair_lap(const FPair<T> &x, const FPair<T> &xl, const FPair<T> &xr) {
  const T m2 = vset<T>(-2.f);
  T s, e1, e2;
  FPair<T> g;
  two_sum(xl.h, xr.h, s, e1);
  two_sum_m(s, m2, x.h, g.h, e2);
  g.l = vadd(vfma(m2, x.l, vadd(xl.l, xr.l)), vadd(e1, e2));
  return g;
}

// The rows of n = -D that are linear in the increments d: all but the Roessler chain's z.  nd, df: tau dx
// = df - nd (Roessler).
template <int MODEL, typename T, int RANGE>
__device__ __forceinline__ void split_linear(const FPair<T> *d, const FPair<T> &xl, const FPair<T> &xr,
                                             const StageCoef<T> &c, FPair<T> *n, T &nd, T &df,
                                             const FPair<T> &xl2 = {}, const FPair<T> &xr2 = {}) {
  const T m1 = vset<T>(-1.f);
  const FPair<T> g = pair_lap(d[0], xl, xr);
  T np, e, ne;
  mul_coef(c.kt, vmul(m1, c.kt.h), g, np, e);  // kappa tau lap = e - np
  if constexpr (RANGE == 2) {
    T np2, e2, s;
    mul_coef(c.k2, vmul(m1, c.k2.h), pair_lap(d[0], xl2, xr2), np2, e2);
    two_sum(np, np2, s, ne);
    np = s;
    e = vsub(vadd(e, e2), ne);
  }
  if constexpr (MODEL == ROESSLER) {
    const T ntau = vmul(m1, c.tau.h);
    FPair<T> w;  // dy + dz
    T we, nw, f;
    two_sum(d[1].h, d[2].h, w.h, we);
    w.l = vadd(vadd(d[1].l, d[2].l), we);
    mul_coef(c.tau, ntau, w, nw, f);
    two_diff(np, nw, n[0].h, ne);
    n[0].l = vadd(vsub(ne, e), f);
    mul_coef(c.tau, ntau, d[0], nd, df);
    mul_coef(c.at, vmul(m1, c.at.h), d[1], np, e);
    two_sum(nd, np, n[1].h, ne);
    n[1].l = vsub(ne, vadd(df, e));
  } else {
    T nq, f;  // w2 tau dq = f - nq
    mul_coef(c.at, vmul(m1, c.at.h), d[0], nq, f);
    two_diff(np, nq, n[1].h, ne);
    n[1].l = vadd(vsub(ne, e), f);
    mul_coef(c.tau, vmul(m1, c.tau.h), d[1], n[0].h, e);  // tau dp = e - n
    n[0].l = vmul(m1, e);
  }
}

// n = -D for the stage increments d (85 FP32 operations per site; harmonic 40).
template <int MODEL, typename T>
__device__ __forceinline__ void split_stage(const FPair<T> *d, const FPair<T> &xl, const FPair<T> &xr,
                                            const SplitBase<T> &b, const StageCoef<T> &c, FPair<T> *n) {
  T nd, df;  // delta = tau dx = df - nd
  split_linear<MODEL, T, 1>(d, xl, xr, c, n, nd, df);
  if constexpr (MODEL == ROESSLER) {
    const T m1 = vset<T>(-1.f);
    const T ntau = vmul(m1, c.tau.h);
    T nz, q, ne;  // zeta = tau dz = q - nz
    mul_coef(c.tau, ntau, d[2], nz, q);
    T pz = vmul(c.tau.h, d[2].h);  // = -nz
    FPair<T> t;  // (x - c) + delta
    T te;
    two_diff(b.t.h, nd, t.h, te);
    t.l = vadd(vadd(te, b.t.l), df);
    const T nzh = vmul(m1, b.z.h);
    const T p1 = vmul(nzh, nd);  // z delta = p1 - g1
    T g1 = vfma(b.z.h, nd, p1);
    g1 = vfma(nzh, df, g1);
    g1 = vfma(b.z.l, nd, g1);
    const T p2 = vmul(nz, t.h);  // zeta t = e2 - p2
    T e2 = vfma(pz, t.h, p2);
    e2 = vfma(pz, t.l, e2);
    e2 = vfma(q, t.h, e2);
    two_diff(p2, p1, n[2].h, ne);
    n[2].l = vsub(vadd(ne, g1), e2);
  }
}

// Bookkeeping after stage j = 1, 2, 3 (the RK stages 2 to 4): the next increments d and the
// running sum N = -(2 D2 + 2 D3 + D4), of which stages 1 and 2 hold half.
template <typename T>
__device__ __forceinline__ void split_update(int j, const FPair<T> &k1, const FPair<T> &n, FPair<T> &d, FPair<T> &N) {
  T e;
  if (j == 1) {
    N = n;
    d = pair_sub(k1, n);
  } else if (j == 2) {
    T s;
    two_sum(N.h, n.h, s, e);
    N = {s, vadd(vadd(N.l, n.l), e)};
    d = pair_sub(k1, n);
    d.h = vadd(d.h, d.h);
    d.l = vadd(d.l, d.l);
  } else {
    const T two = vset<T>(2.f);
    T s;
    two_sum_m(n.h, two, N.h, s, e);
    N = {s, vadd(vfma(two, N.l, n.l), e)};
  }
}
// a + c v and a - c v for a coefficient pair c.
template <typename T> __device__ __forceinline__ FPair<T> pair_fma(const FPair<T> &c, T nch, const FPair<T> &v, const FPair<T> &a) {
  T np, e, ne;
  FPair<T> r;
  mul_coef(c, nch, v, np, e);
  two_diff(a.h, np, r.h, ne);
  r.l = vadd(vadd(a.l, e), ne);
  return r;
}
template <typename T> __device__ __forceinline__ FPair<T> pair_fnma(const FPair<T> &c, T nch, const FPair<T> &v, const FPair<T> &a) {
  T np, e, ne;
  FPair<T> r;
  mul_coef(c, nch, v, np, e);
  two_sum(a.h, np, r.h, ne);
  r.l = vadd(vsub(a.l, e), ne);
  return r;
}
// c v.
template <typename T> __device__ __forceinline__ FPair<T> pair_mul(const FPair<T> &c, T nch, const FPair<T> &v) {
  T np, e;
  mul_coef(c, nch, v, np, e);
  return {vmul(c.h, v.h), e};
}
// y + (tau / 3) (6 K1 - N).
__device__ __forceinline__ double split_final(double y, double k1, double N, double six, double w) {
  return fma(w, fma(six, k1, -N), y);
}

}  // namespace rk4d
