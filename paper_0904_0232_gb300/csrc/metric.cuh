// Device metric module for the Cartesian Kerr-Schild form of the Kerr metric.
//
//   g_mn = eta_mn + f k_m k_n,   f = 2 m r^3 / (r^4 + a^2 z^2)                 (Eq. 4)
//   k = ((r x - a y)/(r^2 + a^2), (r y + a x)/(r^2 + a^2), z / r, 1)          (Eq. 5, dt -> dx^4)
//   r^4 - (R^2 - a^2) r^2 - a^2 z^2 = 0                                        (Eq. 6)
//
// k is null for eta (that is Eq. 6), so |k_spatial| = 1, det g = -1 and
// g^mn = eta^mn - f k^m k^n with k^m = (k_x, k_y, k_z, -1).  Everything below uses those
// closed forms; the gradients of r, f and k are written out by the chain rule.
#pragma once

#include <cuda_runtime.h>

namespace grpic {

// Division and square root used by the metric functions.  IeeeOps is the compiler's own
// operators (the default everywhere); a caller that needs less than full precision can pass a
// cheaper policy with the same three members.
struct IeeeOps {
  template <typename S>
  __device__ static __forceinline__ S rcp(S x) { return S(1) / x; }
  template <typename S>
  __device__ static __forceinline__ S div(S a, S b) { return a / b; }
  template <typename S>
  __device__ static __forceinline__ S root(S x) { return sqrt(x); }
};

// IEEE 754 binary32 -> binary64, exact, with integer operations only (sign, exponent rebiased
// by 1023 - 127 = 896, mantissa shifted by 29).  Zero and subnormal inputs give a signed zero
// (the FP32 push runs with subnormals flushed); infinities and NaNs keep their class.  On this
// GPU the hardware conversions run on the reduced-rate FP64 pipe.
__device__ __forceinline__ double widen(float f) {
  const unsigned u = __float_as_uint(f);
  const unsigned e = (u >> 23) & 0xffu;
  unsigned hi = u & 0x80000000u, lo = 0u;
  if (e != 0u) {
    const unsigned m = u & 0x7fffffu;
    hi |= ((e == 0xffu ? 0x7ffu : e + 896u) << 20) | (m >> 3);
    lo = m << 29;
  }
  return __hiloint2double((int)hi, (int)lo);
}

// IEEE 754 binary64 -> binary32 with round-to-nearest-even, with integer operations for every
// result in the normal binary32 range (the 29 dropped mantissa bits decide; a carry may step the
// exponent, to infinity at the top, as the rounding rule says) and for zeros; other inputs
// (subnormal or out-of-range results, infinities, NaNs) take the hardware conversion.
__device__ __forceinline__ float narrow(double d) {
  const unsigned hi = (unsigned)__double2hiint(d), lo = (unsigned)__double2loint(d);
  const unsigned e = (hi >> 20) & 0x7ffu;
  if (e == 0u && (hi & 0xfffffu) == 0u && lo == 0u) return __uint_as_float(hi & 0x80000000u);  // +-0
  if (e < 897u || e > 1150u) return __double2float_rn(d);
  unsigned r = (hi & 0x80000000u) | ((e - 896u) << 23) | ((hi & 0xfffffu) << 3) | (lo >> 29);
  const unsigned rest = lo & 0x1fffffffu;
  if (rest > 0x10000000u || (rest == 0x10000000u && (r & 1u))) ++r;
  return __uint_as_float(r);
}

// floor of x as an integer and in T.  FP64: from the bits (the FP64 pipe, which would also do the conversions, stays
// free); negative, huge and non-finite x take the conversions.
__device__ __forceinline__ void floor_split(float x, int& i, float& fl) {
  i = (int)floorf(x);
  fl = (float)i;
}
__device__ __forceinline__ void floor_split(double x, int& i, double& fl) {
  const int hi = __double2hiint(x), e = (hi >> 20) - 1023;
  if ((unsigned)hi < 0x41400000u) {  // 0 <= x < 2^21
    const int drop = 20 - max(e, 0);
    const int mask = e < 0 ? 0 : (int)(0xffffffffu << drop);
    i = e < 0 ? 0 : ((hi & 0xfffff) | 0x100000) >> drop;
    fl = __hiloint2double(hi & mask, 0);
  } else {
    i = (int)floor(x);
    fl = (double)i;
  }
}

// FP64 reciprocal, quotient and square root for evaluations whose results are rounded to FP32
// afterwards (the FP32-mixed policy near the hole), where IEEE rounding of the last FP64 bit
// buys nothing: an FP32 estimate (the approximate reciprocal / reciprocal square root, relative
// error a few 2^-23) refined by one FP64 Newton step -- y <- y + y (1 - x y) for 1/x, and
// s <- s + (x - s^2) y / 2 with s = x y, y ~ 1/sqrt x, for sqrt x (Heron).  A Newton step
// squares the relative error.  Arguments outside [1e-30, 1e30] in magnitude (and non-positive
// square-root arguments) take the IEEE operations.
struct SeededOps64 {
  __device__ static __forceinline__ double rcp(double x) {
    const float xf = narrow(x);
    if (!(fabsf(xf) >= 1e-30f && fabsf(xf) <= 1e30f)) return 1.0 / x;
    const double y = widen(__fdividef(1.f, xf));
    return fma(y, fma(-x, y, 1.0), y);
  }
  __device__ static __forceinline__ double div(double a, double b) { return a * rcp(b); }
  __device__ static __forceinline__ double root(double x) {
    const float xf = narrow(x);
    if (!(xf >= 1e-30f && xf <= 1e30f)) return sqrt(x);
    const double y = widen(rsqrtf(xf));
    const double s = x * y;
    return fma(0.5 * y, fma(-s, s, x), s);
  }
};

// FP64 reciprocal, square root and reciprocal square root, rounded as well as the IEEE operations' to a hundredth of
// a unit in the last place, with 1, 2 and 3 FP64 operations (3 for a root and its reciprocal together).  This GPU
// issues one FP64 warp instruction per 16 cycles and SM, 64 times slower than FP32 and integer ones, and its FP64
// kernels are bound by their count (IEEE 1/x, sqrt x and 1/sqrt x take about 9, 10 and 20), so everything else is
// done beside the FP64 pipe:
//   1. the argument's mantissa as two floats xh + xl (46 bits), y0 ~ xh^-1/2 (or xh^-1) from the FP32 approximation,
//      r = 1 - x y0^2 (1 - x y0) in FP32 with fused multiply-adds, whose rounding (2^-24 of r ~ 2^-21) leaves
//      y = y0 (1 + r/2 + 3 r^2/8) (y0 (1 + r + r^2)) within about 2^-44; the sum is an integer addition to y0's bits;
//   2. in FP64 the residuals: 1 - x y; with s = x y, x - s^2 and 1 - s y.  s is rounded, s = x y (1 + n), which the
//      first of these holds twice and the second once: e = 2 (1 - s y) - (x - s^2) / x = 1 - x y^2 to order n^2;
//   3. the first-order step y (1 + e), s (1 + (x - s^2) / 2x) or y (1 + e/2), whose correction is below 2^12 units in
//      the last place: formed in FP32, rounded to an integer and added to the bits (in FP64 where either side of that
//      is not in the result's binade, whose unit it is in).  The truncation is of order e^2.
// So the result is the exact one rounded, but for the FP32 correction's own error of below 2^-7 units (measured over
// 5e7 arguments: 0.500 units off at most, rms 4.7e-17 relative as IEEE; 1/sqrt x in two IEEE operations 1.49 and
// 6.7e-17).  Arguments lie in 2^-890 .. 2^890, and root gives 0 for 0 and subnormals.  Others give no useful value,
// and callers screen them (or use CheckedOps64).
// Few instructions count as well: the push's two copies of them lie at the limit of the instruction cache.
struct FastOps64 {
 private:
  // the upper 23 of a double's mantissa bits under the exponent field `field` of a float, and the 23 after them as a
  // float of that scale
  __device__ static __forceinline__ void split(int hi, int lo, unsigned field, float* xh, float* xl) {
    *xh = __uint_as_float((__funnelshift_l((unsigned)lo, (unsigned)hi, 3) & 0x7fffffu) | field);
    const unsigned base = field - (23u << 23);
    *xl = __uint_as_float(base | (((unsigned)lo & 0x1fffffffu) >> 6)) - __uint_as_float(base);
  }
  // y0 + c (y0 in [0.5, 1]) as a double, its exponent field raised by field (a high word)
  __device__ static __forceinline__ double assemble(float y0, float c, int field) {
    const long long bits = ((long long)__float_as_uint(y0) << 29) + ((long long)field << 32);
    return __longlong_as_double(bits + __float2int_rn(c * 0x1p53f));
  }
  // v as a float, its exponent field lowered by field (a high word) and 0 where that is too small
  __device__ static __forceinline__ float small_float(double v, int field) {
    const int hi = __double2hiint(v);
    const unsigned m = (unsigned)max((hi & 0x7fffffff) - field, 0);
    return __uint_as_float(__funnelshift_l((unsigned)__double2loint(v), m, 3) | ((unsigned)hi & 0x80000000u));
  }
  static constexpr int kNoField = 896 << 20;  // between the fields of a double and a float of one value
  // v moved by n units, where v and the result both have the exponent field (a high word) that n's unit belongs to
  __device__ static __forceinline__ bool add_units(double v, float n, int field, double* out) {
    *out = __longlong_as_double(__double_as_longlong(v) + __float2int_rn(n));
    return (((__double2hiint(v) ^ field) | (__double2hiint(*out) ^ field)) >> 20) == 0;
  }
  struct Start {
    double y;   // x^-1/2 within 2^-43
    float yf;   // y 2^h to FP32, in [0.5, 1], where x 4^-h is in [1, 4)
    int x, r;   // exponent fields of 4^h and 2^h (high words)
  };
  __device__ static __forceinline__ Start rsqrt_start(double x) {
    const int hi = __double2hiint(x), lo = __double2loint(x);
    Start b;
    b.x = ((hi - 0x00100000) | 0x00100000) & 0x7ff00000;
    b.r = (int)((unsigned)b.x >> 1) + (1023 << 19);
    float xh, xl;
    split(hi, lo, (127u << 23) + ((~(unsigned)hi & 0x00100000u) << 3), &xh, &xl);
    const float y0 = fminf(fmaxf(rsqrtf(xh), 0.5f), 1.f);
    const float t = __fmul_rn(xh, y0);
    float r = __fmaf_rn(-t, y0, 1.f);
    r = __fmaf_rn(-__fmaf_rn(xh, y0, -t), y0, r);
    r = __fmaf_rn(-__fmul_rn(xl, y0), y0, r);
    const float c = y0 * (r * __fmaf_rn(0.375f, r, 0.5f));
    b.y = assemble(y0, c, kNoField + (1023 << 20) - b.r);
    b.yf = __fadd_rn(y0, c);
    return b;
  }
  // d 4^-h to FP32
  __device__ static __forceinline__ float scaled(const Start& b, double d) {
    return small_float(d, b.x + (kNoField - (1023 << 20)));
  }
  // root of x from s = x y, d = x - s^2 (s (d / x) / 2 in units of 2^(h - 52): (d 4^-h) (y 2^h) / 2 2^52)
  __device__ static __forceinline__ double root_of(double x, const Start& b, double s, double d, float df) {
    double v;
    if (!add_units(s, df * (b.yf * 0x1p51f), b.r, &v)) v = root_apart(s, d, b.y);
    return (__double2hiint(x) & 0x7fffffff) < 0x00100000 ? 0.0 : v;
  }
  // and its reciprocal from also e1 = 1 - s y
  __device__ static __forceinline__ double rsqrt_of(const Start& b, double d, float df, double e1) {
    const float e = __fmaf_rn(2.f, small_float(e1, kNoField), -(df * __fmul_rn(b.yf, b.yf)));
    double v;
    if (!add_units(b.y, e * (b.yf * 0x1p52f), (2045 << 20) - b.r, &v)) v = rsqrt_apart(b.y, d, e1);
    return v;
  }
  // across a power of two (out of line with their operations, which would be issued, predicated off, for every
  // argument)
  __device__ static __noinline__ double rcp_apart(double y, double e) { return fma(y, e, y); }
  __device__ static __noinline__ double root_apart(double s, double d, double y) { return fma(0.5 * y, d, s); }
  __device__ static __noinline__ double rsqrt_apart(double y, double d, double e1) {
    return fma(0.5 * y, fma(2.0, e1, -d * y * y), y);
  }

 public:
  __device__ static __forceinline__ double rcp(double x) {
    const int hi = __double2hiint(x), lo = __double2loint(x), field = hi & 0x7ff00000;
    float xh, xl, y0;
    split(hi, lo, 127u << 23, &xh, &xl);
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y0) : "f"(xh));
    y0 = fminf(fmaxf(y0, 0.5f), 1.f);
    float r = __fmaf_rn(-xh, y0, 1.f);
    r = __fmaf_rn(-xl, y0, r);
    const float c = y0 * __fmaf_rn(r, r, r);
    const double y = assemble(y0, c, kNoField + (1023 << 20) - field);
    const double e = fma(-x, y, 1.0);
    double v;
    if (!add_units(y, small_float(e, kNoField) * (__fadd_rn(y0, c) * 0x1p53f), (2045 << 20) - field, &v))
      v = rcp_apart(y, e);
    return v;
  }
  __device__ static __forceinline__ double root(double x) {
    const Start b = rsqrt_start(x);
    const double s = x * b.y, d = fma(-s, s, x);
    return root_of(x, b, s, d, scaled(b, d));
  }
  // root(x), and its reciprocal to *ri
  __device__ static __forceinline__ double root_and_rsqrt(double x, double* ri) {
    const Start b = rsqrt_start(x);
    const double s = x * b.y, d = fma(-s, s, x);
    const float df = scaled(b, d);
    *ri = rsqrt_of(b, d, df, fma(-s, b.y, 1.0));
    return root_of(x, b, s, d, df);
  }
  // a / b, its residual taken once: 4 operations, as well rounded as the others (b as for rcp)
  __device__ static __forceinline__ double div(double a, double b) {
    const double y = rcp(b), q = a * y;
    return fma(fma(-b, q, a), y, q);
  }
};

// The same for any argument: those out of FastOps64's range take the IEEE operations, out of line.
struct CheckedOps64 {
  __device__ static __forceinline__ double div(double a, double b) {
    const bool finite = (__double2hiint(a) & 0x7ff00000) != 0x7ff00000;
    return finite && in_range(__double2hiint(b)) ? FastOps64::div(a, b) : ieee_div(a, b);
  }
  __device__ static __forceinline__ double root(double x) {
    return in_range(__double2hiint(x)) ? FastOps64::root(x) : ieee_root(x);
  }

 private:
  // high word of a positive number from 2^-890, below 2^890
  __device__ static __forceinline__ bool in_range(int hi) { return (unsigned)hi - (133u << 20) < 1780u << 20; }
  __device__ static __noinline__ double ieee_div(double a, double b) { return a / b; }
  __device__ static __noinline__ double ieee_root(double x) { return sqrt(x); }
};

// x / 2 for a positive normal x, without an FP64 operation.
__device__ __forceinline__ double halve(double x) {
  return __hiloint2double(__double2hiint(x) - 0x00100000, __double2loint(x));
}

template <typename S>
struct Kerr {
  S r, f;        // r of Eq. 6, f of Eq. 4
  S k0, k1, k2;  // spatial k_m (k_3 = 1)
  S D;           // sqrt((R^2 - a^2)^2 + 4 a^2 z^2) = d(quartic)/d(r^2)
  S inv_r, inv_rho2, inv_sig, inv_D;  // 1/r, 1/(r^2 + a^2), 1/(r^4 + a^2 z^2), 1/D, shared with the derivatives
  bool flat;     // r = 0 (the disk z = 0, R <= a): metric taken flat, its limit there
};

// Non-negative root of Eq. 6 as r^2, written so that neither branch cancels; *D receives
// sqrt((R^2 - a^2)^2 + 4 a^2 z^2).
template <typename S, typename Ops = IeeeOps>
__device__ __forceinline__ S kerr_r2(S x, S y, S z, S a, S* D) {
  const S a2 = a * a;
  const S q = a2 * z * z;
  const S p = x * x + y * y + z * z - a2;
  *D = Ops::root(p * p + S(4) * q);
  return (p >= S(0)) ? S(0.5) * (p + *D) : Ops::div(S(2) * q, *D - p);
}

// f and k of Eqs. 4-5 at (x, y, z) given r^2 from Eq. 6.
template <typename S, typename Ops = IeeeOps>
__device__ __forceinline__ Kerr<S> kerr_from_r2(S x, S y, S z, S m, S a, S r2, S D) {
  Kerr<S> K;
  const S a2 = a * a;
  const S q = a2 * z * z;
  K.D = D;
  if (!(r2 > S(0))) {
    K.flat = true;
    K.r = S(0);
    K.f = S(0);
    K.k0 = S(0);
    K.k1 = S(0);
    K.k2 = S(1);
    return K;
  }
  K.flat = false;
  K.r = Ops::root(r2);
  K.inv_r = Ops::rcp(K.r);
  K.inv_rho2 = Ops::rcp(r2 + a2);
  K.inv_sig = Ops::rcp(r2 * r2 + q);
  K.inv_D = Ops::rcp(D);
  K.f = S(2) * m * K.r * r2 * K.inv_sig;
  K.k0 = (K.r * x - a * y) * K.inv_rho2;
  K.k1 = (K.r * y + a * x) * K.inv_rho2;
  K.k2 = z * K.inv_r;
  return K;
}

template <typename S, typename Ops = IeeeOps>
__device__ __forceinline__ Kerr<S> kerr_eval(S x, S y, S z, S m, S a) {
  S D;
  const S r2 = kerr_r2<S, Ops>(x, y, z, a, &D);
  return kerr_from_r2<S, Ops>(x, y, z, m, a, r2, D);
}

// kerr_eval in FP64 with FastOps64; since the root satisfies Sigma = r^4 + a^2 z^2 = r^2 D, 1 / Sigma and f = 2 m r / D
// need no division.  The root for p = R^2 - a^2 < 0 is out of line (its operations would be issued for every point).
static __device__ __noinline__ double kerr_root_inside(double p, double q4, double D) {
  return halve(FastOps64::div(q4, D - p));
}
__device__ __forceinline__ Kerr<double> kerr_eval_fast(double x, double y, double z, double two_m, double a, double a2,
                                                       double a2_4) {
  Kerr<double> K;
  const double q4 = a2_4 * (z * z);
  const double p = fma(x, x, fma(y, y, fma(z, z, -a2)));
  const double D2 = fma(p, p, q4);
  K.D = FastOps64::root_and_rsqrt(D2, &K.inv_D);
  double r2 = halve(p + K.D);
  if (__double2hiint(p) < 0) r2 = kerr_root_inside(p, q4, K.D);
  if (__double2hiint(D2) < 0x00100000 || __double2hiint(r2) < 0x00100000) {  // r = 0
    K.flat = true;
    K.r = K.f = K.k0 = K.k1 = 0.0;
    K.k2 = 1.0;
    return K;
  }
  K.flat = false;
  K.r = FastOps64::root_and_rsqrt(r2, &K.inv_r);
  K.inv_rho2 = FastOps64::rcp(r2 + a2);
  K.inv_sig = K.inv_D * (K.inv_r * K.inv_r);
  K.f = two_m * K.r * K.inv_D;
  K.k0 = fma(K.r, x, -(a * y)) * K.inv_rho2;
  K.k1 = fma(K.r, y, a * x) * K.inv_rho2;
  K.k2 = z * K.inv_r;
  return K;
}
__device__ __forceinline__ Kerr<double> kerr_eval_fast(double x, double y, double z, double m, double a) {
  const double a2 = a * a;
  return kerr_eval_fast(x, y, z, 2.0 * m, a, a2, 4.0 * a2);
}

// Gamma^a_mn u^m u^n = g^ab (u^m d_m g_bn u^n - 1/2 d_b g_mn u^m u^n) for g = eta + f k k.
// With s = k.u, D_b = u^m d_m k_b, E_b = u^n d_b k_n and d_4 = 0:
//   w_b = (u.df) s k_b + f s D_b + f (u.D) k_b - 1/2 s^2 d_b f - f s E_b
//   Gamma u u = eta^ab w_b - f k^a (k^b w_b)
// with grad r from the implicit quartic, r_x = x r / D, r_y = y r / D, r_z = z (r^2 + a^2) / (r D), and without forming
// d_i k_j: with u.r = u^i d_i r, k_x = (r x - a y) / rho^2 and so on,
//   D_x = [x u.r + r u^x - a u^y - 2 r (u.r) k_x] / rho^2,  D_y alike,  D_z = (u^z - k_z u.r) / r,
//   E_j = A d_j r + ((r u^x + a u^y) / rho^2, (r u^y - a u^x) / rho^2, u^z / r)_j,
//   A = [u^x x + u^y y - 2 r (u^x k_x + u^y k_y)] / rho^2 - u^z k_z / r,
// and d_r f = f (3 / r - 4 r / D).
__device__ __forceinline__ void christoffel_uu_fast(const Kerr<double>& K, double x, double y, double z, double a,
                                                    const double u[4], double out[4]) {
  if (K.flat) {
    out[0] = out[1] = out[2] = out[3] = 0.0;
    return;
  }
  const double r = K.r, f = K.f, k0 = K.k0, k1 = K.k1, k2 = K.k2, ir = K.inv_r, ip = K.inv_rho2;
  const double rD = r * K.inv_D, two_r = r + r, a2 = a * a;
  const double rx = x * rD, ry = y * rD, rz = z * (fma(r, r, a2) * (K.inv_D * ir));
  const double fr = f * fma(3.0, ir, -4.0 * rD);
  const double fx = fr * rx, fy = fr * ry, fz = fma(fr, rz, -2.0 * a2 * z * (f * K.inv_sig));
  const double ur = fma(u[0], rx, fma(u[1], ry, u[2] * rz));
  const double t = two_r * ur;
  const double p0 = r * u[0], p1 = r * u[1];
  const double D0 = fma(-t, k0, fma(x, ur, fma(-a, u[1], p0))) * ip;
  const double D1 = fma(-t, k1, fma(y, ur, fma(a, u[0], p1))) * ip;
  const double D2 = fma(-k2, ur, u[2]) * ir;
  const double uk = fma(u[0], k0, u[1] * k1), u2i = u[2] * ir;
  const double A = fma(fma(-two_r, uk, fma(u[0], x, u[1] * y)), ip, -(k2 * u2i));
  const double E0 = fma(A, rx, fma(a, u[1], p0) * ip);
  const double E1 = fma(A, ry, fma(-a, u[0], p1) * ip);
  const double E2 = fma(A, rz, u2i);
  const double s = fma(k2, u[2], uk) + u[3];
  const double uf = fma(u[0], fx, fma(u[1], fy, u[2] * fz));
  const double uD = fma(u[0], D0, fma(u[1], D1, u[2] * D2));
  const double c1 = fma(uf, s, f * uD), fs = f * s, hs2 = -0.5 * s * s;
  const double w0 = fma(c1, k0, fma(fs, D0 - E0, hs2 * fx));
  const double w1 = fma(c1, k1, fma(fs, D1 - E1, hs2 * fy));
  const double w2 = fma(c1, k2, fma(fs, D2 - E2, hs2 * fz));
  const double kw = fma(k0, w0, fma(k1, w1, fma(k2, w2, -c1)));
  const double fk = f * kw;
  out[0] = fma(-fk, k0, w0);
  out[1] = fma(-fk, k1, w1);
  out[2] = fma(-fk, k2, w2);
  out[3] = fk - c1;
}

// Field tensor at a point from the prognostic pair: covariant b = (F_yz, F_zx, F_xy) and
// contravariant d = (F^x4, F^y4, F^z4).  Lowering F with g = eta + f k k gives, for the
// spatial block, F_cov = M F^sp M + f (d k^T - k d^T) with M = I + f k k^T, so
//   alpha = b - f (d x k),  h = (F^yz, F^zx, F^xy) = [alpha + f k (k.alpha)] / (1 + f),
// and the covariant electric part e_i = F_i4 = f (k x h)_i + (f - 1) d_i - f k_i (k.d).
template <typename S>
__device__ __forceinline__ void contra_spatial(S f, S k0, S k1, S k2, const S b[3], const S d[3], S h[3]) {
  const S al0 = b[0] - f * (d[1] * k2 - d[2] * k1);
  const S al1 = b[1] - f * (d[2] * k0 - d[0] * k2);
  const S al2 = b[2] - f * (d[0] * k1 - d[1] * k0);
  const S ka = f * (k0 * al0 + k1 * al1 + k2 * al2);
  const S inv = S(1) / (S(1) + f);
  h[0] = (al0 + ka * k0) * inv;
  h[1] = (al1 + ka * k1) * inv;
  h[2] = (al2 + ka * k2) * inv;
}

// contra_spatial in FP64: with G = f / (1 + f) the same tensor is h = b - G [b + d x k - k (k.b)].
__device__ __forceinline__ void contra_spatial_fast(double f, double k0, double k1, double k2, const double b[3],
                                                    const double d[3], double h[3]) {
  const double G = f * FastOps64::rcp(1.0 + f);
  const double kb = fma(k0, b[0], fma(k1, b[1], k2 * b[2]));
  h[0] = fma(-G, fma(-k0, kb, b[0]) + fma(d[1], k2, -(d[2] * k1)), b[0]);
  h[1] = fma(-G, fma(-k1, kb, b[1]) + fma(d[2], k0, -(d[0] * k2)), b[1]);
  h[2] = fma(-G, fma(-k2, kb, b[2]) + fma(d[0], k1, -(d[1] * k0)), b[2]);
}

// Lorentz part of Eq. 15, (q/m) F^a_b u^b = (q/m) F^ac u_c, with u_c = g_cb u^b:
//   u_i = u^i + f s k_i, u_4 = -u^4 + f s;  (q/m)[(u_cov x h)_i + d_i u_4],  -(q/m) d.u_cov
template <typename S>
__device__ __forceinline__ void lorentz(S qm, S f, S k0, S k1, S k2, const S h[3], const S d[3], const S u[4],
                                        S out[4]) {
  const S s = k0 * u[0] + k1 * u[1] + k2 * u[2] + u[3];
  const S fs = f * s;
  const S c0 = u[0] + fs * k0, c1 = u[1] + fs * k1, c2 = u[2] + fs * k2;
  const S c3 = fs - u[3];
  out[0] = qm * (c1 * h[2] - c2 * h[1] + d[0] * c3);
  out[1] = qm * (c2 * h[0] - c0 * h[2] + d[1] * c3);
  out[2] = qm * (c0 * h[1] - c1 * h[0] + d[2] * c3);
  out[3] = -qm * (d[0] * c0 + d[1] * c1 + d[2] * c2);
}

// Eq. 16: gamma = [u^4/c + sqrt((u^4/c)^2 + 4 a^4 dt / (2c))] / 2; a negative argument or a
// non-positive result falls back to u^4/c (the caller counts it).
template <typename S, typename Ops = IeeeOps>
__device__ __forceinline__ S gamma_step(S u4, S a4, S inv_c, S dt, bool* fallback) {
  const S w = u4 * inv_c;
  const S arg = w * w + S(2) * a4 * dt * inv_c;
  S g = S(-1);
  if (arg >= S(0)) g = S(0.5) * (w + Ops::root(arg));
  if (!(g > S(0))) {
    *fallback = true;
    return w;
  }
  *fallback = false;
  return g;
}

}  // namespace grpic
