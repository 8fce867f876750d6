// mhd_device.cuh -- device numerics of the CT-MHD step (FP64, sm_103a).
//
// On GB300 the FP64 pipe retires 2 DFMA per SM per clock (measured 0.63 T DFMA/s over 152 SMs;
// 0.53 T of adds or multiplies), 1/64 of the FP32 rate; a DMNMX or DSETP costs a full FP64 issue slot. Every
// comparison, min/max, |x| and sign test below therefore runs on the integer pipe, on the
// IEEE-754 bit pattern: for non-NaN doubles, the key  b ^ ((b >> 63) & 0x7fff...f)  of the bit
// pattern b orders like the value (with -0 just below +0), and for non-negative values the raw
// pattern already does. Only genuine arithmetic is issued to the FP64 pipe.
#pragma once
#include <cstdint>

#include "mhd_fixed.cuh"

namespace mhd {

using ::fma;  // the double overload stays visible beside the Dual one below

enum { REC_PC = 0, REC_PLM_MC = 1, REC_PLM_MINMOD = 2, REC_PPM = 3, REC_PPM_EP = 4 };
enum { RS_HLL = 0, RS_HLLD = 1, RS_LLF = 2 };
enum { EMF_Q26 = 0, EMF_FS18 = 1, EMF_B25A = 2 };

// ------------------------------------------------------------------------------------------
// Integer-pipe comparisons on doubles
// ------------------------------------------------------------------------------------------
__device__ __forceinline__ long long dbits(double x) { return __double_as_longlong(x); }
__device__ __forceinline__ double dfrom(long long b) { return __longlong_as_double(b); }
// The sign-bit operations below are inline PTX on the high 32-bit word, with the masks as
// immediates: written in C++, a mask of the sign bit is recognised as |x|, copysign, -x or a test
// against zero and issued to the FP64 pipe, and a 64-bit mask constant would hold two registers.
__device__ __forceinline__ double vabs(double x) {
  double r;
  asm("{\n\t.reg .b32 l, h;\n\tmov.b64 {l, h}, %1;\n\tand.b32 h, h, 0x7FFFFFFF;\n\tmov.b64 %0, {l, h};\n\t}"
      : "=d"(r) : "d"(x));
  return r;
}
// |m| carrying the sign of s
__device__ __forceinline__ double with_sign(double m, double s) {
  double r;
  asm("{\n\t.reg .b32 l, h, t, g;\n\tmov.b64 {l, h}, %1;\n\tmov.b64 {t, g}, %2;\n\t"
      "and.b32 h, h, 0x7FFFFFFF;\n\tand.b32 g, g, 0x80000000;\n\tor.b32 h, h, g;\n\tmov.b64 %0, {l, h};\n\t}"
      : "=d"(r) : "d"(m), "d"(s));
  return r;
}
// x with its sign flipped when neg (the value of x * -1)
__device__ __forceinline__ double neg_if(bool neg, double x) {
  double r;
  asm("{\n\t.reg .b32 l, h;\n\tmov.b64 {l, h}, %1;\n\txor.b32 h, h, %2;\n\tmov.b64 %0, {l, h};\n\t}"
      : "=d"(r) : "d"(x), "r"(neg ? 0x80000000u : 0u));
  return r;
}
// bit pattern of |x|
__device__ __forceinline__ long long mag_bits(double x) { return dbits(vabs(x)); }
// total-order key: for non-NaN doubles it orders like the value, with -0 just below +0 (the
// magnitude bits of a negative pattern are flipped)
__device__ __forceinline__ long long okey(double x) {
  const long long b = dbits(x);
  return b ^ (long long)((unsigned long long)(b >> 63) >> 1);
}
// max/min return the first argument on ties (as in the method's tie rule).
__device__ __forceinline__ double vmax(double a, double b) { return okey(a) >= okey(b) ? a : b; }
__device__ __forceinline__ double vmin(double a, double b) { return okey(a) <= okey(b) ? a : b; }
// for a, b >= 0 (or +-0) the raw bit pattern orders like the value
__device__ __forceinline__ double pmax(double a, double b) { return dbits(a) >= dbits(b) ? a : b; }
__device__ __forceinline__ double pmin(double a, double b) { return dbits(a) <= dbits(b) ? a : b; }
__device__ __forceinline__ bool gt0(double x) { return dbits(x) > 0; }   // x > 0
// x < 0 (not -0): sign bit set and a non-zero magnitude, one unsigned compare (forming -x
// instead would cost an FP64 issue slot)
__device__ __forceinline__ bool lt0(double x) { return (unsigned long long)dbits(x) > 0x8000000000000000ULL; }
__device__ __forceinline__ bool ge0(double x) { return okey(x) >= -1; }  // x >= 0 (either zero)
__device__ __forceinline__ bool le0(double x) { return !gt0(x); }
__device__ __forceinline__ bool vgt(double a, double b) { return okey(a) > okey(b); }
__device__ __forceinline__ bool is_zero(double x) { return mag_bits(x) == 0; }
// strictly of the same sign, both non-zero
__device__ __forceinline__ bool same_sign(double a, double b) {
  return (gt0(a) && gt0(b)) || (lt0(a) && lt0(b));
}
__device__ __forceinline__ bool finite_d(double x) {
  return (mag_bits(x) >> 52) != 0x7ff;
}
// Reciprocal, reciprocal square root and square root without the IEEE divide/sqrt sequences
// (which cost several FP64 issue slots each): a seed y0 good to about 2^-30, made on the FP32 and
// integer pipes, and one Newton step, y0 (1 + e) with e = 1 - x y0, or y0 (1 + e/2) with
// e = 1 - x y0^2 (2 and 3 FP64 instructions; the hardware's FP64 seeds are good to 2^-20 only and
// take 3 and 5).
// The seed: the significand m (in [1, 4) for the square root, with an even exponent) is split into a
// float mh and a remainder ml; the hardware's single-precision approximation f0 of 1/mh or
// 1/sqrt(mh), in [1/2, 1], has the residual r = 1 - m f0 or 1 - m f0^2, formed by fused
// multiply-adds; the correction f0 r or f0 r / 2 is added to f0's bits as an integer multiple of
// 2^-32. Exponents at the ends of the range, zero, infinities and NaN take the hardware's FP64 seed
// and one more term of the series, as does a negative argument of a root.
// Measured (256^3 turbulence step): face sweeps 21.0 -> 19.5 ms, left/right edge sweeps 6.26 -> 5.91,
// flag pass 1.17 -> 1.05; the 128^3 Alfven wave's face sweeps 4.67 -> 4.30. Largest differences from
// IEEE results over 2^28 arguments of every binade (mhd_math_check): reciprocal and root 2.0, reciprocal
// root 2.4 x 2^-53.
__device__ __forceinline__ unsigned hi_word(double x) { return (unsigned)__double2hiint(x); }
__device__ __forceinline__ double seed_bits(float f0, float c32, unsigned hi_scale) {
  // f0 + c32 2^-32, its exponent shifted by hi_scale (a multiple of 2^20 in the high word)
  const int ci = __float_as_int(c32 + 12582912.0f) - 0x4B400000;  // nearest integer
  const long long b = ((long long)__float_as_int(f0) << 29) + ((long long)ci << 21);
  return __hiloint2double((int)((unsigned)(b >> 32) + hi_scale), (int)b);
}
__device__ __forceinline__ double rcp_seed(double x) {
  const unsigned hi = hi_word(x), lo = (unsigned)__double2loint(x);
  const float mh = __int_as_float((int)((__funnelshift_l(lo, hi, 3) & 0x7fffffu) | 0x3f800000u));
  const float ml = __int_as_float((int)(((lo << 3) >> 9) | 0x3f800000u)) - 1.0f;  // in units of 2^-23
  float f0;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(f0) : "f"(mh));
  f0 = fmaxf(f0, 0.5f);
  const float r = fmaf(ml * -1.1920928955078125e-07f, f0, fmaf(-mh, f0, 1.0f));
  const double y = seed_bits(f0, f0 * r * 4294967296.0f, ((896u + 1023u) << 20) - (hi & 0x7ff00000u));
  return __hiloint2double(__double2hiint(y) | (int)(hi & 0x80000000u), __double2loint(y));
}
__device__ __forceinline__ double rsqrt_seed(double x) {  // x > 0
  const unsigned hi = hi_word(x), lo = (unsigned)__double2loint(x);
  const unsigned odd = ~hi & 0x00100000u;  // the exponent's parity (1023 is odd): m in [2, 4)
  const unsigned one = 0x3f800000u + (odd << 3);
  const float mh = __int_as_float((int)((__funnelshift_l(lo, hi, 3) & 0x7fffffu) | one));
  const float ml = __int_as_float((int)(((lo << 3) >> 9) | one)) - __int_as_float((int)one);
  float f0;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(f0) : "f"(mh));
  f0 = fmaxf(f0, 0.5f);
  const float p = f0 * f0, pe = fmaf(f0, f0, -p);
  const float r = fmaf(ml * -1.1920928955078125e-07f, p, fmaf(-mh, pe, fmaf(-mh, p, 1.0f)));
  const int k2 = (int)(hi & 0x7ff00000u) - (1023 << 20) - (int)odd;  // 2 k, in the exponent's place
  return seed_bits(f0, f0 * r * 2147483648.0f, (896u << 20) - (unsigned)((k2 >> 1) & ~0xfffff));
}
// (functions of their own, not inlined: short enough to be predicated, their FP64 instructions would
// be issued, and take the pipe, for every lane that does not need them)
static __device__ __noinline__ double rcp_any(double x) {
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double e = fma(-x, y, 1.0);
  return fma(y, fma(e, e, e), y);
}
static __device__ __noinline__ double rsqrt_any(double x) {
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double e = fma(-(x * y), y, 1.0);
  return fma(y * e, fma(0.375, e, 0.5), y);
}
static __device__ __noinline__ double sqrt_any(double x) {
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double g = x * y;
  const double e = fma(-g, y, 1.0);
  const double r = fma(g * e, fma(0.375, e, 0.5), g);
  return is_zero(x) ? 0.0 : r;
}
__device__ __forceinline__ double rcp(double x) {
  if (((hi_word(x) >> 20) & 0x7ff) - 2u > 2042u) return rcp_any(x);
  const double y = rcp_seed(x);
  return fma(y, fma(-x, y, 1.0), y);
}
// x / 2 of a normal number above the smallest binades
__device__ __forceinline__ double half_normal(double x) {
  return __hiloint2double(__double2hiint(x) - (1 << 20), __double2loint(x));
}
__device__ __forceinline__ double rsqrt_(double x) {
  if ((hi_word(x) >> 20) - 2u > 2042u) return rsqrt_any(x);
  const double y = rsqrt_seed(x);
  return fma(half_normal(y), fma(-(x * y), y, 1.0), y);
}
// sqrt(x) for x > 0, and 0 for x = 0: with g = x y0 and e = 1 - g y0, sqrt(x) = g (1 + e/2); the
// rounding of g enters halved, since e is formed from the rounded g
__device__ __forceinline__ double sqrt_(double x) {
  if ((hi_word(x) >> 20) - 2u > 2042u) return sqrt_any(x);
  const double y = rsqrt_seed(x);
  const double g = x * y;
  return fma(half_normal(g), fma(-g, y, 1.0), g);
}

// ------------------------------------------------------------------------------------------
// Forward-mode dual number (value + one tangent) for the adjoint kernels' local Jacobians. Every
// decision (comparison, min/max, sign, limiter branch) is taken on the value exactly as in the
// double code, so a derivative is the derivative on the branch the forward pass took.
// ------------------------------------------------------------------------------------------
struct Dual {
  double v, t;
  __device__ __forceinline__ Dual() {}
  __device__ __forceinline__ Dual(double x) : v(x), t(0.0) {}  // NOLINT: constants promote
  __device__ __forceinline__ Dual(double x, double dx) : v(x), t(dx) {}
};
__device__ __forceinline__ Dual operator+(Dual a, Dual b) { return Dual(a.v + b.v, a.t + b.t); }
__device__ __forceinline__ Dual operator-(Dual a, Dual b) { return Dual(a.v - b.v, a.t - b.t); }
__device__ __forceinline__ Dual operator-(Dual a) { return Dual(-a.v, -a.t); }
__device__ __forceinline__ Dual operator*(Dual a, Dual b) { return Dual(a.v * b.v, fma(a.t, b.v, a.v * b.t)); }
// mixed forms with a constant operand (no tangent arithmetic for the constant's zero tangent)
__device__ __forceinline__ Dual operator*(double a, Dual b) { return Dual(a * b.v, a * b.t); }
__device__ __forceinline__ Dual operator*(Dual a, double b) { return Dual(a.v * b, a.t * b); }
__device__ __forceinline__ Dual operator+(Dual a, double b) { return Dual(a.v + b, a.t); }
__device__ __forceinline__ Dual operator+(double a, Dual b) { return Dual(a + b.v, b.t); }
__device__ __forceinline__ Dual operator-(Dual a, double b) { return Dual(a.v - b, a.t); }
__device__ __forceinline__ Dual operator-(double a, Dual b) { return Dual(a - b.v, -b.t); }
__device__ __forceinline__ Dual& operator+=(Dual& a, Dual b) { a = a + b; return a; }
__device__ __forceinline__ Dual fma(Dual a, Dual b, Dual c) {
  return Dual(fma(a.v, b.v, c.v), fma(a.t, b.v, fma(a.v, b.t, c.t)));
}
__device__ __forceinline__ Dual fma(double a, Dual b, Dual c) { return Dual(fma(a, b.v, c.v), fma(a, b.t, c.t)); }
__device__ __forceinline__ Dual fma(Dual a, double b, Dual c) { return Dual(fma(a.v, b, c.v), fma(a.t, b, c.t)); }
__device__ __forceinline__ Dual fma(Dual a, Dual b, double c) {
  return Dual(fma(a.v, b.v, c), fma(a.t, b.v, a.v * b.t));
}
__device__ __forceinline__ double val(double x) { return x; }
__device__ __forceinline__ double val(const Dual& x) { return x.v; }
__device__ __forceinline__ Dual vmax(Dual a, Dual b) { return okey(a.v) >= okey(b.v) ? a : b; }
__device__ __forceinline__ Dual vmin(Dual a, Dual b) { return okey(a.v) <= okey(b.v) ? a : b; }
__device__ __forceinline__ Dual pmax(Dual a, Dual b) { return dbits(a.v) >= dbits(b.v) ? a : b; }
__device__ __forceinline__ Dual pmin(Dual a, Dual b) { return dbits(a.v) <= dbits(b.v) ? a : b; }
__device__ __forceinline__ Dual vabs(Dual x) {
  const bool neg = dbits(x.v) < 0;
  return Dual(vabs(x.v), neg_if(neg, x.t));
}
__device__ __forceinline__ bool gt0(const Dual& x) { return gt0(x.v); }
__device__ __forceinline__ bool lt0(const Dual& x) { return lt0(x.v); }
__device__ __forceinline__ bool ge0(const Dual& x) { return ge0(x.v); }
__device__ __forceinline__ bool vgt(const Dual& a, const Dual& b) { return vgt(a.v, b.v); }
__device__ __forceinline__ bool is_zero(const Dual& x) { return is_zero(x.v); }
__device__ __forceinline__ bool same_sign(const Dual& a, const Dual& b) { return same_sign(a.v, b.v); }
// |m| with the sign of s
__device__ __forceinline__ Dual with_sign(Dual m, Dual s) {
  const bool flip = (dbits(m.v) < 0) != (dbits(s.v) < 0);
  return Dual(with_sign(m.v, s.v), neg_if(flip, m.t));
}
__device__ __forceinline__ Dual rcp(Dual x) {
  const double r = rcp(x.v);
  return Dual(r, -x.t * r * r);
}
__device__ __forceinline__ Dual rsqrt_(Dual x) {
  const double r = rsqrt_(x.v);
  return Dual(r, -0.5 * x.t * r * r * r);
}
// the value of sqrt_, derivative rsqrt(x) / 2; both 0 at x = 0
__device__ __forceinline__ Dual sqrt_(Dual x) {
  return Dual(sqrt_(x.v), is_zero(x.v) ? 0.0 : 0.5 * rsqrt_(x.v) * x.t);
}

// x / 2 exactly as the FP64 multiply by 0.5 rounds it (ties to even), on the integer pipe: one
// less in the exponent above the smallest normal binade; below it (where a double is its bit
// pattern times 2^-1074) the magnitude's integer is halved with ties to even; zero, infinity and
// NaN pass through.
__device__ __forceinline__ double halve(double x) {
  const long long mag = mag_bits(x);
  long long r;
  if (mag >= (2LL << 52)) r = mag >= 0x7ff0000000000000LL ? mag : mag - (1LL << 52);
  else r = (mag >> 1) + (mag & (mag >> 1) & 1);
  return with_sign(dfrom(r), x);
}
__device__ __forceinline__ Dual halve(Dual x) { return Dual(halve(x.v), halve(x.t)); }
__device__ __forceinline__ Dual neg_if(bool neg, Dual x) { return Dual(neg_if(neg, x.v), neg_if(neg, x.t)); }

// ------------------------------------------------------------------------------------------
// Periodic line of points along one axis
// ------------------------------------------------------------------------------------------
struct Line {
  long long base;    // linear index of position 0 along the axis
  long long stride;  // linear-index step along the axis
  int n;             // points along the axis (periodic)
  __device__ __forceinline__ long long at(int p) const {
    p %= n;
    if (p < 0) p += n;
    return base + (long long)p * stride;
  }
};

// ------------------------------------------------------------------------------------------
// Sliding-window 1D reconstruction (Sec. 2.2). A Rec walks along a line of cell (or face)
// values. init() takes the LB + LA values at positions m0-LB .. m0+LA-1; each step() then
// takes the value at m + LA and returns the left/right states of the interface between
// points m-1 and m (left = upper value of point m-1, right = lower value of point m). Every
// point's slope, interface value and limiter run exactly once per sweep.
// FACE: the caller is a face sweep (PPM-EP's choice of pipe, ppm_ep_face).
// For sweeps that keep their windows in shared memory: each() visits the NS doubles of the state,
// and code holds NB more bits.
// ------------------------------------------------------------------------------------------
template <int R> struct Rec;

template <> struct Rec<REC_PC> {
  static constexpr int LB = 1, LA = 0, NS = 1, NB = 0;
  double prev;
  int code;
  template <class F> __device__ __forceinline__ void each(F f) { f(0, prev); }
  template <bool FACE>
  __device__ __forceinline__ void init(const double* q) { prev = q[0]; }
  template <bool FACE>
  __device__ __forceinline__ void step(double qn, double& L, double& R) {
    L = prev;
    R = qn;
    prev = qn;
  }
};

// half of the monotonised-central slope: sgn * min(|dl|, |dr|, |dl + dr| / 4)
template <class T>
__device__ __forceinline__ T half_slope_mc(T dl, T dr) {
  if (!same_sign(dl, dr)) return T(0.0);
  T m = pmin(vabs(dl), vabs(dr));
  m = pmin(m, 0.25 * vabs(dl + dr));
  return with_sign(m, dl);
}
// half of the minmod slope: sgn * min(|dl|, |dr|) / 2
template <class T>
__device__ __forceinline__ T half_slope_minmod(T dl, T dr) {
  if (!same_sign(dl, dr)) return T(0.0);
  return with_sign(halve(pmin(vabs(dl), vabs(dr))), dl);
}

template <int R> struct RecPLM {
  static constexpr int LB = 2, LA = 1, NS = 3, NB = 0;
  double qb, dl, aRprev;  // q[m], q[m] - q[m-1], upper value of point m-1
  int code;
  template <class F> __device__ __forceinline__ void each(F f) {
    f(0, qb);
    f(1, dl);
    f(2, aRprev);
  }
  __device__ __forceinline__ double hs(double a, double b) const {
    return R == REC_PLM_MC ? half_slope_mc(a, b) : half_slope_minmod(a, b);
  }
  template <bool FACE>
  __device__ __forceinline__ void init(const double* q) {
    const double e0 = q[1] - q[0], e1 = q[2] - q[1];
    aRprev = q[1] + hs(e0, e1);
    qb = q[2];
    dl = e1;
  }
  template <bool FACE>
  __device__ __forceinline__ void step(double qn, double& L, double& Rt) {
    const double dr = qn - qb;
    const double h = hs(dl, dr);
    L = aRprev;
    Rt = qb - h;
    aRprev = qb + h;
    qb = qn;
    dl = dr;
  }
};
template <> struct Rec<REC_PLM_MC> : RecPLM<REC_PLM_MC> {};
template <> struct Rec<REC_PLM_MINMOD> : RecPLM<REC_PLM_MINMOD> {};

// Colella & Woodward 1984: van Leer limited slope (their Eqs. 1.7-1.8), interface value
// (Eq. 1.6) and monotonicity constraints (Eq. 1.10), arranged to reuse the one-sided
// differences: the slope is carried doubled, dq2 = 2 dq = sgn min(|dl + dr|, 4|dl|, 4|dr|), the
// interface value between points 0 and 1 is q0 + (q1 - q0)/2 - (dq2_1 - dq2_0)/12, and with
// s1 = aR - a, s2 = a - aL (same sign unless a is an extremum) the tests of Eq. 1.10 become sign
// tests: with da = aR - aL = s1 + s2 (sign of s1) and a6 = 6 (a - (aL + aR)/2) = 3 (s2 - s1),
// da a6 > da^2 <=> da (a6 - da) > 0 <=> s2 - 2 s1 has the sign of s1, and
// -da^2 > da a6 <=> da (a6 + da) < 0 <=> 2 s2 - s1 has the opposite sign; the corrections are
// 3a - 2aR = a - 2 s1 and 3a - 2aL = a + 2 s2.

// Bit pattern of 2|x| from the bit pattern b >= 0 of |x|, exactly and on the integer pipe: zero
// and subnormals double by a shift of the mantissa (which carries into the exponent where the
// result becomes normal), normals by one more in the exponent, and 2|x| >= 2^1024 (or a NaN)
// gives infinity.
__device__ __forceinline__ long long twice_bits(long long b) {
  if (b < (1LL << 52)) return b << 1;
  if (b >= (2046LL << 52)) return 0x7ff0000000000000LL;
  return b + (1LL << 52);
}
// 4 m for m >= 0, exact (two doublings)
__device__ __forceinline__ double times4(double m) { return dfrom(twice_bits(twice_bits(dbits(m)))); }
__device__ __forceinline__ Dual times4(Dual m) { return Dual(times4(m.v), 4.0 * m.t); }

__device__ __forceinline__ double vl_slope2(double dl, double dr) {
  if (!same_sign(dl, dr)) return 0.0;
  const double s = dl + dr;
  const double m = pmin(vabs(s), times4(pmin(vabs(dl), vabs(dr))));
  return with_sign(m, s);
}
// With s1, s2 of one sign, u = s2 - 2 s1 = (a6 - da)/2 has the sign of s1 exactly when
// |s2| > 2|s1|, and v = 2 s2 - s1 = (a6 + da)/2 the sign of -s1 exactly when 2|s2| < |s1|: the two
// tests compare bit patterns (one more in the exponent is the doubling), and the one correction
// that applies is a single FMA.
enum { PPM_FLAT = 0, PPM_FIX_L = 1, PPM_FIX_R = 2, PPM_KEEP = 3 };
// which constraint applies for s1 = aR - a, s2 = a - aL
__device__ __forceinline__ int ppm_mono_case(double s1, double s2) {
  // (unsigned: the doubling of an infinity or a NaN stays the larger)
  const unsigned long long m1 = (unsigned long long)mag_bits(s1), m2 = (unsigned long long)mag_bits(s2), two = 1ULL << 52;
  if ((dbits(s1) ^ dbits(s2)) < 0 || m1 == 0 || m2 == 0) return PPM_FLAT;  // a is an extremum
  if (m2 > m1 + two) return PPM_FIX_L;                                     // aL = 3a - 2aR = a - 2 s1
  if (m2 + two < m1) return PPM_FIX_R;                                     // aR = 3a - 2aL = a + 2 s2
  return PPM_KEEP;
}
__device__ __forceinline__ void ppm_mono(double a, double s1, double s2, double& aL, double& aR) {
  const int c = ppm_mono_case(s1, s2);
  if (c == PPM_FLAT) {
    aL = a;
    aR = a;
  } else if (c != PPM_KEEP) {
    const bool l = c == PPM_FIX_L;
    const double r = fma(l ? -2.0 : 2.0, l ? s1 : s2, a);
    if (l) aL = r; else aR = r;
  }
}

static __device__ __noinline__ double ppm_offset_any(double dl, double d, double dn) {
  return fma(vl_slope2(dl, d) - vl_slope2(d, dn), 1.0 / 12.0, halve(d));
}
__device__ __forceinline__ void ppm_split(double dl, double d, double dn, double& r, double& s) {
  const unsigned long long bd = (unsigned long long)dbits(d);
  const unsigned e = (unsigned)(bd >> 52) & 0x7ff;
  if (e - 128u > 1911u && (bd << 1) != 0) {  // out of the fixed-point form's range
    r = ppm_offset_any(dl, d, dn);
    s = __dsub_rn(d, r);
    return;
  }
  unsigned long long br, bs;
  ppm_split_bits((unsigned long long)dbits(dl), bd, (unsigned long long)dbits(dn), br, bs);
  r = dfrom((long long)br);
  s = dfrom((long long)bs);
}

template <> struct Rec<REC_PPM> {
  static constexpr int LB = 3, LA = 2, NS = 7, NB = 0;
  double q1, q2;      // q[m], q[m+1]
  double dl, dq;      // q[m] - q[m-1], q[m+1] - q[m]
  double s2;          // q[m] - f1
  double f1;          // interface value at m - 1/2
  double aRprev;      // upper value of point m-1
  int code;
  template <class F> __device__ __forceinline__ void each(F f) {
    f(0, q1);
    f(1, q2);
    f(2, dl);
    f(3, dq);
    f(4, s2);
    f(5, f1);
    f(6, aRprev);
  }
  template <bool FACE>
  __device__ __forceinline__ void init(const double* v) {  // v = q[m0-3 .. m0+1]
    const double e0 = v[1] - v[0], e1 = v[2] - v[1], e2 = v[3] - v[2], e3 = v[4] - v[3];
    double ra, sa, rb, sb;
    ppm_split(e0, e1, e2, ra, sa);
    ppm_split(e1, e2, e3, rb, sb);
    const double fb = v[2] + rb;
    double aL = v[1] + ra, aR = fb;
    ppm_mono(v[2], rb, sa, aL, aR);
    aRprev = aR;
    q1 = v[3];
    q2 = v[4];
    dl = e2;
    dq = e3;
    s2 = sb;
    f1 = fb;
  }
  template <bool FACE>
  __device__ __forceinline__ void step(double qn, double& L, double& R) {
    const double dn = qn - q2;
    double r, s;
    ppm_split(dl, dq, dn, r, s);
    const double f2 = q1 + r;
    double aL = f1, aR = f2;
    ppm_mono(q1, r, s2, aL, aR);
    L = aRprev;
    R = aL;
    aRprev = aR;
    q1 = q2;
    q2 = qn;
    dl = dq;
    dq = dn;
    s2 = s;
    f1 = f2;
  }
};

// PPM-EP, the extremum-preserving PPM that Sec. 2.2 cites (Rider, Greenough & Kamm 2007) without
// defining it; the reading taken: the fourth-order interface value
// (7 (q_j + q_{j+1}) - (q_{j-1} + q_{j+2})) / 12 is bounded by its two cells (median form), and a
// cell's parabola takes the CW84 constraints of PPM above, except at smooth extrema. An interface
// lies at an extremum when two of the three differences around it (d_{j-1/2}, d_{j+1/2},
// d_{j+3/2}, d_{k+1/2} = q_{k+1} - q_k) have strictly opposite signs, a cell when one of its two
// interfaces does; "smooth" means the curvatures D_k = d_{k+1/2} - d_{k-1/2} of the two cells of
// the interface (of the cell and its two neighbours) are all > 0 or all < 0. Differences and
// curvatures are formed as differences of differences (no FMA), so their signs are exactly those of
// the definition evaluated in plain FP64.
// Only the signs of differences and curvatures are used: they are carried as 2-bit codes
// (1 positive, 2 negative, 0 zero), decided on the integer pipe.
__device__ __forceinline__ int sgn_code(double x) { return (int)gt0(x) | ((int)lt0(x) << 1); }
__device__ __forceinline__ bool opp_code(int a, int b) { return (a | b) == 3; }
__device__ __forceinline__ bool same_code(int a, int b) { return a == b && a != 0; }
// an interface lies at an extremum: two of the differences around it of strictly opposite sign
__device__ __forceinline__ bool ext_code(int sm, int s0, int sp) {
  return opp_code(sm, s0) || opp_code(s0, sp) || opp_code(sm, sp);
}
// which of a, b, c is the median, ties resolved as vmin / vmax resolve them: 0, 1 or 2
template <class T>
__device__ __forceinline__ int median3_pick(T a, T b, T c) {
  const long long ka = okey(val(a)), kb = okey(val(b)), kc = okey(val(c));
  const int lo = ka <= kb ? 0 : 1, hi = ka >= kb ? 0 : 1;
  const long long klo = lo == 0 ? ka : kb, khi = hi == 0 ? ka : kb;
  const int m = khi <= kc ? hi : 2;
  const long long km = m == 2 ? kc : khi;
  return klo >= km ? lo : m;
}
static __device__ __noinline__ double ppm_ep_offset_any(double dl, double d, double dn) {
  return fma(dl - dn, 1.0 / 12.0, halve(d));
}
__device__ __forceinline__ void ppm_ep_split(double dl, double d, double dn, double& r, double& s) {
  const unsigned long long bl = (unsigned long long)dbits(dl), bd = (unsigned long long)dbits(d),
                           bn = (unsigned long long)dbits(dn);
  const int el = (int)(bl >> 52) & 0x7ff, ed = (int)(bd >> 52) & 0x7ff, en = (int)(bn >> 52) & 0x7ff;
  const int e = max(ed, max(el, en));
  if ((unsigned)e - 128u > 1911u) {
    const bool zero = ((bl | bd | bn) << 1) == 0;
    r = zero ? 0.0 : ppm_ep_offset_any(dl, d, dn);
    s = zero ? 0.0 : __dsub_rn(d, r);
    return;
  }
  unsigned long long br, bs;
  ppm_ep_split_bits(bl, bd, bn, e, el, ed, en, br, bs);
  r = dfrom((long long)br);
  s = dfrom((long long)bs);
}
// r and s of the interface between qa and qb (f = qa + r); keep: it lies at a smooth
// extremum (no bound), else f is bounded by the two cells. pick: 0 the fourth-order value, 1 qa, 2 qb.
// FIXED: r and s on the integer pipe. The face sweeps take that form (128^3 Alfven wave: 3.97 ms a step
// against 4.29), the edge sweeps the FP64 one: they do little else, and the integer pipe would bound
// them (bottom/top 0.53 ms against 0.38, with B25a's sweeps at 96^3 0.69 against 0.58).
template <bool FIXED>
__device__ __forceinline__ double ppm_ep_face(double qa, double qb, double dl, double d, double dn, bool keep,
                                              int& pick, double& r, double& s) {
  if (FIXED) {
    ppm_ep_split(dl, d, dn, r, s);
  } else {
    r = fma(dl - dn, 1.0 / 12.0, halve(d));
    s = __dsub_rn(d, r);
  }
  const double f = qa + r;
  pick = 0;
  if (!keep) {
    const int k = median3_pick(qa, f, qb);
    pick = k == 0 ? 1 : (k == 1 ? 0 : 2);
  }
  if (pick != 0) {
    r = pick == 1 ? 0.0 : d;
    s = pick == 1 ? d : 0.0;
  }
  return pick == 0 ? f : (pick == 1 ? qa : qb);
}
// sign code of a - b: a comparison (the rounded difference of two doubles has the sign of the exact
// one). Where a or b is not a number the difference is that NaN, with its sign: a NaN in b compares as
// far on the other side of everything.
__device__ __forceinline__ int cmp_code(double a, double b) {
  const long long ka = okey(a), k = okey(b);
  const long long kb = (hi_word(b) & 0x7fffffffu) > 0x7ff00000u ? ~k : k;
  const bool z = is_zero(a) && is_zero(b);  // +0 and -0 are equal
  return z ? 0 : ((int)(ka > kb) | ((int)(ka < kb) << 1));
}

template <> struct Rec<REC_PPM_EP> {
  static constexpr int LB = 3, LA = 2, NS = 7, NB = 4;
  double q1, q2;      // q[m], q[m+1]
  double dl, dq;      // q[m] - q[m-1], q[m+1] - q[m]
  double s2;          // q[m] - f1
  double f1;          // interface value at m - 1/2
  double aRprev;      // upper value of point m-1
  int code;           // bits 0-1: sign code of the curvature of point m; bit 2: it is that of point m-1
                      // too, and not 0; bit 3: interface m - 1/2 lies at an extremum
  template <class F> __device__ __forceinline__ void each(F f) {
    f(0, q1);
    f(1, q2);
    f(2, dl);
    f(3, dq);
    f(4, s2);
    f(5, f1);
    f(6, aRprev);
  }
  template <bool FACE>
  __device__ __forceinline__ void init(const double* v) {  // v = q[m0-3 .. m0+1]
    const double e0 = v[1] - v[0], e1 = v[2] - v[1], e2 = v[3] - v[2], e3 = v[4] - v[3];
    const int s0 = sgn_code(e0), s1 = sgn_code(e1), sb = sgn_code(e2), s3 = sgn_code(e3);
    // curvature codes of points m0-2, m0-1, m0
    const int ka = cmp_code(e1, e0), kb = cmp_code(e2, e1), kc = cmp_code(e3, e2);
    const bool xa = ext_code(s0, s1, sb), xb = ext_code(s1, sb, s3);
    int p;
    double ra, sa, rb;
    const double fa = ppm_ep_face<FACE>(v[1], v[2], e0, e1, e2, xa && same_code(ka, kb), p, ra, sa);   // m0 - 3/2
    const double fb = ppm_ep_face<FACE>(v[2], v[3], e1, e2, e3, xb && same_code(kb, kc), p, rb, s2);  // m0 - 1/2
    double aL = fa, aR = fb;
    if (!((xa || xb) && same_code(ka, kb) && same_code(kb, kc))) ppm_mono(v[2], rb, sa, aL, aR);
    aRprev = aR;
    q1 = v[3];
    q2 = v[4];
    dl = e2;
    dq = e3;
    f1 = fb;
    code = kc | ((int)same_code(kb, kc) << 2) | ((int)xb << 3);
  }
  template <bool FACE>
  __device__ __forceinline__ void step(double qn, double& L, double& R) {
    const double dn = qn - q2;  // q[m+2] - q[m+1]
    const int c1 = code & 3, cn = cmp_code(dn, dq);  // points m, m+1
    const bool same01 = code & 4, x1 = code & 8, same1n = same_code(c1, cn);
    const bool x2 = ext_code(sgn_code(dl), sgn_code(dq), sgn_code(dn));
    int p;
    double r, s;
    const double f2 = ppm_ep_face<FACE>(q1, q2, dl, dq, dn, x2 && same1n, p, r, s);  // m + 1/2
    double aL = f1, aR = f2;
    if (!((x1 || x2) && same01 && same1n)) ppm_mono(q1, r, s2, aL, aR);
    L = aRprev;
    R = aL;
    aRprev = aR;
    q1 = q2;
    q2 = qn;
    dl = dq;
    dq = dn;
    s2 = s;
    f1 = f2;
    code = cn | ((int)same1n << 2) | ((int)x2 << 3);
  }
};

// ------------------------------------------------------------------------------------------
// The same reconstructions with a warp's lanes along the line: a lane holds face m (between points
// m - 1 and m), the lane before it face m - 1, and what a walk would carry from face to face comes
// from the lanes before, across a pass of 8 faces from the previous pass's values. step() takes the
// points m .. m + LA (PC: m - 1 and m), prev[NP] with this lane's values of the previous pass
// (replaced by those of this pass) and returns the interface's states. The values are those of Rec
// bit for bit. Every lane of the warp calls it. One pass of 8 points ahead of the first face fills
// prev (its own prev may hold anything).
// ------------------------------------------------------------------------------------------
struct LaneWalk {
  int k;           // this lane's place in its row of 8
  int src1, src2;  // the lanes that hold places k - 1 and k - 2 (mod 8)
  __device__ __forceinline__ double up1(double cur, double prev) const {
    return __shfl_sync(0xffffffffu, k == 7 ? prev : cur, src1);
  }
  __device__ __forceinline__ double up2(double cur, double prev) const {
    return __shfl_sync(0xffffffffu, k >= 6 ? prev : cur, src2);
  }
  __device__ __forceinline__ int up1(int cur, int prev) const {
    return __shfl_sync(0xffffffffu, k == 7 ? prev : cur, src1);
  }
};
template <int R> struct LaneRec;
template <> struct LaneRec<REC_PC> {
  static constexpr int NP = 0, FIRST = -1, NQ = 2, NB = 0;
  __device__ __forceinline__ static void step(const LaneWalk&, const double* q, double*, int&, double& L, double& R) {
    L = q[0];
    R = q[1];
  }
};
template <int RC> struct LanePLM {
  static constexpr int NP = 2, FIRST = 0, NQ = 2, NB = 0;
  __device__ __forceinline__ static void step(const LaneWalk& w, const double* q, double* prev, int&, double& L,
                                              double& R) {
    const double dr = q[1] - q[0];
    const double dl = w.up1(dr, prev[0]);
    const double h = RC == REC_PLM_MC ? half_slope_mc(dl, dr) : half_slope_minmod(dl, dr);
    const double aR = q[0] + h;
    L = w.up1(aR, prev[1]);
    R = q[0] - h;
    prev[0] = dr;
    prev[1] = aR;
  }
};
template <> struct LaneRec<REC_PLM_MC> : LanePLM<REC_PLM_MC> {};
template <> struct LaneRec<REC_PLM_MINMOD> : LanePLM<REC_PLM_MINMOD> {};
template <> struct LaneRec<REC_PPM> {
  static constexpr int NP = 4, FIRST = 0, NQ = 3, NB = 0;
  __device__ __forceinline__ static void step(const LaneWalk& w, const double* q, double* prev, int&, double& L,
                                              double& R) {
    const double dn = q[2] - q[1];
    const double dq = w.up1(dn, prev[0]), dl = w.up2(dn, prev[0]);
    double r, s;
    ppm_split(dl, dq, dn, r, s);
    const double f2 = q[0] + r;
    const double s2 = w.up1(s, prev[1]);
    double aL = w.up1(f2, prev[2]), aR = f2;
    ppm_mono(q[0], r, s2, aL, aR);
    L = w.up1(aR, prev[3]);
    R = aL;
    prev[0] = dn;
    prev[1] = s;
    prev[2] = f2;
    prev[3] = aR;
  }
};
template <> struct LaneRec<REC_PPM_EP> {
  static constexpr int NP = 4, FIRST = 0, NQ = 3, NB = 4;
  __device__ __forceinline__ static void step(const LaneWalk& w, const double* q, double* prev, int& code, double& L,
                                              double& R) {
    const double dn = q[2] - q[1];
    const double dq = w.up1(dn, prev[0]), dl = w.up2(dn, prev[0]);
    const int c1 = cmp_code(dq, dl), cn = cmp_code(dn, dq);  // curvatures of points m, m + 1
    const bool x2 = ext_code(sgn_code(dl), sgn_code(dq), sgn_code(dn)), same1n = same_code(c1, cn);
    int p;
    double r, s;
    const double f2 = ppm_ep_face<true>(q[0], q[1], dl, dq, dn, x2 && same1n, p, r, s);
    const double s2 = w.up1(s, prev[1]);
    double aL = w.up1(f2, prev[2]), aR = f2;
    const int mine = (int)same1n | ((int)x2 << 1), before = w.up1(mine, code);
    const bool same01 = before & 1, x1 = before & 2;
    if (!((x1 || x2) && same01 && same1n)) ppm_mono(q[0], r, s2, aL, aR);
    L = w.up1(aR, prev[3]);
    R = aL;
    prev[0] = dn;
    prev[1] = s;
    prev[2] = f2;
    prev[3] = aR;
    code = mine;
  }
};

// ------------------------------------------------------------------------------------------
// Riemann problem on one face, in the face frame (n, t1, t2).
// W = {rho, u_n, u_t1, u_t2, p, b_t1, b_t2}; bn = stored face field.
// ------------------------------------------------------------------------------------------
template <class T> struct FaceStateT {
  T rho, u, v, w, p, by, bz;
};
using FaceState = FaceStateT<double>;

template <class T> struct PhysFluxT {
  T U[5], F[5];
  T pt, e, cf2, b2;  // cf2: the square of the fast magnetosonic speed along the normal
  T A;               // 2 rho cf2
};
using PhysFlux = PhysFluxT<double>;

// a + b with no product fused into it: the larger-speed decision (fast_left) compares the two sides,
// and equal states have to tie however the code around them is compiled
__device__ __forceinline__ double add_rn(double a, double b) { return __dadd_rn(a, b); }
// a b that is not fused into a sum it enters
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ Dual add_rn(Dual a, Dual b) { return Dual(__dadd_rn(a.v, b.v), a.t + b.t); }

// Total pressure and the fast magnetosonic speed of Eq. (waves:fast-speed) along the normal, as
// A = 2 rho c_f^2 = P + b^2 + sqrt((P + b^2)^2 - 4 P b_n^2) with P = gamma p: neither the
// discriminant nor A needs 1/rho.
template <class T>
__device__ __forceinline__ void phys_speed_a(const FaceStateT<T>& s, T bn2, double gam, PhysFluxT<T>& o) {
  const T b2 = fma(s.by, s.by, fma(s.bz, s.bz, bn2));
  o.b2 = b2;
  o.pt = s.p + halve(b2);
  const T P = gam * s.p;
  const T Sp = add_rn(P, b2);
  T disc = fma(Sp, Sp, -(times4(bn2) * P));  // 4 bn^2 exactly, on the integer pipe
  disc = pmax(disc, T(0.0));
  o.A = Sp + sqrt_(disc);
}
// the same with the square of the speed itself
template <class T>
__device__ __forceinline__ void phys_speed(const FaceStateT<T>& s, T bn, double gam, PhysFluxT<T>& o) {
  phys_speed_a(s, bn * bn, gam, o);
  o.cf2 = halve(rcp(s.rho)) * o.A;
}
// Which side has the larger fast speed, decided on A_L rho_R against A_R rho_L (no quotient); plain
// tells whether both products and x = A rho / 2 of that side are positive normal numbers.
template <class T>
__device__ __forceinline__ bool fast_left(const FaceStateT<T>& sl, const FaceStateT<T>& sr, const PhysFluxT<T>& L,
                                          const PhysFluxT<T>& R, T& ah, T& x, bool& plain) {
  const double tl = val(L.A) * val(sr.rho), tr = val(R.A) * val(sl.rho);
  const bool left = dbits(tl) >= dbits(tr);
  ah = halve(left ? L.A : R.A);
  x = ah * (left ? sl.rho : sr.rho);
  const unsigned a = (unsigned)__double2hiint(tl) - 0x00100000u, b = (unsigned)__double2hiint(tr) - 0x00100000u,
                 c = (unsigned)__double2hiint(val(x)) - 0x00100000u;
  plain = max(max(a, b), c) < 0x7fe00000u;
  return left;
}
// The same for states whose products under- or overflow, a density or pressure below zero, infinities
// and NaN (not inlined: see the reciprocals): the larger of the quotients A / (2 rho), which for a
// negative density loses against the other side's.
template <class T>
__device__ __noinline__ T fast_max_any(T rl, T rr, T Al, T Ar, bool& left) {
  const T cl = halve(rcp(rl)) * Al, cr = halve(rcp(rr)) * Ar;
  left = dbits(val(cl)) >= dbits(val(cr));
  return sqrt_(left ? cl : cr);
}
// The larger of the two fast speeds, sqrt(A / (2 rho)) of that side = (A/2) / sqrt(rho A/2): one
// reciprocal square root in the place of two reciprocals and a square root (7 FP64 instructions
// against 9; 9 against 14 with the hardware's FP64 seeds).
template <class T>
__device__ __forceinline__ T fast_max(const FaceStateT<T>& sl, const FaceStateT<T>& sr, const PhysFluxT<T>& L,
                                      const PhysFluxT<T>& R) {
  bool plain;
  T ah, x;
  bool left = fast_left(sl, sr, L, R, ah, x, plain);
  if (!plain) return fast_max_any(sl.rho, sr.rho, L.A, R.A, left);
  return vabs(ah) * rsqrt_(x);
}

// Conserved vector and ideal-MHD flux of Eq. (mhd:conservation-laws) in the face frame, with e_tot
// in the energy flux (needs b2 and pt from phys_speed).
template <class T>
__device__ __forceinline__ void phys_flux(const FaceStateT<T>& s, T bn, double gm1inv, PhysFluxT<T>& o) {
  const T bn2 = bn * bn;
  const T u2 = fma(s.u, s.u, fma(s.v, s.v, s.w * s.w));
  const T e = fma(s.p, gm1inv, halve(fma(s.rho, u2, o.b2)));
  const T ub = fma(s.u, bn, fma(s.v, s.by, s.w * s.bz));
  const T mu = s.rho * s.u;
  o.U[0] = s.rho;
  o.U[1] = mu;
  o.U[2] = s.rho * s.v;
  o.U[3] = s.rho * s.w;
  o.U[4] = e;
  o.F[0] = mu;
  o.F[1] = fma(mu, s.u, o.pt - bn2);
  o.F[2] = fma(mu, s.v, -bn * s.by);
  o.F[3] = fma(mu, s.w, -bn * s.bz);
  o.F[4] = fma(e + o.pt, s.u, -ub * bn);
  o.e = e;
}

// HLL-type two-state flux; inv = 1 / (ap + am), or 0 when ap + am = 0 (then the left flux).
template <class T>
__device__ __forceinline__ void two_state(const PhysFluxT<T>& L, const PhysFluxT<T>& R, T ap,
                                          T am, T inv, bool zero, T* F) {
  if (zero) {
    for (int v = 0; v < 5; ++v) F[v] = L.F[v];
    return;
  }
  const T wl = ap * inv, wr = am * inv, wd = ap * am * inv;
  for (int v = 0; v < 5; ++v) F[v] = fma(wl, L.F[v], fma(wr, R.F[v], -wd * (R.U[v] - L.U[v])));
}

// Star state on one side of the contact (MK05 Eqs. 43-48), its energy apart.
template <class T> struct StarT {
  T rs, vs, ws, bys, bzs;
};
__device__ __forceinline__ int expo(double x) { return (int)((unsigned long long)dbits(x) >> 52) & 0x7ff; }
// whether the tangential state changes across the fast wave: |dd| > 1e-12 (m su + bn2), with
// dd = m ssm - bn2. Settled on exponents for all but nearly degenerate states (m su + bn2 is below
// 2^(1 + max(e_m + e_su + 2, e_bn2 + 1)), 1e-12 below 2^-39), without the FP64 instructions.
static __device__ __noinline__ bool star_regular_any(double dd, double m, double su, double bn2) {
  return vgt(vabs(dd), 1e-12 * fma(m, su, bn2));
}
__device__ __forceinline__ bool star_regular(double dd, double m, double su, double bn2) {
  const int top = max(expo(m) + expo(su) - 1023 + 2, expo(bn2) + 1);
  if (expo(dd) >= top - 38) return true;
  return star_regular_any(dd, m, su, bn2);
}
// m = rho su is the mass flux through the outer wave S, su = S - u, d = S_M - u, ssm = S - S_M;
// ssminv receives 1 / ssm
template <class T>
__device__ __forceinline__ void star_state(const FaceStateT<T>& q, T m, T su, T d, T ssm, T bn, T bn2, T& ssminv,
                                           StarT<T>& o) {
  ssminv = rcp(ssm);
  o.rs = m * ssminv;
  const T dd = fma(m, ssm, -bn2);
  if (!star_regular(val(dd), val(m), val(su), val(bn2))) {  // no tangential change across the fast wave
    o.vs = q.v;
    o.ws = q.w;
    o.bys = q.by;
    o.bzs = q.bz;
  } else {
    const T ddinv = rcp(dd);
    const T cv = bn * d * ddinv;
    const T cb = fma(m, su, -bn2) * ddinv;
    o.vs = fma(-q.by, cv, q.v);
    o.ws = fma(-q.bz, cv, q.w);
    o.bys = q.by * cb;
    o.bzs = q.bz * cb;
  }
}

// Whether the face (x/t = 0) lies inside the rotational wave S*_side = S_M -/+ |b_n| / sqrt(rho*)
// (MK05 Eq. 51) on the side `left` of the contact (S_M >= 0 on the left): S*_left < 0 and
// S*_right >= 0 compared as (rho* S_M) S_M against b_n^2, without the square root (both sides are
// non-negative, so the bit patterns order them). The reverse sweep takes the same decision.
template <class T>
__device__ __forceinline__ bool hlld_in_rotational(bool left, T SM, T rs, T bn2) {
  const double sm = val(SM);
  const long long q = dbits(val(rs) * sm * sm), b = dbits(val(bn2));
  return left ? q < b : q <= b;
}

template <class T>
__device__ __forceinline__ FaceStateT<T> pick(bool left, const FaceStateT<T>& a, const FaceStateT<T>& b) {
  FaceStateT<T> r;
  r.rho = left ? a.rho : b.rho;
  r.u = left ? a.u : b.u;
  r.v = left ? a.v : b.v;
  r.w = left ? a.w : b.w;
  r.p = left ? a.p : b.p;
  r.by = left ? a.by : b.by;
  r.bz = left ? a.bz : b.bz;
  return r;
}

// Miyoshi & Kusano (2005) HLLD without the Minoshima fixes. Outside the fan (S_L > 0 or S_R < 0)
// the flux is that side's physical flux; inside it the face x/t = 0 lies on the side of the
// contact given by sgn(S_M), and only that side's star state is formed, and the other side's star
// state and the double-star state (MK05 Eqs. 49-63) only when the face lies inside that side's
// rotational wave.
// The Rankine-Hugoniot relations behind the star states make every one of their fluxes
// (F + S (U* - U), and F* + S* (U** - U*)) the physical flux of the state at x/t = 0, with S_M for
// its normal velocity and p_t* for its total pressure. So the branches only form that state
// (density, tangential velocity and field, energy, u . b), and one flux is formed at the end by all
// lanes of a warp together: in the fan 90 FP64 instructions a face (speeds and flux, counted on the
// formulas), in the double-star region 132; 105 and 154 with reciprocals of 3 instructions and roots of
// 5, against 143 and 218 when the flux vectors were differenced across the waves (with fast_max and
// sqrt_ the 256^3 turbulence step took 46.9 ms against 49.4, the 128^3 Alfven step 8.43 against 9.64,
// 96 subsonic patches 19.9 against 22.8). MK05 Eqs. 38 and 41 are taken relative to the side's own
// velocity: d = S_M - u = (m_o (u_R - u_L) + p_L - p_R) / (m_R - m_L) with the other side's mass flux
// m_o, and p_t* = p_t + m d.
// A component of the double-star state differs from the star state a of its side by
// x = (sqrt(rho_b*) (v_b - v_a) + s (B_b - B_a)) / (sqrt(rho_a*) + sqrt(rho_b*)) in the velocity and
// by s sqrt(rho_a*) x in the field (MK05 Eqs. 59-62, b the other side's star state, s = sgn(b_n)
// on the left and -sgn(b_n) on the right).
template <class T>
__device__ __forceinline__ void hlld(const FaceStateT<T>& sl, const FaceStateT<T>& sr, T bn, T bn2, double gm1inv,
                                     const PhysFluxT<T>& L, const PhysFluxT<T>& R, T SL, T SR, T* F) {
  const bool supL = gt0(SL);
  const bool fan = !supL && !lt0(SR);
  T suL = 0.0, suR = 0.0, mL = 0.0, mR = 0.0, du = 0.0, dpt = 0.0, nL = 0.0, dinv = 0.0, SM = 0.0;
  if (fan) {
    suL = SL - sl.u;
    suR = SR - sr.u;
    mL = suL * sl.rho;  // mass fluxes through the outer waves
    mR = suR * sr.rho;
    dinv = rcp(mR - mL);
    du = sr.u - sl.u;
    dpt = L.pt - R.pt;
    nL = fma(mR, du, dpt);
    SM = fma(nL, dinv, sl.u);
  }
  const bool left = fan ? ge0(SM) : supL;
  const FaceStateT<T> q = pick(left, sl, sr);
  const T b2 = left ? L.b2 : R.b2;
  T pt = left ? L.pt : R.pt;
  // the state at x/t = 0: outside the fan the side's own
  T rho = q.rho, un = q.u, v = q.v, w = q.w, by = q.by, bz = q.bz;
  T e = fma(q.p, gm1inv, halve(fma(q.rho, fma(q.u, q.u, fma(q.v, q.v, q.w * q.w)), b2)));
  T ub = fma(q.u, bn, fma(q.v, q.by, q.w * q.bz));
  if (fan) {
    const T su = left ? suL : suR, m = left ? mL : mR;
    const T nS = left ? nL : fma(mL, du, dpt);
    const T d = nS * dinv;  // S_M - u of the side
    const T ptS = fma(m, d, pt);
    const T ssm = su - d;
    T ssminv;
    StarT<T> a;
    star_state(q, m, su, d, ssm, bn, bn2, ssminv, a);
    const T vbs = fma(SM, bn, fma(a.vs, a.bys, a.ws * a.bzs));
    const T es = fma(bn, ub - vbs, fma(ptS, SM, fma(su, e, -(pt * q.u)))) * ssminv;
    rho = a.rs;
    un = SM;
    pt = ptS;
    v = a.vs;
    w = a.ws;
    by = a.bys;
    bz = a.bzs;
    e = es;
    ub = vbs;
    if (hlld_in_rotational(left, SM, a.rs, bn2)) {
      // the other side's star state (its density, tangential velocity and field)
      const FaceStateT<T> qo = pick(!left, sl, sr);
      const T suo = left ? suR : suL, mo = left ? mR : mL;
      const T ssmo = suo - (SM - qo.u);
      T oinv;
      StarT<T> o;
      star_state(qo, mo, suo, SM - qo.u, ssmo, bn, bn2, oinv, o);
      const T sq = sqrt_(a.rs), sqo = sqrt_(o.rs);
      const T inv = rcp(sq + sqo);
      // b_n != 0 here (with b_n = 0 there is no rotational wave), so s = +-1 is a sign flip
      const bool neg = lt0(bn) == left;
      const T xv = fma(sqo, o.vs - a.vs, neg_if(neg, o.bys - a.bys)) * inv;
      const T xw = fma(sqo, o.ws - a.ws, neg_if(neg, o.bzs - a.bzs)) * inv;
      const T ssq = neg_if(neg, sq);
      v = a.vs + xv;
      w = a.ws + xw;
      by = fma(ssq, xv, a.bys);
      bz = fma(ssq, xw, a.bzs);
      ub = fma(SM, bn, fma(v, by, w * bz));
      e = fma(ssq, ub - vbs, es);
    }
  }
  const T mu = rho * un;
  F[0] = mu;
  F[1] = fma(mu, un, pt - bn2);
  F[2] = fma(mu, v, -(bn * by));
  F[3] = fma(mu, w, -(bn * bz));
  F[4] = fma(e + pt, un, -(ub * bn));
}

// Full face solve: flux of {rho, m_n, m_t1, m_t2, e}, alpha+/-, and (with_us) the Q26 face velocity.
template <int RS, class T>
__device__ __forceinline__ void riemann(const FaceStateT<T>& sl, const FaceStateT<T>& sr, T bn,
                                        double gam, double gm1inv, T* F, T& ap,
                                        T& am, T& ustar, bool with_us = true) {
  PhysFluxT<T> L, R;
  const T bn2 = bn * bn;
  T SL = 0.0, SR = 0.0;
  if (RS == RS_LLF) {
    phys_speed(sl, bn, gam, L);
    phys_speed(sr, bn, gam, R);
    const T a = pmax(vabs(sl.u) + sqrt_(L.cf2), vabs(sr.u) + sqrt_(R.cf2));
    ap = a;
    am = a;
  } else {
    phys_speed_a(sl, bn2, gam, L);
    phys_speed_a(sr, bn2, gam, R);
    // Eq. (alpha-pm) = MK05 Eq. 67 speeds
    const T cmax = fast_max(sl, sr, L, R);
    const T umax = vmax(sl.u, sr.u), umin = vmin(sl.u, sr.u);
    SR = umax + cmax;
    SL = umin - cmax;
    ap = vmax(0.0, SR);
    // max(0, -SL), a speed that is not a number kept: -SL is cmax - umin, without forming it
    am = (unsigned long long)dbits(val(SL)) <= 0x7ff0000000000000ULL ? T(0.0) : neg_if(dbits(val(SL)) < 0, SL);
  }
  if (RS == RS_HLLD) {
    hlld(sl, sr, bn, bn2, gm1inv, L, R, SL, SR, F);  // (reads L, R's pt and b2 only)
    if (!with_us) return;
  }
  const T sum = ap + am;
  const bool zero = is_zero(sum);
  const T inv = zero ? 0.0 : rcp(sum);
  if (RS != RS_HLLD) {
    phys_flux(sl, bn, gm1inv, L);
    phys_flux(sr, bn, gm1inv, R);
    two_state(L, R, ap, am, inv, zero, F);
  }
  // Eq. (q26-facevel)
  ustar = zero ? sl.u : fma(ap, sl.u, am * sr.u) * inv;
}

}  // namespace mhd
