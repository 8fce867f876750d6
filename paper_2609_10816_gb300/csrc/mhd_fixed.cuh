// mhd_fixed.cuh -- the interface offsets of PPM and PPM-EP in fixed point, on the integer pipe: bit
// patterns of doubles in and out, so that a host compiler takes the file as well (the test of their
// accuracy against exact arithmetic runs without a GPU).
#pragma once
#ifndef __CUDACC__
#define __host__
#define __device__
#define __forceinline__ inline
#endif

namespace mhd {

// The interface value on the integer pipe. With d = q1 - q0 across the interface and the
// differences dl, dn on either side, the interface lies r = d/2 + (dq2_0 - dq2_1)/12 above q0 and
// s = d - r below q1. The limited slopes never exceed 4|d| in size, so everything is a fixed-point
// number in units of d's exponent: |d| is its 53-bit significand times 2^7 (in [2^59, 2^60)), the
// neighbours are shifted to the same scale (differences of the other sign to 0, and those of at
// least 2^3 |d|'s binade clamped there, where the limiter takes 4|d| whatever they are), and sums,
// minima and the division by 12 are 64-bit integer operations. r and s lie in [|d|/6, 5|d|/6] with
// d's sign, so each is normalised by a shift of 4 to 7 bits and rounded once (to nearest; the bits
// shifted out and the division leave an error below a sixteenth of that rounding unit).
// The FP64 pipe takes 64 cycles for an instruction of a warp and the integer pipe 2: per value
// reconstructed this leaves 3 FP64 instructions (the new difference, q0 + r, and the monotonicity
// correction) of 8, for about 60 more integer ones. The 256^3 bottom/top edge sweeps, which only
// reconstruct, took 1.9 ms a step against 3.2, and a face 119 FP64 instructions against 150.
// Against exact arithmetic the errors of r and s stay below 1.125 x 2^-53 of themselves (half a unit and
// a sixteenth; tests/test_fixed_point.py). FP64 instructions: 2 to 4.4.
__host__ __device__ __forceinline__ unsigned long long dmag_fixed(unsigned long long b, int right) {
  return (((b & 0x000fffffffffffffULL) | 0x0010000000000000ULL) << 10) >> right;
}
__host__ __device__ __forceinline__ unsigned long long fixed_slope2(unsigned long long n, unsigned long long d) {
  const unsigned long long m = 4 * (n < d ? n : d), s = n + d;
  return s < m ? s : m;
}
// the double nearest to x 2^(e - 1082) with the sign bit `sign`, for x in [2^55, 2^60)
__host__ __device__ __forceinline__ unsigned long long fixed_to_bits(unsigned long long x, int e,
                                                                     unsigned long long sign) {
  const unsigned hi = (unsigned)(x >> 32);
#ifdef __CUDA_ARCH__
  const int sh = 11 - __clz(hi);  // the leading bit is bit 32 + 31 - clz: to bit 52
#else
  const int sh = 11 - __builtin_clz(hi);
#endif
  return (((x + (1u << (sh - 1))) >> sh) + ((unsigned long long)(unsigned)(e - 8 + sh) << 52)) | sign;
}
// t / 12 to within 3, with 2^64 / 12 = 0x15555555_55555555
__host__ __device__ __forceinline__ long long twelfth(long long t) {
  const int th = (int)(t >> 32);
  const unsigned tl = (unsigned)t;
  return (long long)th * 0x15555555 + (long long)(((unsigned long long)tl * 0x15555555u) >> 32) +
         (((long long)th * 0x55555555) >> 32);
}
// bit patterns of r and s from those of dl, d, dn, for the exponent field of d in [128, 2039] or
// d = 0 (then both are 0)
__host__ __device__ __forceinline__ void ppm_split_bits(unsigned long long bl, unsigned long long bd,
                                                        unsigned long long bn, unsigned long long& r,
                                                        unsigned long long& s) {
  const int e = (int)(bd >> 52) & 0x7ff, el = (int)(bl >> 52) & 0x7ff, en = (int)(bn >> 52) & 0x7ff;
  int kl = e - el + 3, kn = e - en + 3;
  kl = kl < 0 ? 0 : (kl > 63 ? 63 : kl);
  kn = kn < 0 ? 0 : (kn > 63 ? 63 : kn);
  if ((long long)(bl ^ bd) < 0) kl = 63;
  if ((long long)(bn ^ bd) < 0) kn = 63;
  const unsigned long long fd = dmag_fixed(bd, 3);
  const unsigned long long d0 = fixed_slope2(dmag_fixed(bl, kl), fd), d1 = fixed_slope2(dmag_fixed(bn, kn), fd);
  const unsigned long long x = (fd >> 1) + (unsigned long long)twelfth((long long)(d0 - d1));
  const unsigned long long sign = bd & 0x8000000000000000ULL;
  const bool zero = (bd << 1) == 0;
  r = zero ? 0 : fixed_to_bits(x, e, sign);
  s = zero ? 0 : fixed_to_bits(fd - x, e, sign);
}

// The fourth-order value (7 (qa + qb) - (qc + qd)) / 12 lies r = d/2 + (dl - dn)/12 above qa, with
// d = qb - qa and the differences dl before qa and dn after qb, and s = d - r below qb. Formed on the
// integer pipe like PPM's (ppm_split_bits): the three differences are shifted to the largest one's
// exponent (its significand times 2^7), so r and s are good to 5 x 2^-59 of it before their one rounding
// (tests/test_fixed_point.py; FP64 instructions round three times at 2^-53 of d and dl - dn), and two
// FP64 instructions fewer are issued per value than with the sum formed in FP64.
__host__ __device__ __forceinline__ long long dsigned_fixed(unsigned long long b, int right) {
  const unsigned long long m = (((b & 0x000fffffffffffffULL) | 0x0010000000000000ULL) << 7) >> (right > 63 ? 63 : right);
  return (long long)b < 0 ? -(long long)m : (long long)m;
}
// the double nearest to x 2^(e - 1082), for |x| < 2^62 and e >= 128
__host__ __device__ __forceinline__ unsigned long long signed_fixed_to_bits(long long x, int e) {
  const unsigned long long m = (unsigned long long)(x < 0 ? -x : x);
  if (m == 0) return 0;
#ifdef __CUDA_ARCH__
  const int sh = 11 - __clzll((long long)m);  // the leading bit to bit 52
#else
  const int sh = 11 - __builtin_clzll(m);
#endif
  const unsigned long long q = sh > 0 ? (m + (1ULL << (sh - 1))) >> sh : m << -sh;
  return (q + ((unsigned long long)(unsigned)(e - 8 + sh) << 52)) | ((unsigned long long)x & 0x8000000000000000ULL);
}
// bit patterns of r and s from those of dl, d, dn, for the largest exponent field e of the three in
// [128, 2039]
__host__ __device__ __forceinline__ void ppm_ep_split_bits(unsigned long long bl, unsigned long long bd,
                                                           unsigned long long bn, int e, int el, int ed, int en,
                                                           unsigned long long& r, unsigned long long& s) {
  const long long fl = dsigned_fixed(bl, e - el), fd = dsigned_fixed(bd, e - ed), fn = dsigned_fixed(bn, e - en);
  const long long x = (fd >> 1) + twelfth(fl - fn);
  r = signed_fixed_to_bits(x, e);
  s = signed_fixed_to_bits(fd - x, e);
}

}  // namespace mhd
