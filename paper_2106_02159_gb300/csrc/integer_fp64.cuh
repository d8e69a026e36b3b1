// FP64 additions, divisions and square roots on the integer units, with IEEE 754's
// results (rounded to nearest even) for every operand.
//
// GB300 issues an FP64 warp instruction per 19 cycles and SM (per 63 cycles and
// warp); a division takes 7.4 and a square root 7.5 of them. The row kernels are
// held by that pipe while the integer units, 38 times as fast, idle. A step of the
// 998k-vertex cylinder took 5.11 ms with all of it on the FP64 pipe, 4.50 with the
// additions of k_visc, k_alpha, k_low and k_lim1 here, 4.21 with the divisions and
// roots of k_prep, k_visc, k_alpha, k_low and the line searches too (375k in 3D 7.93,
// 7.48, 6.91; 62k 0.823 and, with the divisions, 0.755).
#pragma once
#include <cuda_runtime.h>

namespace eh {

__device__ __forceinline__ unsigned hi_word(double x) { return (unsigned)__double2hiint(x); }
__device__ __forceinline__ unsigned lo_word(double x) { return (unsigned)__double2loint(x); }
// a + b on the FP64 pipe, for a rarely taken branch: a call, which the compiler
// neither evaluates ahead of the branch nor turns into a predicated instruction
// (that would occupy the pipe whether its predicate holds or not)
static __device__ __noinline__ double add_fp64_cold(double a, double b) { return __dadd_rn(a, b); }
// a + b rounded to nearest even on the integer units: IEEE addition for every
// pair of doubles (the larger magnitude's exponent field within [70, 2045];
// others, infinities and NaN go to the FP64 pipe). The larger significand is held
// with 10 guard bits, the smaller shifted to it with a sticky bit, the sum
// renormalised and rounded. ~60 integer instructions, 30 cycles of an SM per
// warp, against 19 on the FP64 pipe -- but on units that the row kernels leave
// idle: 8 of these beside 16 FP64 FMAs take 335 cycles, 8 FP64 additions beside
// them 461. (Compared with the FP64 pipe on 2.5e9 pairs: exponents apart by
// 0 to 140, cancellation, ties, zeros, subnormals.)
// On the operands' words: a sign flipped or cleared on a double would become an
// FP64 instruction again.
__device__ __forceinline__ double add_words(unsigned ah, unsigned al, unsigned bh, unsigned bl) {
  unsigned xa = ah & 0x7fffffffu, xb = bh & 0x7fffffffu;
  const bool swap = xa < xb || (xa == xb && al < bl);
  {
    unsigned t = ah;
    ah = swap ? bh : ah;
    bh = swap ? t : bh;
    t = al;
    al = swap ? bl : al;
    bl = swap ? t : bl;
    t = xa;
    xa = swap ? xb : xa;
    xb = swap ? t : xb;
  }
  const unsigned ea = xa >> 20, eb = xb >> 20;
  if (ea - 70u > 1975u) {
    return add_fp64_cold(__hiloint2double((int)ah, (int)al), __hiloint2double((int)bh, (int)bl));
  }
  const unsigned d = min(ea - eb, 63u);
  const unsigned mah = (ah & 0xfffffu) | 0x100000u, mbh = (bh & 0xfffffu) | (min(eb, 1u) << 20);
  const unsigned long long ma = ((unsigned long long)mah << 32 | al) << 10, mb = ((unsigned long long)mbh << 32 | bl) << 10;
  const unsigned long long sh = mb >> d;
  const unsigned long long x = sh | (unsigned)((sh << d) != mb);  // sticky
  const unsigned long long sx = (unsigned long long)(long long)((int)(ah ^ bh) >> 31);
  const unsigned long long R = ma + ((x ^ sx) - sx);
  const int lz = __clzll((long long)R);
  const unsigned long long N = R << (lz & 63), m = N >> 11;
  const unsigned up = ((unsigned)N & 0x7ffu) + ((unsigned)m & 1u) > 0x400u;
  const unsigned long long r = ((unsigned long long)(ea - (unsigned)lz) << 52) + m + up;
  const unsigned hi = (unsigned)(r >> 32) | (ah & 0x80000000u);
  return R == 0 ? 0.0 : __hiloint2double((int)hi, (int)(unsigned)r);
}
__device__ __forceinline__ double add_alu(double a, double b) {
  return add_words(hi_word(a), lo_word(a), hi_word(b), lo_word(b));
}
__device__ __forceinline__ double sub_alu(double a, double b) {
  return add_words(hi_word(a), lo_word(a), hi_word(b) ^ 0x80000000u, lo_word(b));
}
__device__ __forceinline__ double add_abs_alu(double a, double b) {  // |a| + |b|
  return add_words(hi_word(a) & 0x7fffffffu, lo_word(a), hi_word(b) & 0x7fffffffu, lo_word(b));
}
static __device__ __noinline__ double div_fp64_cold(double a, double b) { return __ddiv_rn(a, b); }
static __device__ __noinline__ double sqrt_fp64_cold(double a) { return __dsqrt_rn(a); }
// a / b rounded to nearest even on the integer units, for every pair of doubles
// (subnormal, zero, infinite or NaN operands and quotients near the range's ends go
// to the FP64 pipe): a long division of the significands with digits of 18, 18 and
// 17 bits. With D in [1, 2), the FP32 reciprocal of D's leading 24 bits is above 1/D
// by less than 2^-23 through the bits left out and by at most 2^-24 (1 ulp) through
// its own error; lessened by 2^-22 it never exceeds 1/D, so each digit is at most the
// true one, and short of it by less than 1.2: the remainder stays in [0, 1.2 D) and
// fits 64 bits, and one comparison completes the 54-bit quotient, whose last bit
// rounds (a quotient of doubles is never halfway between two). ~65 integer
// instructions, against 7.4 slots of 19 cycles on the FP64 pipe. (Compared with the FP64 division on 3e8
// pairs on the CPU, the reciprocal off by up to one ulp either way, and 1.2e9 on
// the GPU; the square root likewise.)
__device__ __forceinline__ double div_alu(double a, double b) {
  const unsigned ah = hi_word(a), al = lo_word(a), bh = hi_word(b), bl = lo_word(b);
  const unsigned ea = (ah >> 20) & 0x7ffu, eb = (bh >> 20) & 0x7ffu, e0 = ea - eb + 1023u;
  if (ea - 1u >= 2046u || eb - 1u >= 2046u || e0 - 2u >= 2045u) return div_fp64_cold(a, b);
  const unsigned long long N = (unsigned long long)((ah & 0xfffffu) | 0x100000u) << 32 | al;
  const unsigned long long D = (unsigned long long)((bh & 0xfffffu) | 0x100000u) << 32 | bl, nD = 0ull - D;
  const unsigned less = N < D;
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(__uint_as_float(0x3f800000u | ((unsigned)(D >> 29) & 0x7fffffu))));
  const unsigned R = (__float_as_uint(r) << 8) + (0x80000000u - 1024u);  // units of 2^-32
  unsigned long long rem = (N << less) - D;
  const unsigned d1 = __umulhi((unsigned)(rem >> 22), R) >> 12;
  rem = (rem << 18) + d1 * nD;
  const unsigned d2 = __umulhi((unsigned)(rem >> 22), R) >> 12;
  rem = (rem << 18) + d2 * nD;
  const unsigned d3 = __umulhi((unsigned)(rem >> 22), R) >> 13;
  rem = (rem << 17) + d3 * nD;
  const unsigned long long q = (1ull << 53) + ((unsigned long long)d1 << 35) + ((unsigned long long)d2 << 17) + d3 +
                               (rem >= D ? 1u : 0u);
  const unsigned long long x = ((unsigned long long)(e0 - less - 1u) << 52) + ((q + 1) >> 1);
  return __hiloint2double((int)((unsigned)(x >> 32) | ((ah ^ bh) & 0x80000000u)), (int)(unsigned)x);
}
// sqrt(a) rounded to nearest even in the same way (negative, subnormal, zero,
// infinite or NaN a: the FP64 pipe): digits of 19, 18 and 17 bits from an FP32
// reciprocal root lessened by 2^-22, each short by less than 2.2; the remainder
// a - s^2 is kept exactly.
__device__ __forceinline__ double sqrt_alu(double a) {
  const unsigned ah = hi_word(a), al = lo_word(a), ea = ah >> 20;
  if (ea - 1u >= 2046u) return sqrt_fp64_cold(a);
  const unsigned odd = (ea & 1u) ^ 1u;
  const unsigned long long X = ((unsigned long long)((ah & 0xfffffu) | 0x100000u) << 32 | al) << odd;  // [1, 4) 2^52
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;"
      : "=f"(r)
      : "f"(__uint_as_float(((127u + odd) << 23) | ((ah & 0xfffffu) << 3) | (al >> 29))));
  const unsigned Y = (__float_as_uint(r) << 8) + (0x80000000u - 1024u);  // units of 2^-32
  const unsigned s1 = __umulhi((unsigned)(X >> 22), Y) >> 12;
  unsigned long long rem = X - ((unsigned long long)s1 * s1 << 16);
  const unsigned d2 = __umulhi((unsigned)(rem >> 5), Y) >> 12;
  const unsigned long long s2 = ((unsigned long long)s1 << 18) + d2;
  rem = (rem << 20) - d2 * (((unsigned long long)s1 << 19) + d2);
  const unsigned d3 = __umulhi((unsigned)(rem >> 8), Y) >> 12;
  unsigned long long s3 = (s2 << 17) + d3;
  rem = (rem << 34) - d3 * ((s2 << 18) + d3);
  s3 += rem > 2 * s3 ? 1u : 0u;
  const unsigned long long x = ((unsigned long long)(((ea + 1023u - odd) >> 1) - 1u) << 52) + ((s3 + 1) >> 1);
  return __longlong_as_double((long long)x);
}
// a - b on the integer units where a and b have the same sign and exponent (their
// bit patterns' difference is then the exact result's significand: nothing is
// rounded), an FP64 subtraction otherwise: the same value always. For the
// differences of neighbouring densities, streamwise momenta and energies, which
// rarely cross a power of two: ~26 integer instructions run beside the FP64
// pipe instead of one of its 19-cycle slots (k_low 397 -> 386 us, k_lim1 419 ->
// 391 us on the 998k cylinder; 609 -> 485 and 679 -> 634 us in 3D).
__device__ __forceinline__ double sub_near(double a, double b) {
  const int ah = __double2hiint(a), bh = __double2hiint(b);
  const unsigned e = ((unsigned)ah >> 20) & 0x7ffu;
  if ((unsigned)(ah ^ bh) >> 20 != 0 || e - 65u >= 0x7ffu - 65u) {
    return add_fp64_cold(a, -b);
  }
  const long long d = __double_as_longlong(a) - __double_as_longlong(b);
  const long long sg = d >> 63;
  const unsigned long long m = (unsigned long long)((d ^ sg) - sg);
  const int sh = __clzll((long long)m) - 11;
  const unsigned long long r = ((unsigned long long)(e - 1 - sh) << 52) + (m << sh);
  const unsigned long long sign = ((unsigned long long)sg ^ (unsigned long long)__double_as_longlong(a)) & 0x8000000000000000ull;
  return m == 0 ? 0.0 : __longlong_as_double((long long)(r | sign));
}

}  // namespace eh
