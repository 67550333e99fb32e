// FP64 contractions in 64-bit integer arithmetic.
//
// GB300 has two FP64 lanes per SM and clock against 64 or more 32-bit integer
// multiply-add lanes, so a contraction sum_k a_k g_k whose factors are known once per row
// (a) and once per cell (g) is taken in fixed point: each factor is an integer of B bits
// times a power of two, the power shared by a row or by a cell, and the products are
// summed exactly in two 64-bit integers, then rounded once to FP64.
//
//   x = f 2^(e - B),  |x| < 2^e,  f = h 2^29 + l,  -2^28 <= l < 2^28,  |h| <= 2^(B - 29)
//   sum a g = 2^(ea + eg + 58 - 2B) [ sum ah gh + 2^-29 sum (ah gl + al gh) + ... ]
//
// (three 32 x 32 -> 64 multiply-adds per term; the dropped al gl terms are below
// 2^(56 - 2B) of the scales each). Both sums stay within 63 bits for K 4^(B - 29) < 2^63:
// B = 59 for K <= 7, B = 58 for K <= 31. Rounding the factors and dropping al gl costs at
// most K 2^-B of 2^(ea + eg) in all; FP64 multiply-adds cost K 2^-53 of the partial sums.
// The fixed point is thus the more accurate one wherever an entry's own terms are not more
// than 2^(B - 53) below the scales. The callers take a cell only where that holds for every
// entry (each by its own rule, on the factors themselves); other cells take the FP64
// multiply-adds. Factors a that are zero but for rounding are held to 2^-B of their row.
#pragma once

#include <cuda_runtime.h>

namespace ffc {

// |x| < 2^fix_exponent(x) for finite x; 1025 for infinities and NaN
__device__ __forceinline__ int fix_exponent(double x) {
  return int((unsigned(__double2hiint(x)) >> 20) & 0x7ffu) - 1022;
}

__device__ __forceinline__ bool fix_nonzero(double x) {
  return ((unsigned(__double2hiint(x)) << 1) | unsigned(__double2loint(x))) != 0u;
}

// the exponent of a nonzero x, or `zero`
__device__ __forceinline__ int fix_exponent_or(double x, int zero) { return fix_nonzero(x) ? fix_exponent(x) : zero; }

// Smallest exponent of a reference-tensor row: a row of zeros takes it, so that with cell
// exponents from -900 up the constants of the conversions below keep normal exponents.
constexpr int FIX_ROW_MIN = -100;
// Smallest cell exponent with narrow and with wide factors: a wide sum can be as small as 2^-121
// of its scales, and the exponent field of the conversion below must not pass zero there.
constexpr int FIX_CELL_MIN = -900, FIX_CELL_MIN_WIDE = -700;

// x 2^(B - e) rounded to the nearest integer (halves away from zero), |x| < 2^e, 52 <= B <= 59
template <int B>
__device__ __forceinline__ long long fix_round(double x, int e) {
  static_assert(B >= 52 && B <= 59, "the significand is shifted left by B - 52, then right");
  const int hw = __double2hiint(x);
  const int ex = int((unsigned(hw) >> 20) & 0x7ffu);
  const unsigned mh = (unsigned(hw) & 0xfffffu) | (ex ? 1u << 20 : 0u);
  const unsigned long long m = (static_cast<unsigned long long>(mh) << 32 | unsigned(__double2loint(x))) << (B - 52);
  const int sh = e + 1022 - (ex ? ex : 1);  // >= 0
  const long long f = static_cast<long long>(((m >> (sh < 63 ? sh : 63)) + 1) >> 1);
  const long long s = hw >> 31;
  return (f ^ s) - s;
}

// The two parts (h, l) of a fixed-point factor. The empty asm hides that they came from a
// 64-bit value: otherwise the compiler keeps the sign-extended value across a loop and
// multiplies 64 x 64 bits (four multiply-adds for one).
__device__ __forceinline__ int2 fix_split(long long f) {
  const long long h64 = (f + (1ll << 28)) >> 29;
  int h = int(h64), l = int(f - (h64 << 29));
  asm("" : "+r"(h), "+r"(l));
  return make_int2(h, l);
}
template <int B>
__device__ __forceinline__ int2 fix_parts(double x, int e) {
  return fix_split(fix_round<B>(x, e));
}

// The same with 29 bits more, for factors g that differ by many orders of magnitude within one
// cell: x = (h 2^58 + m 2^29 + l) 2^(e - B - 29) cut towards zero.
template <int B>
__device__ __forceinline__ int4 fix_parts_wide(double x, int e) {
  constexpr unsigned MASK = (1u << 29) - 1u;
  const int hw = __double2hiint(x);
  const int ex = int((unsigned(hw) >> 20) & 0x7ffu);
  const unsigned mh = (unsigned(hw) & 0xfffffu) | (ex ? 1u << 20 : 0u);
  const unsigned long long m = (static_cast<unsigned long long>(mh) << 32 | unsigned(__double2loint(x))) << (B - 53);
  const int sh = e + 1022 - (ex ? ex : 1);  // >= 0
  const long long s = hw >> 31;
  const long long f = static_cast<long long>(m >> (sh < 63 ? sh : 63));
  const int low = int(unsigned(sh <= 29 ? m << (29 - sh) : m >> (sh < 92 ? sh - 29 : 63)) & MASK);
  const int2 p = fix_split((f ^ s) - s);
  int l = (low ^ int(s)) - int(s);
  asm("" : "+r"(l));
  return make_int4(p.x, p.y, l, 0);
}

// The partial sums of a contraction, the middle one in two chains (a chain's latency, not
// the multipliers, would bound a thread otherwise); `mid` starts at half a unit of the
// final shift.
struct FixAcc {
  long long hi = 0, mid = 1ll << 28, mid2 = 0;
  __device__ __forceinline__ void add(int2 a, int2 g) {
    hi += static_cast<long long>(a.x) * g.x;
    mid += static_cast<long long>(a.x) * g.y;
    mid2 += static_cast<long long>(a.y) * g.x;
  }
  __device__ __forceinline__ long long sum() const { return hi + ((mid + mid2) >> 29); }
};

// The partial sums with wide factors g, in units 2^58, 2^29 and 1 of the last: five multiply-adds
// per term, and the dropped al gl below 2^-89 of the scales. Up to 10 terms for B = 58, also of
// factors g that are sums of two with half the magnitude.
struct FixAccWide {
  long long hi = 0, mid = 0, lo = 0;
  __device__ __forceinline__ void add(int2 a, int4 g) {
    hi += static_cast<long long>(a.x) * g.x;
    mid += static_cast<long long>(a.x) * g.y;
    mid += static_cast<long long>(a.y) * g.x;
    lo += static_cast<long long>(a.x) * g.z;
    lo += static_cast<long long>(a.y) * g.y;
  }
};

// A magnitude of three words (w2 the highest, zero only for zero) rounded to a double: normalised
// to a leading one at bit 31 of w2 and cut to 53 bits, and the next bit (halves away from zero)
// and the exponent field `expo`, one less than that of bit 31, are added: the leading one
// completes the field, and so does a carry of the rounding.
__device__ __forceinline__ double fix_pack(unsigned w2, unsigned w1, unsigned w0, unsigned sign, int expo) {
  const unsigned sh = unsigned(__clz(int(w2)));  // 32 only for zero
  const unsigned nh = __funnelshift_l(w1, w2, sh), nl = __funnelshift_l(w0, w1, sh);
  const unsigned up = (nl >> 10) & 1u;
  const unsigned lo = __funnelshift_r(nl, nh, 11) + up;
  unsigned hi = (nh >> 11) + (lo < up ? 1u : 0u) + (unsigned(expo) - (sh << 20));
  if (w2 == 0) hi = 0;  // then lo is 0 too
  return __hiloint2double(int(hi | sign), int(lo));
}

// v 2^ulog rounded to the nearest double, |v| < 2^63, for results with normal exponents;
// `e20` is ulog << 20. Two forms, which a kernel can mix so that two pipes share the work.
// This one is on the integer pipes.
__device__ __forceinline__ double fix_to_double(long long v, int e20) {
  const long long s = v >> 63;
  const unsigned long long m = static_cast<unsigned long long>((v ^ s) - s);
  unsigned mh = unsigned(m >> 32), ml = unsigned(m);
  int expo = e20 + (1085 << 20);
  if (mh == 0) {
    mh = ml;
    ml = 0;
    expo -= 32 << 20;
  }
  return fix_pack(mh, ml, 0u, unsigned(s >> 32) & 0x80000000u, expo);
}

// The same for wide sums, `e20` for the unit of `hi`. A negative sum's magnitude is taken as its
// one's complement, less by 2^-58 units.
__device__ __forceinline__ double fix_to_double(const FixAccWide& a, int e20) {
  constexpr long long MASK = (1ll << 29) - 1;
  const long long mid = a.mid + (a.lo >> 29);
  const long long v = a.hi + (mid >> 29), s = v >> 63;
  const unsigned long long m = static_cast<unsigned long long>(v ^ s);
  const unsigned long long f = static_cast<unsigned long long>(((mid & MASK) << 29 | (a.lo & MASK)) ^ s) << 6;
  unsigned w2 = unsigned(m >> 32), w1 = unsigned(m), w0 = unsigned(f >> 32);
  int expo = e20 + (1085 << 20);
  if (m == 0) {
    w2 = w0;
    w1 = unsigned(f);
    w0 = 0;
    expo -= 64 << 20;
  }
  if (w2 == 0) {
    w2 = w1;
    w1 = w0;
    w0 = m == 0 ? 0u : unsigned(f);
    expo -= 32 << 20;
  }
  return fix_pack(w2, w1, w0, unsigned(s >> 32) & 0x80000000u, expo);
}

// On the FP64 pipe: the top 52 bits and the low 12 are placed in the significands of two
// doubles of fixed exponent (T = 1.5 2^52 u + top u with u = 2^(ulog + 12), and L = 2^52
// 2^ulog + low 2^ulog), so T - (1.5 2^52 + 2^40) u = top u - 2^52 2^ulog is exact and
// adding L rounds once: two FP64 additions and no normalisation.
__device__ __forceinline__ double fix_to_double_fp64(long long v, int e20) {
  const long long top = v >> 12;
  const int base = e20 + (1087 << 20);
  const double T = __hiloint2double(int(top >> 32) + base + 0x80000, int(top));
  const double c = __hiloint2double(base + 0x80100, 0);
  const double L = __hiloint2double(e20 + (1075 << 20), int(v) & 0xfff);
  return (T - c) + L;
}

}  // namespace ffc
