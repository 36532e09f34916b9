// mt_fixed.cuh -- the flux sum of MT_MIXED, sum_j P_ij (M_j - M_i) with
// binary32 P and binary64 masses (Eq. 4), in exact integer arithmetic.
//
// The binary64 pipe takes ~19 cycles of a multiprocessor per warp instruction
// (one sixty-fourth of the binary32 rate), so the four binary64 operations per
// ordered pair and species pair hold it for ~76 cycles, while the ~30 integer
// instructions here take ~8 issue cycles of the four schedulers.
//
// Masses become 61-bit integers in units of u = 2^(E - 1083), E the largest
// biased exponent among the staged masses of the species.  A mass other than
// zero is marked if it loses bits below u or lies more than 2^16 below the
// largest: its last bit is set, and it is off by less than u.  (Small masses
// that keep every bit are common: a reaction leaves differences of larger ones,
// on their coarse grid.  Marking every mass below 2^-7 of the largest made the
// one-kernel step 3-8 % slower.)  Differences are exact, P's 24-bit significand
// times a difference is exact in 96 bits, and the products are shifted by P's
// exponent and added in 96 bits (unit 2^-29 u): one rounding, to binary64, at
// the end, where the binary64 form rounds every difference and every term.
//   A row of c terms without a marked mass: its sum is off by less than
// c 2^-29 u, its new mass M' = M + sum / 2 by half of that; its nonzero masses
// are at least 2^44 u.
//   A row with one: the marks would make the sum wrong by up to 2 sum_j P u.  In
// the first tier such a row is summed in binary64 (without one, M' is zero or at
// least 2^43 u P, P the largest of its nonzero neighbours', 2^-20 at the least
// there, and off by c 2^-73 / P of itself).  In the dense tiles the marked masses'
// rests (fix_rest) are summed beside it in binary32: of 512 terms, a chunk, within
// 2^9 2^-24 sum_j P u, so M' is off by 2^-15 u, and a row whose M' is not at least
// 2^38 u (FixAcc::keeps) is summed in binary64.  So a sum that is kept costs M' no
// more than about one rounding more.
//   Everything is summed in binary64 when E is out of range (infinities, NaNs,
// masses near the ends of binary64's range), where weights fall below e^-6.9
// (cutoffs far beyond the kernel's width) and in systems that hold a
// realisation of more than 2^20 particles (row sums that large could take P
// below 2^-30; Dev::fix): just above 2^20 particles a step takes 1.05 times as
// long at one per unit length, and 3.2 times at 200 (1.43 -> 4.59 ms).
#pragma once

#include "mt_pair.cuh"

namespace mt {

// Biased exponent of a mass for the maximum E: 0 for a zero.
__device__ __forceinline__ int fix_exponent(unsigned long long bits) {
  return (int)((bits >> 52) & 0x7ff);
}

// The E in use for a maximum exponent (all zeros: any will do), and whether
// the integer form covers it: results keep within binary64's normal range.
__device__ __forceinline__ int fix_scale(int emax) { return emax == 0 ? 1023 : emax; }
__device__ __forceinline__ bool fix_covers(int E) { return E >= 200 && E <= 2030; }

// A mass in units of 2^(E - 1083); odd if it is marked.
__device__ __forceinline__ long long to_fix(unsigned long long bits, int E) {
  const int e = fix_exponent(bits);
  const unsigned long long m =
      ((bits & ((1ULL << 52) - 1)) | ((unsigned long long)(e != 0) << 52)) << 8;
  const int sh = E - (e != 0 ? e : 1);
  unsigned long long v = m >> (sh < 63 ? sh : 63);
  if (sh > 7 && m != 0) v |= sh > 16 || (v << sh) != m ? 1 : 0;
  return (long long)bits < 0 ? -(long long)v : (long long)v;
}

// What a marked mass is off by, M / u - to_fix (between -1 and 1; binary32).
__device__ __forceinline__ float fix_rest(unsigned long long bits, int E) {
  const int e = fix_exponent(bits);
  const unsigned long long m =
      ((bits & ((1ULL << 52) - 1)) | ((unsigned long long)(e != 0) << 52)) << 8;
  const int sh = E - (e != 0 ? e : 1);
  if (sh <= 7 || m == 0) return 0.0f;
  const unsigned long long v = m >> (sh < 63 ? sh : 63);
  float f = 0.0f;  // the bits below u
  if (sh < 64)
    f = __uint2float_rn((unsigned int)(m << (64 - sh) >> 32)) * 0x1p-32f;
  else if (sh < 150)
    f = __uint2float_rn((unsigned int)(m >> 32)) * __int_as_float((159 - sh) << 23);
  if ((v & 1) == 0 && (sh > 16 || (v << sh) != m)) f -= 1.0f;
  return (long long)bits < 0 ? -f : f;
}

// 1: marked, 2: negative.
__device__ __forceinline__ int fix_flags(long long v) {
  return (int)(v & 1) | (v < 0 ? 2 : 0);
}

// P (or 2 P; in [2^-30, 2]) as a 31-bit integer and a right shift: P = p 2^-29
// after the shift.
struct FixP {
  unsigned int p;
  int s;
};
__device__ __forceinline__ FixP fix_p(float P) {
  const unsigned int u = __float_as_uint(P);
  return {((u & 0x7fffffu) | 0x800000u) << 7, 128 - (int)(u >> 23)};
}

// 96-bit sum of (difference p) >> s.
struct FixAcc {
  unsigned int a0 = 0, a1 = 0, a2 = 0;
  __device__ __forceinline__ void add(long long diff, FixP f) {
    const unsigned long long t0 = (unsigned long long)(unsigned int)diff * f.p;
    const long long t1 = (long long)(int)(diff >> 32) * (int)f.p + (long long)(t0 >> 32);
    const unsigned int x0 = (unsigned int)t0, x1 = (unsigned int)t1;
    const int x2 = (int)(t1 >> 32);
    const unsigned int y0 = __funnelshift_r(x0, x1, f.s), y1 = __funnelshift_r(x1, x2, f.s);
    const int y2 = x2 >> f.s;
    asm("add.cc.u32 %0, %0, %3;\n\taddc.cc.u32 %1, %1, %4;\n\taddc.u32 %2, %2, %5;"
        : "+r"(a0), "+r"(a1), "+r"(a2)
        : "r"(y0), "r"(y1), "r"(y2));
  }
  // Adds a binary32 sum of P times rests (fix_rest), in units of u.
  __device__ __forceinline__ void add_rest(float rest) {
    const long long r = __float2ll_rn(rest * 0x1p29f);
    const unsigned int x0 = (unsigned int)r, x1 = (unsigned int)(r >> 32);
    const unsigned int x2 = (unsigned int)(r >> 63);
    asm("add.cc.u32 %0, %0, %3;\n\taddc.cc.u32 %1, %1, %4;\n\taddc.u32 %2, %2, %5;"
        : "+r"(a0), "+r"(a1), "+r"(a2)
        : "r"(x0), "r"(x1), "r"(x2));
  }
  // Whether the sum of up to 512 terms and their rests is kept: the new mass it
  // gives, M' = mass + sum / 2^halvings, is at least 2^38 u; or both are zero,
  // which without marked or negative masses, or (one: a P times u is at least one
  // unit of the sum) without negative ones, says that every mass of the row is.
  // In units of 8 u, by integers: two binary64 instructions per chunk and species
  // made the dense step 1.4 % slower.
  __device__ __forceinline__ bool keeps(long long mass, int halvings, int flags, bool one) const {
    const long long next =
        (mass >> 3) + ((long long)((unsigned long long)a2 << 32 | a1) >> halvings);
    if (((next ^ (next >> 63)) >> 35) != 0) return true;
    return (mass | a0 | a1 | a2) == 0 && (flags == 0 || (flags == 1 && one));
  }
  // The sum in binary64 (rounded to nearest even), masses in units of
  // 2^(E - 1083).
  __device__ __forceinline__ double value(int E) const {
    unsigned int b0 = a0, b1 = a1, b2 = a2;
    const unsigned int neg = (unsigned int)((int)a2 >> 31);
    asm("add.cc.u32 %0, %3, %6;\n\taddc.cc.u32 %1, %4, 0;\n\taddc.u32 %2, %5, 0;"
        : "=r"(b0), "=r"(b1), "=r"(b2)
        : "r"(a0 ^ neg), "r"(a1 ^ neg), "r"(a2 ^ neg), "r"(neg & 1u));
    // the leading bit to the top of 96 bits
    int t = 95;
    if (b2 == 0) {
      b2 = b1;
      b1 = b0;
      b0 = 0;
      t -= 32;
    }
    if (b2 == 0) {
      b2 = b1;
      b1 = b0;
      b0 = 0;
      t -= 32;
    }
    if (b2 == 0) return 0.0;
    const int z = __clz((int)b2);
    t -= z;
    b2 = __funnelshift_l(b1, b2, z);
    b1 = __funnelshift_l(b0, b1, z);
    b0 <<= z;
    const unsigned long long top = (unsigned long long)b2 << 32 | b1 | (b0 != 0 ? 1u : 0u);
    const unsigned long long q = (top + 0x3ff + ((top >> 11) & 1)) >> 11;  // 53 bits, or a carry
    const unsigned long long carry = top > 0xfffffffffffffbffULL ? 1ULL << 53 : 0;
    const unsigned long long mant = q | carry;
    // 2^52 <= mant <= 2^53: its leading bit adds one to the exponent field
    return __longlong_as_double(
        (long long)((((unsigned long long)(t + E - 90)) << 52) + mant) |
        (long long)((unsigned long long)(neg & 1u) << 63));
  }
};

}  // namespace mt
