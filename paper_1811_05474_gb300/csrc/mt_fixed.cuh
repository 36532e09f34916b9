// mt_fixed.cuh -- the flux sum of MT_MIXED, sum_j P_ij (M_j - M_i) with
// binary32 P and binary64 masses (Eq. 4), in exact integer arithmetic.
//
// The binary64 pipe takes ~19 cycles of a multiprocessor per warp instruction
// (one sixty-fourth of the binary32 rate), so the four binary64 operations per
// ordered pair and species pair hold it for ~76 cycles, while the ~30 integer
// instructions here take ~8 issue cycles of the four schedulers.
//
// Masses become 61-bit integers in units of 2^(E - 1083), E the largest
// biased exponent among the staged masses of the species; the 53-bit
// significand of any mass of at least 2^-7 of the largest one is kept
// exactly.  A smaller mass may lose bits below that unit; its last bit is then
// set, which marks it.  Differences are exact, P's 24-bit significand times a
// difference is exact in 96 bits, and the products are shifted by P's exponent
// and added in 96 bits (unit 2^-29 of the masses'): one rounding, to binary64,
// at the end, where the binary64 form rounds every difference and every term.
// A row that holds a marked mass and no mass of at least 2^-2 of the largest
// staged one is summed in binary64 instead (its result may be as small as
// the unit lets through), and so is everything when E is out of range
// (infinities, NaNs, masses near the ends of binary64's range).  Weights below
// e^-6.9 (cutoffs far beyond the kernel's width) and realisations of more than
// 2^20 particles (row sums that large could take P below 2^-30) keep the
// binary64 form throughout (Dev::fix).
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

// A mass in units of 2^(E - 1083); odd if bits were lost.
__device__ __forceinline__ long long to_fix(unsigned long long bits, int E) {
  const int e = fix_exponent(bits);
  const unsigned long long m =
      ((bits & ((1ULL << 52) - 1)) | ((unsigned long long)(e != 0) << 52)) << 8;
  const int sh = E - (e != 0 ? e : 1);
  unsigned long long v = sh < 64 ? m >> (sh < 63 ? sh : 63) : 0;
  if (sh > 7 && m != 0) {
    const bool lost = sh >= 63 || (v << sh) != m || (v & 1);
    v = (v & ~1ULL) | (lost ? 1 : 0);
  }
  return (long long)bits < 0 ? -(long long)v : (long long)v;
}

// Magnitude bits of a fixed mass's high word, to be ORed over a row: a mass
// of at least 2^-2 of the largest has one of the bits 26 .. 28.
__device__ __forceinline__ unsigned int fix_size(long long v) {
  const int h = (int)(v >> 32);
  return (unsigned int)(h ^ (h >> 31));
}
__device__ __forceinline__ bool fix_large(unsigned int size) { return (size >> 26) != 0; }

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
