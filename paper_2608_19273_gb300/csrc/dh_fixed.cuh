// Sums of several FP64 numbers in 64-bit fixed point on the integer pipe.
//
// GB300 issues one FP64 warp instruction per 64 clocks and SM sub-partition (2 lanes per clock
// and SM) but an integer one every other clock, and the two run beside each other (measured: 8
// DFMAs per thread take 310 ns per warp and sub-partition alone and with 128 integer operations
// beside them).  A sum of n terms is therefore formed on the integer pipe:
//   * e = the largest exponent among the terms;
//   * every term becomes a signed 64-bit integer in units of 2^(e - 1075 - SH): its 53-bit
//     significand shifted left by SH guard bits and right by its distance from e (about a dozen
//     integer instructions);
//   * the integers are added exactly (small integer weights are shifts and adds);
//   * one conversion rounds the sum to FP64 (to nearest), and its exponent takes the unit.
// A term loses only what lies below 2^-SH units in the last place of the largest term, where a
// chain of FP64 additions rounds at every partial sum: the error is at most the number of terms
// (by weight) times 2^-SH ulp of the largest term plus half an ulp of the result.
// Negative terms are complemented bit by bit (-x - 1, one unit off -x); the callers count those units
// and add them back, so that terms are cut towards zero and terms that fit are exact.
// The caller checks fx_ok(e): terms that are infinite, NaN or so large or small that an exponent
// could leave the normal range take the FP64 operations instead.
#pragma once

#include <cuda_runtime.h>

namespace dh {

// Exponent of x in place (bits 20..30 of the high word).
__device__ __forceinline__ int fx_exp(double x) { return __double2hiint(x) & 0x7ff00000; }

// Whether terms of largest exponent e (in place) can be summed: e in [80, 2030] (biased).
__device__ __forceinline__ bool fx_ok(int e) { return (unsigned)(e - (80 << 20)) <= (unsigned)((2030 - 80) << 20); }

// -1 for a term that fx_align complements, else 0: subtracting it from the aligned term adds the
// unit back, so that terms that fit are exact and -x is aligned to minus what x is.
__device__ __forceinline__ int fx_neg(double x) { return __double2hiint(x) >> 31; }

// x in units of 2^(e - 1075 - SH), towards minus infinity (zeros and terms 2^-63 below e give 0
// or -1; 0 < SH < 11).
template <int SH>
__device__ __forceinline__ long long fx_align(double x, int e) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const unsigned d = (unsigned)(e - (int)(hi & 0x7ff00000u)) >> 20;
  const unsigned s = (unsigned)((int)hi >> 31);
  const unsigned h = (__funnelshift_l(lo, hi, SH) & ((0x100000u << SH) - 1u)) | (0x100000u << SH);
  const unsigned long long m = ((unsigned long long)(h ^ s) << 32) | ((lo << SH) ^ s);
  long long r;
  asm("shr.s64 %0, %1, %2;" : "=l"(r) : "l"(m), "r"(d));  // (a count above 63 shifts by 64: the sign is left)
  return r;
}

// The FP64 number nearest to t units of 2^(e - 1075 - SH).
template <int SH>
__device__ __forceinline__ double fx_value(long long t, int e) {
  const double f = __ll2double_rn(t);
  const int hi = __double2hiint(f) + (e - ((1075 + SH) << 20));
  return t == 0 ? 0.0 : __hiloint2double(hi, __double2loint(f));
}

// p[0] + .. + p[NP-1] - m[0] - .. - m[NM-1], with NP + NM <= 24 (five bits above the 53 + 5 of a
// term): about 13 integer instructions per term and one conversion, instead of NP + NM - 1 FP64
// additions.  With NP = NM and p[i] = m[i] the sum is exactly 0 in either form.  A term that lies far
// below the largest loses bits even where the largest ones cancel: where that can happen (the pressures
// beside the momentum fluxes of a slow flow), the caller passes the difference as one term.
template <int NP, int NM>
__device__ __forceinline__ double fx_sum(const double (&p)[NP], const double (&m)[NM]) {
  static_assert(NP + NM <= 24 && NM <= NP, "room for the terms");
  constexpr int SH = 5;
  int e = 0;
#pragma unroll
  for (int i = 0; i < NP; ++i) e = max(e, fx_exp(p[i]));
#pragma unroll
  for (int i = 0; i < NM; ++i) e = max(e, fx_exp(m[i]));
  if (!fx_ok(e)) {
    long long any = 0;  // zeros (a quantity at rest) are the usual case here
#pragma unroll
    for (int i = 0; i < NP; ++i) any |= __double_as_longlong(p[i]);
#pragma unroll
    for (int i = 0; i < NM; ++i) any |= __double_as_longlong(m[i]);
    if ((any & 0x7fffffffffffffffll) == 0) return 0.0;
    double s = 0.0;
#pragma unroll
    for (int i = 0; i < NP; ++i) s += i < NM ? p[i] - m[i < NM ? i : 0] : p[i];
    return s;
  }
  long long t = 0;
  int neg = 0;  // the unit that each complemented term lacks: sums of terms that fit are exact
#pragma unroll
  for (int i = 0; i < NP; ++i) {
    t += fx_align<SH>(p[i], e);
    neg -= fx_neg(p[i]);
  }
#pragma unroll
  for (int i = 0; i < NM; ++i) {
    t -= fx_align<SH>(m[i], e);
    neg += fx_neg(m[i]);
  }
  return fx_value<SH>(t + neg, e);
}

}  // namespace dh
