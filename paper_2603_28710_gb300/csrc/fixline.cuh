// Contractions of the FP64 operator in 64-bit fixed point, in place of chains of FP64 fused
// multiply-adds.
//
// GB300 retires 2 FP64 operations per clock and SM, but 64 32x32-bit integer multiply-adds
// with a 64-bit sum (measured 1.67 against 51 thread operations per clock and SM).  The
// sweeps, the lift and the trace interpolation are contractions with constant tables, so
// they run on the integer pipe with an accuracy above that of an FP64 chain:
//   * the values that enter a contraction share an exponent e, that of the largest of them
//     (sweep and lift: of one variable's fluxes in the whole element; traces: of the line),
//     and become fixed-point numbers v of 59 or 60 bits, cut into two limbs, v = f1 2^31 + f0
//     (0 <= f0 < 2^31);
//   * the tables are fixed-point numbers of at most 61 bits per sum of |entries|, cut
//     likewise, q = q1 2^31 + q0 (|q0| <= 2^30);
//   * sum q v = 2^62 sum q1 f1 + 2^31 sum (q1 f0 + q0 f1) + sum q0 f0; the first two are exact
//     in 64 bits (the host checks the bounds when it makes the tables); of the last only its
//     mean 2^30 sum q0 is kept, as the start value of the second (with half a unit of the
//     first for rounding; zeros start with the half unit alone, so that they give zeros);
//   * the result is rounded to FP64 once.
// Error before that rounding: typically 2^-59 of the largest value times the table's row sum.
// An FP64 chain rounds once per term, each time by up to 2^-53 of its partial sum; emulated
// on random lines its error is 4 to 10 times larger.
// Values that hold Inf or NaN, or are too large or too small for the exponent range (about
// 10^-290 to 10^303), go through the FP64 chain, so non-finite values spread as they do there.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "adg_internal.h"

namespace adg {

// Upper 31 bits of |x|: its magnitude as an ordered integer, its exponent field from bit 20.
__device__ __forceinline__ int abs_hi(double x) { return __double2hiint(x) & 0x7FFFFFFF; }

// Exponent of the largest magnitude (abs_hi); zeros take the smallest one.
__device__ __forceinline__ int fixed_exponent(const FixedScale& s, int max_hi) {
  return max(max_hi >> 20, s.elo);
}
// Whether the magnitude is outside of the range in which 60 bits below it and the results are
// normal numbers (zero is inside): the values then go through the FP64 chain.
__device__ __forceinline__ bool fixed_outside(const FixedScale& s, int max_hi) {
  return (max_hi >> 20) > s.ehi || (unsigned)(max_hi - 1) < (unsigned)((s.elo << 20) - 1);
}

// (hi, lo) -> -(hi, lo) where the top bit of s is set
__device__ __forceinline__ void negate_if(unsigned s, unsigned& lo, unsigned& hi) {
  asm("{\n\t.reg .pred p;\n\t"
      "setp.lt.s32 p, %2, 0;\n\t"
      "@p sub.cc.u32 %0, 0, %0;\n\t"
      "@p subc.u32 %1, 0, %1;\n\t}"
      : "+r"(lo), "+r"(hi)
      : "r"(s));
}

// Limbs {f1, f0} of x: x = (f1 2^31 + f0) 2^(es - 1086), truncated, for exponents below es - 3
// (zeros and subnormals become 0: their shift is 64 or more).
__device__ __forceinline__ int2 fixed_limbs(double x, int es) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const unsigned t1 = __funnelshift_l(lo, hi, 11) | 0x80000000u;  // mantissa, top bit set
  const unsigned long long t = ((unsigned long long)t1 << 32) | (lo << 11);
  const unsigned sh = (unsigned)(es - (int)((hi >> 20) & 0x7FFu));
  unsigned long long v;
  asm("shr.u64 %0, %1, %2;" : "=l"(v) : "l"(t), "r"(sh));  // 0 for shifts of 64 and more
  unsigned v0 = (unsigned)v, v1 = (unsigned)(v >> 32);
  negate_if(hi, v0, v1);
  return make_int2((int)__funnelshift_r(v0, v1, 31), (int)(v0 & 0x7FFFFFFFu));
}

// c + a b: one wide multiply-add.  (Written in C: inline PTX mad.wide takes two instructions,
// and so does a product whose operands the compiler knows the sign or range of; the limbs are
// therefore made opaque where they are computed.)
__device__ __forceinline__ long long mad_wide(int a, int b, long long c) { return c + (long long)a * b; }
__device__ __forceinline__ void opaque(int2& f) { asm("" : "+r"(f.x), "+r"(f.y)); }

// I 2^(eb - 1086) rounded to FP64 with integer operations (64-bit conversions run at the
// FP64 rate).  eb lies in 64..2045, so that every result is a normal number or zero.
__device__ __forceinline__ double fixed_to_double(long long I, int eb) {
  unsigned lo = (unsigned)I, hi = (unsigned)((unsigned long long)I >> 32);
  const unsigned sgn = hi & 0x80000000u;
  negate_if(hi, lo, hi);
  if (hi == 0) {  // small result: by one word
    hi = lo;
    lo = 0;
    eb -= 32;
  }
  const int n = __clz((int)hi);  // top bit to bit 62: the rounding below cannot overflow
  const unsigned top = __funnelshift_l(lo, hi, n);
  const unsigned h = top >> 1;
  const unsigned long long t =
      (((unsigned long long)h << 32) | __funnelshift_r(lo << n, top, 1)) + 0x200ull;
  unsigned b = (unsigned)(t >> 42);
  if (h != 0) b += (unsigned)(eb - 1 - n) << 20;
  return __hiloint2double((int)(b | sgn), (int)(t >> 10));
}

// Accumulator of a sweep: 2^62 a + 2^31 m (exponent shift of the limbs: kSweepShift).
constexpr int kSweepShift = 5, kTraceShift = 4;
struct FixedAcc {
  long long a, m;
};
__device__ __forceinline__ void fixed_fma(int2 q, int2 f, FixedAcc& t) {
  t.a = mad_wide(q.x, f.x, t.a);
  t.m = mad_wide(q.x, f.y, t.m);
  t.m = mad_wide(q.y, f.x, t.m);
}
__device__ __forceinline__ double fixed_result(const FixedAcc& t, const FixedScale& s, int e) {
  return fixed_to_double(t.a + (t.m >> 31), e + s.eout);
}

// Start value of the middle limb sum for values of exponent e.
constexpr long long kFixedHalf = 1ll << 30;
__device__ __forceinline__ long long fixed_start(const FixedScale& s, int e, long long c) {
  return e > s.elo ? c : kFixedHalf;
}

// Traces at both ends of a line of N nodes (low end -1, high end +1).
template <int N>
__device__ __forceinline__ void line_traces(const FixedTrace& T, const OpTables* tab,
                                            const double (&x)[N], double& lo, double& hi) {
  int m = 0;
#pragma unroll
  for (int a = 0; a < N; ++a) m = max(m, abs_hi(x[a]));
  const int e = fixed_exponent(T.s, m);
  if (fixed_outside(T.s, m)) {
    lo = hi = 0.0;
#pragma unroll
    for (int a = 0; a < N; ++a) {
      lo = fma(tab->Tm[a], x[a], lo);
      hi = fma(tab->Tp[a], x[a], hi);
    }
    return;
  }
  int2 f[N];
#pragma unroll
  for (int a = 0; a < N; ++a) {
    f[a] = fixed_limbs(x[a], e + kTraceShift);
    opaque(f[a]);
  }
#pragma unroll
  for (int side = 0; side < 2; ++side) {
    long long s = fixed_start(T.s, e, T.c[side]);
#pragma unroll
    for (int a = 0; a < N; ++a) {
      s = mad_wide(T.t[side][a].x, f[a].y, s);
      s = mad_wide(T.t[side][a].y, f[a].x, s);
    }
    s >>= 31;
#pragma unroll
    for (int a = 0; a < N; ++a) s = mad_wide(T.t[side][a].x, f[a].x, s);
    (side ? hi : lo) = fixed_to_double(s, e + T.s.eout);
  }
}

}  // namespace adg
