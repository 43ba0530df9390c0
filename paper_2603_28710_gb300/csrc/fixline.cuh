// Contractions of the FP64 operator in 64-bit fixed point, in place of chains of FP64 fused
// multiply-adds.
//
// GB300 retires 2 FP64 operations per clock and SM, but 64 32x32-bit integer multiply-adds
// with a 64-bit sum (measured 1.67 against 51 thread operations per clock and SM).  The
// sweeps, the lift and the trace interpolation are contractions with constant tables, so
// they run on the integer pipe with an accuracy above that of an FP64 chain:
//   * the values of a line of nodes (sweep and lift: N fluxes and the two face fluxes) share an
//     exponent e, that of the largest of them, and become fixed-point numbers v of 61 bits, cut
//     into two limbs, v = f1 2^31 + f0 (0 <= f0 < 2^31);
//   * the tables are fixed-point numbers of at most 61 bits per row sum of |entries|, with a scale
//     of its own for every direction, cut likewise, q = q1 2^31 + q0 (|q0| <= 2^30);
//   * sum q v = 2^62 sum q1 f1 + 2^31 sum (q1 f0 + q0 f1) + sum q0 f0; the first two are exact
//     in 64 bits (the host checks the bounds when it makes the tables); of the last only its
//     mean 2^30 sum q0 is kept, as the start value of the second (with half a unit of the last
//     bit kept, for rounding);
//   * a node adds up its lines as 64-bit integers, shifted to the largest of their exponents, and
//     rounds to FP64 once.
// Error before that rounding: typically 2^-60 of a line's largest value times the table's row
// sum.  An FP64 chain rounds once per term, each time by up to 2^-53 of its partial sum.
// Emulated on lines with random values, values over eight orders of magnitude, single large nodes
// and faces, small rows of nodes and stretched elements, for all degrees: the root mean square
// error of every node is 0.02 to 1.0 of the chain's there.
// Lines whose values hold Inf or NaN, or are too large or too small for the exponent range (about
// 10^-290 to 10^303), keep FP64 values and chains, so non-finite values spread as they do there;
// so do lines whose middle one of an odd number of nodes stands out (line_exponent).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "adg_internal.h"

namespace adg {

// Upper 31 bits of |x|: its magnitude as an ordered integer, its exponent field from bit 20.
__device__ __forceinline__ int abs_hi(double x) { return __double2hiint(x) & 0x7FFFFFFF; }

// Whether the magnitude is outside of the range in which the bits below it and the results are
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

// Limbs {f1, f0} of x: x = (f1 2^31 + f0) 2^(es - 1086), truncated, for exponents up to es - 3
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

// c + a b, a 32x32-bit product added to 64 bits.  Written in C, and with operands that the compiler
// knows nothing about (opaque), as measured, us per volume launch: 48^3 p=3 765, with mad.wide as
// inline PTX 919, without the barrier behind the limbs of a trace line 790; 256^2 p=4 117, 135, 120.
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

// Exponent of the limbs of values whose largest exponent is e.
__device__ __forceinline__ int limb_exponent(int e) { return max(e, kFixedMinExp) + 64 - kFixedValueBits; }

// Accumulator of a line: 2^62 a + 2^31 m.
struct FixedAcc {
  long long a, m;
};
__device__ __forceinline__ void fixed_fma(int2 q, int2 f, FixedAcc& t) {
  t.a = mad_wide(q.x, f.x, t.a);
  t.m = mad_wide(q.x, f.y, t.m);
  t.m = mad_wide(q.y, f.x, t.m);
}
// The sum with FRAC bits below 2^62.
template <int FRAC>
__device__ __forceinline__ long long fixed_sum(const FixedAcc& t) {
  return (t.a << FRAC) + (t.m >> (31 - FRAC));
}

// ---- sweeps and lift ------------------------------------------------------------------
// Exponent of a line's sums as stored for its nodes: 64 to 2045, 0 for a line of zeros,
// or kChainLine, larger than those and with a bit of its own, for a line that keeps its FP64 values.
constexpr int kChainLine = 2048;

// Exponent of a line of N fluxes and the two face fluxes behind them (direction scale s); es:
// that of its limbs.  The middle one of an odd number of nodes has the weight zero in its own
// row, so the other values set that row's accuracy: where it exceeds them by more than 2^5 the
// line keeps its FP64 values (the bits that a fixed-point sum has beyond a chain's).
template <int N>
__device__ __forceinline__ int line_exponent(const double (&x)[N + 2], const FixedScale& s, int& es) {
  int m = 0, mid = 0;
#pragma unroll
  for (int a = 0; a < N + 2; ++a) {
    if (N % 2 == 1 && a == N / 2) mid = abs_hi(x[a]);
    else m = max(m, abs_hi(x[a]));
  }
  const bool lone = (mid >> 20) > (m >> 20) + 5;
  m = max(m, mid);
  es = limb_exponent(m >> 20);
  if (lone || fixed_outside(s, m)) return kChainLine;
  return m == 0 ? 0 : (m >> 20) + s.eout;
}
// es again from the exponent of the sums
__device__ __forceinline__ int limbs_of_line(int ex, const FixedScale& s) { return limb_exponent(ex - s.eout); }

// Adds a line's sum of exponent ex to a sum of exponent e >= ex.  (A line of zeros has ex = 0 and
// e >= 64 beside other lines: a shift by 64 or more leaves the sign alone.)
__device__ __forceinline__ void add_line(const FixedAcc& t, int ex, int e, long long& sum) {
  long long r;
  asm("shr.s64 %0, %1, %2;" : "=l"(r) : "l"(fixed_sum<kSweepFrac>(t)), "r"(e - ex));
  sum += r;
}
// Value of a sum of lines of exponent e (0: lines of zeros only).
__device__ __forceinline__ double line_result(long long sum, int e) {
  return e > 0 ? fixed_to_double(sum, e) : 0.0;
}

// ---- traces ---------------------------------------------------------------------------
// Traces at both ends of a line of N nodes (low end -1, high end +1).
template <int N>
__device__ __forceinline__ void line_traces(const FixedTrace& T, const OpTables* tab,
                                            const double (&x)[N], double& lo, double& hi) {
  int m = 0;
#pragma unroll
  for (int a = 0; a < N; ++a) m = max(m, abs_hi(x[a]));
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
    f[a] = fixed_limbs(x[a], limb_exponent(m >> 20));
    opaque(f[a]);
  }
#pragma unroll
  for (int side = 0; side < 2; ++side) {
    FixedAcc t{0, m > 0 ? T.c[side] : fixed_half(kTraceFrac)};
#pragma unroll
    for (int a = 0; a < N; ++a) fixed_fma(T.t[side][a], f[a], t);
    (side ? hi : lo) = fixed_to_double(fixed_sum<kTraceFrac>(t), (m >> 20) + T.s.eout);
  }
}

}  // namespace adg
