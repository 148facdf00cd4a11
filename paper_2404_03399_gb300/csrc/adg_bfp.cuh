// Local block fixed point: FP64 fields in memory, the element arithmetic of the nonlinear
// stages in 57-bit integers.
//
// On this part a warp's FP64 instruction holds the SM's FP64 pipe for 16 clocks (2 lanes per
// clock per SM), a 32 x 32 -> 64-bit integer product the heavy FMA pipe of one of the four
// sub-partitions for 4, and shifts and adds run beside it. A stage evaluated in FP64 is bound
// by that pipe (73-84 FP64 instructions per element at p = 4), so the stages here load FP64
// values, bring each element to a scale of its neighbourhood, work in integers, and round once
// to FP64 when the step is done.
//
// An element's values are X = x 2^(57 - E), |x| < 2^E over the element and the two beside it, so
// |X| < 2^57 at the start of the step; every intermediate value is checked to stay below 2^58,
// and what comes from a neighbour is shifted from its scale. Squares and face fluxes are held in
// units of 2^(2E - 56): G = X^2 2^-58. An operator coefficient c is C = round(c 2^(58 - sc)),
// |C| <= 2^58, split as in adg_fixed.cuh, and sums of products are rounded once.
//
// Against FP64: a value's unit is 2^-56 of the largest one beside it, FP64's roundings are
// 2^-53 of a value each, and the integer path is taken only where every non-zero element reaches
// 2^-kBfSpan of that largest value. The span is where the error of an element, over its own
// largest value, stays below that of the FP64 stages: emulated in integers and compared with
// 113-bit arithmetic over p = 1..4, Courant numbers 0.002 to 0.05, 20 and 200 steps, on smooth
// fields and on rough ones whose patches of four elements differ by up to 50 (rms over the
// elements, integer over FP64): SSP-RK3 0.17 at equal patches, 0.18 to 0.26 at a ratio of 8 and
// at most 1.00 beyond with a span of 4; the 2N schemes, whose FP64 stages round once or twice,
// 0.45 (five stages) to 0.72 (RK2) at equal patches, at most 0.89 at 8 and 1.06 beyond with a
// span of 3. The means of the products that sums leave out, and (in the 2N schemes) roundings
// that send every half up, add up step by step: with them RK2 reached 1.9 after 200 steps.
// SSP-RK3 keeps the latter (2 to 4% of a step to even out), since its FP64 stages lose a unit
// of 2^-54 a step in 1/3 + 2/3: it stays below 0.1. With a span of 6 and the scale of the
// elements up to a stage count away, RK2 reached 8.8 at a ratio of 50 and SSP-RK3 2.1.
// The reverse step, whose scale and span are those of SSP-RK3: 0.18 to 0.23 with alike elements,
// at most 0.79 at any ratio and on waves through zero, at most 0.40 over 500 steps. (Its
// products rounded to a unit of 2^-57 of their bound, where smooth fields leave them far
// below it, and without the low limbs' product, it reached 4 on such a wave at a Courant
// number of 0.01 and p = 3, 22 at 0.05.)
//
// A simple zero of a smooth field leaves its element within a third of its neighbours, inside
// both spans. Forward Euler takes FP64: its stage is one rounding, which the integer path also
// ends with. Warps with an element outside the span (or exponents near the ends of the FP64
// range, NaN, infinities, growth past the headroom within a step, Courant numbers whose
// coefficients do not fit) take the FP64 stages.
//
// With one scale per warp instead of per element the warps at a smooth wave's zeros did (the
// gradient on 65536 elements, 100 steps: 3.00 ms, 2.91 ms with a scale per element; without a
// zero the scales per element cost 4% on 2^20 elements).
#pragma once

#include "adg_fixed.cuh"

namespace adg {
namespace {

// exponent of an element below its scale on the integer path, by the scheme (2N or SSP-RK3)
template <bool LS>
constexpr int kBfSpan = LS ? 3 : 4;
constexpr int kBfMinE = 600;    // biased exponents of the scales
constexpr int kBfMaxE = 1400;
constexpr int kBfTop = 58;      // every intermediate value below 2^kBfTop

// x 2^(1079 - be) rounded to an integer: |x| < 2^(be - 1022) gives |X| < 2^57. Exponents
// below be - 63 (zeros and subnormals among them: be >= kBfMinE) give 0.
__device__ __forceinline__ long long bf_from(double x, int be) {
  const int hi = __double2hiint(x);
  const unsigned lo = (unsigned)__double2loint(x);
  const int e = (hi >> 20) & 0x7ff;
  const unsigned mh = ((unsigned)hi & 0xfffffu) | 0x100000u;
  int d = be - e;
  d = d > 63 ? 63 : d;
  const unsigned long long m =
      (unsigned long long)fx_join(lo << 5, __funnelshift_l(lo, mh, 5));   // mantissa 2^5
  const long long M = (long long)(((m >> d) + 1) >> 1);
  const long long s = (long long)(hi >> 31);
  return (M ^ s) - s;
}

// y 2^sigma rounded to nearest even, for results inside the normal range (the integer path's
// exponents keep them there) or zero.
__device__ __forceinline__ double bf_to(long long y, int sigma) {
  const long long s = y >> 63;
  const unsigned long long a = (unsigned long long)((y ^ s) - s);   // < 2^62
  const int lz = __clzll((long long)a);
  const unsigned long long nrm = a << (lz - 1);   // leading one in bit 62: no carry out
  const unsigned long long m = (nrm + 0x1ffull + ((nrm >> 10) & 1ull)) >> 10;   // <= 2^53
  // the leading one of m adds one to the exponent field
  const unsigned long long r = m + ((unsigned long long)(unsigned)(1085 + sigma - lz) << 52);
  return a == 0 ? 0.0 : __longlong_as_double((long long)(r | ((unsigned long long)s << 63)));
}

// X^2 2^-58 (|X| < 2^58), rounded, with the mean (a third of a unit) of the xl^2 2^-58 left out:
// below 7/6 units of error.
constexpr long long kSquareRound = (1ll << 27) + (1ll << 28) / 3;
__device__ __forceinline__ long long bf_square(int xh, int xl) {
  return fx_mul(xh, xh) + ((fx_mul(xh, xl) + kSquareRound) >> 28);
}

// Local Lax-Friedrichs flux 1/4 (a^2 + b^2) - 1/2 max(|a|, |b|) (b - a) of the traces a = u^-,
// b = u^+ with squares ga, gb, in the squares' units. With the larger trace x the last product
// is +-(a b - x^2): one product and no magnitudes (the sign is x's, and the other one for b);
// equal traces give a b = a^2 exactly. EVEN: halves go up or down by a bit of gb.
template <bool EVEN>
__device__ __forceinline__ long long bf_llf(long long a, long long b, long long ga, long long gb) {
  int ah, al, bh, bl;
  fx_split(a, ah, al);
  fx_split(b, bh, bl);
  const long long ab =
      fx_mul(ah, bh) + ((fx_mul(ah, bl) + fx_mul(al, bh) + 2 * kSquareRound) >> 29);
  const bool left = ga >= gb;
  const long long t = left ? ab - ga : gb - ab;
  const long long s = (long long)((int)((left ? a : b) >> 32) >> 31);   // 0 or -1
  return (ga + gb - 2 * ((t ^ s) - s) + 2 - (EVEN ? (gb >> 1) & 1 : 0)) >> 2;
}

// 1/3 as limbs of round(2^58 / 3).
constexpr long long kThird = ((1ll << 58) - 1) / 3;
constexpr int kThirdLo = (int)(((kThird & 0x1FFFFFFF) ^ 0x10000000) - 0x10000000);
constexpr int kThirdHi = (int)((kThird - kThirdLo) >> 29);

// The high word of a bound on |y| as fx_mag gives it: OR-ed over the values of a step, its bits
// from kBfTop up show growth past the headroom (two instructions less per value than in 64 bits).
__device__ __forceinline__ unsigned bf_mag(long long y) {
  const int h = (int)(y >> 32);
  return (unsigned)(h ^ (h >> 31));
}
constexpr unsigned kBfOver = 1u << (kBfTop - 32);

// v 2^-d (d < 0: a left shift; the caller has checked that the result fits).
__device__ __forceinline__ long long bf_shift(long long v, int d) {
  return d >= 0 ? v >> d : (long long)((unsigned long long)v << (-d));
}

// A neighbour's value v brought to this lane's unit, d exponents above the neighbour's (rounded);
// raises `mag` past the headroom where it does not stay below 2^Top.
template <int Top = kBfTop>
__device__ __forceinline__ long long bf_bring(long long v, int d, unsigned &mag) {
  if (d == 0) return v;
  d = d > 62 ? 62 : d;
  if (d > 0) return (v + (1ll << (d - 1))) >> d;
  if (d < -Top || (fx_mag(v) >> (Top + d)) != 0) {
    mag |= v ? kBfOver : 0u;
    return 0;
  }
  return (long long)((unsigned long long)v << (-d));
}

// The largest of x over the lanes within n of this one.
__device__ __forceinline__ int bf_window_max(int x, int n) {
  for (int k = 0; k < n; ++k)
    x = max(x, max(__shfl_up_sync(0xffffffffu, x, 1), __shfl_down_sync(0xffffffffu, x, 1)));
  return x;
}

}  // namespace
}  // namespace adg
