// Scalars of the coarse CG: the reciprocals of its step lengths, its stopping
// test, and the power of two that keeps its sums away from the ends of the
// exponent range.
#pragma once

#include <cstdint>

// 1 / b, within one unit in the last place of the rounded reciprocal, for
// 2^-1021 <= |b| <= 2^1021 (which cg_shift sees to): the hardware's reciprocal
// approximation y and one third-order step y (1 + e + e^2), e = 1 - b y
// (Halley's iteration for 1 / b).  Three dependent FP64 operations of 68 clocks
// each in the chain that bounds an iteration of about 5000 clocks, where the
// IEEE division takes 590; dividing was measured at 4 to 8% of a solve (343 rows
// 216 -> 234 us, 3375 rows 449 -> 467 us), and the cycles' error against 64-bit
// references is the same to three digits either way: x and r move by the same
// step, so its rounding only turns the search direction.
__device__ __forceinline__ double cg_recip(double b) {
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(b));
  double d = fma(-b, y, 1.0);
  d = fma(d, d, d);
  return fma(y, d, y);
}

// The CG's sums are squares of its vectors, which it reduces by the tolerance:
// with a load of norm 1e-143 r.r falls to 1e-310, its reciprocal is infinite,
// and even the quotient of two such sums has lost its bits (an iterate of a
// load of norm 1e-150 was off by factors of 1e56 to 1e99).  So where b.b lies
// outside 2^-400 .. 2^400 (cg_in_range) the load is multiplied by the power of
// two that brings its largest entry to [1, 2), and the solution divided by it:
// exact, and the same bits as for a load in ordinary units.  Tolerances are
// taken to be CG_RTOL_MIN at least, far below what moves a bit of x.
constexpr double CG_RTOL_MIN = 1e-60;
__device__ __forceinline__ uint32_t cg_exponent(double v) { return ((uint32_t)__double2hiint(v) >> 20) & 0x7ffu; }
__device__ __forceinline__ bool cg_in_range(double bb) { return cg_exponent(bb) - 623u <= 800u; }
// The factor for a largest exponent field m of the load's entries (in bounds of
// the exponent range, also for its reciprocal); 1 for infinities and NaN.
__device__ __forceinline__ double cg_shift(uint32_t m) {
  const int e = m == 0x7ffu ? 1023 : 2046 - (int)(m < 1u ? 1u : m > 2023u ? 2023u : m);
  return __hiloint2double(e << 20, 0);
}

// The test sqrt(rr) > thr, set up once for a thr: rr (>= 0, or not a number) is
// compared as an integer with thr^2 (1 +- 1e-14), and only between the two, or
// where thr^2 is near the ends of the exponent range, the square root (650
// clocks) is taken.
struct CgTest {
  double thr;
  long long lo, hi;
};
__device__ __forceinline__ CgTest cg_test(double thr) {
  CgTest t{thr, 0, 0x7ff0000000000000ll};
  const double t2 = thr * thr;
  if (t2 > 1e-280 && t2 < 1e280) {
    t.lo = __double_as_longlong(t2 * (1.0 - 1e-14));
    t.hi = __double_as_longlong(t2 * (1.0 + 1e-14));
  }
  return t;
}
static __device__ __noinline__ bool cg_above_sqrt(double rr, double thr) { return sqrt(rr) > thr; }
__device__ __forceinline__ bool cg_above(double rr, const CgTest& t) {
  const long long b = __double_as_longlong(rr);
  if (b > t.hi && b < 0x7ff0000000000000ll) return true;
  if (b < t.lo) return false;
  return cg_above_sqrt(rr, t.thr);
}
