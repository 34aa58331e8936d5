// fixed64.cuh - 64-bit fixed point on the integer pipes, for sums of FP64 values.
//
// An FP64 instruction holds a scheduler's FP64 unit for 64 cycles, while the integer
// pipes take one every cycle or two: an FP64 addition costs as much as some fifty integer
// instructions.  A group of doubles (the populations of a shell, or the terms of one
// relaxation) is brought to a common exponent, that of its largest member, and added as
// 64-bit integers, with B = 56 or 60 bits below that exponent: a member within 2^-3 (2^-7) of
// the largest keeps its 53 bits, a smaller one loses less than 2^-B of that power of two,
// where an FP64 sum rounds every partial sum at 2^-53 of itself.  Integer sums do not depend
// on their order.
//
// top: the largest (high word & 0x7fffffff) of the group; its exponent field e bounds
// |v| < 2^(e - 1022).  A value v is held as trunc(v 2^(B - (e - 1022))) with B bits.
// Groups with an exponent field of 2000 or more (|v| >= 2^977, Inf, NaN) are the caller's
// (fx_regular: the moments of such a cell are NaN); fields below 64 count as 64 (|v| < 2^-1014 is held as 0).
#pragma once

namespace lbm {

__device__ __forceinline__ int fx_top(double v) { return __double2hiint(v) & 0x7fffffff; }
__device__ __forceinline__ bool fx_regular(int top) { return top < (2000 << 20); }
__device__ __forceinline__ int fx_exponent(int top) { return max(top >> 20, 64); }

// v with B bits below 2^(e - 1022): 63 - B + e(v)'s distance is the right shift.
template <int B>
__device__ __forceinline__ long long fx_from(double v, int e) {
  const unsigned h = (unsigned)__double2hiint(v), l = (unsigned)__double2loint(v);
  const int r = min(e + (63 - B) - (int)((h >> 20) & 0x7ffu), 63);
  const unsigned mh = (__funnelshift_l(l, h, 10) & 0x3fffffffu) | 0x40000000u;   // 1.f at bit 62
  const unsigned long long m = ((unsigned long long)mh << 32) | (l << 10);
  const long long s = (long long)((int)h >> 31);
  return ((long long)(m >> r) ^ s) - s;
}
// The double nearest to i (B bits below 2^(e - 1022)), of two equally near ones the even: a
// sum of doubles of one exponent has a few bits more than 53 and often ends in a tie, which
// must not always go the same way (away from zero, it cost a relaxing flow 4e-18 of its mass
// a step).
template <int B>
__device__ __forceinline__ double fx_to(long long i, int e) {
  const long long s = i >> 63;
  const unsigned long long u = (unsigned long long)((i ^ s) - s);
  const int lz = __clzll((long long)u);
  const unsigned long long m = u << (lz & 63);
  const unsigned long long f0 = m >> 11;
  const unsigned rest = ((unsigned)m << 21) | ((unsigned)f0 & 1u);
  const unsigned long long f = f0 + (rest > 0x80000000u);     // 53 bits, rounded
  const int exponent = e + (63 - B) + 1 - lz;                 // field of the leading bit
  unsigned long long bits = ((unsigned long long)(unsigned)(exponent - 1) << 52) + f;
  bits |= (unsigned long long)s & 0x8000000000000000ull;
  return __longlong_as_double(u == 0 ? 0ll : (long long)bits);
}
// a f / 2^62 to the nearest integer, for |a| < 2^62 and an even factor f in [0, 2^63) with
// |a f| < 2^125: the wide products of the halves ah, al (a = 2^32 ah + 2 al + a0) and fh, fl.
// A relaxation repeated at one omega adds up whatever its product leaves out or rounds one
// way, so nothing is left out but bits below 2^-29 of a unit, and of two equally near
// integers (omega = 1.5 has them often) al's last bit chooses.  0 gives 0.
__device__ __forceinline__ long long fx_mul(long long a, long long f) {
  const int fh = (int)(f >> 32), fl = (int)((unsigned)f >> 1);
  const int ah = (int)(a >> 32), al = (int)((unsigned)a >> 1), a0 = (int)a & 1;
  const unsigned low = (unsigned)(((long long)al * fl) >> 31) + (1u << 28) - (unsigned)(al & 1);
  const long long t = (long long)ah * fl + ((long long)al * fh + (low + (unsigned)(a0 * (fh >> 1))));
  return (long long)ah * fh * 4 + (t >> 29);
}

}  // namespace lbm
