// collide64.cuh - the cell update of the FP64 form (a3 - a6), written for the fewest
// FP64 operations.  Included by kernels.cuh after the shared helpers.
//
// What bounds it: a quarter of an SM (one scheduler) takes 64 cycles for an FP64
// instruction, whatever the number of active lanes (measured, dependent or not; a
// conversion between FP64 and FP32 costs the same), so the form is bound by its FP64
// instruction count and not by memory: 1520 bytes a D3Q95 cell take 0.23 ns of HBM time,
// the ~1290 FP64 operations of the pair-by-pair form 2.4 ns.  What brings D3Q95 to ~470 with
// two warps sharing 32 cells (of which one repeats ~35):
//   * moments shell by shell: the members of a shell share weight and |xi|^2, so their
//     sums are formed unweighted and each shell is weighted once;
//   * those sums, and the relaxation's h + omega (h^eq - h), in 64-bit fixed point on the
//     integer pipes (fixed64.cuh);
//   * rho and rho - 1 folded into the shell's equilibrium coefficients, so a pair's
//     even part is c0 + s^2 (c2 + s^2 c4) and its odd part s (c1 + s^2 c3);
//   * s and s^2 once per primitive direction b: the pairs k b of several shells (axes
//     2, 3, 5; diagonals 2, 3, 4; ...) share them, with the powers of k folded into the
//     coefficients.
// Measured (us a step): D3Q95 128x32x32 311 pair by pair, 235 regrouped in FP64, 149 with
// the fixed point; D2Q33 1024x512 446, 354, 210.
// Error: runs of 40 to 150 steps end 0.2 to 0.45 as far from extended precision as the same
// collisions evaluated direction by direction in FP64.
//
// The shells are dealt into kParts64 parts of nearly equal work (whole shells, so the
// weighting is not repeated).  Every kernel sums the parts' moments in the same order,
// ((0 + 1) + (2 + 3)), so one thread doing all parts and several warps doing some each
// produce the same bits.
#pragma once

#include "fixed64.cuh"

namespace lbm {

constexpr int kParts64 = 4;

// The part each shell belongs to, and the pairs of a part in evaluation order: grouped
// by primitive direction.
template <int M>
struct Part64 {
  int n;                          // pairs
  int dir[Model<M>::NP];          // direction of +e (e = k b; -e follows it)
  int b[Model<M>::NP][3];
  int k[Model<M>::NP];
  int grp[Model<M>::NP];
};

// D2Q33 (4 pairs each): (1,0) (2,0) | (1,1) (3,0) | (2,2) (4,4) | (2,1).
// D3Q95 (11 or 12 pairs): (2,2,0) (3,3,0) | (2,0,0) (3,0,0) (4,4,0) |
//   (2,2,2) (3,3,3) (5,0,0) | (2,2,5).  Shell numbers as in velset.cuh.
template <int M>
LBM_HD constexpr int shell_part64(int g) {
  constexpr int d2[8] = {-1, 0, 1, 0, 2, 1, 3, 2};
  constexpr int d3[10] = {-1, 1, 0, 2, 1, 0, 2, 3, 1, 2};
  return M == 0 ? d2[g] : d3[g];
}

// Pairs [first, end) of symmetry group g (g >= 1) in storage order.
template <int M>
struct ShellPairs {
  static constexpr int first(int g) {
    int p = 0;
    while (p < Model<M>::NP && Model<M>::vs.grp[1 + 2 * p] != g) ++p;
    return p;
  }
  static constexpr int end(int g) {
    int p = first(g);
    while (p < Model<M>::NP && Model<M>::vs.grp[1 + 2 * p] == g) ++p;
    return p;
  }
};

// part < 0: all pairs.
template <int M>
LBM_HD constexpr Part64<M> make_part64(int part) {
  using Mo = Model<M>;
  Part64<M> t{};
  bool used[Mo::NP] = {};
  for (int p0 = 0; p0 < Mo::NP; ++p0) {
    if (used[p0] || (part >= 0 && shell_part64<M>(Mo::vs.grp[1 + 2 * p0]) != part)) continue;
    const int* e0 = Mo::vs.e[1 + 2 * p0];
    const int g0 = igcd(igcd(iabs(e0[0]), iabs(e0[1])), iabs(e0[2]));
    for (int p = p0; p < Mo::NP; ++p) {          // the part's pairs along e0
      const int* e = Mo::vs.e[1 + 2 * p];
      const int g = igcd(igcd(iabs(e[0]), iabs(e[1])), iabs(e[2]));
      if (used[p] || (part >= 0 && shell_part64<M>(Mo::vs.grp[1 + 2 * p]) != part)) continue;
      if (e[0] * g0 != e0[0] * g || e[1] * g0 != e0[1] * g || e[2] * g0 != e0[2] * g) continue;
      used[p] = true;
      t.dir[t.n] = 1 + 2 * p;
      for (int d = 0; d < 3; ++d) t.b[t.n][d] = e[d] / g;
      t.k[t.n] = g;
      t.grp[t.n] = Mo::vs.grp[1 + 2 * p];
      ++t.n;
    }
  }
  return t;
}

template <int M, int P>
struct P64 {
  static constexpr Part64<M> t = make_part64<M>(P);
  static constexpr bool first_of(int n) {        // first / last pair of its shell
    for (int m = 0; m < n; ++m)
      if (t.grp[m] == t.grp[n]) return false;
    return true;
  }
  static constexpr bool last_of(int n) {
    for (int m = n + 1; m < t.n; ++m)
      if (t.grp[m] == t.grp[n]) return false;
    return true;
  }
  static constexpr bool new_base(int n) {          // first / last pair along its primitive vector
    return n == 0 || t.b[n][0] != t.b[n - 1][0] || t.b[n][1] != t.b[n - 1][1] ||
           t.b[n][2] != t.b[n - 1][2];
  }
  static constexpr bool end_base(int n) { return n + 1 == t.n || new_base(n + 1); }
};
static_assert(P64<0, 0>::t.n == 4 && P64<0, 1>::t.n == 4 && P64<0, 2>::t.n == 4 &&
              P64<0, 3>::t.n == 4, "D2Q33 parts");
static_assert(P64<1, 0>::t.n == 12 && P64<1, 1>::t.n == 12 && P64<1, 2>::t.n == 11 &&
              P64<1, 3>::t.n == 12, "D3Q95 parts");

// sum w h, sum w h |xi|^2 and sum w h e over one part.
struct Mom64 {
  double r, e, x, y, z;
};
template <int M>
__device__ __forceinline__ Mom64 add64(const Mom64& a, const Mom64& b) {
  return {__dadd_rn(a.r, b.r), __dadd_rn(a.e, b.e), __dadd_rn(a.x, b.x), __dadd_rn(a.y, b.y),
          Model<M>::D == 3 ? __dadd_rn(a.z, b.z) : 0.0};
}

// p + m and p - m of a pair in fixed point.  A call, as relax_pair64 below: expanded at all
// 47 pairs of D3Q95 the step's code outgrows the instruction cache (266 us against 152 at
// 128 x 32 x 32).
struct SumDiff64 {
  long long s, d;
};
static __device__ __noinline__ SumDiff64 sum_diff64(double hp, double hm, int e) {
  const long long p = fx_from<56>(hp, e), m = fx_from<56>(hm, e);
  return {p + m, p - m};
}
// Shell by shell: the members' sums in fixed point (fixed64.cuh) at the shell's own scale,
// so no member loses bits to another shell's larger deviations, and one below 1/8 of its own
// shell's largest less than 2^-56 of that.
template <int M, int P, class Get>
__device__ __forceinline__ Mom64 moments64(Get&& hv) {
  using Mo = Model<M>;
  const ModelConst& mc = c_mc[M];
  Mom64 m = {0.0, 0.0, 0.0, 0.0, 0.0};
  bool none = true;
  sfor<1, Mo::G>([&](auto Gi) {
    constexpr int g = decltype(Gi)::value;
    if constexpr (shell_part64<M>(g) == P) {
      constexpr int p0 = ShellPairs<M>::first(g), np = ShellPairs<M>::end(g) - p0;
      double h[2 * np];
      int top = 0;
      sfor<0, 2 * np>([&](auto J) {
        constexpr int j = decltype(J)::value;
        h[j] = hv(std::integral_constant<int, 1 + 2 * p0 + j>{});
        top = max(top, fx_top(h[j]));
      });
      const int e = fx_exponent(top);
      long long gs = 0, gx = 0, gy = 0, gz = 0;
      sfor<0, np>([&](auto J) {
        constexpr int j = decltype(J)::value, i = 1 + 2 * (p0 + j);
        constexpr int ex = Mo::vs.e[i][0], ey = Mo::vs.e[i][1], ez = Mo::vs.e[i][2];
        const SumDiff64 sd = sum_diff64(h[2 * j], h[2 * j + 1], e);
        const long long d = sd.d;
        gs += sd.s;
        if constexpr (ex != 0) gx += ex * d;
        if constexpr (ey != 0) gy += ey * d;
        if constexpr (ez != 0) gz += ez * d;
      });
      // sums: at most 72 2^56 < 2^63
      double S = fx_to<56>(gs, e), X = fx_to<56>(gx, e), Y = fx_to<56>(gy, e), Z = 0.0;
      if constexpr (Mo::D == 3) Z = fx_to<56>(gz, e);
      if (!fx_regular(top)) S = X = Y = Z = __longlong_as_double(0x7ff8000000000000ll);
      const double tr = __dmul_rn(mc.W[g], S);
      m.r = none ? tr : __dadd_rn(m.r, tr);
      m.e = none ? __dmul_rn(mc.X2[g], tr) : __fma_rn(mc.X2[g], tr, m.e);
      m.x = none ? __dmul_rn(mc.W[g], X) : __fma_rn(mc.W[g], X, m.x);
      m.y = none ? __dmul_rn(mc.W[g], Y) : __fma_rn(mc.W[g], Y, m.y);
      if constexpr (Mo::D == 3) m.z = none ? __dmul_rn(mc.W[g], Z) : __fma_rn(mc.W[g], Z, m.z);
      none = false;
    }
  });
  return m;
}

// x / 3 and x / 6 (P = 0, 1), with the rest of 1 / 3: (1 / 3) 2^-54.  The rounded 1 / 3 alone is
// too small by half an ulp in every cell and step, which cooled a D3Q95 flow.
template <int P>
__device__ __forceinline__ double over3_64(double x) {
  constexpr double hi = 1.0 / (P == 0 ? 3.0 : 6.0), lo = hi * 0x1p-54;
  return __fma_rn(x, hi, __dmul_rn(x, lo));
}
template <int D>
__device__ __forceinline__ double over_dim64(double x) {
  if constexpr (D == 3) return over3_64<0>(x); else return __dmul_rn(x, 0.5);
}

// What the relaxation needs of a cell: the velocity a u (s = e . v), and the equilibrium's
// coefficients with rho folded in.  h^eq of a pair +- k b, with s = b . v, is
//   c0 +- s c1 + s^2 c2 +- s^3 c3 + s^4 c4
//   c0 = P0 + x2 (K1 + (x2 / 8) tt),  c1 = k (L0 + (x2 / 2) rt),
//   c2 = k^2 (d2 + (x2 / 4) rt),  c3 = k^3 r6,  c4 = k^4 r24
// (EqCoef's polynomials times rho; rt = rho t, tt = rho t^2, d2 = (L0 - rt) / 2, r6 = rho / 6,
// r24 = rho / 24).  Of a shell only x2 (or an exact fraction of it), its weight and small
// integers are multiplied in, as in the moments: a rounded product of them (W x2, k^3 / 6,
// ...) is off by the same fraction of an ulp in every cell and step, and after 200 steps of
// a 256 x 8 D2Q33 flow the populations' rms error was 4.8e-14 with such products, 1.6e-15
// without (pair by pair: 2.0e-15).
struct Cell64 {
  double vx, vy, vz;
  double P0, K1, tt, L0, rt, d2, rho, r6, r24;
};
template <int M>
__device__ __forceinline__ Cell64 cell64(const Mom64& m) {
  constexpr int D = Model<M>::D;
  const double a = c_mc[M].a;
  Cell64 c;
  c.rho = __dadd_rn(1.0, m.r);
  const double ir = 1.0 / c.rho;
  const double air = __dmul_rn(a, ir);
  const double ux = __dmul_rn(air, m.x), uy = __dmul_rn(air, m.y);
  const double uz = D == 3 ? __dmul_rn(air, m.z) : 0.0;
  double q = __fma_rn(ux, ux, __dmul_rn(uy, uy));
  if constexpr (D == 3) q = __fma_rn(uz, uz, q);
  // theta - 1 = ((E - D rho) / rho - |u|^2) / D
  const double t = over_dim64<D>(__fma_rn(__fma_rn(-(double)D, m.r, m.e), ir, -q));
  c.vx = __dmul_rn(a, ux);
  c.vy = __dmul_rn(a, uy);
  c.vz = D == 3 ? __dmul_rn(a, uz) : 0.0;
  c.rt = __dmul_rn(c.rho, t);
  c.tt = __dmul_rn(c.rt, t);
  const double K0m1 =
      __fma_rn(t, __fma_rn(t, 0.125 * D * (D + 2), __fma_rn(q, 0.25 * (D + 2), -0.5 * D)),
               __dmul_rn(q, __fma_rn(q, 0.125, -0.5)));
  c.P0 = __fma_rn(c.rho, K0m1, m.r);
  c.K1 = __dmul_rn(c.rt, __fma_rn(t, -0.25 * (D + 2), __fma_rn(q, -0.25, 0.5)));
  c.L0 = __fma_rn(c.rt, -0.5 * (D + 2), __dmul_rn(c.rho, __fma_rn(q, -0.5, 1.0)));
  c.d2 = __dmul_rn(__dsub_rn(c.L0, c.rt), 0.5);
  c.r6 = over3_64<1>(c.rho);
  c.r24 = __dmul_rn(c.r6, 0.25);
  return c;
}

// h + omega (h^eq - h) of a pair's two members, h^eq = ev +- od: in fixed point at the
// scale of the largest of the four terms (about 160 integer instructions for six at the FP64
// rate); om is omega in units of 2^-62.  The error is at most six units of 2^-60 of that
// term's power of two (five from the terms' truncation, half a one from the product),
// against omega 2^-53 of it in FP64; a smaller omega than 2^-6 (0 must return h as it is)
// keeps the FP64 operations (tested on om: an FP64 comparison would cost as much as an
// addition).
struct Two64 {
  double p, m;
};
static __device__ __noinline__ Two64 relax_pair_any(double ev, double od, double hp, double hm,
                                                    double omega) {
  return {__fma_rn(omega, __dsub_rn(__dadd_rn(ev, od), hp), hp),
          __fma_rn(omega, __dsub_rn(__dsub_rn(ev, od), hm), hm)};
}
static __device__ __noinline__ Two64 relax_pair64(double ev, double od, double hp, double hm,
                                              double omega, long long om) {
  const int top = max(max(fx_top(ev), fx_top(od)), max(fx_top(hp), fx_top(hm)));
  if (!fx_regular(top) || om < (1ll << 56)) return relax_pair_any(ev, od, hp, hm, omega);
  const int e = fx_exponent(top);
  const long long v = fx_from<60>(ev, e), o = fx_from<60>(od, e);
  const long long p = fx_from<60>(hp, e), m = fx_from<60>(hm, e);
  // |v + o - p| < 3 2^60; times omega < 2: below 6 2^60
  return {fx_to<60>(p + fx_mul(v + o - p, om), e), fx_to<60>(m + fx_mul(v - o - m, om), e)};
}

template <int K>
__device__ __forceinline__ double times64(double v) {
  if constexpr (K == 1) return v; else return __dmul_rn((double)K, v);
}

// The relaxation h' = h + omega (h^eq - h) of one part's pairs.
template <int M, int P, class Get, class Store>
__device__ __forceinline__ void relax64(const Cell64& c, double omega, Get&& hv, Store&& st) {
  using T = P64<M, P>;
  const ModelConst& mc = c_mc[M];
  const long long om = fx_from<63>(omega, 1023);   // omega < 2 = 2^(1023 - 1022)
  double s = 0.0, s2 = 0.0;
  sfor<0, T::t.n>([&](auto I) {
    constexpr int n = decltype(I)::value;
    constexpr int g = T::t.grp[n], k = T::t.k[n], i = T::t.dir[n];
    if constexpr (T::new_base(n)) {
      s = edot<double, T::t.b[n][0], T::t.b[n][1], T::t.b[n][2]>(c.vx, c.vy, c.vz);
      s2 = __dmul_rn(s, s);
    }
    // the shell's coefficients: the same expressions for each of its pairs, which the
    // compiler forms once
    const double c0 = __fma_rn(mc.X2[g], __fma_rn(mc.X2o8[g], c.tt, c.K1), c.P0);
    const double c1 = times64<k>(__fma_rn(mc.X2o2[g], c.rt, c.L0));
    const double c2 = times64<k * k>(__fma_rn(mc.X2o4[g], c.rt, c.d2));
    const double c3 = times64<k * k * k>(c.r6);
    const double c4 = times64<k * k * k * k>(c.r24);
    const double ev = __fma_rn(s2, __fma_rn(s2, c4, c2), c0);
    const double od = __dmul_rn(s, __fma_rn(s2, c3, c1));
    const double hp = hv(std::integral_constant<int, i>{});
    const double hm = hv(std::integral_constant<int, i + 1>{});
    const Two64 r = relax_pair64(ev, od, hp, hm, omega, om);
    st(std::integral_constant<int, i>{}, r.p);
    st(std::integral_constant<int, i + 1>{}, r.m);
  });
}

// The four parts' sums and the rest direction (deviation h0).
template <int M>
__device__ __forceinline__ Mom64 total64(const Mom64& p01, const Mom64& p23, double h0) {
  Mom64 m = add64<M>(p01, p23);
  m.r = __fma_rn(c_mc[M].W[0], h0, m.r);
  return m;
}
__device__ __forceinline__ double relax_rest64(const Cell64& c, double omega, double h0) {
  return __fma_rn(omega, __dsub_rn(c.P0, h0), h0);
}

// a3 - a6 of one cell by one thread: hm(I) / hr(I) return direction I's population for
// the moments and for the relaxation (the same values; a kernel may read them again).
template <int M, class GetM, class GetR, class Store>
__device__ __forceinline__ void collide64(GetM&& hm, GetR&& hr, double omega, Store&& st) {
  constexpr std::integral_constant<int, 0> rest{};
  const Mom64 p0 = moments64<M, 0>(hm), p1 = moments64<M, 1>(hm);
  const Mom64 p01 = add64<M>(p0, p1);
  const Mom64 p2 = moments64<M, 2>(hm), p3 = moments64<M, 3>(hm);
  const Cell64 c = cell64<M>(total64<M>(p01, add64<M>(p2, p3), hm(rest)));
  st(rest, relax_rest64(c, omega, hr(rest)));
  relax64<M, 0>(c, omega, hr, st);
  relax64<M, 1>(c, omega, hr, st);
  relax64<M, 2>(c, omega, hr, st);
  relax64<M, 3>(c, omega, hr, st);
}

}  // namespace lbm
