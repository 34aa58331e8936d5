// contract.cuh - the contraction of adjoint populations lambda with the derivatives of the
// equilibrium, in FP64 or in double-float (FF) on the FP32 pipe.  Included by
// adjoint_kernels.cuh.
//
// Needed are, with f_i^eq = w_i rho P(s_i; q, t) (the polynomial of the file header of
// kernels.cuh),
//   Lr = sum w lambda P,  Sq = sum w lambda dP/dq,  St = sum w lambda dP/dt,
//   V = sum w lambda dP/ds e.
// On a shell A0, A1, A2 are polynomials in x2 = |xi|^2, and along a primitive vector b the
// pairs k b of several shells have x2 = beta k^2 with one beta, so lambda enters a
// direction b only through four sums over k (ls, ld the pair's sum and difference):
//   b0 = sum W k^2 ls, d = sum W k^4 ls, c0 = sum W k ld, e = sum W k^3 ld,
// and the s-independent terms through the shell totals of ls.  The polynomial work is then
// done once per primitive vector (25 for the 47 pairs of D3Q95, 8 for D2Q33's 16), and
// the cell's q and t are applied once at the end:
//   S1c = sum s c0, S1e = sum s beta e, S2b = sum s^2 b0, S2d = sum s^2 beta d,
//   S3 = sum s^3 e, S4 = sum s^4 d.
// About 600 operations for a D3Q95 cell against 1900 pair by pair.
#pragma once

namespace lbm {

// Arithmetic of the two number types (double-float not renormalised between operations).
__device__ __forceinline__ double nadd(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ double nsub(double a, double b) { return __dsub_rn(a, b); }
__device__ __forceinline__ double nmul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ double nfma(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ FF nadd(FF a, FF b) { return fu_add(a, b); }
__device__ __forceinline__ FF nsub(FF a, FF b) { return fu_add(a, ff_neg(b)); }
__device__ __forceinline__ FF nmul(FF a, FF b) { return fu_mul(a, b); }
__device__ __forceinline__ FF nfma(FF a, FF b, FF c) { return fu_add(c, fu_mul(a, b)); }
// A compile-time constant; its double-float form is the exact split.
template <class R>
__device__ __forceinline__ R ncst(double v) {
  if constexpr (std::is_same<R, FF>::value) {
    const float h = (float)v;
    return FF{h, (float)(v - (double)h)};
  } else {
    return v;
  }
}
// K v for a small integer, and acc + K v
template <int K, class R>
__device__ __forceinline__ R nscale(R v) {
  if constexpr (K == 1) return v;
  else if constexpr (std::is_same<R, FF>::value) return fu_scale<K>(v);
  else return K == -1 ? -v : __dmul_rn((double)K, v);
}
template <int K, class R>
__device__ __forceinline__ R naxpy(R v, R acc) {
  if constexpr (std::is_same<R, FF>::value) return fu_add(acc, fu_scale<K>(v));
  else return xaxpy<K>(v, acc);
}
template <int EX, int EY, int EZ, class R>
__device__ __forceinline__ R ndot(R x, R y, R z) {
  if constexpr (std::is_same<R, FF>::value) return ff_edot<EX, EY, EZ>(x, y, z);
  else return edot<double, EX, EY, EZ>(x, y, z);
}
// Weights of shell g: W, W x2, W x2^2, and W k^m (m = 1 .. 4).
template <class R>
struct ShellW {
  static __device__ __forceinline__ R W(const ModelConst& mc, int g) {
    if constexpr (std::is_same<R, FF>::value) return FF{mc.Wf[g], mc.Wlo[g]}; else return mc.W[g];
  }
  static __device__ __forceinline__ R WX2(const ModelConst& mc, int g) {
    if constexpr (std::is_same<R, FF>::value) return FF{mc.WX2f[g], mc.WX2lo[g]}; else return mc.WX2[g];
  }
  static __device__ __forceinline__ R WX4(const ModelConst& mc, int g) {
    if constexpr (std::is_same<R, FF>::value) return FF{mc.WX4f[g], mc.WX4lo[g]}; else return mc.WX4[g];
  }
  // W k^m v (and acc + W k^m v): from the table w[g] = W k^m in FP64; from v = W v0 times
  // the integer KM = k^m in double-float
  template <int KM>
  static __device__ __forceinline__ R first(const double* w, int g, R v) {
    if constexpr (std::is_same<R, FF>::value) return nscale<KM>(v); else return __dmul_rn(w[g], v);
  }
  template <int KM>
  static __device__ __forceinline__ R more(const double* w, int g, R v, R acc) {
    if constexpr (std::is_same<R, FF>::value) return naxpy<KM>(v, acc); else return __fma_rn(w[g], v, acc);
  }
};

template <class R>
struct Contraction {
  R a0, x2, x4;                  // sum W ls, sum W x2 ls, sum W x2^2 ls over the shells
  R S1c, S1e, S2b, S2d, S3, S4;
  R Vx, Vy, Vz;
};
// The cell's coefficients V needs (EqCoef): L0, L1, M0, M1, and a^2.
template <class R>
struct ContractCell {
  R vx, vy, vz;                  // a u: s = b . v
  R L0, L1, M0x2, M1x2;          // M0x2 = 2 M0, M1x2 = 2 M1
  R aa;                          // a^2: beta = a^2 |b|^2
};

// The pairs of list T (a P64): lam(i) is lambda of direction i.
template <int M, class T, class R, class Lam>
__device__ __forceinline__ Contraction<R> contract(const ContractCell<R>& c, Lam&& lam) {
  constexpr int D = Model<M>::D;
  constexpr bool kScale = std::is_same<R, FF>::value;
  const ModelConst& mc = c_mc[M];
  const R zero = ncst<R>(0.0);
  Contraction<R> o = {zero, zero, zero, zero, zero, zero, zero, zero, zero, zero, zero, zero};
  R shell[Model<M>::G];
  R b0 = zero, d = zero, c0 = zero, e = zero;
  sfor<0, T::t.n>([&](auto I) {
    constexpr int n = decltype(I)::value;
    constexpr int g = T::t.grp[n], i = T::t.dir[n], k = T::t.k[n];
    constexpr int bx = T::t.b[n][0], by = T::t.b[n][1], bz = T::t.b[n][2];
    constexpr bool only = T::new_base(n) && T::end_base(n);
    const R lp = lam(std::integral_constant<int, i>{});
    const R lm = lam(std::integral_constant<int, i + 1>{});
    const R ls = nadd(lp, lm), ld = nsub(lp, lm);
    shell[g] = T::first_of(n) ? ls : nadd(shell[g], ls);
    if constexpr (T::last_of(n)) {
      o.a0 = nfma(ShellW<R>::W(mc, g), shell[g], o.a0);
      o.x2 = nfma(ShellW<R>::WX2(mc, g), shell[g], o.x2);
      o.x4 = nfma(ShellW<R>::WX4(mc, g), shell[g], o.x4);
    }
    // double-float: one product by W, scaled exactly; FP64: the weights hold k^m
    const R ws = kScale ? nmul(ShellW<R>::W(mc, g), ls) : ls, wd = kScale ? nmul(ShellW<R>::W(mc, g), ld) : ld;
    if constexpr (T::new_base(n)) {
      b0 = ShellW<R>::template first<k * k>(mc.Wk2, g, ws);
      d = only && k == 1 ? b0 : ShellW<R>::template first<k * k * k * k>(mc.Wk4, g, ws);
      c0 = ShellW<R>::template first<k>(mc.Wk, g, wd);
      e = only && k == 1 ? c0 : ShellW<R>::template first<k * k * k>(mc.Wk3, g, wd);
    } else {
      b0 = ShellW<R>::template more<k * k>(mc.Wk2, g, ws, b0);
      d = ShellW<R>::template more<k * k * k * k>(mc.Wk4, g, ws, d);
      c0 = ShellW<R>::template more<k>(mc.Wk, g, wd, c0);
      e = ShellW<R>::template more<k * k * k>(mc.Wk3, g, wd, e);
    }
    if constexpr (T::end_base(n)) {
      constexpr double b2 = bx * bx + by * by + bz * bz;
      const R beta = nmul(ncst<R>(b2), c.aa);
      const R s = ndot<bx, by, bz>(c.vx, c.vy, c.vz);
      const R s2 = nmul(s, s);
      const R se = nmul(s, e), sd = nmul(s2, d);
      o.S1c = nfma(s, c0, o.S1c);
      o.S1e = nfma(beta, se, o.S1e);
      o.S2b = nfma(s2, b0, o.S2b);
      o.S2d = nfma(beta, sd, o.S2d);
      o.S3 = nfma(s2, se, o.S3);
      o.S4 = nfma(s2, sd, o.S4);
      const R ve = nfma(e, nfma(s2, ncst<R>(0.5), nmul(beta, c.L1)), nmul(c0, c.L0));
      const R vo = nfma(d, nfma(s2, ncst<R>(1.0 / 6.0), nmul(beta, c.M1x2)), nmul(b0, c.M0x2));
      const R v = nfma(s, vo, ve);
      if constexpr (bx != 0) o.Vx = naxpy<bx>(v, o.Vx);
      if constexpr (by != 0) o.Vy = naxpy<by>(v, o.Vy);
      if constexpr (D == 3 && bz != 0) o.Vz = naxpy<bz>(v, o.Vz);
    }
  });
  return o;
}

// Lr, Sq and St of the sums (the rest direction's W lambda already in a0).
template <int D, class R>
__device__ __forceinline__ void contract_finish(const Contraction<R>& o, R q, R t, R L0, R L1, R M0,
                                                R M1, R& Lr, R& Sq, R& St) {
  // A0 = K0 + x2 K1 + x2^2 K2 (EqCoef)
  const R hq = nmul(ncst<R>(0.25), q), ht = nmul(ncst<R>(0.25), t);
  const R K0m1 = nadd(nmul(t, nadd(nadd(nmul(ncst<R>(0.125 * D * (D + 2)), t),
                                        nmul(ncst<R>(D + 2.0), hq)), ncst<R>(-0.5 * D))),
                      nmul(q, nadd(nmul(ncst<R>(0.5), hq), ncst<R>(-0.5))));
  const R K1 = nmul(t, nsub(nsub(ncst<R>(0.5), hq), nmul(ncst<R>(D + 2.0), ht)));
  const R K2 = nmul(ncst<R>(0.5), nmul(t, ht));
  Lr = nadd(o.a0, nmul(K0m1, o.a0));
  Lr = nfma(K1, o.x2, Lr);
  Lr = nfma(K2, o.x4, Lr);
  Lr = nfma(M0, o.S2b, Lr);
  Lr = nfma(M1, o.S2d, Lr);
  Lr = nfma(L0, o.S1c, Lr);
  Lr = nfma(L1, o.S1e, Lr);
  Lr = nfma(ncst<R>(1.0 / 24.0), o.S4, Lr);
  Lr = nfma(ncst<R>(1.0 / 6.0), o.S3, Lr);
  // dP/dq = -1/2 + q/4 + t (D + 2 - x2)/4 - s/2 - s^2/4
  Sq = nmul(o.a0, nadd(nadd(ncst<R>(-0.5), hq), nmul(ncst<R>(D + 2.0), ht)));
  Sq = nsub(Sq, nmul(ht, o.x2));
  Sq = nfma(ncst<R>(-0.5), o.S1c, Sq);
  Sq = nfma(ncst<R>(-0.25), o.S2b, Sq);
  // dP/dt = (x2 - D)/2 + (D+2-x2) q/4 + t (x2^2 - 2(D+2) x2 + D(D+2))/4
  //         + s (x2-D-2)/2 + s^2 (x2-D-4)/4
  St = nmul(o.a0, nadd(nadd(ncst<R>(-0.5 * D), nmul(ncst<R>(D + 2.0), hq)),
                       nmul(ncst<R>(D * (D + 2.0)), ht)));
  St = nfma(o.x2, nsub(nsub(ncst<R>(0.5), hq), nmul(ncst<R>(2.0 * (D + 2)), ht)), St);
  St = nfma(ht, o.x4, St);
  St = nfma(ncst<R>(0.25), nfma(ncst<R>(-(D + 4.0)), o.S2b, o.S2d), St);
  St = nfma(ncst<R>(0.5), nfma(ncst<R>(-(D + 2.0)), o.S1c, o.S1e), St);
}

}  // namespace lbm
