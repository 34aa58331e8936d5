// adjoint_kernels.cuh - sm_103a kernels of the discrete adjoint (templates).
//
// Included by k_storage.inl after kernels.cuh (which supplies the model table,
// codecs, equilibrium coefficients and helpers).
#pragma once

#include "kernels.cuh"
#include "contract.cuh"

namespace lbm {

// ----------------------------------------------------------------- adjoint
// Discrete adjoint of one pull stream-collide step (exact transpose; k_adjoint in FP32 for
// the FP32, FP16 and BF16 forms, k_adjoint64 for the FP64 form).  Variables are derivatives with respect to the
// physical populations f.  With nu_n(x, j) = dL/dg^(n)_j(x) for the populations
// gathered by step n and lambda_{n+1}(x, i) = dL/dS_{n+1}(x, i) = nu_{n+1}(x + e_i, i):
//   nu_n(x, j) = (1 - omega) lambda_j + omega (alpha + beta . xi_j + gamma |xi_j|^2)
// because f^eq depends on g only through M = (rho, j, E) with dM/dg_j = (1, xi_j, |xi_j|^2)
// (the collision Jacobian has rank D + 2 beyond its diagonal).  alpha, beta,
// gamma = sum_i lambda_i d f_i^eq / dM, through f_i^eq = w_i rho P(s_i; q, t):
//   dP/ds = A1 + 2 A2 s + s^2/2 + s^3/6
//   dP/dq = Bq - s/2 - s^2/4,            Bq = -1/2 + q/4 + t (D+2-x2)/4
//   dP/dt = Bt + Ct s + Dt s^2,          Bt = (x2-D)/2 + (D+2-x2) q/4 + t (x2^2 - 2(D+2) x2 + D(D+2))/4
//                                        Ct = (x2-D-2)/2, Dt = (x2-D-4)/4
// and the chain rule from (rho, u, theta) to M:
//   d u/d rho = -u/rho, d u/d j = 1/rho, d theta/d rho = (q - D theta)/(D rho),
//   d theta/d j = -2 u/(D rho), d theta/d E = 1/(D rho).
// dL/domega of the step is sum_i lambda_i (f_i^eq - g_i) = rho Lrho - sum_i lambda_i w_i (1 + h_i).
template <class R, int D>
struct EqGrad {
  R q, t;
  __device__ __forceinline__ EqGrad(R q_, R t_) : q(q_), t(t_) {}
  __device__ __forceinline__ R Bq(R x2) const {
    return R(-0.5) + q * R(0.25) + t * (R(D + 2) - x2) * R(0.25);
  }
  __device__ __forceinline__ R Bt(R x2) const {
    return (x2 - R(D)) * R(0.5) + (R(D + 2) - x2) * q * R(0.25) +
           t * (x2 * x2 - R(2 * (D + 2)) * x2 + R(D * (D + 2))) * R(0.25);
  }
  static __device__ __forceinline__ R Ct(R x2) { return (x2 - R(D + 2)) * R(0.5); }
  static __device__ __forceinline__ R Dt(R x2) { return (x2 - R(D + 4)) * R(0.25); }
};


__device__ __forceinline__ double block_sum_128(double v, double* sh) {
  v = warp_sum(v);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (lane == 0) sh[wid] = v;
  __syncthreads();
  double r = 0;
  if (threadIdx.x == 0)
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) r += sh[w];
  return r;
}

#ifndef LBM_ADJ_MINB
#define LBM_ADJ_MINB 4
#endif
// The FP32 adjoint commits its lambda copies in this many groups and waits for each
// just before pass 1 needs it, so the later groups' latency overlaps pass 1 (1.75
// adjoint steps per forward step against 1.78 with one wait for all; 2, 3 or 6
// groups measured 1.76).
// Unroll factor of the shell loops of passes 2 and 3 (1.74 adjoint steps per forward
// step at 2, 1.75 at 1, 1.78 at 3).
#ifndef LBM_ADJ_UNROLL
#define LBM_ADJ_UNROLL 2
#endif
constexpr int kAdjUnroll = LBM_ADJ_UNROLL;
#ifndef LBM_ADJ_GROUPS
#define LBM_ADJ_GROUPS 4
#endif
// The Q gathered lambda_i of a thread live in dynamic shared memory (lambda_i of thread t at
// word i * 128 + t: conflict-free), which leaves the registers to the gather offsets and the
// sums (Q floats in registers on top of them spill at 128 registers a thread).
constexpr int kAdjThreads = 128;
template <int M, class L>
constexpr int adj_smem_bytes() {
  return Model<M>::Q * kAdjThreads * (int)sizeof(L);
}
// Address of population i at a cell: the element index in 32 bits when every index
// of a state copy fits them (NARROW), which saves the per-population 64-bit offset
// arithmetic; else the population's array first, then the cell.  (A macro: passed
// through a helper function, the 64-bit form compiled to a different register
// allocation, 168 registers with spills against 128 without.)
#define LBM_POP(base, i, cell)                                                                \
  (NARROW ? (base) + (uint32_t)((uint32_t)(i) * (uint32_t)g.ncell + (uint32_t)(cell))         \
          : (base) + (size_t)(i) * g.ncell + (cell))
template <int M, class S, class L, bool kFirst, bool NARROW>
__global__ void __launch_bounds__(kAdjThreads, LBM_ADJ_MINB)
    k_adjoint(const S* __restrict__ state, const L* __restrict__ nu_next,
              const double* __restrict__ dldrho, L* __restrict__ nu_out,
              double* __restrict__ omega_acc, Grid g, double omega) {
  using Mo = Model<M>;
  using Rt = L;
  static_assert(std::is_same<L, float>::value, "the FP64 form has k_adjoint64");
  constexpr int D = Mo::D, RR = Mo::R, NP = Mo::NP;
  // the lambda copies are committed in kGroups groups of kPerGroup pairs; pass 1
  // waits for each group just before its first pair
  constexpr int kGroups = LBM_ADJ_GROUPS;
  constexpr int kPerGroup = (NP + kGroups - 1) / kGroups;
  const ModelConst& mc = c_mc[M];
  __shared__ double sh[4];
  extern __shared__ __align__(16) unsigned char adj_dyn[];
  wait_prior_grid();     // programmatic launch: the previous step's writes are visible after this
  allow_next_grid();

  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  const int y = blockIdx.y, z = blockIdx.z;
  const bool active = x < g.nx;
  double om_part = 0.0;
  if (active) {
    int xo[2 * RR + 1], yo[2 * RR + 1], zo[2 * RR + 1];
    neighbour_offsets<D, RR>(x, y, z, g.nx, g.ny, g.nz, g.nxy, xo, yo, zo);
    const size_t self = ((size_t)z * g.ny + y) * g.nx + x;
    Rt l1 = Rt(0);
    if constexpr (kFirst) l1 = (Rt)dldrho[self];
    // lambda_i(x) = nu_next(x + e_i, i): one value per direction for the first step
    // of the sweep (dL/drho_N, the same for every i), else gathered.
    const Rt* const lam_s = reinterpret_cast<const Rt*>(adj_dyn) + threadIdx.x;
    auto lam = [&](int i) -> Rt {
      if constexpr (kFirst) return l1;
      else return lam_s[i * kAdjThreads];
    };
    if constexpr (!kFirst) {
      // FP32: the lambda gather goes global -> shared by cp.async, which holds no
      // registers while in flight; each thread waits for its own copies only.
      Rt* const dst = reinterpret_cast<Rt*>(adj_dyn) + threadIdx.x;
      cp_async4(dst, nu_next + self);
      sfor<0, NP>([&](auto P) {
        constexpr int p = decltype(P)::value;
        constexpr int ip = 1 + 2 * p, im = 2 + 2 * p;
        constexpr int ex = Mo::vs.e[ip][0], ey = Mo::vs.e[ip][1], ez = Mo::vs.e[ip][2];
        const int cm = zo[ez + RR] + yo[ey + RR] + xo[ex + RR];   // x - e_ip
        const int cp = zo[RR - ez] + yo[RR - ey] + xo[RR - ex];   // x + e_ip
        cp_async4(dst + ip * kAdjThreads, LBM_POP(nu_next, ip, cp));
        cp_async4(dst + im * kAdjThreads, LBM_POP(nu_next, im, cm));
        if constexpr (kGroups > 1 && (p % kPerGroup == kPerGroup - 1 || p + 1 == NP))
          cp_async_commit();
      });
      if constexpr (kGroups <= 1) cp_async_wait_all();
    }
    // pass 1: forward moments of g (gathered from x - e_i) and sum lambda_i f_i
    Rt rs, es = Rt(0), jx = Rt(0), jy = Rt(0), jz = Rt(0), sg;
    {
      const Rt h0 = (Rt)Codec<S>::ld(state + self);
      if constexpr (!kFirst && kGroups > 1) cp_async_wait_group<kGroups - 1>();
      rs = gW<Rt>(mc, 0) * h0;
      sg = gW<Rt>(mc, 0) * lam(0) * (Rt(1) + h0);
    }
    // Shell by shell: the weight and |xi|^2 are common to a shell, so the pair
    // terms are summed unweighted and each shell's totals are weighted once.
    Rt gs = Rt(0), gjx = Rt(0), gjy = Rt(0), gjz = Rt(0), gsg = Rt(0);
    sfor<0, NP>([&](auto P) {
      constexpr int p = decltype(P)::value;
      constexpr int ip = 1 + 2 * p, im = 2 + 2 * p;
      constexpr int gg = Mo::vs.grp[ip];
      constexpr int ex = Mo::vs.e[ip][0], ey = Mo::vs.e[ip][1], ez = Mo::vs.e[ip][2];
      constexpr bool first = (p == 0) || (Mo::vs.grp[ip - 2] != gg);
      constexpr bool last = (p + 1 == NP) || (Mo::vs.grp[ip + 2] != gg);
      if constexpr (!kFirst && kGroups > 1 && p > 0 && p % kPerGroup == 0)
        cp_async_wait_group<kGroups - 1 - p / kPerGroup>();
      const int cm = zo[ez + RR] + yo[ey + RR] + xo[ex + RR];   // x - e_ip
      const int cp = zo[RR - ez] + yo[RR - ey] + xo[RR - ex];   // x + e_ip
      const Rt hp = (Rt)Codec<S>::ld(LBM_POP(state, ip, cm));
      const Rt hm = (Rt)Codec<S>::ld(LBM_POP(state, im, cp));
      if constexpr (first) gs = gjx = gjy = gjz = gsg = Rt(0);
      const Rt sp = hp + hm, dm = hp - hm;
      gs += sp;
      if constexpr (ex != 0) gjx += Rt(ex) * dm;
      if constexpr (ey != 0) gjy += Rt(ey) * dm;
      if constexpr (ez != 0) gjz += Rt(ez) * dm;
      const Rt lp = lam(ip), lm = lam(im);
      gsg += lp * hp + lm * hm + (lp + lm);               // lambda_p f_p / w + lambda_m f_m / w
      if constexpr (last) {
        const Rt w = gW<Rt>(mc, gg);
        const Rt tr = w * gs;
        rs += tr;
        es += gX2<Rt>(mc, gg) * tr;
        jx += w * gjx;
        jy += w * gjy;
        jz += w * gjz;
        sg += w * gsg;
      }
    });
    // Linearisation point: the forward moments and temperature of g.  Plain sums in
    // the arithmetic type suffice here (they fix where the Jacobian is taken, to
    // ~1e-7 relative in FP32; the gradients are compared at 1e-4).
    const Rt rho_r = Rt(1) + rs;
    const Rt ir_r = __fdividef(1.0f, rho_r);
    const double rho_d = (double)rho_r;
    const Rt ux = gA<Rt>(mc) * jx * ir_r;
    const Rt uy = gA<Rt>(mc) * jy * ir_r;
    const Rt uz = (D == 3) ? gA<Rt>(mc) * jz * ir_r : Rt(0);
    const Rt q = ux * ux + uy * uy + uz * uz;
    const Rt t = ((es - Rt(D) * rs) * ir_r - q) * Rt(1.0 / D);
    const Rt theta = Rt(1) + t;
    const EqCoef<Rt, D> cf(q, t);
    const EqGrad<Rt, D> gr(q, t);
    const Rt a_r = gA<Rt>(mc);
    const Rt uax = a_r * ux, uay = a_r * uy, uaz = a_r * uz;

    // pass 2: contractions with lambda
    Rt Lr = gW<Rt>(mc, 0) * lam(0) * cf.K0;
    Rt Sq = gW<Rt>(mc, 0) * lam(0) * gr.Bq(Rt(0));
    Rt St = gW<Rt>(mc, 0) * lam(0) * gr.Bt(Rt(0));
    Rt Vx = Rt(0), Vy = Rt(0), Vz = Rt(0);
    // Per shell, with ls = lambda_p + lambda_m, ld = lambda_p - lambda_m and s = xi_p . u:
    //   sum ls P = A0 m0 + A2 m2 + m4 / 24 + A1 n1 + n3 / 6,
    //   sum ls dP/dq = Bq m0 - m2 / 4 - n1 / 2,  sum ls dP/dt = Bt m0 + Dt m2 + Ct n1,
    // with m0 = sum ls, m2 = sum ls s^2, m4 = sum ls s^4, n1 = sum ld s, n3 = sum ld s^3;
    // the vector term keeps one v = ld (A1 + s^2/2) + ls s (2 A2 + s^2/6) per pair.
    Rt m0 = Rt(0), m2 = Rt(0), m4 = Rt(0), n1 = Rt(0), n3 = Rt(0);
    Rt gvx = Rt(0), gvy = Rt(0), gvz = Rt(0);
    // Passes 2 and 3 loop over each shell's pairs (lattice vectors from constant memory):
    // unrolled over all pairs the kernel outgrows the instruction cache.
    sfor<1, Mo::G>([&](auto Gi) {
      constexpr int gg = decltype(Gi)::value;
      const Rt x2 = gX2<Rt>(mc, gg);
      const Rt A1 = cf.A1(x2), A2 = cf.A2(x2);
      m0 = m2 = m4 = n1 = n3 = gvx = gvy = gvz = Rt(0);
#pragma unroll kAdjUnroll
      for (int p = ShellPairs<M>::first(gg); p < ShellPairs<M>::end(gg); ++p) {
        const int ip = 1 + 2 * p, im = 2 + 2 * p;
        const Rt ex = mc.ef[ip][0], ey = mc.ef[ip][1], ez = mc.ef[ip][2];
        const Rt s = ex * uax + ey * uay + ez * uaz;
        const Rt s2 = s * s;
        const Rt lp = lam(ip), lm = lam(im);
        const Rt ls = lp + lm, ld = lp - lm;
        const Rt tl = ls * s2, tu = ld * s;
        m0 += ls;
        m2 += tl;
        m4 += tl * s2;
        n1 += tu;
        n3 += tu * s2;
        const Rt v = ld * (A1 + s2 * Rt(0.5)) + (ls * s) * (Rt(2) * A2 + s2 * Rt(1.0 / 6.0));
        gvx += ex * v;
        gvy += ey * v;
        gvz += ez * v;
      }
      const Rt w = gW<Rt>(mc, gg);
      Lr += w * (cf.A0(x2) * m0 + A2 * m2 + m4 * Rt(1.0 / 24.0) + A1 * n1 + n3 * Rt(1.0 / 6.0));
      Sq += w * (gr.Bq(x2) * m0 - m2 * Rt(0.25) - n1 * Rt(0.5));
      St += w * (gr.Bt(x2) * m0 + EqGrad<Rt, D>::Dt(x2) * m2 + EqGrad<Rt, D>::Ct(x2) * n1);
      Vx += w * gvx;
      Vy += w * gvy;
      Vz += w * gvz;
    });
    // chain rule to the moments (arithmetic type; the omega term in FP64)
    const Rt Lux = rho_r * (a_r * Vx + Rt(2) * ux * Sq);
    const Rt Luy = rho_r * (a_r * Vy + Rt(2) * uy * Sq);
    const Rt Luz = (D == 3) ? rho_r * (a_r * Vz + Rt(2) * uz * Sq) : Rt(0);
    const Rt Lt = rho_r * St;
    const Rt iDr = ir_r * Rt(1.0 / D);
    const Rt alpha = Lr - (ux * Lux + uy * Luy + uz * Luz) * ir_r + Lt * (q - Rt(D) * theta) * iDr;
    const Rt bx = Lux * ir_r - Rt(2) * Lt * ux * iDr;
    const Rt by = Luy * ir_r - Rt(2) * Lt * uy * iDr;
    const Rt bz = Luz * ir_r - Rt(2) * Lt * uz * iDr;
    const Rt gam = Lt * iDr;
    om_part = fma(rho_d, (double)Lr, -(double)sg);

    // pass 3: nu_n(x, j)
    const Rt om1 = (Rt)(1.0 - omega);
    const Rt om = (Rt)omega;
    const Rt oa = om * alpha, og = om * gam;
    const Rt obx = om * a_r * bx, oby = om * a_r * by, obz = om * a_r * bz;
    nu_out[self] = om1 * lam(0) + oa;
    sfor<1, Mo::G>([&](auto Gi) {
      constexpr int gg = decltype(Gi)::value;
      const Rt ev = oa + og * gX2<Rt>(mc, gg);
#pragma unroll kAdjUnroll
      for (int p = ShellPairs<M>::first(gg); p < ShellPairs<M>::end(gg); ++p) {
        const int ip = 1 + 2 * p, im = 2 + 2 * p;
        const Rt od = mc.ef[ip][0] * obx + mc.ef[ip][1] * oby + mc.ef[ip][2] * obz;
        *LBM_POP(nu_out, ip, self) = om1 * lam(ip) + (ev + od);
        *LBM_POP(nu_out, im, self) = om1 * lam(im) + (ev - od);
      }
    });
  }
  const double bsum = block_sum_128(om_part, sh);
  if (threadIdx.x == 0) {
    const size_t b = ((size_t)blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
    omega_acc[b] += bsum;
  }
}

#undef LBM_POP

// The adjoint step of the FP64 form: the same derivatives as k_adjoint with the FP64
// instructions counted (see collide64.cuh and contract.cuh): the forward moments shell by
// shell, the contractions once per primitive vector; ~600 FP64 operations a D2Q33 cell
// against ~900 pair by pair.  Linear cell index, 32 cells per block, shared by WARPS = 1, 2
// or 4 warps as in k_stream_collide64; but a warp sums its own parts before the warps' sums
// meet, so the last bits of a gradient depend on WARPS (the forward step's do not).
template <int M, bool kFirst, int WARPS>
__global__ void __launch_bounds__(32 * WARPS, 8 / WARPS)
    k_adjoint64(const double* __restrict__ state, const double* __restrict__ nu_next,
                const double* __restrict__ dldrho, double* __restrict__ nu_out,
                double* __restrict__ omega_acc, Grid g, double omega) {
  using Mo = Model<M>;
  constexpr int D = Mo::D, RR = Mo::R, PW = kParts64 / WARPS;
  const ModelConst& mc = c_mc[M];
  wait_prior_grid();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const unsigned cell = blockIdx.x * 32u + lane;
  const bool active = cell < (unsigned)g.ncell;
  const unsigned at0 = active ? cell : 0;
  const unsigned row = at0 / (unsigned)g.nx;
  const int x = (int)(at0 - row * (unsigned)g.nx);
  const int z = D == 3 ? (int)(row / (unsigned)g.ny) : 0;
  const int y = (int)row - z * g.ny;
  int xo[2 * RR + 1], yo[2 * RR + 1], zo[2 * RR + 1];
  neighbour_offsets<D, RR>(x, y, z, g.nx, g.ny, g.nz, g.nxy, xo, yo, zo);
  const size_t nc = (size_t)g.ncell;
  auto hv = [&](auto I) {                  // gathered from x - e_i
    constexpr int i = decltype(I)::value;
    constexpr int ex = Mo::vs.e[i][0], ey = Mo::vs.e[i][1], ez = Mo::vs.e[i][2];
    return __ldg(state + (size_t)i * nc + (zo[ez + RR] + yo[ey + RR] + xo[ex + RR]));
  };
  const double l1 = kFirst ? dldrho[at0] : 0.0;
  // lambda_i = nu_next(x + e_i, i), used three times: kept in shared memory (each thread its
  // own copies, of its warp's directions)
  extern __shared__ __align__(16) double stage64[];
  double* const mine = stage64 + lane;
  if constexpr (!kFirst) {
    sfor<0, Mo::Q>([&](auto I) {
      constexpr int i = decltype(I)::value;
      constexpr int ex = Mo::vs.e[i][0], ey = Mo::vs.e[i][1], ez = Mo::vs.e[i][2];
      constexpr int p = i == 0 ? -1 : shell_part64<M>(Mo::vs.grp[i]);
      if (WARPS == 1 || i == 0 || p / PW == warp)
        cp_async8(mine + 32 * i, nu_next + (size_t)i * nc + (zo[RR - ez] + yo[RR - ey] + xo[RR - ex]));
    });
    cp_async_wait_all();
  }
  auto lam = [&](auto I) -> double {
    if constexpr (kFirst) return l1;
    else return mine[32 * decltype(I)::value];
  };
  __shared__ double xch[WARPS][7][32];
  // sums over the warps, in order; the value of warp w is in xch[w][k]
  auto total = [&](int k) {
    double v = xch[0][k][lane];
    for (int w = 1; w < WARPS; ++w) v = __dadd_rn(v, xch[w][k][lane]);
    return v;
  };

  // pass 1: forward moments, and sum w lambda h over the pairs
  Mom64 m = {};
  double lh = 0.0;
  auto dot = [&](auto Pi) {
    using T = P64<M, decltype(Pi)::value>;
    double gl[Mo::G];
    sfor<0, T::t.n>([&](auto I) {
      constexpr int n = decltype(I)::value, gg = T::t.grp[n], i = T::t.dir[n];
      constexpr std::integral_constant<int, i> ip{};
      constexpr std::integral_constant<int, i + 1> im{};
      const double p = T::first_of(n) ? __dmul_rn(lam(ip), hv(ip)) : __fma_rn(lam(ip), hv(ip), gl[gg]);
      gl[gg] = __fma_rn(lam(im), hv(im), p);
      if constexpr (T::last_of(n)) lh = __fma_rn(mc.W[gg], gl[gg], lh);
    });
  };
  auto pass1 = [&](auto Wi) {
    constexpr int p0 = decltype(Wi)::value * PW;
    m = moments64<M, p0>(hv);
    dot(std::integral_constant<int, p0>{});
    sfor<1, PW>([&](auto K) {
      constexpr int p = p0 + decltype(K)::value;
      m = add64<M>(m, moments64<M, p>(hv));
      dot(std::integral_constant<int, p>{});
    });
  };
  sfor<0, WARPS>([&](auto Wi) {
    if (warp == decltype(Wi)::value) pass1(Wi);
  });
  if constexpr (WARPS > 1) {
    xch[warp][0][lane] = m.r;
    xch[warp][1][lane] = m.e;
    xch[warp][2][lane] = m.x;
    xch[warp][3][lane] = m.y;
    xch[warp][4][lane] = m.z;
    xch[warp][5][lane] = lh;
    __syncthreads();
    m = {total(0), total(1), total(2), total(3), D == 3 ? total(4) : 0.0};
    lh = total(5);
    __syncthreads();
  }
  const double h0 = hv(std::integral_constant<int, 0>{}), lam0 = lam(std::integral_constant<int, 0>{});
  m.r = __fma_rn(mc.W[0], h0, m.r);
  const double rho = 1.0 + m.r, ir = 1.0 / rho, a = mc.a;
  const double ux = a * m.x * ir, uy = a * m.y * ir, uz = D == 3 ? a * m.z * ir : 0.0;
  const double q = ux * ux + uy * uy + uz * uz;
  const double t = ((m.e - D * m.r) * ir - q) * (1.0 / D);
  // EqCoef's L0, L1, M0, M1
  const double L1 = 0.5 * t, M1 = 0.25 * t;
  const double L0 = fma(t, -0.5 * (D + 2), fma(q, -0.5, 1.0));
  const double M0 = fma(t, -0.5, 0.5 * L0);

  // pass 2: contractions of lambda
  const ContractCell<double> cc = {a * ux, a * uy, a * uz, L0, L1, 2.0 * M0, L1, a * a};
  double s6[7] = {};                       // Lr, Sq, St, V, sum w lambda
  auto pass2 = [&](auto Pi) {
    constexpr int p = decltype(Pi)::value;
    Contraction<double> o = contract<M, P64<M, p>, double>(cc, lam);
    if constexpr (p == 0) o.a0 = __fma_rn(mc.W[0], lam0, o.a0);
    return o;
  };
  auto sum2 = [&](auto Wi) {
    constexpr int p0 = decltype(Wi)::value * PW;
    Contraction<double> o = pass2(std::integral_constant<int, p0>{});
    sfor<1, PW>([&](auto K) {
      const Contraction<double> w = pass2(std::integral_constant<int, p0 + decltype(K)::value>{});
      o = {o.a0 + w.a0, o.x2 + w.x2, o.x4 + w.x4, o.S1c + w.S1c, o.S1e + w.S1e, o.S2b + w.S2b,
           o.S2d + w.S2d, o.S3 + w.S3, o.S4 + w.S4, o.Vx + w.Vx, o.Vy + w.Vy, o.Vz + w.Vz};
    });
    contract_finish<D, double>(o, q, t, L0, L1, M0, M1, s6[0], s6[1], s6[2]);
    s6[3] = o.Vx;
    s6[4] = o.Vy;
    s6[5] = o.Vz;
    s6[6] = o.a0;
  };
  sfor<0, WARPS>([&](auto Wi) {
    if (warp == decltype(Wi)::value) sum2(Wi);
  });
  if constexpr (WARPS > 1) {
#pragma unroll
    for (int k = 0; k < 7; ++k) xch[warp][k][lane] = s6[k];
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 7; ++k) s6[k] = total(k);
  }
  const double Lr = s6[0], Sq = s6[1], St = s6[2], Vx = s6[3], Vy = s6[4], Vz = s6[5];
  // chain rule to the moments (as in k_adjoint)
  const double Lux = rho * (a * Vx + 2.0 * ux * Sq), Luy = rho * (a * Vy + 2.0 * uy * Sq);
  const double Luz = D == 3 ? rho * (a * Vz + 2.0 * uz * Sq) : 0.0;
  const double Lt = rho * St, iDr = ir * (1.0 / D);
  const double alpha = Lr - (ux * Lux + uy * Luy + uz * Luz) * ir + Lt * (q - D * (1.0 + t)) * iDr;
  const double bx = Lux * ir - 2.0 * Lt * ux * iDr, by = Luy * ir - 2.0 * Lt * uy * iDr;
  const double bz = Luz * ir - 2.0 * Lt * uz * iDr;
  const double gam = Lt * iDr;

  // pass 3: nu_n(x, j)
  const double om1 = 1.0 - omega;
  const double oa = omega * alpha, og = omega * gam, oma = omega * a;
  const double obx = oma * bx, oby = oma * by, obz = oma * bz;
  auto pass3 = [&](auto Pi) {
    using T = P64<M, decltype(Pi)::value>;
    double od = 0.0;
    sfor<0, T::t.n>([&](auto I) {
      constexpr int n = decltype(I)::value, i = T::t.dir[n], gg = T::t.grp[n], k = T::t.k[n];
      if constexpr (T::new_base(n))
        od = edot<double, T::t.b[n][0], T::t.b[n][1], T::t.b[n][2]>(obx, oby, obz);
      const double ev = __fma_rn(og, mc.X2[gg], oa);
      const double vp = __fma_rn((double)k, od, ev), vm = __fma_rn(-(double)k, od, ev);
      const double lp = lam(std::integral_constant<int, i>{});
      const double lm = lam(std::integral_constant<int, i + 1>{});
      if (active) {
        nu_out[(size_t)i * nc + cell] = __fma_rn(om1, lp, vp);
        nu_out[(size_t)(i + 1) * nc + cell] = __fma_rn(om1, lm, vm);
      }
    });
  };
  sfor<0, WARPS>([&](auto Wi) {
    constexpr int w = decltype(Wi)::value;
    if (warp == w) sfor<0, PW>([&](auto K) { pass3(std::integral_constant<int, w * PW + decltype(K)::value>{}); });
  });
  // The next step's blocks are let in only now: placed while this step's blocks still fill
  // part of the SMs they bunch up on the others, and one scheduler with two warps sets the
  // step's time (D3Q95 33 x 17 x 15: 65 us a step against 52, D2Q33 200 x 40: 29 against 24).
  allow_next_grid();
  if (warp == 0) {
    if (active) nu_out[cell] = __fma_rn(om1, lam0, oa);
    // dL/domega: rho Lr - sum w lambda (1 + h)
    const double om = rho * Lr - (s6[6] + __fma_rn(mc.W[0] * lam0, h0, lh));
    const double sum = warp_sum(active ? om : 0.0);
    if (lane == 0) omega_acc[blockIdx.x] += sum;
  }
}

// dL/d(rho0, U0, T0): lambda_0(x, i) = nu0(x + e_i, i) contracted with the derivatives of
// f_i^eq(rho, u, theta) at the initial fields: FP64 for the FP64 form; double-float on the
// FP32 pipe for the others, whose lambda is FP32 (~46 significant bits, against lambda's 24,
// which set the error of the gradients: their rms distance from the FP64 oracle's, 3e-8 to
// 1e-6, is the same to five digits with the contraction in FP64).  In FP64 the contraction is bound by the FP64 pipe (64 cycles an instruction and
// scheduler): 9.8 ms for 128^3 D3Q95 cells, as long as 22 adjoint steps.
template <int M, class L>
__global__ void __launch_bounds__(128)
    k_grad_init(const L* __restrict__ nu0, const double* __restrict__ fields,
                double* __restrict__ d_rho, double* __restrict__ d_U, double* __restrict__ d_T,
                Grid g) {
  using Mo = Model<M>;
  constexpr int D = Mo::D, RR = Mo::R;
  constexpr bool kFF = std::is_same<L, float>::value;
  using R = typename std::conditional<kFF, FF, double>::type;
  const ModelConst& mc = c_mc[M];
  const unsigned cell = blockIdx.x * blockDim.x + threadIdx.x;
  if (cell >= (unsigned)g.ncell) return;
  const unsigned row = cell / (unsigned)g.nx;
  const int x = (int)(cell - row * (unsigned)g.nx);
  const int z = D == 3 ? (int)(row / (unsigned)g.ny) : 0;
  const int y = (int)row - z * g.ny;
  int xo[2 * RR + 1], yo[2 * RR + 1], zo[2 * RR + 1];
  neighbour_offsets<D, RR>(x, y, z, g.nx, g.ny, g.nz, g.nxy, xo, yo, zo);
  const size_t n = (size_t)g.ncell;
  auto field = [&](int k) -> R {
    if constexpr (kFF) return ff_from(fields[k * n + cell]); else return fields[k * n + cell];
  };
  R a, iT0;
  if constexpr (kFF) { a = {mc.af, mc.alo}; iT0 = {mc.iT0f, mc.iT0lo}; }
  else { a = mc.a; iT0 = 1.0 / mc.T0; }
  const R rho = field(0);
  const R ux = nmul(a, field(1)), uy = nmul(a, field(2));
  const R uz = D == 3 ? nmul(a, field(3)) : ncst<R>(0.0);
  const R t = nadd(nmul(iT0, field(D + 1)), ncst<R>(-1.0));
  R q = nfma(ux, ux, nmul(uy, uy));
  if constexpr (D == 3) q = nfma(uz, uz, q);
  const R L1 = nmul(ncst<R>(0.5), t), M1 = nmul(ncst<R>(0.25), t);
  const R L0 = nsub(nsub(ncst<R>(1.0), nmul(ncst<R>(0.5), q)), nmul(ncst<R>(0.5 * (D + 2)), t));
  const R M0 = nmul(ncst<R>(0.5), nsub(L0, t));
  const ContractCell<R> cc = {nmul(a, ux), nmul(a, uy), nmul(a, uz), L0, L1, nsub(L0, t), L1, nmul(a, a)};
  auto lam = [&](auto I) -> R {
    constexpr int i = decltype(I)::value;
    constexpr int ex = Mo::vs.e[i][0], ey = Mo::vs.e[i][1], ez = Mo::vs.e[i][2];
    const L v = __ldg(nu0 + (size_t)i * n + (zo[RR - ez] + yo[RR - ey] + xo[RR - ex]));
    if constexpr (kFF) return FF{v, 0.f}; else return v;
  };
  Contraction<R> o = contract<M, P64<M, -1>, R>(cc, lam);
  o.a0 = nfma(ShellW<R>::W(mc, 0), lam(std::integral_constant<int, 0>{}), o.a0);
  R Lr, Sq, St;
  contract_finish<D, R>(o, q, t, L0, L1, M0, M1, Lr, Sq, St);
  auto put = [&](double* p, size_t at, R v) {
    if constexpr (kFF) p[at] = ff_to_double(v); else p[at] = v;
  };
  if (d_rho) put(d_rho, cell, Lr);
  if (d_U) {
    const R ar = nmul(a, rho), Sq2 = nmul(ncst<R>(2.0), Sq);
    put(d_U, cell, nmul(ar, nfma(a, o.Vx, nmul(ux, Sq2))));
    put(d_U, n + cell, nmul(ar, nfma(a, o.Vy, nmul(uy, Sq2))));
    if constexpr (D == 3) put(d_U, 2 * n + cell, nmul(ar, nfma(a, o.Vz, nmul(uz, Sq2))));
  }
  if (d_T) put(d_T, cell, nmul(nmul(rho, St), iT0));
}

// Fixed-order sum of n FP64 partials by one block of 256 threads.
static __global__ void __launch_bounds__(256) k_sum_reduce(const double* __restrict__ partials,
                                                           long long n, double* __restrict__ out) {
  double acc = 0;
  for (long long b = threadIdx.x; b < n; b += blockDim.x) acc += partials[b];
  __shared__ double sh[8];
  acc = warp_sum(acc);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double v = 0;
    for (int w = 0; w < 8; ++w) v += sh[w];
    *out = v;
  }
}

}  // namespace lbm
