// fixed64.cuh and collide64.cuh evaluated on the host: the device intrinsics they use, and
// entry points for ctypes (g++ -ffp-contract=off; see test_fixed64_host.py).
#include <algorithm>
#include <cmath>
#include <cstring>
#include <type_traits>
#include <utility>

#define __host__
#define __device__
#define __forceinline__ inline
#define __noinline__
#include "velset.cuh"

using std::max;
using std::min;
static inline long long __double_as_longlong(double d) {
  long long v;
  std::memcpy(&v, &d, 8);
  return v;
}
static inline double __longlong_as_double(long long v) {
  double d;
  std::memcpy(&d, &v, 8);
  return d;
}
static inline int __double2hiint(double d) { return (int)(__double_as_longlong(d) >> 32); }
static inline int __double2loint(double d) { return (int)__double_as_longlong(d); }
static inline unsigned __funnelshift_l(unsigned lo, unsigned hi, unsigned s) {
  return s ? (hi << s) | (lo >> (32 - s)) : hi;
}
static inline int __clzll(unsigned long long v) { return v ? __builtin_clzll(v) : 64; }
static inline double __dadd_rn(double a, double b) { return a + b; }
static inline double __dsub_rn(double a, double b) { return a - b; }
static inline double __dmul_rn(double a, double b) { return a * b; }
static inline double __fma_rn(double a, double b, double c) { return std::fma(a, b, c); }

namespace lbm {
// What collide64.cuh reads of the model tables (common.h has the whole).
struct ModelConst {
  double W[10], X2[10], X2o2[10], X2o4[10], X2o8[10], a;
};
static ModelConst c_mc[2];
template <int I, int N, class F>
inline void sfor(F&& f) {
  if constexpr (I < N) {
    f(std::integral_constant<int, I>{});
    sfor<I + 1, N>(f);
  }
}
template <class R, int EX, int EY, int EZ>
inline double edot(double x, double y, double z) {
  double s = EX * x;
  if constexpr (EY != 0) s = EX ? std::fma((double)EY, y, s) : EY * y;
  if constexpr (EZ != 0) s = EX || EY ? std::fma((double)EZ, z, s) : EZ * z;
  return s;
}
}  // namespace lbm

#include "collide64.cuh"

using namespace lbm;

template <int M>
static void collide(double* h, double omega) {
  double out[Model<M>::Q];
  auto hv = [&](auto I) { return h[decltype(I)::value]; };
  collide64<M>(hv, hv, omega, [&](auto I, double v) { out[decltype(I)::value] = v; });
  std::memcpy(h, out, sizeof out);
}

extern "C" {
void host_setup(int m, const double* w, double a) {
  const auto& vs = m ? Model<1>::vs : Model<0>::vs;
  ModelConst& mc = c_mc[m];
  mc.a = a;
  for (int i = 0; i < vs.Q; ++i) {
    const int g = vs.grp[i], *v = vs.e[i];
    mc.W[g] = w[i];
    mc.X2[g] = a * a * (v[0] * v[0] + v[1] * v[1] + v[2] * v[2]);
    mc.X2o2[g] = mc.X2[g] / 2.0;
    mc.X2o4[g] = mc.X2[g] / 4.0;
    mc.X2o8[g] = mc.X2[g] / 8.0;
  }
}
// The lattice vectors in storage order, three components each.
void host_velocities(int m, int* e) {
  const auto& vs = m ? Model<1>::vs : Model<0>::vs;
  for (int i = 0; i < 3 * vs.Q; ++i) e[i] = vs.e[i / 3][i % 3];
}
// One collision of each of n cells, h[cell][Q], in place.
void host_collide(int m, double* h, long n, double omega) {
  for (long c = 0; c < n; ++c) m ? collide<1>(h + c * Model<1>::Q, omega) : collide<0>(h + c * Model<0>::Q, omega);
}
double host_fx_to(long long i, int e) { return fx_to<60>(i, e); }
long long host_fx_from(double v, int e) { return fx_from<60>(v, e); }
long long host_fx_mul(long long a, double omega) { return fx_mul(a, fx_from<63>(omega, 1023)); }
void host_relax(double ev, double od, double* hp, double* hm, double omega) {
  const Two64 r = relax_pair64(ev, od, *hp, *hm, omega, fx_from<63>(omega, 1023));
  *hp = r.p;
  *hm = r.m;
}
}
