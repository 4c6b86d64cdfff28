// One site's plaquettes and one spatial site's time line, for the reductions of
// single lattices and of batches (k_batch_measure), all in su2_kernels.cu.
// Read-only loads unless a kernel can start beside one that writes links (NC =
// false; see pdl_wait).
// Paper: Cardoso & Bicudo, arXiv:1010.4834.
#pragma once

#include "su2_internal.h"

namespace su2 {

// The sixteen links one site's six plaquettes use: its own four and, for each
// direction mu, the three U_nu(x + mu) with nu != mu.
template <int P> struct PlaqLinks { Quat<typename Real<P>::T> u[4], n[4][3]; };

template <int P>
__device__ __forceinline__ void plaq_load(const Links<P>& L, const Geom& g, int s, PlaqLinks<P>& k, int& p) {
  const Site x = site_from_index(g, (uint32_t)s);
  p = parity(x);
  const int q = p ^ 1;
  const int h = s >> 1;
  const int hm[4] = {hidx(g, shifted<0, +1>(g, x)), hidx(g, shifted<1, +1>(g, x)), hidx(g, shifted<2, +1>(g, x)),
                     hidx(g, shifted<3, +1>(g, x))};
#pragma unroll
  for (int mu = 0; mu < 4; ++mu) k.u[mu] = L.ld(2 * mu + p, h);
#pragma unroll
  for (int mu = 0; mu < 4; ++mu) {
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      const int nu = j < mu ? j : j + 1;
      k.n[mu][j] = L.ld(2 * nu + q, hm[mu]);
    }
  }
}

// U_nu(x + mu) among the loaded links.
template <int P>
__device__ __forceinline__ const Quat<typename Real<P>::T>& plaq_nb(const PlaqLinks<P>& k, int mu, int nu) {
  return k.n[mu][nu < mu ? nu : nu - 1];
}

template <int P>
__device__ __forceinline__ void plaq_sums(const PlaqLinks<P>& k, typename Real<P>::T& ss, typename Real<P>::T& ts) {
  using R = typename Real<P>::T;
  ss = R(0);
  ts = R(0);
#pragma unroll
  for (int mu = 0; mu < 4; ++mu) {
#pragma unroll
    for (int nu = mu + 1; nu < 4; ++nu) {
      const R v = qdot(qmul(k.u[mu], plaq_nb<P>(k, mu, nu)), qmul(k.u[nu], plaq_nb<P>(k, nu, mu)));
      if (nu == 3) ts += v; else ss += v;
    }
  }
}

// One plaquette in fixed point (FP64, units of 2^-58): each neighbour link
// enters one plaquette of its site and is converted there.
template <int MU, int NU>
__device__ __forceinline__ int64_t plaq_fixed(const Links<kF64>& L, int q, const FixQuat& umu, const FixQuat& unu,
                                              int h_pmu, int h_pnu, FixBad& bad) {
  const FixQuat a = fix_mul(umu, fix_of(L.ld(2 * NU + q, h_pmu), 0, bad));
  const FixQuat b = fix_mul(unu, fix_of(L.ld(2 * MU + q, h_pnu), 0, bad));
  return fix_dot(a, b, 0);
}

// The sums (spatial, space-time planes) of a site with links that plaq_fixed
// refuses, out of line, a rolled loop over the planes: in fixed point with any
// components, then in FP64.
static __device__ __noinline__ double2 plaq_other(Links<kF64> L, int p, int h, int h0, int h1, int h2, int h3) {
  const int q = p ^ 1;
  double sum[2];
  FixBad bad{0u, 0u};
  for (int fp64 = 0; fp64 < 2; ++fp64) {
    sum[0] = sum[1] = 0.0;
#pragma unroll 1
    for (int k = 0; k < 6; ++k) {
      const int nu = k < 1 ? 1 : k < 3 ? 2 : 3, mu = nu == 1 ? 0 : nu == 2 ? k - 1 : k - 3;
      const int hm = mu == 0 ? h0 : mu == 1 ? h1 : h2, hn = nu == 1 ? h1 : nu == 2 ? h2 : h3;
      const Quat<double> a = L.ld(2 * mu + p, h), b = L.ld(2 * nu + q, hm), c = L.ld(2 * nu + p, h), d = L.ld(2 * mu + q, hn);
      const double v = fp64 ? qdot(qmul(a, b), qmul(c, d))
                            : fix_to_double(fix_dot(fix_mul(fix_of<true>(a, 0, bad), fix_of<true>(b, 0, bad)),
                                                    fix_mul(fix_of<true>(c, 0, bad), fix_of<true>(d, 0, bad)), 0));
      if (nu == 3) sum[1] += v;
      else sum[0] += v;
      if (!fp64 && !fix_ok(bad)) break;
    }
    if (fix_ok(bad)) break;
  }
  return make_double2(sum[0], sum[1]);
}

// The two sums (spatial and space-time planes) of site s.
template <int P>
__device__ __forceinline__ void plaq_site(const Links<P>& L, const Geom& g, int s, float& ss, float& ts) {
  PlaqLinks<P> k;
  int p;
  plaq_load<P>(L, g, s, k, p);
  plaq_sums<P>(k, ss, ts);
}

__device__ __forceinline__ void plaq_site(const Links<kF64>& L, const Geom& g, int s, double& ss, double& ts) {
  const Site x = site_from_index(g, (uint32_t)s);
  const int p = parity(x), q = p ^ 1, h = s >> 1;
  const int h0 = hidx(g, shifted<0, +1>(g, x)), h1 = hidx(g, shifted<1, +1>(g, x)),
            h2 = hidx(g, shifted<2, +1>(g, x)), h3 = hidx(g, shifted<3, +1>(g, x));
  FixBad bad{0u, 0u};
  const FixQuat u0 = fix_of(L.ld(0 + p, h), 0, bad), u1 = fix_of(L.ld(2 + p, h), 0, bad),
                u2 = fix_of(L.ld(4 + p, h), 0, bad), u3 = fix_of(L.ld(6 + p, h), 0, bad);
  const int64_t s01 = plaq_fixed<0, 1>(L, q, u0, u1, h0, h1, bad), s02 = plaq_fixed<0, 2>(L, q, u0, u2, h0, h2, bad),
                s12 = plaq_fixed<1, 2>(L, q, u1, u2, h1, h2, bad);
  const int64_t s03 = plaq_fixed<0, 3>(L, q, u0, u3, h0, h3, bad), s13 = plaq_fixed<1, 3>(L, q, u1, u3, h1, h3, bad),
                s23 = plaq_fixed<2, 3>(L, q, u2, u3, h2, h3, bad);
  ss = fix_to_double(s01 + s02 + s12);
  ts = fix_to_double(s03 + s13 + s23);
  if (__builtin_expect(!fix_ok(bad), 0)) {
    const double2 v = plaq_other(L, p, h, h0, h1, h2, h3);
    ss = v.x;
    ts = v.y;
  }
}

// The product of `seg` time links: link t is element e0 + t nsig_h of b0 (t
// even) or b1 (t odd).  FP64 multiplies in fixed point (su2_fixed.cuh), and
// again in FP64 if a link is not a unit quaternion.
template <int P, int CP, bool NC>
__device__ __forceinline__ Quat<typename Real<P>::T> time_line(const typename Links<P, CP>::E* b0,
                                                               const typename Links<P, CP>::E* b1, uint32_t e0,
                                                               uint32_t nsig_h, int seg) {
  using R = typename Real<P>::T;
  using LT = Links<P, CP>;
  constexpr int C = 8;
  Quat<R> pr = qone<R>();
  if constexpr (P == kF64) {
    FixQuat f = fix_one();
    bool bad = false;
    for (int t = 0; t < seg; t += 2) {
      const Quat<R> u = LT::template ldp<NC>(b0, e0 + nsig_h * (uint32_t)t);
      const Quat<R> v = t + 1 < seg ? LT::template ldp<NC>(b1, e0 + nsig_h * (uint32_t)(t + 1)) : qone<R>();
      f = fix_mul(fix_mul(f, fix_unit_link(u, bad)), fix_unit_link(v, bad));
    }
    pr = qmake<R>(fix_to_double(fix_value(f.w)), fix_to_double(fix_value(f.x)), fix_to_double(fix_value(f.y)),
                  fix_to_double(fix_value(f.z)));
    if (__builtin_expect(bad, 0)) {
      pr = qone<R>();
#pragma unroll 1
      for (int t = 0; t < seg; ++t) pr = qmul(pr, LT::template ldp<NC>((t & 1) ? b1 : b0, e0 + nsig_h * (uint32_t)t));
    }
  } else {
    int t = 0;
    for (; t + C <= seg; t += C) {
      Quat<R> u[C];
#pragma unroll
      for (int j = 0; j < C; ++j) u[j] = LT::template ldp<NC>((j & 1) ? b1 : b0, e0 + nsig_h * (uint32_t)(t + j));
#pragma unroll
      for (int j = 0; j < C; ++j) pr = qmul(pr, u[j]);
    }
    for (; t < seg; ++t) pr = qmul(pr, LT::template ldp<NC>((t & 1) ? b1 : b0, e0 + nsig_h * (uint32_t)t));
  }
  return pr;
}

}  // namespace su2
