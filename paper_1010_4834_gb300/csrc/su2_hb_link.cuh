// One link's heat-bath update (Section 2, Eqs. 5-9, 11) and over-relaxation
// update, shared by the substep kernel (su2_heatbath.cuh), the fused parity-pair
// kernel (su2_pair.cu), the over-relaxation kernel (su2_kernels.cu) and the batched
// kernel (su2_batch_kernel.cuh).  The heat bath of a lattice leaves the same links by
// every schedule; how batches compare with it is said at SU2_COMPILER_FUSES
// (su2_device.cuh).
// Paper: Cardoso & Bicudo, arXiv:1010.4834.
//
// Every lane makes the link's first a0 trial inline.  A link that rejects it
// goes to a block-wide shared-memory queue (its W = Sigma/k, alpha, index and
// site), which the block later finishes with trials 2, 3, ... (hb_drain): a
// warp then does not wait on its slowest lane's trial loop.  The draws and
// their order are those of the plain loop, so only the schedule differs.  A
// full queue falls back to finishing the link inline.
//
// With MEAS the update also adds Tr(U_MU(x) L(x)^dagger)/2 to `plaq`, with L
// the staple's partial sum over NU < MU and U the link's final value (the
// accepted draw as stored, or the kept old link); see k_heatbath.
#pragma once

#include "su2_kernel_util.cuh"

namespace su2 {

template <class R> struct PlainAcc {
  R s = R(0);
  __device__ __forceinline__ void add(R v) { s += v; }
  __device__ __forceinline__ double value() const { return (double)s; }
};

// Queue entries are 16-byte aligned (FP32: 28 -> 32 bytes), so an entry
// moves in a few wide shared-memory accesses: 64^4 FP32 sweep 1412 -> 1407
// us, F16Q 1610 -> 1592 us.
template <class R, bool MEAS> struct __align__(16) Deferred {
  WOf<R> w;
  R alpha;
  int h;
  uint32_t site;
};
template <class R> struct __align__(16) Deferred<R, true> {
  WOf<R> w;
  R alpha;
  int h;
  uint32_t site;
  Quat<R> lower;
};

template <class R, bool MEAS>
__device__ __forceinline__ int finish_deferred(const Deferred<R, MEAS>& d, uint4 ctr, const HBParams& hp,
                                               Quat<R>* out) {
  A0Of<R> a0;
  uint4 rt;
  const int n =
      sample_a0_from<R>(2, d.alpha, trial_inv2a(d.alpha), trial_e(d.alpha, hp.sampler), ctr, hp, &a0, &rt);
  if (n) *out = compose_link<R>(a0, d.w, ctr, rt, hp);
  return n;
}

// Direction and parity of a substep: compile-time for FP32 / F16Q (MU, PAR >= 0,
// so that every class index is a constant), run-time for FP64 (MU = PAR =
// kRuntime; see staple_fixed).
constexpr int kRuntime = -1;
struct Substep { int mu, p; };
template <int MU, int PAR> __device__ __forceinline__ Substep substep_of(const Substep& s) {
  return Substep{MU >= 0 ? MU : s.mu, PAR >= 0 ? PAR : s.p};
}

// The addressing that goes with it.
template <int P, int CP> constexpr int hb_addr = P == kF64 ? (int)kFlat : CP;
// The template arguments of direction MU, parity PAR.
template <int P, int MU> constexpr int hb_dir = P == kF64 ? kRuntime : MU;

// Update link h of class (MU, PAR).  Rejected first trials go to queue slot
// atomicAdd(qn, 1) when it is below CAP.  MCG: the staple's loads of the
// other-parity MU class bypass L1 (the fused pair kernel writes that class
// earlier in the same launch).  NC: read-only loads; the persistent batched
// kernel, whose other CTAs write links during the launch, loads coherently.
template <int P, int MU, bool MEAS, int PAR, bool MCG, int CAP, int CP, bool NC = true>
__device__ __forceinline__ void hb_link(const Links<P, CP>& L, const Geom& g, Substep sub, int h, uint32_t tag, uint32_t sweep,
                                        typename Real<P>::T beta, const HBParams& hp,
                                        Deferred<typename Real<P>::T, MEAS>* queue, int* qn,
                                        PlainAcc<typename Real<P>::T>& plaq) {
  sub = substep_of<MU, PAR>(sub);
  const int mu = sub.mu, p = sub.p;
  using R = typename Real<P>::T;
  using Def = Deferred<R, MEAS>;
  const Site x = site_from_half(g, (uint32_t)h, p);
  Quat<R> lower;
  const Frame<R> f = link_frame<P, MU, MEAS, NC, CP, MCG>(L, g, x, h, mu, p, beta, lower);
  const R alpha = f.alpha;
  const uint32_t site = philox_site(g, x);
  const uint4 ctr = make_uint4(site, tag, sweep, 0u);
  if (!(alpha >= R(1e-12))) {
    uint4 c = ctr;
    c.w = 1u;
    const Quat<R> nl = haar_from<R>(philox(c, hp.rk));
    if constexpr (MEAS) plaq.add(qdot_rn(L.put(2 * mu + p, h, nl), lower));
    else L.st(2 * mu + p, h, nl);
    return;
  }
  const R inv2a = trial_inv2a(alpha);
  const R e = trial_e(alpha, hp.sampler);
  const WOf<R> w = f.w;
  A0Of<R> a0;
  uint4 rt;
  if (trial_a0<R>(alpha, inv2a, e, ctr, 1, hp, &a0, &rt)) {
    const Quat<R> nl = compose_link<R>(a0, w, ctr, rt, hp);
    if constexpr (MEAS) plaq.add(qdot_rn(L.put(2 * mu + p, h, nl), lower));
    else L.st(2 * mu + p, h, nl);
  } else if (hp.max_tries > 1) {
    const int slot = atomicAdd(qn, 1);
    Def d;
    d.w = w;
    d.alpha = alpha;
    d.h = h;
    d.site = site;
    if constexpr (MEAS) d.lower = lower;
    if (slot < CAP) {
      queue[slot] = d;
    } else {
      Quat<R> nl;
      const int n = finish_deferred<R, MEAS>(d, ctr, hp, &nl);
      if constexpr (MEAS) plaq.add(qdot_rn(n ? L.put(2 * mu + p, h, nl) : ldl<P, NC>(L, 2 * mu + p, h), lower));
      else if (n) L.st(2 * mu + p, h, nl);
    }
  } else {
    if constexpr (MEAS) plaq.add(qdot_rn(ldl<P, NC>(L, 2 * mu + p, h), lower));
  }
}

// Finish the queue entries i = threadIdx.x, threadIdx.x + blockDim.x, ... < n.
template <int P, int MU, bool MEAS, int PAR, int CP, bool NC = true>
__device__ __forceinline__ void hb_drain(const Links<P, CP>& L, Substep sub, const Deferred<typename Real<P>::T, MEAS>* queue, int n,
                                         uint32_t tag, uint32_t sweep, const HBParams& hp,
                                         PlainAcc<typename Real<P>::T>& plaq) {
  sub = substep_of<MU, PAR>(sub);
  const int mu = sub.mu, p = sub.p;
  using R = typename Real<P>::T;
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    const Deferred<R, MEAS> d = queue[i];
    Quat<R> nl;
    const int t = finish_deferred<R, MEAS>(d, make_uint4(d.site, tag, sweep, 0u), hp, &nl);
    if constexpr (MEAS) plaq.add(qdot_rn(t ? L.put(2 * mu + p, d.h, nl) : ldl<P, NC>(L, 2 * mu + p, d.h), d.lower));
    else if (t) L.st(2 * mu + p, d.h, nl);
  }
}

// FP64 in fixed point; false if a link is outside fix_link's (ANY: fix_any_link's)
// range.
template <bool NC, bool ANY, int CP>
__device__ __forceinline__ bool or_fixed(const Links<kF64, CP>& L, const Geom& g, const Site& x, int h, int mu, int p,
                                         const Quat<double>& u) {
  FixSum s;
  Quat<double> lower;
  FixBad bad{0u, 0u};
  const bool ok = staple_fixed<false, NC, false, ANY>(L, g, x, h, mu, p, 4, s, lower);
  const FixQuat ud = fix_of<ANY>(u, -1, bad);
  if (!ok || !fix_ok(bad)) return false;
  const Frame<double> f = staple_frame(s, 1.0);
  if (f.alpha == 0.0) return true;
  s = fix_zero();
  fix_mac(s, fix_mul(f.w, ud), f.w);
  L.st(2 * mu + p, h, fix_sum_to_double(s));
  return true;
}
// The links that it refuses, out of line.
template <bool NC, int CP>
static __device__ __noinline__ void or_other(Links<kF64, CP> L, const Geom& g, Site x, int h, int mu, int p) {
  const Quat<double> u = ldl<kF64, NC>(L, 2 * mu + p, h);
  if (or_fixed<NC, true>(L, g, x, h, mu, p, u)) return;
  Quat<double> lower;
  const Quat<double> sig = staple_rolled<NC, false>(L, g, x, h, mu, p, 4, lower);
  const double k2 = qdot(sig, sig);
  if (!(k2 >= Math<double>::kTiny)) return;
  const Quat<double> w = qscale(sig, Math<double>::rsqrt(k2));
  L.st(2 * mu + p, h, qmul(qmul_nd(w, u), w));
}

// One over-relaxation update (Section 2, Eq. 10 with W = Sigma/|Sigma| for
// the orientation of Eq. 11): U' = W U^dagger W keeps Tr(U Sigma^dagger).
// Unlike a heat-bath link, U' is built from the old link, so rounding would
// accumulate over many over-relaxation sweeps: in FP32 each step multiplies
// |U| by |W|^2 = 1 + O(2^-22), a random walk of about 1e-5 after a thousand
// sweeps.  FP32 (and the F16Q arithmetic, whose stores are normalised again
// on load) therefore normalises U' before storing it; in FP64 the walk (2e-15
// rms in |U|^2 after a hundred sweeps, 9e-15 after a thousand) is let be and
// the update is stored as computed, like the oracle's.  NC: read-only loads
// (no other block of the launch writes these links).
template <int P, int MU, int PAR, bool NC, int CP>
__device__ __forceinline__ void or_link(const Links<P, CP>& L, const Geom& g, Substep sub, int h) {
  sub = substep_of<MU, PAR>(sub);
  const int mu = sub.mu, p = sub.p;
  using R = typename Real<P>::T;
  using M = Math<R>;
  const Site x = site_from_half(g, (uint32_t)h, p);
  if constexpr (P == kF64) {
    const Quat<R> u = ldl<P, NC>(L, 2 * mu + p, h);
    if (__builtin_expect(!or_fixed<NC, false>(L, g, x, h, mu, p, u), 0)) or_other<NC>(L, g, x, h, mu, p);
  } else {
    const Quat<R> sig = staple<P, MU, 0xF, NC>(L, g, x, h, p);
    const R k2 = qdot_rn(sig, sig);
    if (!(k2 >= M::kTiny)) return;
    const Quat<R> w = qscale(sig, M::rsqrt(k2));
    const Quat<R> u = ldl<P, NC>(L, 2 * mu + p, h);   // the staple's registers are free
    Quat<R> v = qmul_rn(qmul_nd_rn(w, u), w);
    v = qscale(v, M::rsqrt(qdot_rn(v, v)));
    L.st(2 * mu + p, h, v);
  }
}

}  // namespace su2
