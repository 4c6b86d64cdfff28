// Kernels of the SU(2) heat-bath Monte Carlo for sm_103a, except the heat-bath
// substep itself (su2_heatbath.cuh, su2_pair.cu) and batched sweeps
// (su2_batch_kernel.cuh): start configurations, the
// over-relaxation substep, the fused plaquette / Polyakov reductions, APE
// smearing, Wilson loops and the canonical-layout conversions.  Paper: Cardoso & Bicudo,
// arXiv:1010.4834 (Sections 2 and 4).
//
// None of this work is a dense contraction (2x2 SU(2) products in
// registers), so everything runs on the FP32/FP64 pipes; the sweep is bound
// by HBM traffic and ALU issue.  Reductions are fused into the measurement
// kernels: per-thread sums (compensated when the arithmetic is FP32), FP64
// warp shuffles, one partial per block and a last-block finisher that adds
// the partials in a fixed order, so a result is reproducible run to run.
#define SU2_COMPILER_FUSES
#include <algorithm>
#include <atomic>
#include <cfloat>
#include <mutex>
#include <type_traits>

#include "su2_batch.h"
#include "su2_hb_link.cuh"
#include "su2_internal.h"
#include "su2_kernel_util.cuh"
#include "su2_measure.cuh"

namespace su2 {

static std::atomic<uint64_t> g_launches{0};
static thread_local int g_capturing = 0;
void count_launches(uint64_t n) {
  if (!g_capturing) g_launches.fetch_add(n, std::memory_order_relaxed);
}
uint64_t launches_total() { return g_launches.load(std::memory_order_relaxed); }
CaptureScope::CaptureScope() { ++g_capturing; }
CaptureScope::~CaptureScope() { --g_capturing; }

// ---------------------------------------------------------------------------
// Device info and launch shapes
// ---------------------------------------------------------------------------
const DeviceInfo& device_info() {
  // filled once per device; concurrent first calls from several host
  // threads wait on the device's once_flag
  static DeviceInfo info[64];
  static std::once_flag once[64];
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev < 0 || dev >= 64) dev = 0;
  std::call_once(once[dev], [dev]() {
    cudaDeviceGetAttribute(&info[dev].sms, cudaDevAttrMultiProcessorCount, dev);
    cudaDeviceGetAttribute(&info[dev].l2_bytes, cudaDevAttrL2CacheSize, dev);
    if (info[dev].sms <= 0) info[dev].sms = 1;
  });
  return info[dev];
}

Geom make_geom(const int n[4]) {
  Geom g;
  for (int i = 0; i < 4; ++i) g.n[i] = n[i];
  g.n0h = n[0] / 2;
  g.vh = (int64_t)n[0] * n[1] * n[2] * n[3] / 2;
  g.st[0] = 0;
  g.st[1] = 1;
  g.st[2] = n[1];
  g.st[3] = n[1] * n[2];
  for (int d = 0; d < 4; ++d) g.wr[d] = d ? g.st[d] * (n[d] - 1) : 0;
  for (int d = 0; d < 4; ++d) {
    g.hst[d] = d ? g.n0h * g.st[d] : 0;
    g.hwr[d] = d ? g.n0h * g.wr[d] : 0;
  }
  g.f_n0h = FastDiv((uint32_t)g.n0h);
  g.f_n1 = FastDiv((uint32_t)n[1]);
  g.f_n2 = FastDiv((uint32_t)n[2]);
  g.f_n0 = FastDiv((uint32_t)n[0]);
  g.site0 = 0;
  return g;
}

size_t scratch_bytes() {
  return kScratchPartials * sizeof(double) + 256 + kScratchOut * sizeof(double) + 256;
}

// ---------------------------------------------------------------------------
// Start configurations (Section 4 kernel list: cold start U = 1, hot start a
// random element of SU(2) on every link, read here as Haar via Philox draw 0 of sweep index
// 0xFFFFFFFF).  One thread per (site, direction).
// ---------------------------------------------------------------------------
template <int P>
__global__ void __launch_bounds__(kThreads) k_init(Links<P> L, Geom g, int start,
                                                   const __grid_constant__ RoundKeys rk,
                                                   uint32_t lattice_tag) {
  using R = typename Real<P>::T;
  const int64_t V = 2 * g.vh;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t w = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; w < 4 * V; w += stride) {
    const int mu = (int)(w / V);
    const uint32_t s = (uint32_t)(w - (int64_t)mu * V);
    const Site x = site_from_index(g, s);
    Quat<R> q = qone<R>();
    if (start) q = haar_from<R>(philox(make_uint4(s + g.site0, (uint32_t)mu | lattice_tag, 0xFFFFFFFFu, 0u), rk));
    L.st(2 * mu + parity(x), hidx(g, x), q);
  }
}

// ---------------------------------------------------------------------------
// Over-relaxation substep (Section 2, Eq. 10): or_link (su2_hb_link.cuh) on
// every link of direction MU and parity PAR.
// ---------------------------------------------------------------------------
template <int P, int MU, int PAR>
__global__ void __launch_bounds__(kThreads, Occ<P>::hb)
    k_overrelax(Links<P, hb_addr<P, kClassPtr>> L, const __grid_constant__ Geom g, Substep sub) {
  const int stride = gridDim.x * blockDim.x;
  for (int h = blockIdx.x * blockDim.x + threadIdx.x; h < g.vh; h += stride) or_link<P, MU, PAR, true>(L, g, sub, h);
}

// ---------------------------------------------------------------------------
// Plaquette (Section 2, Eqs. 12-13): per site the six (1/2) Re Tr
// U_mu(x) U_nu(x+mu) U_mu(x+nu)^dagger U_nu(x)^dagger = (A B^dagger)_0 with
// A = U_mu(x) U_nu(x+mu), B = U_nu(x) U_mu(x+nu): the dot product A.B.
// out[0] all, out[1] spatial, out[2] space-time means.
// ---------------------------------------------------------------------------
template <int P>
__device__ __forceinline__ void plaquette_sum(const Links<P>& L, const Geom& g, int64_t s0, int64_t V, double* partials,
                                              unsigned int* counter, double* out) {
  using R = typename Real<P>::T;
  Acc<R> sp, tm;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  // the plaquettes of the V sites from s0 on (all sites: s0 = 0, V = volume);
  // 64-bit loop index: V may come within one stride of 2^31
  for (int64_t s = s0 + (int64_t)blockIdx.x * blockDim.x + threadIdx.x; s < s0 + V; s += stride) {
    R ss0, ts0;
    plaq_site(L, g, (int)s, ss0, ts0);
    sp.add(ss0);
    tm.add(ts0);
  }
  double v[2] = {sp.value(), tm.value()};
  if (block_partial<2>(v, partials, counter, blockIdx.x, gridDim.x)) {
    double tot[2];
    final_sum<2>(partials, gridDim.x, tot);
    if (threadIdx.x == 0) {
      const double n3 = 3.0 * (double)V;
      out[0] = (tot[0] + tot[1]) / (2.0 * n3);
      out[1] = tot[0] / n3;
      out[2] = tot[1] / n3;
      *counter = 0;
    }
  }
}

template <int P>
__global__ void __launch_bounds__(kThreads) k_plaquette(Links<P> L, Geom g, int64_t s0, int64_t V,
                                                        double* partials, unsigned int* counter, double* out) {
  plaquette_sum<P>(L, g, s0, V, partials, counter, out);
}

// FP64 at 128 registers a thread, two blocks an SM.
template <>
__global__ void __launch_bounds__(kThreads, 2) k_plaquette<kF64>(Links<kF64> L, Geom g, int64_t s0, int64_t V,
                                                                 double* partials, unsigned int* counter, double* out) {
  plaquette_sum<kF64>(L, g, s0, V, partials, counter, out);
}

// ---------------------------------------------------------------------------
// Polyakov loop (Section 2, Eqs. 14-15): per spatial site the product of the
// time links in increasing t; mean of (1/2) Tr over the spatial sites.  Site
// s = xs + Nsigma t has half-index (xs >> 1) + (Nsigma/2) t.
//
// A block takes kThreads / G consecutive time lines, and each line is split
// into G consecutive segments of nt / G >= 8 links (G a power of two <= 8
// dividing nt, as large as that allows).  Warp group q loads segment q of
// every line of the block in chunks of 8 (all loads of a chunk issued
// before the products; each load instruction of a warp reads 32 consecutive
// spatial sites at one t), and the segment products are multiplied in t
// order through shared memory.  With one line per thread the kernel kept
// one chunk in flight per thread at 120 registers and ran at under half the
// copy bandwidth (ncu, 64^4: 24% warps active, long-scoreboard stalls 11 per
// issue).  After a measured sweep the last block also finishes the sweep's
// plaquette, records both in the history ring and advances the sweep
// counter (SweepEpilogue), which saves two launches per sweep.
// ---------------------------------------------------------------------------
template <int P> struct PolyMinBlocks { static constexpr int value = 4; };
template <> struct PolyMinBlocks<kF64> { static constexpr int value = 2; };

template <int P, bool NC>
__global__ void __launch_bounds__(kThreads, PolyMinBlocks<P>::value)
    k_polyakov(Links<P, kClassPtr> L, Geom g, int lg, double* partials, unsigned int* counter, double* out,
               SweepEpilogue ep, int early) {
  using R = typename Real<P>::T;
  using LT = Links<P, kClassPtr>;
  __shared__ Quat<R> seg_prod[kThreads];
  Acc<R> acc;
  const int nsig = g.n[0] * g.n[1] * g.n[2];
  const uint32_t nsig_h = (uint32_t)(nsig / 2);
  const int G = 1 << lg;
  const int lines = kThreads >> lg;  // lines per block, a multiple of 32
  const int seg = g.n[3] >> lg;
  const int q = threadIdx.x / lines;
  const int l = threadIdx.x - q * lines;
  const int t0 = q * seg;
  const int zero = pdl_wait();
  if (early) pdl_trigger();
  for (int first = blockIdx.x * lines + zero; first < nsig; first += gridDim.x * lines) {
    const int xs = first + l;
    Quat<R> pr = qone<R>();
    if (xs < nsig) {
      const Site x = site_from_index(g, (uint32_t)xs);
      const uint32_t hh = (uint32_t)(xs >> 1);
      // the time links of x alternate between the two parity classes: b0
      // holds those at t of the parity of t0, b1 the others
      const bool swap = (parity(x) ^ (t0 & 1)) != 0;
      const typename LT::E* b0 = swap ? L.cls_base(7) : L.cls_base(6);
      const typename LT::E* b1 = swap ? L.cls_base(6) : L.cls_base(7);
      const uint32_t e0 = hh + nsig_h * (uint32_t)t0;
      pr = time_line<P, kClassPtr, NC>(b0, b1, e0, nsig_h, seg);
    }
    if (G > 1) {
      seg_prod[threadIdx.x] = pr;
      __syncthreads();
      if (q == 0) {
        for (int k = 1; k < G; ++k) pr = qmul(pr, seg_prod[k * lines + l]);
      }
      __syncthreads();
    }
    if (q == 0 && xs < nsig) acc.add(pr.w);
  }
  double v[1] = {acc.value()};
  if (block_partial<1>(v, partials, counter, blockIdx.x, gridDim.x)) {
    double tot[1];
    final_sum<1>(partials, gridDim.x, tot);
    // every thread reads the counter here; thread 0 advances it only after
    // the barriers inside plaquette_from_block_sums
    double* row = ep.meas ? ep.hist + 4 * (size_t)(*(volatile uint32_t*)ep.sweep % (uint32_t)kHistRing) : nullptr;
    if (threadIdx.x == 0) {
      (row ? row[3] : out[0]) = tot[0] / (double)nsig;
      *counter = 0;
    }
    if (ep.meas) {
      plaquette_from_block_sums(ep.meas, kMeasStride, ep.nb, ep.volume, row);
      if (threadIdx.x == 0) *ep.sweep += 1u;
    }
  }
}

// ---------------------------------------------------------------------------
// Plaquette or Polyakov loop of every lattice of a batch in one launch: block b
// takes a share of one lattice (blocks[b]) and the last block of a lattice
// adds its blocks' sums in a fixed order.  With a launch and a device copy per
// lattice, the two measurements of 64 lattices of 8^4 to 24^3 x 6 took 1.5 ms more
// (eight sweeps and both: 3.79 against 2.30 ms).
// ---------------------------------------------------------------------------
// A block's sum of (1/2) Tr over its share of a lattice's time lines, split into
// segments as in k_polyakov (which, as a caller of this, took other registers and
// with them 1 us more of a measured sweep: 32^3x4, F16Q).
template <int P>
__device__ __forceinline__ double polyakov_lines(const Links<P>& L, const Geom& g, int lg, int block, int nblocks) {
  using R = typename Real<P>::T;
  using LT = Links<P>;
  __shared__ Quat<R> seg_prod[kThreads];
  Acc<R> acc;
  const int nsig = g.n[0] * g.n[1] * g.n[2];
  const uint32_t nsig_h = (uint32_t)(nsig / 2);
  const int G = 1 << lg;
  const int lines = kThreads >> lg;  // lines per block, a multiple of 32
  const int seg = g.n[3] >> lg;
  const int q = threadIdx.x / lines;
  const int l = threadIdx.x - q * lines;
  const int t0 = q * seg;
  for (int first = block * lines; first < nsig; first += nblocks * lines) {
    const int xs = first + l;
    Quat<R> pr = qone<R>();
    if (xs < nsig) {
      const Site x = site_from_index(g, (uint32_t)xs);
      const uint32_t hh = (uint32_t)(xs >> 1);
      // the time links of x alternate between the two parity classes: b0
      // holds those at t of the parity of t0, b1 the others
      const bool swap = (parity(x) ^ (t0 & 1)) != 0;
      const typename LT::E* b0 = swap ? L.cls_base(7) : L.cls_base(6);
      const typename LT::E* b1 = swap ? L.cls_base(6) : L.cls_base(7);
      const uint32_t e0 = hh + nsig_h * (uint32_t)t0;
      pr = time_line<P, kFlat, true>(b0, b1, e0, nsig_h, seg);
    }
    if (G > 1) {
      seg_prod[threadIdx.x] = pr;
      __syncthreads();
      if (q == 0) {
        for (int k = 1; k < G; ++k) pr = qmul(pr, seg_prod[k * lines + l]);
      }
      __syncthreads();
    }
    if (q == 0 && xs < nsig) acc.add(pr.w);
  }
  return acc.value();
}

template <int P, bool POLY>
__global__ void __launch_bounds__(kThreads, measure_blocks_per_sm(P))
    k_batch_measure(const BatchLattice* __restrict__ desc, const BatchBlock4* __restrict__ blocks, double* partials,
                    unsigned int* counters, double* out) {
  using R = typename Real<P>::T;
  const BatchBlock4 b = blocks[blockIdx.x];
  const Geom& g = desc[b.lattice].g;
  Links<P> L;
  L.set(desc[b.lattice].links, g.vh);
  constexpr int NV = POLY ? 1 : 2;
  double v[NV];
  if constexpr (POLY) {
    v[0] = polyakov_lines<P>(L, g, polyakov_segments(g.n[3]), b.rank, b.count);
  } else {
    Acc<R> sp, tm;
    for (int s = b.rank * kThreads + (int)threadIdx.x; s < (int)(2 * g.vh); s += b.count * kThreads) {
      R ss, ts;
      plaq_site(L, g, s, ss, ts);
      sp.add(ss);
      tm.add(ts);
    }
    v[0] = sp.value();
    v[NV - 1] = tm.value();
  }
  if (block_partial<NV>(v, partials, counters + b.lattice, blockIdx.x, b.count)) {
    double tot[NV];
    final_sum<NV>(partials + (size_t)(blockIdx.x - b.rank) * NV, b.count, tot);
    if (threadIdx.x == 0) {
      if constexpr (POLY) {
        out[b.lattice] = tot[0] / (double)(g.n[0] * g.n[1] * g.n[2]);
      } else {
        const double n3 = 3.0 * (double)(2 * g.vh);
        double* o = out + 3 * (size_t)b.lattice;
        o[0] = (tot[0] + tot[NV - 1]) / (2.0 * n3);
        o[1] = tot[0] / n3;
        o[2] = tot[NV - 1] / n3;
      }
      counters[b.lattice] = 0;
    }
  }
}

// ---------------------------------------------------------------------------
// APE smearing step (Section 2, Eq. 19), Jacobi: spatial link (x, mu) ->
// P[(1-alpha) U + (alpha/4) (four spatial staples)], P = normalisation; a sum
// with vanishing norm keeps U.
//
// One thread per site updates all three spatial links.  For a pair mu < nu
// the two forward staple terms share one product: with
// A = U_nu(x+mu) U_mu(x+nu)^dag, link mu gets U_nu(x) A^dag and link nu gets
// U_mu(x) A.  Per site that is 27 link loads and 21 products instead of 39
// and 24 for three independent link updates, and one site decode instead of
// three.  Each link's staple terms are added nu ascending, forward then
// backward.  blockIdx.y = parity.
// ---------------------------------------------------------------------------
// binary16 links enter as stored and each product of three is scaled to unit
// norm (qacc_unit), as in the heat bath's staples.
template <int P, bool NC>
__device__ __forceinline__ Quat<typename Real<P>::T> ape_link(const Links<P, kClassPtr>& L, int cls, int h) {
  if constexpr (P == kF16Q) return ld_raw<P, NC, false>(L, cls, h);
  else return ldl<P, NC>(L, cls, h);
}
// s += a b^dagger, s += a b
template <int P, class Q> __device__ __forceinline__ void ape_acc_nd(Q& s, const Q& a, const Q& b) {
  if constexpr (P == kF16Q) qacc_unit(s, qmul_nd(a, b));
  else qacc_mul_nd(s, a, b);
}
template <int P, class Q> __device__ __forceinline__ void ape_acc(Q& s, const Q& a, const Q& b) {
  if constexpr (P == kF16Q) qacc_unit(s, qmul(a, b));
  else qacc_mul(s, a, b);
}

template <int P, int MU, int NU, bool NC>
__device__ __forceinline__ void ape_pair(const Links<P, kClassPtr>& L, int h, int p, const int (&dp)[3], const int (&dm)[3],
                                         const Quat<typename Real<P>::T>& umu, const Quat<typename Real<P>::T>& unu,
                                         Quat<typename Real<P>::T>& smu, Quat<typename Real<P>::T>& snu) {
  using R = typename Real<P>::T;
  const int q = p ^ 1;
  auto link = [&](int cls, int i) { return ape_link<P, NC>(L, cls, i); };
  const Quat<R> a = qmul_nd(link(2 * NU + q, h + dp[MU]), link(2 * MU + q, h + dp[NU]));
  const int hn = h + dm[NU], hm = h + dm[MU];  // x - nu, x - mu
  // link mu, term nu: forward U_nu(x) A^dag, backward U_nu(x-nu)^dag U_mu(x-nu) U_nu(x-nu+mu)
  ape_acc_nd<P>(smu, unu, a);
  ape_acc<P>(smu, qmul_dn(link(2 * NU + q, hn), link(2 * MU + q, hn)), link(2 * NU + p, hn + dp[MU]));
  // link nu, term mu: forward U_mu(x) A, backward U_mu(x-mu)^dag U_nu(x-mu) U_mu(x-mu+nu)
  ape_acc<P>(snu, umu, a);
  ape_acc<P>(snu, qmul_dn(link(2 * MU + q, hm), link(2 * NU + q, hm)), link(2 * MU + p, hm + dp[NU]));
}

template <int P, int CP>
__device__ __forceinline__ void ape_store(const Links<P, CP>& dst, int cls, int h, const Quat<typename Real<P>::T>& u,
                                          const Quat<typename Real<P>::T>& sig, typename Real<P>::T c0,
                                          typename Real<P>::T c1) {
  using R = typename Real<P>::T;
  const Quat<R> q = qmake<R>(c0 * u.w + c1 * sig.w, c0 * u.x + c1 * sig.x, c0 * u.y + c1 * sig.y,
                             c0 * u.z + c1 * sig.z);
  const R n2 = qdot(q, q);
  dst.st(cls, h, n2 >= Math<R>::kTiny ? qscale(q, Math<R>::rsqrt(n2)) : u);
}

#ifndef SU2_APE3_MINB
#define SU2_APE3_MINB 3
#endif
// The sites of parity PAR (a template parameter, so every class index is a
// compile-time constant for the per-class base pointers).
template <int P, int PAR, bool NC>
__device__ __forceinline__ void ape_sites(const Links<P, kClassPtr>& src, const Links<P, kClassPtr>& dst, const Geom& g,
                                          typename Real<P>::T c0, typename Real<P>::T c1, int zero) {
  using R = typename Real<P>::T;
  constexpr int p = PAR;
  const int vh = (int)g.vh;
  const int stride = gridDim.x * blockDim.x;
  for (int h = blockIdx.x * blockDim.x + threadIdx.x + zero; h < vh; h += stride) {
    const Site x = site_from_half(g, (uint32_t)h, p);
    // half-index steps to the six spatial neighbours; the index of x + a + b
    // is h + step(a) + step(b) for steps in different directions
    const int dp[3] = {half_step<0, +1>(g, x), half_step<1, +1>(g, x), half_step<2, +1>(g, x)};
    const int dm[3] = {half_step<0, -1>(g, x), half_step<1, -1>(g, x), half_step<2, -1>(g, x)};
    Quat<R> u0 = ape_link<P, NC>(src, 0 + p, h), u1 = ape_link<P, NC>(src, 2 + p, h), u2 = ape_link<P, NC>(src, 4 + p, h);
    Quat<R> s0 = qmake<R>(0, 0, 0, 0), s1 = s0, s2 = s0;
    ape_pair<P, 0, 1, NC>(src, h, p, dp, dm, u0, u1, s0, s1);
    ape_pair<P, 0, 2, NC>(src, h, p, dp, dm, u0, u2, s0, s2);
    ape_pair<P, 1, 2, NC>(src, h, p, dp, dm, u1, u2, s1, s2);
    if constexpr (P == kF16Q) {
      u0 = qscale(u0, rsqrtf(qdot(u0, u0)));
      u1 = qscale(u1, rsqrtf(qdot(u1, u1)));
      u2 = qscale(u2, rsqrtf(qdot(u2, u2)));
    }
    ape_store<P>(dst, 0 + p, h, u0, s0, c0, c1);
    ape_store<P>(dst, 2 + p, h, u1, s1, c0, c1);
    ape_store<P>(dst, 4 + p, h, u2, s2, c0, c1);
  }
}

// FP64: one link a thread, its four staples in fixed point (su2_fixed.cuh).
// Sharing the forward products among a site's three links as above keeps three
// sums of 16 registers and spilled 2 KB a thread; the nine further loads and
// conversions cost less.
// Links that fix_link refuses are computed in FP64 at once: a second conversion, as in
// the heat bath, would cost all fields 2% here, and out of line 1.8 us a step (20 x 12
// x 18 x 10: 18.0 -> 19.8); a cold 24^3x32 takes 398 us a step for 149.
template <bool NC>
__device__ __forceinline__ void ape_links_fixed(const Links<kF64>& src, const Links<kF64>& dst, const Geom& g, int mu,
                                                int p, double c0, double c1) {
  const int vh = (int)g.vh;
  const int stride = gridDim.x * blockDim.x;
  for (int h = blockIdx.x * blockDim.x + threadIdx.x; h < vh; h += stride) {
    const Site x = site_from_half(g, (uint32_t)h, p);
    FixSum s;
    Quat<double> sig;
    if (__builtin_expect(staple_fixed<false, NC, false>(src, g, x, h, mu, p, 3, s, sig), 1))
      sig = fix_sum_to_double(s);
    else
      sig = staple_rolled<NC, false>(src, g, x, h, mu, p, 3, sig);
    ape_store<kF64>(dst, 2 * mu + p, h, ldl<kF64, NC>(src, 2 * mu + p, h), sig, c0, c1);
  }
}

template <int P, bool NC>
__global__ void __launch_bounds__(kThreads, P == kF64 ? 2 : SU2_APE3_MINB)
    k_ape(Links<P, hb_addr<P, kClassPtr>> src, Links<P, hb_addr<P, kClassPtr>> dst, Geom g, double alpha_d, int early) {
  using R = typename Real<P>::T;
  const int zero = pdl_wait();
  if (early) pdl_trigger();
  const R alpha = (R)alpha_d;
  const R c0 = R(1) - alpha, c1 = R(0.25) * alpha;
  if constexpr (P == kF64) {
    ape_links_fixed<NC>(src, dst, g, (int)(blockIdx.y >> 1) + zero, (int)(blockIdx.y & 1), c0, c1);
  } else {
    if (blockIdx.y == 0) ape_sites<P, 0, NC>(src, dst, g, c0, c1, zero);
    else ape_sites<P, 1, NC>(src, dst, g, c0, c1, zero);
  }
}

template <int P>
__global__ void __launch_bounds__(kThreads) k_copy_spatial(Links<P> src, Links<P> dst) {
  const int64_t n = 6 * src.vh;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
    const int cls = (int)(i / src.vh);
    const int j = (int)(i - cls * src.vh);
    dst.st(cls, j, src.ld(cls, j));
  }
}

// ---------------------------------------------------------------------------
// Wilson loops (Section 2, Eq. 18), (1/2) Tr[S_R(x) T_T(x+R mu) S_R(x+T t)^dag
// T_T(x)^dag] = (A B) . (D C) with A = S_R(x), B = T_T(x+R mu), C = S_R(x+T t),
// D = T_T(x).  A thread owns one (site, spatial MU) and a chunk of TC values
// of T; it walks R = 1..rmax extending A and the TC lines C by one link each,
// rebuilds the time line B at x + R mu, and adds the TC loop values into the
// block's shared accumulators (one transposing warp reduction per R).
// blockIdx.y = 3 chunk + mu.  Per-block sums go to `partials`; a second
// kernel adds them per (R, T) in a fixed order.
// ---------------------------------------------------------------------------
constexpr int kWilsonMaxR = 32;
constexpr int kWilsonThreads = 128;

// Walker along the time direction in half-site index space: one step adds
// the half-index stride of a time slice (wrapping at the last slice) and
// flips the parity.
struct TWalk {
  int h, par, x3;
  __device__ __forceinline__ void init(const Geom& g, const Site& y) {
    h = hidx(g, y);
    par = parity(y);
    x3 = y.x3;
  }
  __device__ __forceinline__ void step(int nt, int hts, int hwrap) {
    if (x3 + 1 == nt) { x3 = 0; h -= hwrap; } else { ++x3; h += hts; }
    par ^= 1;
  }
};

template <int P, int TC, int MU>
__device__ __forceinline__ void wilson_site(const Links<P>& Ls, const Links<P>& Lt, const Geom& g, int s,
                                            bool valid, int rmax, int t0, int nT, double* acc) {
  using R = typename Real<P>::T;
  static_assert(TC == 4 || TC == 8 || TC == 16, "T chunk must be 4, 8 or 16");
  const int lane = threadIdx.x & 31;
  const int nt = g.n[3];
  const int hts = g.n0h * g.st[3];
  const int hwrap = hts * (nt - 1);
  const Site x = site_from_index(g, (uint32_t)s);
  Quat<R> D[TC], C[TC];
  {
    TWalk w;
    w.init(g, x);
    Quat<R> pr = qone<R>();
    for (int t = 0; t < t0; ++t) { pr = qmul(pr, Lt.ld(6 + w.par, w.h)); w.step(nt, hts, hwrap); }
#pragma unroll
    for (int j = 0; j < TC; ++j) {
      if (j < nT) { pr = qmul(pr, Lt.ld(6 + w.par, w.h)); w.step(nt, hts, hwrap); }
      D[j] = pr;
      C[j] = qone<R>();
    }
  }
  Quat<R> A = qone<R>();
  Site xr = x;  // x + (r-1) mu at the top of iteration r
  Site zt = x;  // x + (r-1) mu + (t0 + 1) t
  for (int t = 0; t <= t0; ++t) zt = shifted<3, +1>(g, zt);
  for (int r = 1; r <= rmax; ++r) {
    A = qmul(A, Ls.ld(2 * MU + parity(xr), hidx(g, xr)));
    {
      TWalk z;
      z.init(g, zt);
#pragma unroll
      for (int j = 0; j < TC; ++j) {
        if (j < nT) { C[j] = qmul(C[j], Ls.ld(2 * MU + z.par, z.h)); z.step(nt, hts, hwrap); }
      }
    }
    xr = shifted<MU, +1>(g, xr);
    zt = shifted<MU, +1>(g, zt);
    TWalk w;
    w.init(g, xr);
    Quat<R> b = qone<R>();
    for (int t = 0; t < t0; ++t) { b = qmul(b, Lt.ld(6 + w.par, w.h)); w.step(nt, hts, hwrap); }
    R val[TC];
#pragma unroll
    for (int j = 0; j < TC; ++j) {
      val[j] = R(0);
      if (j < nT) {
        b = qmul(b, Lt.ld(6 + w.par, w.h));
        w.step(nt, hts, hwrap);
        if (valid) val[j] = qdot(qmul(A, b), qmul(D[j], C[j]));
      }
    }
    // Sum the TC values over the warp by a transposing butterfly: each of the
    // first log2(TC) stages trades half of a lane's values with its partner,
    // halving the count; the remaining stages finish the sum.  Afterwards the
    // lanes of each group of 32/TC hold the total of one value j = lo.
    int nv = TC;
    int lo = 0;  // this lane's values are j = lo .. lo + nv - 1
#pragma unroll
    for (int off = 16; off >= 1; off >>= 1) {
      if (nv > 1) {
        const bool upper = (lane & off) != 0;
        const int half = nv / 2;
#pragma unroll
        for (int k = 0; k < TC / 2; ++k) {
          if (k < half) {
            const R send = upper ? val[k] : val[k + half];
            const R keep = upper ? val[k + half] : val[k];
            val[k] = keep + __shfl_xor_sync(0xffffffffu, send, off);
          }
        }
        if (upper) lo += half;
        nv = half;
      } else {
        val[0] += __shfl_xor_sync(0xffffffffu, val[0], off);
      }
    }
    if ((lane & (32 / TC - 1)) == 0 && lo < nT) atomicAdd(&acc[(r - 1) * TC + lo], (double)val[0]);
  }
}

template <int P, int TC>
__global__ void __launch_bounds__(kWilsonThreads) k_wilson(Links<P> Ls, Links<P> Lt, Geom g, int rmax,
                                                           int tmax, double* partials) {
  __shared__ double acc[kWilsonMaxR * TC];
  const int mu = blockIdx.y % 3;
  const int chunk = blockIdx.y / 3;
  const int t0 = chunk * TC;
  const int nT = min(TC, tmax - t0);
  for (int i = threadIdx.x; i < kWilsonMaxR * TC; i += blockDim.x) acc[i] = 0.0;
  __syncthreads();
  const int64_t V = 2 * g.vh;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t base = (int64_t)blockIdx.x * blockDim.x; base < V; base += stride) {
    const int64_t s = base + threadIdx.x;
    const bool valid = s < V;
    const int sv = valid ? (int)s : 0;
    if (mu == 0) wilson_site<P, TC, 0>(Ls, Lt, g, sv, valid, rmax, t0, nT, acc);
    else if (mu == 1) wilson_site<P, TC, 1>(Ls, Lt, g, sv, valid, rmax, t0, nT, acc);
    else wilson_site<P, TC, 2>(Ls, Lt, g, sv, valid, rmax, t0, nT, acc);
  }
  __syncthreads();
  const int bid = blockIdx.y * gridDim.x + blockIdx.x;
  const int per = rmax * TC;
  for (int i = threadIdx.x; i < per; i += blockDim.x) partials[(size_t)bid * per + i] = acc[i];
}

// ---------------------------------------------------------------------------
// Wilson loops, time-outer form.  In the (MU, time) plane with coordinates
// (a, t), S_R(a, t) = U_MU(a, t) ... U_MU(a+R-1, t) and T_T(a, t) = U_t(a, t)
// ... U_t(a, t+T-1), the loop of Eq. 18 at (a, t) is
//   W = (1/2) Tr[S_R(a,t) T_T(a+R,t) S_R(a,t+T)^dag T_T(a,t)^dag]
//     = (F . Q),  F = S_R(a,t) T_T(a+R,t),  Q = T_T(a,t) S_R(a,t+T).
// A thread owns one site of a plane (or of a band of its time slices, when
// the whole plane does not fit) staged in shared memory and holds F for RC
// consecutive R in registers.  Stepping T by one multiplies each F by one
// time link and D = T_T(a,t) by one; Q is then rebuilt along R from D with
// one spatial link per R.  That is two quaternion products and a dot product
// per (R, T), where extending every line per (R, T) costs four to five.
// blockIdx.y = (R chunk, T chunk); chunks after the first start from prefix
// products.  Plane rows are stored with `pad` extra columns repeating the
// first ones, so the lines along MU need no periodic wrap test.  Loop values
// go through a transposing warp reduction into per-warp sums of the work
// unit (FP32 or FP64, the arithmetic's precision), which are folded into the
// block's FP64 totals after each unit in a fixed order (no atomics); per-block sums go to `partials` in a fixed layout
// for k_wilson_rt_final.
// ---------------------------------------------------------------------------
constexpr int kWrtT = 16;  // T values per chunk
// The T loop unrolled by two: W(16,16) on 64^4 FP32 21.8 -> 20.4 ms (the
// sixteen F quaternions stay in place across iterations instead of being
// moved back at the loop edge); by four 21.7 ms.
#ifndef SU2_WILSON_TUNROLL
#define SU2_WILSON_TUNROLL 2
#endif
constexpr int kWilsonTUnroll = SU2_WILSON_TUNROLL;


template <int P, int RC, int NTH>
__global__ void __launch_bounds__(NTH, 1) k_wilson_rt(Links<P> Ls, Links<P> Lt, Geom g, int rmax, int tmax,
                                                      int ntc, int pad, int tile, double* partials) {
  using R = typename Real<P>::T;
  static_assert(RC == 8 || RC == 16, "R chunk must be 8 or 16");
  constexpr int NS = RC * kWrtT;  // (R, T) slots of one chunk
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ double acc[NS];               // block totals; slot k belongs to thread k
  __shared__ R wacc[NTH / 32][NS];         // one work unit's sums per warp (in the arithmetic's precision)
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int rc = blockIdx.y / ntc, tc = blockIdx.y - (blockIdx.y / ntc) * ntc;
  const int r0 = rc * RC, t0 = tc * kWrtT;
  const int nR = min(RC, rmax - r0), nT = min(kWrtT, tmax - t0);
  const int nt = g.n[3];
  // a work unit is `tile` consecutive time slices of one plane.  A whole
  // plane (tile == nt) is staged once, rows read modulo nt; a band of slices
  // stages rows tstart .. tstart + nrows - 1 (mod nt), enough for every line
  // its sites start (T up to ntc * kWrtT beyond the last slice), and reads
  // them without a wrap
  const bool whole = tile >= nt;
  const int ntiles = whole ? 1 : (nt + tile - 1) / tile;
  const int nrows = whole ? nt : tile + ntc * kWrtT;
  const int wrap_at = whole ? nt : 0x7fffffff;
  for (int i = threadIdx.x; i < NS; i += NTH) acc[i] = 0.0;
  for (int i = threadIdx.x; i < (NTH / 32) * NS; i += NTH) (&wacc[0][0])[i] = R(0);
  const int ntr0 = g.n[1] * g.n[2], ntr1 = g.n[0] * g.n[2], ntr2 = g.n[0] * g.n[1];
  const int nunits = (ntr0 + ntr1 + ntr2) * ntiles;
  for (int u = blockIdx.x; u < nunits; u += gridDim.x) {
    const int pl = u / ntiles, tstart = (u - pl * ntiles) * tile;
    const int mu = pl < ntr0 ? 0 : (pl < ntr0 + ntr1 ? 1 : 2);
    const int tr = pl - (mu == 0 ? 0 : (mu == 1 ? ntr0 : ntr0 + ntr1));
    const int nm = mu == 0 ? g.n[0] : (mu == 1 ? g.n[1] : g.n[2]);
    const int tn = min(tile, nt - tstart);  // slices whose sites this unit owns
    const int np = nm * tn;
    // rows of W = nm + pad columns: column c holds plane column c mod nm, so
    // every line a, a+1, ..., a + pad - 1 is read without a wrap test; row r
    // holds time slice tstart + r (mod nt), so lines along t need none either
    const int W = nm + pad;
    Quat<R>* us = reinterpret_cast<Quat<R>*>(smem_raw);   // us[c + W r] = U_mu(c mod nm, tstart + r)
    Quat<R>* ut = us + W * nrows;                         // ut[c + W r] = U_t(c mod nm, tstart + r)
    const int n1st = mu == 0 ? g.n[1] : g.n[0];
    const int c1 = tr % n1st, c2 = tr / n1st;
    __syncthreads();  // the previous unit's readers and the warp-sum fold are done
    for (int i = threadIdx.x; i < W * nrows; i += NTH) {
      const int c = i % W, r = i / W;
      const int a = c % nm;
      Site y;
      y.x0 = mu == 0 ? a : c1;
      y.x1 = mu == 0 ? c1 : (mu == 1 ? a : c2);
      y.x2 = mu == 2 ? a : c2;
      y.x3 = (tstart + r) % nt;
      y.row = y.x1 + g.n[1] * (y.x2 + g.n[2] * y.x3);
      const int h = hidx(g, y), par = parity(y);
      us[i] = Ls.ld(2 * mu + par, h);
      ut[i] = Lt.ld(6 + par, h);
    }
    __syncthreads();
    for (int base = 0; base < np; base += NTH) {
      const int i = base + threadIdx.x;
      const bool valid = i < np;
      const int a = valid ? i % nm : 0, t = valid ? i / nm : 0;   // t: local row of the site
      // F[k] = S_{r0+k+1}(a, t) T_{t0}(a+r0+k+1, t),  D = T_{t0}(a, t)
      Quat<R> F[RC];
      {
        const Quat<R>* row = us + a + W * t;
        Quat<R> sp = qone<R>();
        for (int k = 0; k < r0; ++k) sp = qmul(sp, row[k]);
#pragma unroll
        for (int k = 0; k < RC; ++k) {
          sp = qmul(sp, row[r0 + k]);
          F[k] = sp;
        }
      }
      Quat<R> D = qone<R>();
      int tt = t;                                   // row of t + T - 1 for the next T
      for (int j = 0; j < t0; ++j) {
        D = qmul(D, ut[a + W * tt]);
        const Quat<R>* row = ut + a + r0 + 1 + W * tt;
#pragma unroll
        for (int k = 0; k < RC; ++k) F[k] = qmul(F[k], row[k]);
        tt = tt + 1 == wrap_at ? 0 : tt + 1;
      }
#pragma unroll kWilsonTUnroll
      for (int j = 0; j < nT; ++j) {             // T = t0 + j + 1
        D = qmul(D, ut[a + W * tt]);
        {
          const Quat<R>* row = ut + a + r0 + 1 + W * tt;
#pragma unroll
          for (int k = 0; k < RC; ++k) F[k] = qmul(F[k], row[k]);
        }
        tt = tt + 1 == wrap_at ? 0 : tt + 1;     // row of t + T
        const Quat<R>* row = us + a + W * tt;
        Quat<R> Q = D;
        for (int k = 0; k < r0; ++k) Q = qmul(Q, row[k]);
        R val[RC];
#pragma unroll
        for (int k = 0; k < RC; ++k) {
          Q = qmul(Q, row[r0 + k]);
          val[k] = (valid && k < nR) ? qdot(F[k], Q) : R(0);
        }
        int nv = RC, lo = 0;
#pragma unroll
        for (int off = 16; off >= 1; off >>= 1) {
          if (nv > 1) {
            const bool upper = (lane & off) != 0;
            const int half = nv / 2;
#pragma unroll
            for (int k = 0; k < RC / 2; ++k) {
              if (k < half) {
                const R send = upper ? val[k] : val[k + half];
                const R keep = upper ? val[k + half] : val[k];
                val[k] = keep + __shfl_xor_sync(0xffffffffu, send, off);
              }
            }
            if (upper) lo += half;
            nv = half;
          } else {
            val[0] += __shfl_xor_sync(0xffffffffu, val[0], off);
          }
        }
        // owner lanes hold distinct R slots: plain read-modify-write
        if ((lane & (32 / RC - 1)) == 0 && lo < nR) wacc[warp][lo * kWrtT + j] += val[0];
      }
    }
    __syncthreads();
    // fold the warps' sums into the block totals in a fixed order
    for (int k = threadIdx.x; k < NS; k += NTH) {
      double t = 0.0;
#pragma unroll
      for (int w = 0; w < NTH / 32; ++w) {
        t += (double)wacc[w][k];
        wacc[w][k] = R(0);
      }
      acc[k] += t;
    }
  }
  __syncthreads();
  const size_t bid = (size_t)blockIdx.y * gridDim.x + blockIdx.x;
  for (int i = threadIdx.x; i < NS; i += NTH) partials[bid * NS + i] = acc[i];
}

// out[(R-1) tmax + (T-1)] from k_wilson_rt's per-block sums: one block per
// output adds the gx blocks of its (R chunk, T chunk) in a fixed order.
// excess: the sum of the time links' |U|^2 - 1 over all 1/inv terms in units of
// 2^-58 (k_wilson_tg in FP64), or NULL.
template <int RC>
__global__ void __launch_bounds__(kThreads) k_wilson_rt_final(const double* partials, int gx, int ntc, int tmax,
                                                              double inv, const long long* excess, double* out) {
  const int o = blockIdx.x;
  const int r = o / tmax, t = o % tmax;
  const int y = (r / RC) * ntc + t / kWrtT;
  const int slot = (r % RC) * kWrtT + t % kWrtT;
  double a = 0.0;
  for (int bx = threadIdx.x; bx < gx; bx += blockDim.x) a += __ldcg(partials + ((size_t)y * gx + bx) * (RC * kWrtT) + slot);
  const double tot = block_sum(a);
  if (threadIdx.x == 0) {
    const double w = tot * inv;
    out[o] = excess ? w + w * ((double)(t + 1) * ((double)*excess * 0x1p-58 * inv)) : w;
  }
}

// ---------------------------------------------------------------------------
// Wilson loops in temporal gauge.  The loop of Eq. 18 is gauge invariant, so
// it may be evaluated on any gauge transform U'_mu(x) = G(x) U_mu(x)
// G(x+mu)^dag of the links.  In the (MU, time) plane with coordinates (a, t)
// take G(a, 0) = 1 and G(a, t+1) = G(a, t) U_t(a, t) (each product
// normalised, so G stays a unit quaternion): every time line then becomes
// T_T(a, t) = G(a,t)^dag G(a,t+T), and the loop at (a, t) becomes
//   W = (1/2) Tr[S'_R(a,t) S'_R(a,t+T)^dag] = S'_R(a,t) . S'_R(a,t+T),
// with S'_R(a, r) = U'(a, r) U'(a+1, r) ... U'(a+R-1, r) the spatial line of
// the transformed links (the G between neighbouring links cancel).  A time
// line that wraps past the last slice is G(a,t)^dag P(a) G(a,t') with P(a) =
// G(a, Nt) the Polyakov line, so rows Nt + t' of an extended plane hold
// U'(a, Nt + t') = P(a) U'(a, t') P(a+1)^dag and no loop needs a wrap test.
// Per loop that is one dot product (4 FMA) where the direct form needs two
// quaternion products and a dot (36 FMA); the lines cost one product per
// (site, R), shared by all T.
//
// One block per plane at a time.  A warp owns four columns a; lane (k, c),
// k = lane % 4, c = lane / 4, owns of column 4 warp + k the RO = Nt / 8 rows
// c RO .. (c+1) RO - 1 (the rows its loops start from) and the extended
// rows Nt + 2c, Nt + 2c + 1, so every lane starts loops from RO rows and
// every row it reads beyond its own belongs to its warp: the R loop needs no
// block barrier and no lane branches off.  The time links are scanned in
// the same chunks of RO slices (products within a chunk, then a prefix over
// the chunks) and the transformed spatial links U' of the extended plane are
// staged in shared memory; then for R = 1 .. rmax every thread extends its
// RO + 2 lines by one link, publishes them, and adds the dot products with
// the lines 1 .. kTgT rows ahead into sixteen register accumulators (one per
// T), which a transposing warp reduction leaves in a per-(R, warp) slot; the
// block folds the slots into its FP64 totals in a fixed order after the
// plane.  Row strides are 2 mod 4 quaternions and the origin rows of every
// other chunk are shifted (tg_stride, tg_skew_unit), so the 16-byte shared
// accesses of eight lanes (two chunks of four columns) hit distinct banks.
// Per-block sums go to `partials` in the layout k_wilson_rt_final reads (one
// 16 x 16 chunk).
// ---------------------------------------------------------------------------
#ifndef SU2_WILSON_TG
#define SU2_WILSON_TG 1
#endif
constexpr int kTgT = 16;                 // T values in registers; also the rows added past Nt
constexpr int kTgChunks = 8;             // row chunks of a column (lanes per column)
constexpr int kTgCols = 32 / kTgChunks;  // columns of a warp
constexpr int kTgExt = kTgT / kTgChunks; // extended rows a lane owns
constexpr int kTgThreads = 512;          // planes of up to 64 columns

// q / |q| for |q| near one, as q + q d, d = (1 - |q|^2) / 2: a scale factor is
// itself rounded, to 2^-24 below 1 and 2^-23 above, and the approximate root's
// error near 1 has one sign, which came back four times in every loop (16^4 FP32,
// W to 8 x 8, off FP64: 7.8e-7 with the root, 4.1e-7 with a Newton step on it).
// `bad` is raised from |q|^2 off one by 2^-18 on (the links of FP32 chains stay
// within 1.1e-6 = 2^-19.8, products of eight normalised ones as well): below, the
// kernel drops the time links' norms, 2 T 2^-19 of a loop at most (6e-5 at T = 16,
// all links off alike; a chain's links 1.4e-6).  Giving back their mean, as FP64
// does, took W(16,16) on 64^4 from 4.45 to 4.57 ms.
__device__ __forceinline__ Quat<float> qunit(const Quat<float>& q, bool& bad) {
  const float e = fmaf(-q.x, q.x, fmaf(-q.w, q.w, 1.0f)) - fmaf(q.z, q.z, q.y * q.y);
  bad |= !(fabsf(e) <= 0x1p-18f);
  const float d = 0.5f * e;
  return qmake<float>(fmaf(q.w, d, q.w), fmaf(q.x, d, q.x), fmaf(q.y, d, q.y), fmaf(q.z, d, q.z));
}

// The kernel's arithmetic: FP32 quaternions with FP32 sums, or (FP64) the
// 58-bit fixed point of su2_fixed.cuh with 64-bit sums in units of 2^-52 (one
// plane's sum of one (R, T) and warp is below 2^60).  The time links must be unit
// quaternions, in fixed point all links to 2^-29 (`bad` is raised otherwise; NORMS,
// below, takes more).  The gauge transform normalises the time lines, whose links are unit quaternions only to
// FP64 rounding (together about 1e-16 a link below one in a typical store, 1e-15
// on a loop of T = 12); FP64 sums the time links' |U|^2 - 1 on the way (`excess`),
// and the loops of extent T get the factor 1 + T <|U|^2 - 1> back.  That gives back
// the mean norm, not a loop's own: FP64 raises `bad` where a time link's |U|^2 is
// off one by 2^-47 (7e-15; heat-bath links stay within 7e-16), below which the
// difference is within FP64's rounding of the loop (norms 1e-9 up in half of the
// lattice and down in the other half: 2.5e-10 at T = 12).
template <int P> struct TgMath {
  using E = Quat<float>;
  using A = float;
  template <bool> static __device__ __forceinline__ E load(const Links<P>& L, int cls, int h, bool&) {
    return L.ld(cls, h);
  }
  static __device__ __forceinline__ int64_t excess(const E&, bool&) { return 0; }
  static __device__ __forceinline__ E one() { return qone<float>(); }
  static __device__ __forceinline__ E mul(const E& a, const E& b) { return qmul(a, b); }
  static __device__ __forceinline__ E mul_nd(const E& a, const E& b) { return qmul_nd(a, b); }
  static __device__ __forceinline__ E unit(const E& q, bool& bad) { return qunit(q, bad); }
  static __device__ __forceinline__ A dot(const E& a, const E& b, A s) {
    return fma(a.w, b.w, fma(a.x, b.x, fma(a.y, b.y, fma(a.z, b.z, s))));
  }
  static __device__ __forceinline__ double value(A s) { return (double)s; }
};

template <> struct TgMath<kF64> {
  using E = FixQuat;
  using A = int64_t;
  template <bool NORMS> static __device__ __forceinline__ E load(const Links<kF64>& L, int cls, int h, bool& bad) {
    return fix_unit_link<NORMS ? 16 : 28>(L.ld(cls, h), bad);
  }
  // a time link's |q|^2 - 1 in units of 2^-58
  static __device__ __forceinline__ int64_t excess(const E& q, bool& bad) {
    constexpr int64_t most = (int64_t)1 << (kFixFrac - 47);
    const int64_t x = fix_dot(q, q, -((int64_t)1 << kFixFrac));
    bad |= x < -most || x > most;
    return x;
  }
  static __device__ __forceinline__ E one() { return fix_one(); }
  static __device__ __forceinline__ E mul(const E& a, const E& b) { return fix_mul(a, b); }
  static __device__ __forceinline__ E mul_nd(const E& a, const E& b) {
    return fix_mul(a, fix_conj(b));
  }
  // q (3 - |q|^2) / 2: one Newton step, enough while |q|^2 is within 2^-26 of one
  static __device__ __forceinline__ Fix scaled(const Fix& a, int e) {
    return fix_split(fix_value(a) + (((int64_t)a.h * e) >> kFixLow));
  }
  static __device__ __forceinline__ E unit(const E& q, bool&) {
    const int e = (int)(-fix_dot(q, q, -((int64_t)1 << kFixFrac)) >> 1);
    return E{scaled(q.w, e), scaled(q.x, e), scaled(q.y, e), scaled(q.z, e)};
  }
  static __device__ __forceinline__ A dot(const E& a, const E& b, A s) { return s + (fix_dot(a, b, 32) >> 6); }
  static __device__ __forceinline__ double value(A s) { return fix_to_double<52>(s); }
};

// A factor near one: its excess over one and that of its inverse, units of 2^-58.
struct TgNorm { int64_t d, i; };
__device__ __forceinline__ int64_t tg_times(int64_t x, int64_t y) { return x + y + fix_mulhi(x, y * 64); }
__device__ __forceinline__ TgNorm tg_times(const TgNorm& a, const TgNorm& b) {
  return TgNorm{tg_times(a.d, b.d), tg_times(a.i, b.i)};
}
__device__ __forceinline__ Fix tg_scaled(const Fix& a, int64_t x) {
  const int64_t v = fix_value(a);
  return fix_split(v + fix_mulhi(v, x * 64));
}
__device__ __forceinline__ FixQuat tg_scaled(const FixQuat& q, int64_t x) {
  return FixQuat{tg_scaled(q.w, x), tg_scaled(q.x, x), tg_scaled(q.y, x), tg_scaled(q.z, x)};
}
// |q|; q becomes q / |q|.  With e = |q|^2 - 1, |e| <= 2^-16: the square root's and
// its inverse's binomial series to e^3 (e^4 is below 2^-63).
__device__ __forceinline__ TgNorm tg_take_norm(FixQuat& q) {
  const int64_t e = fix_dot(q, q, -((int64_t)1 << kFixFrac));
  const int64_t x = (int64_t)((uint64_t)e << 20);                  // 2^-78
  const int64_t e2 = fix_mulhi(x, x), e3 = fix_mulhi(e2, x);       // 2^-92, 2^-106
  const TgNorm n{(e >> 1) - (e2 >> 37) + (e3 >> 52), ((3 * e2) >> 37) - (e >> 1) - ((5 * e3) >> 52)};
  q = tg_scaled(q, n.i);
  return n;
}

// The value of the lane n below.
__device__ __forceinline__ float tg_lane_up(float v, int n) { return __shfl_up_sync(0xffffffffu, v, n); }
__device__ __forceinline__ Fix tg_lane_up(const Fix& v, int n) {
  return Fix{__shfl_up_sync(0xffffffffu, v.h, n), __shfl_up_sync(0xffffffffu, v.l, n)};
}
__device__ __forceinline__ TgNorm tg_lane_up(const TgNorm& v, int n) {
  return TgNorm{__shfl_up_sync(0xffffffffu, v.d, n), __shfl_up_sync(0xffffffffu, v.i, n)};
}
template <class Q> __device__ __forceinline__ Q tg_lane_up(const Q& q, int n) {
  Q r;
  r.w = tg_lane_up(q.w, n);
  r.x = tg_lane_up(q.x, n);
  r.y = tg_lane_up(q.y, n);
  r.z = tg_lane_up(q.z, n);
  return r;
}

// Site (column a, slice 0) of the plane (mu, c1, c2).
__device__ __forceinline__ Site plane_site(const Geom& g, int mu, int a, int c1, int c2) {
  Site y;
  y.x0 = mu == 0 ? a : c1;
  y.x1 = mu == 0 ? c1 : (mu == 1 ? a : c2);
  y.x2 = mu == 2 ? a : c2;
  y.x3 = 0;
  y.row = y.x1 + g.n[1] * y.x2;
  return y;
}

// Row layout of a staged plane, chunks of RO rows.  Eight lanes of a 16-byte
// shared access are two chunks of four columns, so rows c RO + i and
// (c+1) RO + i must start 4 mod 8 quaternions apart (16 banks), and so must
// the extended rows 2c + e and 2c + 2 + e.  The latter needs a
// row stride S = 2 mod 4; the former then holds for RO = 2 mod 4 and, with
// the origin rows of odd chunks shifted by tg_skew_unit quaternions, for RO
// = 0 mod 4 (shift 4) and RO odd (S = 2 mod 8, shift 2).  S leaves room for
// the shift after the last column.
template <int RO> __host__ __device__ constexpr int tg_skew_unit() { return RO % 4 == 0 ? 4 : (RO % 2 ? 2 : 0); }
template <int RO> __host__ __device__ __forceinline__ int tg_stride(int cols) {
  const int m = RO % 2 ? 8 : 4;
  const int lo = cols + tg_skew_unit<RO>();
  return lo + ((2 - lo % m) + m) % m;
}
// row r of the staged plane: kTgChunks RO origin rows, then the extended ones
template <int RO> __device__ __forceinline__ int tg_row(int r, int stride) {
  return r * stride + (r < kTgChunks * RO ? tg_skew_unit<RO>() * ((r / RO) & 1) : 0);
}

// EXACT: Nt = 8 RO (every origin row starts loops), a constant to the compiler: with
// Nt read at run time the rows' slices took integer divisions in phases 1 and 3
// (48^3x8 FP32, W(1,4): 235 us, so 216; with the prefix over the chunks by
// shuffles instead of through shared memory 186).
// NORMS (FP64): links up to 2^-16 off unit norm (in |U|^2; a configuration stored
// in FP32, say).  A loop carries the product of its time links' norms, N(a, r + T)
// N(a + R, r + T) / (N(a, r) N(a + R, r)) with N(a, r) the norms' product along
// column a up to row r: the lines published to the other lanes get the factor N N
// of their two columns, the lines that loops start from its inverse.
// 32^4, links rounded to FP32, W(16,16): 82 ms multiplied out by the time-outer
// kernel, here 4.7, after the 3.4 of the kernel without NORMS that found them.
// Compiled for even RO.
template <int P, int RO, bool EXACT, bool NORMS>
__global__ void __launch_bounds__(kTgThreads, 1)
    k_wilson_tg(Links<P> Ls, Links<P> Lt, Geom g, int rmax, int tmax, double* partials, double* flag,
                unsigned long long* excess) {
  using M = TgMath<P>;
  using E = typename M::E;
  using A = typename M::A;
  constexpr int NO = kTgChunks * RO;               // origin rows, at least Nt
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ double acc64[16 * kTgT];              // block totals; slot (R-1) kTgT + T-1
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = (int)(blockDim.x >> 5);
  const int nt = EXACT ? NO : g.n[3];
  const int hts = g.n0h * g.st[3];
  for (int i = threadIdx.x; i < 16 * kTgT; i += blockDim.x) acc64[i] = 0.0;
  const int ntr0 = g.n[1] * g.n[2], ntr1 = g.n[0] * g.n[2], ntr2 = g.n[0] * g.n[1];
  const int nunits = ntr0 + ntr1 + ntr2;
  const int c = lane / kTgCols, r0 = c * RO;
  bool bad = false;
  int64_t over = 0;
  // slice of row r: rows past the last slice repeat the first ones
  auto slice = [&](int r) -> int {
    if constexpr (EXACT) {
      return r < NO ? r : (r - NO) % NO;
    } else {
      while (r >= nt) r -= nt;
      return r;
    }
  };
  for (int u = blockIdx.x; u < nunits; u += gridDim.x) {
    const int mu = u < ntr0 ? 0 : (u < ntr0 + ntr1 ? 1 : 2);
    const int tr = u - (mu == 0 ? 0 : (mu == 1 ? ntr0 : ntr0 + ntr1));
    const int nm = mu == 0 ? g.n[0] : (mu == 1 ? g.n[1] : g.n[2]);
    const int n1st = mu == 0 ? g.n[1] : g.n[0];
    const int c1 = tr % n1st, c2 = tr / n1st;
    const int W = nm + rmax - 1;       // columns of the staged plane (column cc is plane column cc mod nm)
    const int SU = tg_stride<RO>(W), SS = tg_stride<RO>(nm);
    E* Ue = reinterpret_cast<E*>(smem_raw);      // Ue[tg_row(r, SU) + cc] = U'(cc, r), r < NO + kTgT
    E* Sb = Ue + (NO + kTgT) * SU + 4;           // Sb[tg_row(r, SS) + a]: G(a, r), then S'_R(a, r)
    E* Pb = Sb + (NO + kTgT) * SS + 4;           // Pb[a] = P(a)
    TgNorm* Nb = reinterpret_cast<TgNorm*>(Pb + nm);   // NORMS: Nb[r nm + a] = N(a, r), r < NO
    TgNorm* Np = Nb + NO * nm;                   // Np[a] = N(a, Nt)
    A* wsum = reinterpret_cast<A*>(NORMS ? (void*)(Np + nm) : (void*)(Pb + nm));   // per R, warp and T
    const int a = kTgCols * warp + lane % kTgCols;
    const bool active = a < nm;
    __syncthreads();  // the previous plane's readers are done
    // (1) this lane's links, loaded together: the time and spatial links of
    // its origin rows and the spatial links that its extended rows repeat;
    // then the time links' products within the chunk
    E us[RO + kTgExt], Q = M::one();
    TgNorm n{0, 0};
    if (active) {
      E ut[RO];
      const Site y = plane_site(g, mu, a, c1, c2);
      const int h0 = hidx(g, y), par0 = parity(y);
#pragma unroll
      for (int i = 0; i < RO; ++i) {
        const int t = slice(r0 + i), h = h0 + hts * t, par = (par0 ^ t) & 1;
        ut[i] = EXACT || r0 + i < nt ? M::template load<NORMS>(Lt, 6 + par, h, bad) : M::one();
        if constexpr (!NORMS) over += M::excess(ut[i], bad);
        us[i] = M::template load<NORMS>(Ls, 2 * mu + par, h, bad);
      }
#pragma unroll
      for (int e = 0; e < kTgExt; ++e) {
        const int t = slice(NO + kTgExt * c + e), h = h0 + hts * t, par = (par0 ^ t) & 1;
        us[RO + e] = M::template load<NORMS>(Ls, 2 * mu + par, h, bad);
      }
      if constexpr (NORMS) {
#pragma unroll
        for (int i = 0; i < RO; ++i) {
          Nb[(r0 + i) * nm + a] = n;
          n = tg_times(n, tg_take_norm(ut[i]));
        }
      }
#pragma unroll
      for (int i = 0; i < RO; ++i) {
        Sb[tg_row<RO>(r0 + i, SS) + a] = Q;
        Q = M::unit(M::mul(Q, ut[i]), bad);
      }
    }
    // (2) prefix over a column's chunks, the warp's lanes: G(a, r) for the
    // thread's rows, P(a) = G(a, Nt).  Products of up to eight unit quaternions,
    // normalised with G.
#pragma unroll
    for (int d = 1; d < kTgChunks; d *= 2) {
      const E before = tg_lane_up(Q, d * kTgCols);
      if (c >= d) Q = M::mul(before, Q);
      if constexpr (NORMS) {
        const TgNorm m = tg_lane_up(n, d * kTgCols);
        if (c >= d) n = tg_times(m, n);
      }
    }
    if (active && c == kTgChunks - 1) {
      Pb[a] = M::unit(Q, bad);
      if constexpr (NORMS) Np[a] = n;
    }
    Q = tg_lane_up(Q, kTgCols);
    if constexpr (NORMS) n = tg_lane_up(n, kTgCols);
    if (active && c > 0) {
#pragma unroll
      for (int i = 0; i < RO; ++i) {
        E* p = Sb + tg_row<RO>(r0 + i, SS) + a;
        *p = M::unit(M::mul(Q, *p), bad);
        if constexpr (NORMS) Nb[(r0 + i) * nm + a] = tg_times(n, Nb[(r0 + i) * nm + a]);
      }
    }
    __syncthreads();
    // (3) U'(a, r) = G(a, t) U_mu(a, t) G(a+1, t)^dag for the lane's rows,
    // conjugated by P on the rows past the last slice; column a + nm (a <
    // rmax - 1) repeats column a
    if (active) {
      const int an = a + 1 == nm ? 0 : a + 1;
#pragma unroll
      for (int i = 0; i < RO + kTgExt; ++i) {
        const int r = i < RO ? r0 + i : NO + kTgExt * c + (i - RO);
        const int gt = tg_row<RO>(slice(r), SS);
        E v = M::mul_nd(M::mul(Sb[gt + a], us[i]), Sb[gt + an]);
        if (EXACT ? i >= RO : r >= nt) v = M::mul_nd(M::mul(Pb[a], v), Pb[an]);
        const int ru = tg_row<RO>(r, SU);
        Ue[ru + a] = v;
        if (a < rmax - 1) Ue[ru + a + nm] = v;
      }
    }
    __syncthreads();  // Sb now holds lines
    // (4) R = 1 .. rmax, warp-synchronous.  The thread's rows start at
    // bu / bs (origin rows, shifted by sk) and bue / bse (extended rows).
    constexpr int unit = tg_skew_unit<RO>();
    const int sk = unit * (c & 1);
    const int bu = r0 * SU + sk + a, bs = r0 * SS + sk + a;
    const int bue = (NO + kTgExt * c) * SU + a, bse = (NO + kTgExt * c) * SS + a;
    const int rows = nt - r0;  // loops start from the first `rows` of the lane's origin rows
    E own[RO];  // the origin rows' lines; the extended rows' stay in Sb (NORMS: in ext)
    E from[NORMS ? RO : 1], ext[NORMS ? kTgExt : 1];   // NORMS: the lines that loops start from
    auto norms = [&](int r, int b) {   // N(a, r) N(b, r)
      TgNorm n{0, 0};
      for (int col : {a, b}) {
        const TgNorm m = Nb[slice(r) * nm + col];
        n = tg_times(n, r < nt ? m : tg_times(m, Np[col]));
      }
      return n;
    };
    A acc[kTgT];
#pragma unroll
    for (int k = 0; k < kTgT; ++k) acc[k] = A(0);
    for (int Rl = 1; Rl <= rmax; ++Rl) {
      if (active) {
#pragma unroll
        for (int i = 0; i < RO; ++i) {
          const E v = Ue[bu + i * SU + Rl - 1];
          own[i] = Rl == 1 ? v : M::mul(own[i], v);
          if constexpr (NORMS) {
            const TgNorm n = norms(r0 + i, a + Rl < nm ? a + Rl : a + Rl - nm);
            Sb[bs + i * SS] = tg_scaled(own[i], n.d);
            from[i] = tg_scaled(own[i], n.i);
          } else {
            Sb[bs + i * SS] = own[i];
          }
        }
#pragma unroll
        for (int e = 0; e < kTgExt; ++e) {
          const E v = Ue[bue + e * SU + Rl - 1];
          E* p = Sb + bse + e * SS;
          if constexpr (NORMS) {
            ext[e] = Rl == 1 ? v : M::mul(ext[e], v);
            *p = tg_scaled(ext[e], norms(NO + kTgExt * c + e, a + Rl < nm ? a + Rl : a + Rl - nm).d);
          } else {
            *p = Rl == 1 ? v : M::mul(*p, v);
          }
        }
      }
      __syncwarp();
      if (active) {
        // origin rows r0 + i, i < RO, against rows r0 + j, j = i + T; the
        // common case, all sixteen T and Nt a multiple of eight, takes a copy
        // without the tests
        auto dots = [&](auto full_c) {
          constexpr bool FULL = decltype(full_c)::value;
#pragma unroll
          for (int j = 1; j < RO + kTgT; ++j) {
            if (!FULL && j >= RO + tmax) break;
            E w;
            if (!NORMS && j < RO) {
              w = own[j < RO ? j : 0];
            } else {
              const int rr = r0 + j;  // chunk c + j / RO while an origin row
              w = Sb[rr * SS + (rr < NO ? unit * ((c + j / RO) & 1) : 0) + a];
            }
#pragma unroll
            for (int i = 0; i < RO; ++i) {
              const int T = j - i;
              if (T >= 1 && T <= kTgT && (FULL || (T <= tmax && (EXACT || i < rows))))
                acc[T - 1] = M::dot(NORMS ? from[NORMS ? i : 0] : own[i], w, acc[T - 1]);
            }
          }
        };
        if (EXACT && tmax == kTgT) dots(std::true_type{});
        else dots(std::false_type{});
      }
      __syncwarp();  // the lines are read before the next R overwrites them
      // this R's sums: a transposing butterfly leaves lanes 2k and 2k+1 the
      // warp total of slot lo; the even lanes store it in this R's slot
      int lo = 0;
#pragma unroll
      for (int lev = 0; lev < 4; ++lev) {
        const int off = 16 >> lev, half = 8 >> lev;
        const bool upper = (lane & off) != 0;
#pragma unroll
        for (int m = 0; m < 8; ++m) {
          if (m < half) {
            const A send = upper ? acc[m] : acc[m + half];
            const A keep = upper ? acc[m + half] : acc[m];
            acc[m] = keep + __shfl_xor_sync(0xffffffffu, send, off);
          }
        }
        if (upper) lo += half;
      }
      acc[0] += __shfl_xor_sync(0xffffffffu, acc[0], 1);
      if ((lane & 1) == 0) wsum[((Rl - 1) * nw + warp) * kTgT + lo] = acc[0];
#pragma unroll
      for (int k = 0; k < kTgT; ++k) acc[k] = A(0);
    }
    __syncthreads();
    // the plane's sums, warps in a fixed order
    for (int s = threadIdx.x; s < rmax * kTgT; s += blockDim.x) {
      double t = 0.0;
      for (int w = 0; w < nw; ++w) t += M::value(wsum[(s / kTgT * nw + w) * kTgT + s % kTgT]);
      acc64[s] += t;
    }
  }
  if (bad) *flag = 1.0;
  if constexpr (P == kF64 && !NORMS) {
    over = warp_sum(over);
    if (lane == 0) atomicAdd(excess, (unsigned long long)over);   // exact in any order
  }
  __syncthreads();
  for (int i = threadIdx.x; i < 16 * kTgT; i += blockDim.x) partials[(size_t)blockIdx.x * 16 * kTgT + i] = acc64[i];
}

// out[(R-1) tmax + (T-1)]: one block per output adds the per-block sums of the
// three directions and all x-blocks of T's chunk, in a fixed order.
template <int TC>
__global__ void __launch_bounds__(kThreads) k_wilson_final(const double* partials, int gx, int rmax, int tmax,
                                                           double inv, double* out) {
  const int o = blockIdx.x;
  const int r = o / tmax, t = o % tmax;
  const int c = t / TC, j = t % TC;
  const int per = rmax * TC;
  const int n = 3 * gx;
  double a = 0.0;
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    const int m = i / gx, bx = i % gx;
    a += __ldcg(partials + (size_t)((3 * c + m) * gx + bx) * per + r * TC + j);
  }
  const double tot = block_sum(a);
  if (threadIdx.x == 0) out[o] = tot * inv;
}

// ---------------------------------------------------------------------------
// Canonical FP64 host layout (site-major, direction, component) <-> store.
// ---------------------------------------------------------------------------
template <int P>
__global__ void __launch_bounds__(kThreads) k_to_canonical(Links<P> L, Geom g, double* c,
                                                           int64_t s0, int64_t ns) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t w = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; w < 4 * ns; w += stride) {
    const uint32_t s = (uint32_t)(s0 + (w >> 2));
    const int mu = (int)(w & 3);
    const Site x = site_from_index(g, s);
    const auto q = L.ld(2 * mu + parity(x), hidx(g, x));
    double* o = c + 4 * w;
    o[0] = q.w; o[1] = q.x; o[2] = q.y; o[3] = q.z;
  }
}

// Two 16-byte loads a link (eight-byte ones, a quarter of each 32-byte sector at a
// time, took 955 us on 64^4 FP32, 3.4 TB/s).
template <int P>
__global__ void __launch_bounds__(kThreads) k_from_canonical(Links<P> L, Geom g, const double* c,
                                                             int64_t s0, int64_t ns, int wide) {
  using R = typename Real<P>::T;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t w = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; w < 4 * ns; w += stride) {
    const uint32_t s = (uint32_t)(s0 + (w >> 2));
    const int mu = (int)(w & 3);
    const Site x = site_from_index(g, s);
    const double* i = c + 4 * w;
    double2 a, b;
    if (wide) {
      a = reinterpret_cast<const double2*>(i)[0];
      b = reinterpret_cast<const double2*>(i)[1];
    } else {
      a = make_double2(i[0], i[1]);
      b = make_double2(i[2], i[3]);
    }
    L.st(2 * mu + parity(x), hidx(g, x), qmake<R>((R)a.x, (R)a.y, (R)b.x, (R)b.y));
  }
}

__global__ void k_add_u32(uint32_t* p, uint32_t v) { *p += v; }

// ---------------------------------------------------------------------------
// Host launchers
// ---------------------------------------------------------------------------
cudaError_t launch_init(const LatticeView& v, int start, PhiloxKey key, uint32_t lattice_tag,
                        cudaStream_t st) {
  const RoundKeys rk = round_keys(key);
  SU2_DISPATCH(v.prec, {
    auto L = links_of<P>(v.links, v.g.vh);
    const int gr = grid_for(k_init<P>, 8 * v.g.vh);
    k_init<P><<<gr, kThreads, 0, st>>>(L, v.g, start, rk, lattice_tag);
  });
  count_launches(1);
  return cudaGetLastError();
}

cudaError_t launch_overrelax(const LatticeView& v, int mu, int parity, cudaStream_t st) {
  SU2_DISPATCH(v.prec, SU2_DISPATCH_MU(mu, {
    auto L = links_of<P, hb_addr<P, kClassPtr>>(v.links, v.g.vh);
    auto launch = [&](auto kernel) {
      kernel<<<grid_for(kernel, v.g.vh), kThreads, 0, st>>>(L, v.g, Substep{mu, parity});
    };
    if (parity == 0) launch(k_overrelax<P, hb_dir<P, MU>, hb_dir<P, 0>>);
    else launch(k_overrelax<P, hb_dir<P, MU>, hb_dir<P, 1>>);
  }));
  count_launches(1);
  return cudaGetLastError();
}

cudaError_t launch_plaquette(const LatticeView& v, const Scratch& s, cudaStream_t st, int64_t s0, int64_t ns) {
  if (ns < 0) ns = 2 * v.g.vh;
  SU2_DISPATCH(v.prec, {
    auto L = links_of<P>(v.links, v.g.vh);
    const int gr = grid_for(k_plaquette<P>, ns);
    k_plaquette<P><<<gr, kThreads, 0, st>>>(L, v.g, s0, ns, s.partials, s.counter, s.out);
  });
  count_launches(1);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Time lines (for the Polyakov loop of a lattice split into time slabs,
// Section 2 Eqs. 14-15): for every spatial site xs in [x0, x0 + nx) the
// product of its time links at slices t0, t0 + 1, ..., t0 + nt - 1 in that
// order, to out[4 (xs - x0) + c] in FP64.
// ---------------------------------------------------------------------------
template <int P>
__global__ void __launch_bounds__(kThreads) k_time_lines(Links<P> L, Geom g, int t0, int nt, int64_t x0, int64_t nx,
                                                         double* out) {
  using R = typename Real<P>::T;
  const int64_t nsig = 2 * g.vh / g.n[3];
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nx; i += stride) {
    const int64_t xs = x0 + i;
    Quat<R> pr = qone<R>();
    for (int t = t0; t < t0 + nt; ++t) {
      const Site x = site_from_index(g, (uint32_t)(xs + nsig * t));
      pr = qmul(pr, L.ld(6 + parity(x), hidx(g, x)));
    }
    double* o = out + 4 * i;
    o[0] = pr.w; o[1] = pr.x; o[2] = pr.y; o[3] = pr.z;
  }
}

cudaError_t launch_time_lines(const LatticeView& v, int t0, int nt, int64_t x0, int64_t nx, double* out,
                              cudaStream_t st) {
  SU2_DISPATCH(v.prec, {
    auto L = links_of<P>(v.links, v.g.vh);
    const int gr = grid_for(k_time_lines<P>, nx);
    k_time_lines<P><<<gr, kThreads, 0, st>>>(L, v.g, t0, nt, x0, nx, out);
  });
  count_launches(1);
  return cudaGetLastError();
}

cudaError_t launch_polyakov(const LatticeView& v, const Scratch& s, cudaStream_t st, const SweepEpilogue* ep) {
  SweepEpilogue e{};
  if (ep) e = *ep;
  SU2_DISPATCH(v.prec, {
    auto L = links_of<P, kClassPtr>(v.links, v.g.vh);
    const int64_t nsig = 2 * v.g.vh / v.g.n[3];
    const int lg = polyakov_segments(v.g.n[3]);
    auto launch = [&](auto kernel) {
      const int gr = grid_for(kernel, nsig << lg);
      return launch_pdl(overlaps(v), kernel, dim3(gr), kThreads, st, L, v.g, lg, s.partials, s.counter, s.out, e, (int)overlaps(v));
    };
    const cudaError_t err = overlaps(v) ? launch(k_polyakov<P, false>) : launch(k_polyakov<P, true>);
    if (err != cudaSuccess) return err;
  });
  count_launches(1);
  return cudaGetLastError();
}

cudaError_t launch_batch_measure(int prec, bool polyakov, const BatchLattice* desc, const BatchBlock4* blocks,
                                 int nblocks, double* partials, unsigned int* counters, double* out,
                                 cudaStream_t st) {
  SU2_DISPATCH(prec, {
    if (polyakov) k_batch_measure<P, true><<<nblocks, kThreads, 0, st>>>(desc, blocks, partials, counters, out);
    else k_batch_measure<P, false><<<nblocks, kThreads, 0, st>>>(desc, blocks, partials, counters, out);
  });
  count_launches(1);
  return cudaGetLastError();
}

cudaError_t launch_ape(const LatticeView& src, void* dst, double alpha, cudaStream_t st) {
  SU2_DISPATCH(src.prec, {
    auto S = links_of<P, hb_addr<P, kClassPtr>>(src.links, src.g.vh);
    auto D = links_of<P, hb_addr<P, kClassPtr>>(dst, src.g.vh);
    // the y-slices (parities; in FP64 link classes) share the machine
    const int slices = P == kF64 ? 6 : 2;
    auto launch = [&](auto kernel) {
      int gx = grid_for(kernel, slices * src.g.vh) / slices;
      if (gx < 1) gx = 1;
      return launch_pdl(overlaps(src), kernel, dim3(gx, slices), kThreads, st, S, D, src.g, alpha, (int)overlaps(src));
    };
    const cudaError_t e = overlaps(src) ? launch(k_ape<P, false>) : launch(k_ape<P, true>);
    if (e != cudaSuccess) return e;
  });
  count_launches(1);
  return cudaGetLastError();
}

cudaError_t launch_copy_spatial(const LatticeView& src, void* dst, cudaStream_t st) {
  SU2_DISPATCH(src.prec, {
    auto S = links_of<P>(src.links, src.g.vh);
    auto D = links_of<P>(dst, src.g.vh);
    const int gr = grid_for(k_copy_spatial<P>, 6 * src.g.vh);
    k_copy_spatial<P><<<gr, kThreads, 0, st>>>(S, D);
  });
  count_launches(1);
  return cudaGetLastError();
}

template <int P> struct WilsonChunk { static constexpr int tc = 16; };
template <> struct WilsonChunk<kF64> { static constexpr int tc = 8; };

// Plane kernel shape per arithmetic precision: T chunk and block size.
#ifndef SU2_WILSON_RT
#define SU2_WILSON_RT 1
#endif
constexpr int kWilsonRtThreads = 512;
// dynamic shared memory of the time-outer kernel: 227 KB per block minus its
// static accumulators (18 KB at RC = 16)
constexpr int kWilsonRtSmemMax = 208 * 1024;

template <int P, int RC>
static cudaError_t launch_wilson_rt_rc(const LatticeView& v, const void* spatial, int rmax, int tmax, int tile,
                                       int smem, const Scratch& s, cudaStream_t st) {
  constexpr int NTH = kWilsonRtThreads;
  // the shared-memory limit is raised once per device (concurrent first
  // calls from several host threads wait on the device's once_flag)
  static std::once_flag attr_once[64];
  static cudaError_t attr_err[64];
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev >= 0 && dev < 64) {
    std::call_once(attr_once[dev], [dev]() {
      attr_err[dev] = cudaFuncSetAttribute(k_wilson_rt<P, RC, NTH>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                           kWilsonRtSmemMax);
    });
    if (attr_err[dev] != cudaSuccess) return attr_err[dev];
  }
  int per_sm = 1;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_wilson_rt<P, RC, NTH>, NTH, smem);
  if (per_sm < 1) per_sm = 1;
  const int nrc = (rmax + RC - 1) / RC, ntc = (tmax + kWrtT - 1) / kWrtT;
  const int nchunks = nrc * ntc;
  const int ntiles = (v.g.n[3] + tile - 1) / tile;
  const int64_t nunits = (int64_t)(v.g.n[1] * v.g.n[2] + v.g.n[0] * v.g.n[2] + v.g.n[0] * v.g.n[1]) * ntiles;
  int64_t gx = ((int64_t)device_info().sms * per_sm + nchunks - 1) / nchunks;
  if (gx > nunits) gx = nunits;
  const int64_t cap = (int64_t)kScratchPartials / (RC * kWrtT) / nchunks;
  if (gx > cap) gx = cap;
  if (gx < 1) gx = 1;
  auto Lt = links_of<P>(v.links, v.g.vh);
  auto Ls = links_of<P>(const_cast<void*>(spatial), v.g.vh);
  k_wilson_rt<P, RC, NTH><<<dim3((unsigned)gx, nchunks), NTH, smem, st>>>(Ls, Lt, v.g, rmax, tmax, ntc, nrc * RC,
                                                                         tile, s.partials);
  count_launches(1);
  const int64_t V = 2 * v.g.vh;
  k_wilson_rt_final<RC><<<rmax * tmax, kThreads, 0, st>>>(s.partials, (int)gx, ntc, tmax, 1.0 / (3.0 * (double)V),
                                                          nullptr, s.out);
  count_launches(1);
  return cudaGetLastError();
}

// The time-outer kernel with as many time slices per work unit as fit in
// shared memory next to the ntc * 16 slices of line overhang (the whole
// plane when it fits); *used = false if not even one slice fits.  FP64 runs
// 8-wide R chunks (register budget).
template <int P>
static cudaError_t launch_wilson_rt(const LatticeView& v, const void* spatial, int rmax, int tmax,
                                    const Scratch& s, cudaStream_t st, bool* used) {
  using R = typename Real<P>::T;
  *used = false;
  if (!SU2_WILSON_RT) return cudaSuccess;
  const int nmax = v.g.n[0] > v.g.n[1] ? (v.g.n[0] > v.g.n[2] ? v.g.n[0] : v.g.n[2])
                                       : (v.g.n[1] > v.g.n[2] ? v.g.n[1] : v.g.n[2]);
  const int rc = (rmax <= 8 || P == kF64) ? 8 : 16;
  const int pad = (rmax + rc - 1) / rc * rc;  // columns a .. a + pad - 1 of a row
  const int overhang = (tmax + kWrtT - 1) / kWrtT * kWrtT;
  const int row_bytes = 2 * (nmax + pad) * (int)sizeof(Quat<R>);
  int tile, smem;
  if (row_bytes * v.g.n[3] <= kWilsonRtSmemMax) {
    tile = v.g.n[3];  // the whole plane, rows read modulo nt
    smem = row_bytes * tile;
  } else {
    tile = kWilsonRtSmemMax / row_bytes - overhang;
    if (tile < 1) return cudaSuccess;
    smem = row_bytes * (tile + overhang);
  }
  *used = true;
  if (rc == 8) return launch_wilson_rt_rc<P, 8>(v, spatial, rmax, tmax, tile, smem, s, st);
  if constexpr (P != kF64) return launch_wilson_rt_rc<P, 16>(v, spatial, rmax, tmax, tile, smem, s, st);
  return cudaErrorInvalidValue;
}

// Whether the time-outer kernel is the faster one below FP64: wide planes, whose
// temporal-gauge block is alone on its SM and waits at its barriers, with so few
// loops that the transform is not made good.  It counts more with few time slices
// and where Nt does not fill the eight row chunks; from R = 5 on the time-outer
// kernel's chunk of eight is well used.  FP32, temporal gauge against time-outer, us:
// 64^3x2 W(16,2) 1150 and 635, W(1,1) 403 and 303; 48^3x10 W(4,1) 297 and 224,
// W(8,8) 511 and 569; 48^3x48 W(16,1) 1155 and 998, W(4,1) 497 and 671.  Up to 32
// columns temporal gauge is faster but for the longest lines at T = 1 (24^3x20
// W(16,1) 1.07 times the other's); at 48^3x12 W(1,1) takes 267 against 313.
static bool time_outer_is_faster(int nmax, int nt, int rmax, int tmax) {
  if (nmax <= 32) return false;
  const bool ragged = nt % kTgChunks != 0;
  if (nt < 16) return tmax <= (rmax >= 5 ? 4 : rmax >= 3 ? 2 : ragged && nt <= 10);
  if (nt < 32) return tmax <= (rmax >= 5 ? 2 : rmax >= 3 && ragged);
  return tmax <= (rmax >= 5);
}

// The temporal-gauge kernel when R and T are at most 16, Nt is at most 64, one
// block holds four columns a warp of the widest plane, and the staged plane
// fits in shared memory; *used = false otherwise.
template <int P, int RO, bool EXACT, bool NORMS>
static cudaError_t launch_wilson_tg_rows(const LatticeView& v, const void* spatial, int rmax, int tmax,
                                         const Scratch& s, double* flag, cudaStream_t st, bool* used) {
  using E = typename TgMath<P>::E;
  *used = false;
  const int nmax = std::max(v.g.n[0], std::max(v.g.n[1], v.g.n[2]));
  const int nr = kTgChunks * RO + kTgT;
  const int nth = (nmax + kTgCols - 1) / kTgCols * 32;
  if (nth > kTgThreads) return cudaSuccess;
  int dev = 0;
  cudaGetDevice(&dev);
  int optin = 0;
  cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  cudaFuncAttributes fa;
  cudaError_t e = cudaFuncGetAttributes(&fa, k_wilson_tg<P, RO, EXACT, NORMS>);
  if (e != cudaSuccess) return e;
  const int64_t smem = ((int64_t)nr * tg_stride<RO>(nmax + rmax - 1) + 4 + (int64_t)nr * tg_stride<RO>(nmax) + 4 +
                        (int64_t)nmax) *
                       (int64_t)sizeof(E) +
                       (int64_t)rmax * (nth / 32) * kTgT * (int64_t)sizeof(typename TgMath<P>::A) +
                       (NORMS ? (int64_t)(kTgChunks * RO + 1) * nmax * (int64_t)sizeof(TgNorm) : 0);
  const int64_t dyn_max = (int64_t)optin - (int64_t)fa.sharedSizeBytes;
  if (smem > dyn_max) return cudaSuccess;
  // raised once per device, as for the time-outer kernel
  static std::once_flag attr_once[64];
  static cudaError_t attr_err[64];
  if (dev >= 0 && dev < 64) {
    const int lim = (int)dyn_max;
    std::call_once(attr_once[dev], [dev, lim]() {
      attr_err[dev] = cudaFuncSetAttribute(k_wilson_tg<P, RO, EXACT, NORMS>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
    });
    if (attr_err[dev] != cudaSuccess) return attr_err[dev];
  }
  int per_sm = 1;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_wilson_tg<P, RO, EXACT, NORMS>, nth, (size_t)smem);
  if (per_sm < 1) per_sm = 1;
  const int64_t nunits = (int64_t)v.g.n[1] * v.g.n[2] + (int64_t)v.g.n[0] * v.g.n[2] + (int64_t)v.g.n[0] * v.g.n[1];
  int64_t gx = (int64_t)device_info().sms * per_sm;
  if (gx > nunits) gx = nunits;
  const int64_t cap = (int64_t)kScratchPartials / (16 * kTgT);
  if (gx > cap) gx = cap;
  *used = true;
  auto Lt = links_of<P>(v.links, v.g.vh);
  auto Ls = links_of<P>(const_cast<void*>(spatial), v.g.vh);
  // a word of the counters' 256 bytes, away from the reductions' own
  unsigned long long* excess = P == kF64 && !NORMS ? reinterpret_cast<unsigned long long*>(s.counter + 32) : nullptr;
  if (excess) e = cudaMemsetAsync(excess, 0, sizeof *excess, st);
  if (e != cudaSuccess) return e;
  k_wilson_tg<P, RO, EXACT, NORMS><<<(unsigned)gx, nth, (size_t)smem, st>>>(Ls, Lt, v.g, rmax, tmax, s.partials, flag, excess);
  count_launches(1);
  const int64_t V = 2 * v.g.vh;
  k_wilson_rt_final<16><<<rmax * tmax, kThreads, 0, st>>>(s.partials, (int)gx, 1, tmax, 1.0 / (3.0 * (double)V),
                                                          reinterpret_cast<const long long*>(excess), s.out);
  count_launches(1);
  return cudaGetLastError();
}

template <int P>
static cudaError_t launch_wilson_tg(const LatticeView& v, const void* spatial, int rmax, int tmax,
                                    const Scratch& s, WilsonLinks links, double* flag, cudaStream_t st, bool* used) {
  *used = false;
  if (!SU2_WILSON_TG || rmax > 16 || tmax > kTgT || links == kWilsonAny) return cudaSuccess;
  if (P != kF64 && time_outer_is_faster(std::max(v.g.n[0], std::max(v.g.n[1], v.g.n[2])), v.g.n[3], rmax, tmax))
    return cudaSuccess;
  auto launch = [&](auto rows) -> cudaError_t {
    constexpr int RO = decltype(rows)::value;
    if constexpr (P == kF64) {
      if (links == kWilsonNear)
        return launch_wilson_tg_rows<P, (RO + 1) / 2 * 2, false, true>(v, spatial, rmax, tmax, s, flag, st, used);
    } else if (v.g.n[3] == kTgChunks * RO) {
      return launch_wilson_tg_rows<P, RO, true, false>(v, spatial, rmax, tmax, s, flag, st, used);
    }
    return launch_wilson_tg_rows<P, RO, false, false>(v, spatial, rmax, tmax, s, flag, st, used);
  };
  switch ((v.g.n[3] + kTgChunks - 1) / kTgChunks) {
    case 1: return launch(std::integral_constant<int, 1>{});
    case 2: return launch(std::integral_constant<int, 2>{});
    case 3: return launch(std::integral_constant<int, 3>{});
    case 4: return launch(std::integral_constant<int, 4>{});
    case 5: return launch(std::integral_constant<int, 5>{});
    case 6: return launch(std::integral_constant<int, 6>{});
    case 7: return launch(std::integral_constant<int, 7>{});
    case 8: return launch(std::integral_constant<int, 8>{});
    default: return cudaSuccess;
  }
}

cudaError_t launch_wilson(const LatticeView& v, const void* spatial, int rmax, int tmax,
                          const Scratch& s, WilsonLinks links, double* flag, cudaStream_t st) {
  if (rmax < 1 || rmax > kWilsonMaxR || tmax < 1) return cudaErrorInvalidValue;
  {
    bool used = false;
    cudaError_t e = cudaSuccess;
    SU2_DISPATCH(v.prec, {
      e = launch_wilson_tg<P>(v, spatial, rmax, tmax, s, links, flag, st, &used);
      if (e == cudaSuccess && !used) e = launch_wilson_rt<P>(v, spatial, rmax, tmax, s, st, &used);
    });
    if (e != cudaSuccess || used) return e;
  }
  // rows too long for even one time slice in shared memory: global-memory kernel
  SU2_DISPATCH(v.prec, {
    constexpr int TC = WilsonChunk<P>::tc;
    auto Lt = links_of<P>(v.links, v.g.vh);
    auto Ls = links_of<P>(const_cast<void*>(spatial), v.g.vh);
    const int nchunks = (tmax + TC - 1) / TC;
    const int64_t V = 2 * v.g.vh;
    int per_sm = 1;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_wilson<P, TC>, kWilsonThreads, 0);
    if (per_sm < 1) per_sm = 1;
    // all (chunk, direction) slices together fill the machine once
    int64_t gx = (int64_t)device_info().sms * per_sm / (3 * nchunks);
    const int64_t need = (V + kWilsonThreads - 1) / kWilsonThreads;
    if (gx > need) gx = need;
    // keep one partial set per block within the scratch buffer
    const int64_t per = (int64_t)rmax * TC;
    const int64_t cap = (int64_t)kScratchPartials / per / (3 * nchunks);
    if (gx > cap) gx = cap;
    if (gx < 1) gx = 1;
    k_wilson<P, TC><<<dim3((unsigned)gx, 3 * nchunks), kWilsonThreads, 0, st>>>(Ls, Lt, v.g, rmax, tmax, s.partials);
    count_launches(1);
    k_wilson_final<TC><<<rmax * tmax, kThreads, 0, st>>>(s.partials, (int)gx, rmax, tmax, 1.0 / (3.0 * (double)V),
                                                         s.out);
  });
  count_launches(1);
  return cudaGetLastError();
}

cudaError_t launch_to_canonical(const LatticeView& v, double* canon, int64_t s0, int64_t ns,
                                cudaStream_t st) {
  SU2_DISPATCH(v.prec, {
    auto L = links_of<P>(v.links, v.g.vh);
    const int gr = grid_for(k_to_canonical<P>, 4 * ns);
    k_to_canonical<P><<<gr, kThreads, 0, st>>>(L, v.g, canon, s0, ns);
  });
  count_launches(1);
  return cudaGetLastError();
}

cudaError_t launch_from_canonical(const LatticeView& v, const double* canon, int64_t s0,
                                  int64_t ns, cudaStream_t st) {
  SU2_DISPATCH(v.prec, {
    auto L = links_of<P>(v.links, v.g.vh);
    const int gr = grid_for(k_from_canonical<P>, 4 * ns);
    // a caller's array need not be 16-byte aligned
    const int wide = reinterpret_cast<uintptr_t>(canon) % 16 == 0;
    k_from_canonical<P><<<gr, kThreads, 0, st>>>(L, v.g, canon, s0, ns, wide);
  });
  count_launches(1);
  return cudaGetLastError();
}

cudaError_t launch_add_u32(uint32_t* p, uint32_t v, cudaStream_t st) {
  k_add_u32<<<1, 1, 0, st>>>(p, v);
  count_launches(1);
  return cudaGetLastError();
}

}  // namespace su2
