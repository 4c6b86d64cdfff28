// The checkerboard heat-bath substep for sm_103a (Section 2 Eqs. 5-9, 11;
// Section 4), with its optional plaquette sum for measured sweeps (the
// Polyakov kernel's last block turns those block sums into the plaquette).
// Paper: Cardoso & Bicudo, arXiv:1010.4834.
#pragma once

#include <type_traits>

#include "su2_hb_link.cuh"
#include "su2_internal.h"
#include "su2_kernel_util.cuh"

namespace su2 {

// ---------------------------------------------------------------------------
// Heat-bath substep (Section 2 Eqs. 5-9, 11; Section 4 checkerboard): one
// thread per link of direction MU on the parity-p sublattice.
//
// Most links accept their first a0 trial, but a warp would repeat the trial
// loop until its slowest lane accepts.  So every lane makes trial 1 inline;
// a link that rejects it goes to a block-wide shared-memory queue (its
// W = Sigma/k, alpha, index and site), which the whole block drains every
// DeferEvery iterations with trials 2, 3, ...  The draws and their order are
// those of the plain loop, so results are identical; only the schedule
// differs.  A full queue falls back to finishing the link inline.
//
// With MEAS (the odd-parity substeps of MU = 1, 2, 3 of a measured sweep) the
// kernel also adds up Tr(U_MU(x) L(x)^dagger)/2 over its links, with L the
// staple's partial sum over NU < MU and U the link's final value (the
// accepted draw as stored, or the kept old link), and writes one sum per
// block to `meas`.  Every plaquette of a plane (NU, MU), NU < MU, holds two
// MU-links on sites of opposite parity, so the odd-parity substep of MU counts
// each of them once; and once that substep has run, every link in directions
// <= MU has its end-of-sweep value.  The three substeps together give the
// plaquette of Eq. 12 after the sweep (planes (0,1), (0,2) and (1,2) the
// spatial part, (NU,3) the space-time part) without another pass over the
// links.
// ---------------------------------------------------------------------------
// Queue capacity: the plaquette-summing variant's entries are larger (they
// carry the partial staple), so it keeps fewer and leaves the SM's L1 share
// of the shared-memory carveout about the same.
// Block size BS: on large lattices blocks of 1024 share one deferral queue
// among more threads, which drain it less often per link (FP32 substep on
// 64^4, 55 k half-sites per SM: 202 us at 256 threads, 194 at 1024); up to
// 48^4 (17 k per SM) 256 is faster (70.9 against 72.2 us; 16^4 12.3
// against 14.0), as more, smaller blocks spread the few block iterations
// evenly over the SMs.  The switch is at SU2_HB_BIG_PER_SM half-lattice
// sites per SM.  FP64, 128 registers a thread: 256 throughout.
#ifndef SU2_HB_BIG_PER_SM
#define SU2_HB_BIG_PER_SM 32768
#endif
#ifndef SU2_HB_LARGE_BS
#define SU2_HB_LARGE_BS 1024
#endif
template <int BS, bool MEAS> struct DeferCap { static constexpr int value = MEAS ? 2 * BS : 4 * BS; };
// Drain interval in block iterations: at the ~5% first-trial rejection of
// beta ~ 2.5 a queue collects about 0.05 * 1024 * interval links, which the
// capacity covers (the plaquette-summing variant's smaller queue, half as
// often); fewer drains mean fewer block-wide barriers.
template <bool MEAS> struct DeferEvery { static constexpr int value = MEAS ? 32 : 64; };

// Minimum resident blocks per SM (the register budget): 1024 threads per SM
// at 64 registers for FP32 / F16Q.
template <int P, int BS> struct HbMinBlocks {
  static constexpr int value = Occ<P>::hb * kThreads / BS > 0 ? Occ<P>::hb * kThreads / BS : 1;
};

// Programmatic dependent launch: a substep is launched with programmatic
// stream serialisation, so the launch of its grid overlaps the end of the
// previous kernel; each block first waits (griddepcontrol.wait, a hardware
// wait for the previous grid to complete and its writes to be visible) and
// reads nothing before.  No kernel triggers its dependents early (the
// implicit trigger at completion).  Sweep times, plain / measured, in us:
// 16^4 26.2 -> 25.2 / 37.9 -> 37.1, 32^3 x 4 31.0 -> 29.9 / 43.6 -> 42.6,
// 64^4 1417.6 -> 1415.3 / 1497.2 -> 1496.4.  An explicit trigger at the
// start of each block lost (64^4 sweep 1427 us, 48^4 measured sweep 512 ->
// 576 us): the next grid's blocks then hold SM slots while they wait.

template <int P, int MU, bool MEAS, int PAR, int BS>
__global__ void __launch_bounds__(BS, HbMinBlocks<P, BS>::value)
    k_heatbath(Links<P, hb_addr<P, kClassPtr>> L, const __grid_constant__ Geom g, Substep sub, const uint32_t* sweep_base, uint32_t sweep_off,
               const __grid_constant__ HBParams hp, double* meas) {
  const int mu = substep_of<MU, PAR>(sub).mu;
  using R = typename Real<P>::T;
  using Def = Deferred<R, MEAS>;
  constexpr int kDeferCap = DeferCap<BS, MEAS>::value;
  constexpr int kHbThreads = BS;
  __shared__ Def queue[kDeferCap];
  __shared__ int qn;
  const int zero = pdl_wait();
  const R beta = (R)hp.beta;
  const uint32_t sweep = (sweep_base ? *sweep_base : 0u) + sweep_off;
  const uint32_t tag = (uint32_t)mu | hp.lattice_tag;
  // MEAS: plaquettes of the planes (NU < MU, MU).  A plain sum: a thread adds
  // vh / (grid size) terms of magnitude <= 2 (about 55 on 64^4), so FP32
  // rounding stays near 1e-6 relative per thread before the FP64 block sums.
  PlainAcc<R> plaq;
  if (threadIdx.x == 0) qn = 0;
  __syncthreads();
  const int vh = (int)g.vh;
  const int stride = gridDim.x * blockDim.x;
  int it = 0;
  for (int base = blockIdx.x * blockDim.x + zero; base < vh; base += stride, ++it) {
    const int h = base + threadIdx.x;
    if (h < vh) hb_link<P, MU, MEAS, PAR, false, kDeferCap>(L, g, sub, h, tag, sweep, beta, hp, queue, &qn, plaq);
    if ((it % DeferEvery<MEAS>::value) == DeferEvery<MEAS>::value - 1 || base + stride >= vh) {
      __syncthreads();
      hb_drain<P, MU, MEAS, PAR>(L, sub, queue, min(qn, kDeferCap), tag, sweep, hp, plaq);
      __syncthreads();
      if (threadIdx.x == 0) qn = 0;
      __syncthreads();
    }
  }
  if (MEAS) {
    __shared__ double shp[kHbThreads / 32];
    const double v = warp_sum(plaq.value());
    if ((threadIdx.x & 31) == 0) shp[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
      double t = 0.0;
      for (int w = 0; w < kHbThreads / 32; ++w) t += shp[w];
      meas[blockIdx.x] = t;
    }
  }
}

// ---------------------------------------------------------------------------
// The substep on lattices of at most one link per resident thread, with room
// for the next grid beside this one.  There the time is the latency of one
// update: launch, gather, draw, store.  So each thread draws its random
// numbers (two trials and their directions, parked in shared memory) before
// it waits for the previous substep, whose links they do not depend on; that
// substep has let this grid start as soon as its own wait was over.  A link
// that rejects both trials (0.25% of Kennedy-Pendleton links at beta ~ 2.5)
// is finished by its warp: the lanes divide into groups, one for each such
// link, whose lanes take consecutive trials, and the first that accepts
// counts.  The trials and their order are those of k_heatbath.  A sweep, k_heatbath
// (of these sizes) and this kernel: 16^4 FP32 25.6 and 21.0 us, 32^3 x 4 29.9 and
// 25.4; without the early start of the next grid 24.6 and 29.3, with it before
// the wait instead of after 27.3 and 30.7.
// ---------------------------------------------------------------------------
// Blocks of 64 in FP64; in FP32 of 128, or of 256 where that puts one block on
// every SM but leaves none with two (16^4: 21.0 against 22.0 us a sweep; 32^3 x 4
// 25.9 against 25.4, 8^4 18.1 against 17.1).
template <int P, int MU, bool MEAS, int PAR, int BS>
__global__ void __launch_bounds__(BS, 2 * SmallPerSM<P>::value / BS)
    k_heatbath_small(Links<P, hb_addr<P, kClassPtr>> L, const __grid_constant__ Geom g, Substep sub, const uint32_t* sweep_base,
                     uint32_t sweep_off, int late, const __grid_constant__ HBParams hp, double* meas) {
  sub = substep_of<MU, PAR>(sub);
  const int mu = sub.mu, p = sub.p;
  constexpr int ND = P == kF64 ? 1 : 2;   // the FP64 direction does not depend on the trial
  using R = typename Real<P>::T;
  union Numbers {
    TrialNumbers<R> kp;
    struct { R u0, u1; };                  // Creutz
  };
  struct Open { R alpha; uint32_t site; int next; };
  __shared__ Numbers numbers[2][BS];
  __shared__ Direction<R> direction[ND][BS];
  __shared__ Open open[BS / 32][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, tid = threadIdx.x;
  const int i = blockIdx.x * BS + tid;
  const bool valid = i < (int)g.vh;
  int h = valid ? i : 0;                   // idle threads keep their warp whole
  const Site x = site_from_half(g, (uint32_t)h, p);
  if (late) {
    h += pdl_wait();
    pdl_trigger();
  }
  // the sweep counter was final before the previous substep passed its wait
  const uint32_t sweep = (sweep_base ? __ldcg(sweep_base) : 0u) + sweep_off;
  const uint4 ctr = make_uint4(philox_site(g, x), (uint32_t)mu | hp.lattice_tag, sweep, 0u);
#pragma unroll(P == kF64 ? 1 : 2)
  for (int n = 0; n < 2; ++n) {
    uint4 c = ctr;
    c.w = (uint32_t)n + 1u;
    const uint4 r = philox(c, hp.rk);
    if (hp.sampler == 0) {
      numbers[n][tid].kp = trial_numbers<R>(r);
    } else {
      numbers[n][tid].u0 = u01<R>(r.x);
      numbers[n][tid].u1 = u01<R>(r.y);
    }
    if (n < ND) direction[n][tid] = draw_direction<R>(ctr, r, hp);
  }
  if (!late) {
    h += pdl_wait();
    pdl_trigger();
  }
  const R beta = (R)hp.beta;
  Quat<R> lower;
  const Frame<R> f = link_frame<P, MU, MEAS, false, hb_addr<P, kClassPtr>, false>(L, g, x, h, mu, p, beta, lower);
  const R alpha = f.alpha;
  Quat<R> nl = qone<R>();
  bool found = false, rejected = false;
  int next = 3;
  if (!(alpha >= R(1e-12))) {
    uint4 c = ctr;
    c.w = 1u;
    nl = haar_from<R>(philox(c, hp.rk));
    found = true;
  } else {
    // numbers that do not serve (fixed-point logarithms at small alpha) leave
    // the link to the loop below from its first trial on
    const bool serve = P != kF64 || hp.sampler != 0 || alpha >= (R)kFixMinAlpha;
    const R inv2a = trial_inv2a(alpha), e = trial_e(alpha, hp.sampler);
    A0Of<R> a0;
#pragma unroll(P == kF64 ? 1 : 2)
    for (int n = 0; n < 2; ++n) {
      if (!found && serve && n < hp.max_tries) {
        const Numbers t = numbers[n][tid];
        if (hp.sampler == 0 ? trial_decide(t.kp, inv2a, &a0) : creutz_decide<R>(t.u0, t.u1, alpha, e, &a0)) {
          nl = compose_from(a0, f.w, direction[n < ND ? n : 0][tid]);
          found = true;
        }
      }
    }
    next = serve ? 3 : 1;
    rejected = !found && next <= hp.max_tries && valid;
  }
  uint32_t mask;
  while ((mask = __ballot_sync(0xffffffffu, rejected)) != 0u) {
    const int m = __popc(mask), lg = 32 - __clz(m - 1);       // 2^lg >= m groups (m = 1: clz(0) = 32)
    const int per = 32 >> lg;                                 // trials a round and link
    const int rank = __popc(mask & ((1u << lane) - 1u));
    if (rejected) open[warp][rank] = Open{alpha, ctr.x, next};
    __syncwarp();
    const int k = lane >> (5 - lg);
    bool accept = false;
    A0Of<R> a0 = 0;
    uint4 rt = make_uint4(0u, 0u, 0u, 0u);
    if (k < m) {
      const Open o = open[warp][k];
      const int n = o.next + (lane & (per - 1));
      uint4 c = ctr;
      c.x = o.site;
      if (n <= hp.max_tries)
        accept = trial_a0<R>(o.alpha, trial_inv2a(o.alpha), trial_e(o.alpha, hp.sampler), c, n, hp, &a0, &rt);
    }
    const uint32_t votes = __ballot_sync(0xffffffffu, accept);
    const uint32_t mine = rejected ? (votes >> (rank * per)) & (0xffffffffu >> (32 - per)) : 0u;
    const int from = mine ? rank * per + __ffs(mine) - 1 : lane;
    a0 = __shfl_sync(0xffffffffu, a0, from);
    rt.x = __shfl_sync(0xffffffffu, rt.x, from);
    rt.y = __shfl_sync(0xffffffffu, rt.y, from);
    rt.z = __shfl_sync(0xffffffffu, rt.z, from);
    rt.w = __shfl_sync(0xffffffffu, rt.w, from);
    if (mine) {
      nl = compose_from(a0, f.w, P == kF64 ? direction[0][tid] : draw_direction<R>(ctr, rt, hp));
      found = true;
      rejected = false;
    } else if (rejected) {
      next += per;
      rejected = next <= hp.max_tries;
    }
    __syncwarp();  // open[] is read before the next round writes it
  }
  R plaq = R(0);
  if (valid) {
    if constexpr (MEAS) plaq = qdot_rn(found ? L.put(2 * mu + p, h, nl) : L.ldc(2 * mu + p, h), lower);
    else if (found) L.st(2 * mu + p, h, nl);
  }
  if constexpr (MEAS) {
    __shared__ double sums[BS / 32];
    const double v = warp_sum((double)plaq);
    if (lane == 0) sums[warp] = v;
    __syncthreads();
    if (tid == 0) {
      double t = 0.0;
      for (int k = 0; k < BS / 32; ++k) t += sums[k];
      meas[blockIdx.x] = t;
    }
  }
}

// ---------------------------------------------------------------------------
// FP64 lattices that leave most of the GPU idle: LANES threads share a link.
// Lane j takes the staple terms j, j + LANES, ... (their fixed-point sums add
// up to the same bits in any order) and trials j + 1, j + 1 + LANES, ...; the
// first trial that accepts counts, as in one thread's loop.  A thread's 4000
// instructions for a link, on one or two warps an SM, are the time of a substep
// there (8^4 measured sweep, one lane: 97 us).
// ---------------------------------------------------------------------------
template <int LANES> __device__ __forceinline__ void lanes_add(FixSum& s) {
#pragma unroll
  for (int o = LANES / 2; o > 0; o >>= 1) {
    s.hw += __shfl_xor_sync(0xffffffffu, s.hw, o);
    s.hx += __shfl_xor_sync(0xffffffffu, s.hx, o);
    s.hy += __shfl_xor_sync(0xffffffffu, s.hy, o);
    s.hz += __shfl_xor_sync(0xffffffffu, s.hz, o);
    s.mw += __shfl_xor_sync(0xffffffffu, s.mw, o);
    s.mx += __shfl_xor_sync(0xffffffffu, s.mx, o);
    s.my += __shfl_xor_sync(0xffffffffu, s.my, o);
    s.mz += __shfl_xor_sync(0xffffffffu, s.mz, o);
  }
}

template <bool MEAS, int LANES>
__global__ void __launch_bounds__(64, 8)
    k_heatbath_lanes(Links<kF64> L, const __grid_constant__ Geom g, Substep sub, const uint32_t* sweep_base, uint32_t sweep_off, int late,
                     const __grid_constant__ HBParams hp, double* meas) {
  const int mu = sub.mu, p = sub.p;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int j = lane & (LANES - 1), group = lane & ~(LANES - 1);
  const int i = (int)((blockIdx.x * 64 + threadIdx.x) / LANES);
  const bool valid = i < (int)g.vh;
  int h = valid ? i : 0;
  const Site x = site_from_half(g, (uint32_t)h, p);
  if (late) {
    h += pdl_wait();
    pdl_trigger();
  }
  const uint32_t sweep = (sweep_base ? __ldcg(sweep_base) : 0u) + sweep_off;
  const uint4 ctr = make_uint4(philox_site(g, x), (uint32_t)mu | hp.lattice_tag, sweep, 0u);
  uint4 c = ctr;
  c.w = (uint32_t)j + 1u;
  uint4 r = philox(c, hp.rk);
  TrialNumbers<double> numbers = trial_numbers<double>(r);
  const Direction<double> direction = draw_direction<double>(ctr, r, hp);
  if (!late) {
    h += pdl_wait();
    pdl_trigger();
  }
  FixSum s = j == 0 ? fix_zero() : FixSum{0, 0, 0, 0, 0, 0, 0, 0}, low = s;
  FixBad bad{0u, 0u};
  const int dmu = half_step_mu(g, x, mu);
#pragma unroll 1
  for (int k = j; k < 6; k += LANES) {
    const TermLinks t = term_links<false, false>(L, g, x, h, dmu, mu, p, k);
    const int odd = -(k & 1);
    fix_mac(s, fix_mul(fix_of(t.a, odd, bad), fix_of(t.b, 0, bad)), fix_of(t.c, ~odd, bad));
    if (MEAS && k < 2 * mu) low = s;   // a lane's terms ascend
  }
  lanes_add<LANES>(s);
  Quat<double> lower = qmake<double>(0, 0, 0, 0);
  if constexpr (MEAS) {
    lanes_add<LANES>(low);
    lower = fix_sum_to_double(low);
  }
  const uint32_t off = __ballot_sync(0xffffffffu, !fix_ok(bad));
  Frame<double> f;
  if (__builtin_expect((off >> group & ((1u << LANES) - 1u)) == 0u, 1)) {
    f = staple_frame(s, hp.beta);
  } else {
    const OtherFrame r = frame_other<false, false>(L, g, x, h, mu, p, hp.beta);
    f = r.f;
    lower = r.lower;
  }
  Quat<double> nl = qone<double>();
  bool found = false, open = valid;
  if (!(f.alpha >= 1e-12)) {
    c.w = 1u;
    nl = haar_from<double>(philox(c, hp.rk));
    found = true;
    open = false;
  }
  const double inv2a = trial_inv2a(f.alpha), e = trial_e(f.alpha, hp.sampler);
  for (int n = j + 1; __any_sync(0xffffffffu, open); n += LANES) {
    int64_t a0 = 0;
    bool accept = false;
    if (open && n <= hp.max_tries) {
      if (n > LANES) {
        c.w = (uint32_t)n;
        r = philox(c, hp.rk);
        if (hp.sampler == 0) numbers = trial_numbers<double>(r);
      }
      accept = hp.sampler != 0 ? creutz_decide<double>(u01<double>(r.x), u01<double>(r.y), f.alpha, e, &a0)
               : f.alpha >= kFixMinAlpha ? trial_decide(numbers, inv2a, &a0) : trial_small_alpha(r, inv2a, &a0);
    }
    const uint32_t mine = __ballot_sync(0xffffffffu, accept) >> group & ((1u << LANES) - 1u);
    a0 = __shfl_sync(0xffffffffu, a0, group + (mine ? __ffs(mine) - 1 : j));
    if (open && mine) {
      nl = compose_from(a0, f.w, direction);
      found = true;
      open = false;
    }
    open = open && n - j + LANES <= hp.max_tries;   // the same in every lane of a link
  }
  const bool writes = valid && j == 0;
  double plaq = 0.0;
  if (writes) {
    if constexpr (MEAS) plaq = qdot_rn(found ? L.put(2 * mu + p, h, nl) : L.ldc(2 * mu + p, h), lower);
    else if (found) L.st(2 * mu + p, h, nl);
  }
  if constexpr (MEAS) {
    __shared__ double sums[2];
    plaq = warp_sum(plaq);
    if (lane == 0) sums[warp] = plaq;
    __syncthreads();
    if (threadIdx.x == 0) meas[blockIdx.x] = sums[0] + sums[1];
  }
}

// ---------------------------------------------------------------------------
// Host launcher for one precision, instantiated in one translation unit each
// (they compile side by side).
// ---------------------------------------------------------------------------
template <int P>
cudaError_t launch_heatbath_prec(const LatticeView& v, int mu, int parity, const uint32_t* sweep_base,
                                 uint32_t sweep_off, const HBParams& hp, cudaStream_t st,
                                 double* meas, int* meas_blocks) {
  if (meas && (mu < 1 || parity != 1 || !meas_blocks)) return cudaErrorInvalidValue;
  SU2_DISPATCH_MU(mu, {
    // FP32 / F16Q: direction and parity are template parameters, so every class
    // index in the kernel is a compile-time constant: per-class base pointers
    auto L = links_of<P, hb_addr<P, kClassPtr>>(v.links, v.g.vh);
    const Substep sub{mu, parity};
    const int64_t sms = device_info().sms;
    const bool large = v.g.vh >= (int64_t)SU2_HB_BIG_PER_SM * sms;
    auto launch = [&](auto kernel, int nthreads, double* m) -> cudaError_t {
      const int gr = grid_for(kernel, v.g.vh, 0, nthreads);
      if (m) {
        if (gr > kMeasStride) return cudaErrorInvalidConfiguration;
        *meas_blocks = gr;
      }
      return launch_pdl(true, kernel, dim3((unsigned)gr), nthreads, st, L, v.g, sub, sweep_base, sweep_off, hp, m);
    };
    const bool small = overlaps(v);
    const bool one_each = v.g.vh > 128 * sms && v.g.vh <= 256 * sms;
    auto launch_small = [&](auto kernel, int nthreads, double* m, int lanes = 1) -> cudaError_t {
      const int gr = (int)((v.g.vh * lanes + nthreads - 1) / nthreads);
      if (m) *meas_blocks = gr;
      // the first substep of a sweep may follow the kernel that advances the sweep counter
      const int late = mu == 0 && parity == 0 && sweep_base != nullptr;
      return launch_pdl(true, kernel, dim3((unsigned)gr), nthreads, st, L, v.g, sub, sweep_base, sweep_off, late, hp, m);
    };
    // blocks of 256, on large FP32 / F16Q lattices of 1024
    auto with_bs = [&](auto meas_c, auto par_c, double* m) -> cudaError_t {
      constexpr bool M = decltype(meas_c)::value;
      constexpr int KM = hb_dir<P, MU>, PP = hb_dir<P, decltype(par_c)::value>;
      if constexpr (P == kF64) {
        // eight lanes a link, or two, while the small kernel's threads allow
        if (small && 8 * v.g.vh <= SmallPerSM<P>::value * sms) return launch_small(k_heatbath_lanes<M, 8>, 64, m, 8);
        if (small && 2 * v.g.vh <= SmallPerSM<P>::value * sms) return launch_small(k_heatbath_lanes<M, 2>, 64, m, 2);
      }
      if (small) {
        constexpr int kBlock = P == kF64 ? 64 : 128, kWide = P == kF64 ? 64 : 256;
        return one_each ? launch_small(k_heatbath_small<P, KM, M, PP, kWide>, kWide, m)
                        : launch_small(k_heatbath_small<P, KM, M, PP, kBlock>, kBlock, m);
      }
      constexpr int kLarge = P == kF64 ? 256 : SU2_HB_LARGE_BS;
      return large ? launch(k_heatbath<P, KM, M, PP, kLarge>, kLarge, m) : launch(k_heatbath<P, KM, M, PP, 256>, 256, m);
    };
    cudaError_t e = cudaSuccess;
    if (meas) {
      if constexpr (MU >= 1) e = with_bs(std::true_type{}, std::integral_constant<int, 1>{}, meas);
    } else if (parity == 0) {
      e = with_bs(std::false_type{}, std::integral_constant<int, 0>{}, nullptr);
    } else {
      e = with_bs(std::false_type{}, std::integral_constant<int, 1>{}, nullptr);
    }
    if (e != cudaSuccess) return e;
  });
  count_launches(1);
  return cudaGetLastError();
}

}  // namespace su2
