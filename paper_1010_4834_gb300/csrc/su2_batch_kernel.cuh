// Batched lattices: many independent lattices of uneven extents and couplings
// swept together by one persistent kernel per call (captured in a CUDA graph).
//
// The heat bath of each lattice follows Section 2 (Eqs. 5-9, 11) and the
// checkerboard of Section 4 exactly as for a single lattice; lattice i uses
// Philox lattice_id = i, so every link's draws are fixed by (lattice, sweep,
// site, direction) and the result does not depend on the schedule below.
//
// Schedule.  The cooperative grid is split into G groups of CTAs.  The
// lattices are dealt to the groups largest first, each to the group with the
// least work so far, and each group gets a share of the CTAs in proportion
// to its work, so that the groups finish together and small lattices do not
// leave most of a group's threads idle.  A group sweeps its lattices one
// after another, all n sweeps of one lattice before the next.  Substeps
// within a lattice are ordered by a barrier among the group's CTAs only,
// which is cheaper than a grid-wide barrier (a one-CTA group needs only the
// block barrier), and the G lattices in flight are re-read from L2 rather
// than HBM between substeps when they fit.  G defaults to one group per
// lattice; su2_batch_tune times candidate G on a scratch copy of the links.
//
// Every barrier wait is bounded twice (global timer and iteration count); a
// wait that runs out raises a device error flag, all blocks leave, and the
// host reports SU2_ETIMEOUT.  Cooperative launch guarantees that all CTAs are
// co-resident.
//
// This header holds the kernel; su2_batch.cu the host side, and one small
// translation unit for each (precision, measured or not) its instantiations,
// which compile side by side.
#pragma once

#include <type_traits>

#include "su2_batch.h"
#include "su2_hb_link.cuh"

namespace su2 {

__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Barrier among the `n` CTAs of one group.  Returns false if any wait timed out.
__device__ __forceinline__ bool group_barrier(GroupBarrier* gb, unsigned int n, BatchCtl* ctl,
                                              unsigned long long timeout_ns) {
  __shared__ int ok;
  __syncthreads();
  // a group of one CTA needs no more than the block barrier (unless a fault
  // is injected, which makes every barrier wait for an arrival that never comes)
  if (n == 1 && ctl->extra == 0) return true;
  if (threadIdx.x == 0) {
    volatile unsigned int* vgen = &gb->gen;
    volatile int* verr = &ctl->err;
    const unsigned int g = *vgen;
    __threadfence();
    const unsigned int arrived = atomicAdd(&gb->count, 1u) + 1u;
    if (arrived == n + ctl->extra) {
      gb->count = 0;
      __threadfence();
      atomicExch(&gb->gen, g + 1u);
    } else {
      // bounded twice over: by the global timer and by an iteration count
      const unsigned long long t0 = global_ns();
      unsigned long long spins = 0;
      while (*vgen == g) {
        if (*verr) break;
        if (global_ns() - t0 > timeout_ns || ++spins > (1ull << 24)) {
          atomicExch(&ctl->err, 1);
          break;
        }
        __nanosleep(100);
      }
    }
    __threadfence();
    ok = *verr == 0;
  }
  __syncthreads();
  return ok != 0;
}

// The deferral queue holds two entries a thread.
template <int BS> struct BatchQueue { static constexpr int value = 2 * BS; };

// A lattice's geometry: FP64 in place, since its out-of-line paths take the address
// (of a copy, that would be one in local memory).
template <int P> using BatchGeom = std::conditional_t<P == kF64, const Geom&, const Geom>;

// One substep (MU, p) of one lattice by the CTAs of a group, each link by
// hb_link with coherent loads (other CTAs of the group wrote the links
// before the last barrier): trial 1 inline, rejected links queued and
// finished by the whole block at the end.  MEAS (odd substeps of MU >= 1 in
// a measured sweep): plaq accumulates Tr(U_MU(x) L(x)^dagger)/2 with L the
// staple's partial sum over NU < MU, as in the single-lattice substep.
template <int P, int MU, int PAR, int BS, bool MEAS>
__device__ __forceinline__ void batch_substep(const Links<P, hb_addr<P, kClassOff>>& L, const Geom& g, Substep sub, int rank, int cpg,
                                              uint32_t sweep, uint32_t tag, typename Real<P>::T beta,
                                              const HBParams& hp, void* queue_mem, int* qn,
                                              PlainAcc<typename Real<P>::T>& plaq) {
  using R = typename Real<P>::T;
  using Def = Deferred<R, MEAS>;
  Def* queue = static_cast<Def*>(queue_mem);
  constexpr int kQ = BatchQueue<BS>::value;
  const int vh = (int)g.vh;
  for (int base = rank * BS; base < vh; base += cpg * BS) {
    const int h = base + threadIdx.x;
    if (h < vh)
      hb_link<P, MU, MEAS, PAR, false, kQ, hb_addr<P, kClassOff>, false>(L, g, sub, h, tag, sweep, beta, hp, queue, qn, plaq);
  }
  __syncthreads();
  hb_drain<P, MU, MEAS, PAR, hb_addr<P, kClassOff>, false>(L, sub, queue, min(*qn, kQ), tag, sweep, hp, plaq);
  __syncthreads();
  if (threadIdx.x == 0) *qn = 0;
}

// One over-relaxation substep (MU, p) of one lattice by the CTAs of a group.
template <int P, int MU, int PAR, int BS>
__device__ __forceinline__ void batch_or_substep(const Links<P, hb_addr<P, kClassOff>>& L, const Geom& g, Substep sub, int rank,
                                                 int cpg) {
  const int vh = (int)g.vh;
  for (int h = rank * BS + (int)threadIdx.x; h < vh; h += cpg * BS) or_link<P, MU, PAR, false>(L, g, sub, h);
}

// Measured sweeps.  The plaquette (Eq. 12) comes from the sweep's odd
// substeps of MU = 1, 2 (spatial planes) and MU = 3 (space-time planes), each
// thread's sums ps and pt; at the end of the last of them every CTA writes
// its block sums to part[4 blockIdx.x + 0, 1].  The Polyakov loop (Eqs.
// 14-15) of the sweep's final links is taken during the first substep of
// the lattice's next sweep, which changes no time link (over-relaxation or
// heat bath of MU = 0): each CTA multiplies the time links of its spatial
// sites in increasing t and writes its sum of (1/2) Tr to
// part[4 blockIdx.x + 2].  After that substep's barrier the group's first
// CTA adds the CTAs' sums (warp 0, a fixed lane assignment and tree) into
// the history; a lattice's last sweep of the call takes its Polyakov loop
// after one more barrier.  Coherent loads throughout: other CTAs of the
// group write links during the launch.
template <int BS>
__device__ __forceinline__ void block_sums_to(double v0, double v1, double* out0, double* out1) {
  __shared__ double sh[BS / 32][2];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  v0 = warp_sum(v0);
  v1 = warp_sum(v1);
  if (lane == 0) {
    sh[warp][0] = v0;
    sh[warp][1] = v1;
  }
  __syncthreads();
  if (warp == 0) {
    const double t0 = warp_sum(lane < BS / 32 ? sh[lane][0] : 0.0);
    const double t1 = warp_sum(lane < BS / 32 ? sh[lane][1] : 0.0);
    if (lane == 0) {
      *out0 = t0;
      if (out1) *out1 = t1;
    }
  }
  __syncthreads();
}

template <int P, int BS>
__device__ __forceinline__ void batch_polyakov_part(const Links<P, kClassOff>& L, const Geom& g, int rank, int cpg,
                                                    double* part) {
  using R = typename Real<P>::T;
  Acc<R> pl;
  const int nsig = g.n[0] * g.n[1] * g.n[2];
  const int nt = g.n[3];
  for (int xs = rank * BS + (int)threadIdx.x; xs < nsig; xs += cpg * BS) {
    const int p0 = parity(site_from_index(g, (uint32_t)xs));   // parity of (xs, t = 0)
    const uint32_t h0 = (uint32_t)xs >> 1, hstep = (uint32_t)nsig >> 1;
    Quat<R> pr = qone<R>();
    // nt is even: the loads of two slices are issued before their products
    for (int t = 0; t < nt; t += 2) {
      const Quat<R> a = L.ldc(6 + p0, h0 + hstep * t);
      const Quat<R> b = L.ldc(6 + (p0 ^ 1), h0 + hstep * (t + 1));
      pr = qmul(qmul(pr, a), b);
    }
    pl.add(pr.w);
  }
  block_sums_to<BS>(pl.value(), 0.0, part + 4 * (size_t)blockIdx.x + 2, nullptr);
}

// The history entry of one sweep from the group's CTA sums (warp 0 of the
// group's first CTA).
__device__ __forceinline__ void batch_history(const double* part, int cta0, int cpg, const Geom& g, double* o) {
  const int lane = threadIdx.x & 31;
  double a = 0.0, b = 0.0, c = 0.0;
  for (int r = lane; r < cpg; r += 32) {
    const double* q = part + 4 * (size_t)(cta0 + r);
    a += __ldcg(q);
    b += __ldcg(q + 1);
    c += __ldcg(q + 2);
  }
  a = warp_sum(a);
  b = warp_sum(b);
  c = warp_sum(c);
  if (lane == 0) {
    const double n3 = 3.0 * (double)(2 * g.vh);
    o[0] = (a + b) / (2.0 * n3);
    o[1] = a / n3;
    o[2] = b / n3;
    o[3] = c / (double)(g.n[0] * g.n[1] * g.n[2]);
  }
}

// 1024 threads per SM (64 registers a thread) for FP32 / F16Q, 512 for FP64.
// MEAS: measured sweeps (su2_batch_sweep_measure), a separate instantiation
// so that the plain sweep's kernel carries none of the measurement.  It runs
// the same number of CTAs per SM (so the same plan) with blocks of 3/4 BS
// threads, which leaves it 85 registers a thread instead of 64: at 64 its
// bookkeeping spilled registers out of the substep loops (16 x 32^3 x 4
// FP32, 100 sweeps without any measurement work: 32.9 against the plain
// kernel's 42.0 G updates/s).
template <int BS, bool MEAS> struct BatchBlock { static constexpr int value = MEAS ? BS * 3 / 4 : BS; };

template <int P, int BS, bool MEAS>
__global__ void __launch_bounds__(BatchBlock<BS, MEAS>::value, (P == kF64 ? 512 : 1024) / BS)
    k_batch_groups(const BatchLattice* __restrict__ desc, const int* __restrict__ order,
                   const int4* __restrict__ plan, const int* __restrict__ cta_group, int nsweeps, int nor,
                   const uint32_t* sweep_base, const __grid_constant__ HBParams hp, GroupBarrier* bars, BatchCtl* ctl,
                   unsigned long long timeout_ns, double* mhist, double* mpart, int nlat) {
  using R = typename Real<P>::T;
  constexpr int kB = BatchBlock<BS, MEAS>::value;  // threads per CTA
  // the deferral queue, sized for the larger (plaquette-carrying) entries
  __shared__ __align__(16) unsigned char queue[BatchQueue<kB>::value * sizeof(Deferred<R, MEAS>)];
  __shared__ int qn;
  PlainAcc<R> ps, pt;  // measured sweep: spatial and space-time plaquette sums
  const int group = cta_group[blockIdx.x];
  if (group < 0) return;
  // plan[group] = (first lattice in `order`, lattices, first CTA, CTAs)
  const int4 pl = plan[group];
  const int cpg = pl.w;
  const int rank = (int)blockIdx.x - pl.z;
  if (threadIdx.x == 0) qn = 0;
  __syncthreads();
  const uint32_t sweep0 = *sweep_base;
  // one substep (mu, p) of lattice l by this group's CTAs
  auto substep = [&](int l, uint32_t sweep, int mu, int p) {
    BatchGeom<P> g = desc[l].g;
    Links<P, hb_addr<P, kClassOff>> L;
    L.set(desc[l].links, g.vh);
    const R beta = (R)desc[l].beta;
    const uint32_t tag = (uint32_t)mu | ((uint32_t)l << 2);
    auto run = [&](auto mu_c, auto par_c, auto meas_c, PlainAcc<R>& plaq) {
      batch_substep<P, decltype(mu_c)::value, decltype(par_c)::value, kB, MEAS && decltype(meas_c)::value>(
          L, g, Substep{mu, p}, rank, cpg, sweep, tag, beta, hp, queue, &qn, plaq);
    };
    using std::integral_constant;
    using No = std::false_type;
    using Yes = std::true_type;
    if constexpr (P == kF64) {
      // one code for all (see staple_fixed); the measured one also where its
      // sum is not wanted would cost the partial staple
      using Rt = integral_constant<int, kRuntime>;
      if (p == 0 || mu == 0 || !MEAS) run(Rt{}, Rt{}, No{}, ps);
      else if (mu < 3) run(Rt{}, Rt{}, Yes{}, ps);
      else run(Rt{}, Rt{}, Yes{}, pt);
      return;
    } else {
    switch (2 * mu + p) {
      case 0: run(integral_constant<int, 0>{}, integral_constant<int, 0>{}, No{}, ps); break;
      case 1: run(integral_constant<int, 0>{}, integral_constant<int, 1>{}, No{}, ps); break;
      case 2: run(integral_constant<int, 1>{}, integral_constant<int, 0>{}, No{}, ps); break;
      case 3: run(integral_constant<int, 1>{}, integral_constant<int, 1>{}, Yes{}, ps); break;
      case 4: run(integral_constant<int, 2>{}, integral_constant<int, 0>{}, No{}, ps); break;
      case 5: run(integral_constant<int, 2>{}, integral_constant<int, 1>{}, Yes{}, ps); break;
      case 6: run(integral_constant<int, 3>{}, integral_constant<int, 0>{}, No{}, pt); break;
      default: run(integral_constant<int, 3>{}, integral_constant<int, 1>{}, Yes{}, pt); break;
    }
    }
  };
  // one lattice at a time, a barrier after each substep: the lattice's links
  // stay in L2 through its sweeps (interleaving the group's lattices between
  // barriers halves the barriers but spills the working set: 32.5 against
  // 35.5 G updates/s for the 64-lattice batch at 32 groups)
  // `nor` over-relaxation sweeps precede each heat-bath sweep
  auto or_substep = [&](int l, int mu, int p) {
    BatchGeom<P> g = desc[l].g;
    Links<P, hb_addr<P, kClassOff>> L;
    L.set(desc[l].links, g.vh);
    if constexpr (P == kF64) {
      batch_or_substep<P, kRuntime, kRuntime, kB>(L, g, Substep{mu, p}, rank, cpg);
      return;
    } else {
    switch (2 * mu + p) {
      case 0: batch_or_substep<P, 0, 0, kB>(L, g, Substep{mu, p}, rank, cpg); break;
      case 1: batch_or_substep<P, 0, 1, kB>(L, g, Substep{mu, p}, rank, cpg); break;
      case 2: batch_or_substep<P, 1, 0, kB>(L, g, Substep{mu, p}, rank, cpg); break;
      case 3: batch_or_substep<P, 1, 1, kB>(L, g, Substep{mu, p}, rank, cpg); break;
      case 4: batch_or_substep<P, 2, 0, kB>(L, g, Substep{mu, p}, rank, cpg); break;
      case 5: batch_or_substep<P, 2, 1, kB>(L, g, Substep{mu, p}, rank, cpg); break;
      case 6: batch_or_substep<P, 3, 0, kB>(L, g, Substep{mu, p}, rank, cpg); break;
      default: batch_or_substep<P, 3, 1, kB>(L, g, Substep{mu, p}, rank, cpg); break;
    }
    }
  };
  // measured sweeps: after the first substep of sweep sw (sw >= 1), the
  // history entry of sweep sw - 1
  auto after_first = [&](int l, int sw) {
    if constexpr (MEAS) {
      if (sw > 0 && rank == 0 && threadIdx.x < 32)
        batch_history(mpart, pl.z, cpg, desc[l].g, mhist + ((size_t)(sw - 1) * nlat + l) * 4);
    }
  };
  auto polyakov_part = [&](int l) {
    const Geom g = desc[l].g;
    Links<P, kClassOff> L;
    L.set(desc[l].links, g.vh);
    batch_polyakov_part<P, kB>(L, g, rank, cpg, mpart);
  };
  for (int li = 0; li < pl.y; ++li) {
    const int l = order[pl.x + li];
    for (int sw = 0; sw < nsweeps; ++sw) {
      bool first = true;
      for (int k = 0; k < nor; ++k)
        for (int mu = 0; mu < 4; ++mu)
          for (int p = 0; p < 2; ++p) {
            or_substep(l, mu, p);
            if constexpr (MEAS) {
              if (first && sw > 0) polyakov_part(l);
            }
            if (!group_barrier(bars + group, (unsigned)cpg, ctl, timeout_ns)) return;
            if (first) after_first(l, sw);
            first = false;
          }
      for (int mu = 0; mu < 4; ++mu)
        for (int p = 0; p < 2; ++p) {
          substep(l, sweep0 + (uint32_t)sw, mu, p);
          if constexpr (MEAS) {
            if (first && sw > 0) polyakov_part(l);
            if (mu == 3 && p == 1) {
              // the sweep's plaquette sums of this CTA
              block_sums_to<kB>(ps.value(), pt.value(), mpart + 4 * (size_t)blockIdx.x,
                                mpart + 4 * (size_t)blockIdx.x + 1);
              ps = PlainAcc<R>();
              pt = PlainAcc<R>();
            }
          }
          if (!group_barrier(bars + group, (unsigned)cpg, ctl, timeout_ns)) return;
          if (first) after_first(l, sw);
          first = false;
        }
    }
    if constexpr (MEAS) {
      // the lattice's last sweep of this call
      if (nsweeps > 0) {
        polyakov_part(l);
        if (!group_barrier(bars + group, (unsigned)cpg, ctl, timeout_ns)) return;
        after_first(l, nsweeps);
        // the next lattice's first substep overwrites these CTA sums only
        // after a barrier that warp 0 of the first CTA reaches after reading them
      }
    }
  }
}

template <int P, bool MEAS>
cudaError_t launch_batch_groups(int bs, int grid, const BatchArgs& a, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3((unsigned)(MEAS ? bs * 3 / 4 : bs));   // BatchBlock
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  auto go = [&](auto kernel) {
    return cudaLaunchKernelEx(&cfg, kernel, a.desc, a.order, a.plan, a.cta_group, a.nsweeps, a.nor, a.sweep_base, a.hp,
                              a.bars, a.ctl, a.timeout_ns, a.mhist, a.mpart, a.nlat);
  };
  return bs == 512 ? go(k_batch_groups<P, 512, MEAS>) : go(k_batch_groups<P, 256, MEAS>);
}

template <int P, bool MEAS> int batch_blocks_per_sm(int bs) {
  int n = 0;
  if (bs == 512)
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_batch_groups<P, 512, MEAS>, BatchBlock<512, MEAS>::value, 0);
  else
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_batch_groups<P, 256, MEAS>, BatchBlock<256, MEAS>::value, 0);
  return n;
}

}  // namespace su2
