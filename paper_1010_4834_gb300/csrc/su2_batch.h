// Data and launch interface of the batched kernel (internal).
#pragma once

#include "su2_internal.h"

namespace su2 {

struct BatchLattice {
  Geom g;
  void* links;
  double beta;
};

// One barrier per group, each on its own 128-byte line.
struct GroupBarrier {
  unsigned int count;
  unsigned int gen;
  unsigned int pad[30];
};

struct BatchCtl {
  int err;             // 1: a barrier wait timed out
  unsigned int extra;  // arrivals a barrier waits for beyond its group (fault injection)
};

// Block sizes the batched kernel is built for (su2_batch_set_block_size,
// searched by su2_batch_tune).
constexpr int kBatchThreads = 256;  // default

// A block of a batched measurement: block `rank` of the `count` that share a
// lattice (consecutive blocks).
struct BatchBlock4 {
  int lattice, rank, count, pad;
};
// Resident blocks of 256 of the batched measurements an SM: 64 registers a thread
// below FP64.
constexpr int measure_blocks_per_sm(int prec) { return prec == kF64 ? 2 : 4; }
// Plaquette means (3 doubles a lattice) or Polyakov loops (1) of every lattice;
// counters: one zero word a lattice, left zero.
cudaError_t launch_batch_measure(int prec, bool polyakov, const BatchLattice* desc, const BatchBlock4* blocks,
                                 int nblocks, double* partials, unsigned int* counters, double* out, cudaStream_t st);

// One launch's arguments (see k_batch_groups).
struct BatchArgs {
  const BatchLattice* desc;
  const int* order;
  const int4* plan;
  const int* cta_group;
  int nsweeps, nor;
  const uint32_t* sweep_base;
  HBParams hp;
  GroupBarrier* bars;
  BatchCtl* ctl;
  unsigned long long timeout_ns;
  double *mhist, *mpart;
  int nlat;
};
// The cooperative launch of the plain or measured kernel with blocks of bs (256
// or 512; the measured kernel's are 3/4 of that), and its blocks per SM.
template <int P, bool MEAS>
cudaError_t launch_batch_groups(int bs, int grid, const BatchArgs& a, cudaStream_t st);
template <int P, bool MEAS> int batch_blocks_per_sm(int bs);

}  // namespace su2
