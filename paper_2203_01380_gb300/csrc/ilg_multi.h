// Multi-lattice steps used by the server: descriptors, shares of work, launcher.
#pragma once

#include <cuda_runtime.h>

#include <cstddef>
#include <cstdint>

#include "ilg_device.cuh"

namespace ilg {

constexpr int kMultiThreads = 1024;  // one block per SM
constexpr uint32_t kMultiRun = 32;   // nodes of a run: what a warp collides at a time

struct LatDesc {
  uint32_t Lx, Ly;
  uint32_t t0;          // step counter at the start of the round
  uint32_t phase;       // 0: buf0 holds the state at t0, 1: buf1 does
  uint32_t replica;
  uint32_t flip, omega_mode, rest_mode;
  uint32_t steps;       // steps this lattice takes in the round
  uint32_t particle;    // 1: particle sampler
  uint16_t* buf0;
  uint16_t* buf1;
  const uint32_t* tables;  // kDevBlockWords words
};

// Runs [run0, run1) of a lattice's nodes, for all steps of the round.
struct WorkShare {
  uint32_t lattice, run0, run1;
};

struct MultiArgs {
  const LatDesc* lat;
  const WorkShare* shares;
  const uint32_t* first;       // block b takes shares [first[b], first[b + 1])
  uint32_t steps;              // steps of the round (of the lattice with most)
  unsigned long long* sync;    // barrier word of the blocks, 0 at start
  uint32_t* fail;              // per lattice: first step of the round that would exceed 65535, ~0 if none
  unsigned long long* cycles;  // per block: cycles at work in the round
  uint32_t* gave_up;           // set to 1 when a wait between blocks gave up
};

size_t multi_smem_bytes();
cudaError_t prepare_multi_kernel();
// cooperative: at most one block per SM
cudaError_t launch_multi_round(const MultiArgs& ma, const StepArgs& common, int blocks, cudaStream_t s);

}  // namespace ilg
