// Multi-lattice steps: one cooperative launch advances every resident lattice of a server by
// the steps of a round.  The lattices' nodes, laid end to end and weighted by what a node of
// each costs, are cut into one equal share per block (one block per SM); a share holds parts
// of few lattices, so a block keeps their alias tables in shared memory for the whole round,
// and a barrier of all blocks separates the steps.  Each lattice keeps its own step counter,
// replica word and two buffers, so its result is the one it would have had alone.
// Bound: integer issue (see collide_warp; 70 % of it while many lattices run).  24 requests of
// 64 to 1024 a side at 5 to 100 per velocity: 52 ms in these launches.  What a step's nodes
// have in common (ten Philox words, ten planes) is read from shared memory where it is used:
// those loads cost next to nothing beside the collision, while some 30 registers for them left it
// short (55.2 ms; one lattice of 1024^2 at 50 per velocity 27.7 / 24.9 us per step, 17.9 / 15.4 at
// omega* = 0.1); one warp makes them for the next step while the others wait at the barrier.  Shares of a lattice
// that wait only for one another (608 blocks of 256 threads) took 80 where this took 63: the
// blocks of different lattices on an SM then wait at different times and leave it half idle.
#include <cuda_runtime.h>

#include "ilg_collide.cuh"
#include "ilg_device.cuh"
#include "ilg_multi.h"
#include "ilg_sync.cuh"

namespace ilg {

namespace {

constexpr uint32_t kMultiRing = 16;   // extension words per lane
constexpr uint32_t kMultiTables = 3;  // lattices whose (packed) tables a block holds
constexpr uint32_t kMultiDescs = 8;   // shares whose descriptors a block holds

// A share's lattice in shared memory, with what a step's nodes have in common: the launch-wide
// Philox words and the planes it reads (velocity i of the collision from plane from[i]: the
// flip F_i(n) = n_{-i}) and writes.
struct ShareDesc {
  WordKeys keys;
  const unsigned char* from[5];
  unsigned char* to[5];
  LatDesc d;
  WorkShare w;

  // one thread: for step sub of the round
  __device__ __forceinline__ void prepare(StepArgs a, uint32_t sub) {
    a.replica = d.replica;
    keys = word_keys(a, d.t0 + sub);
    const bool odd = ((sub + d.phase) & 1u) != 0;
    const size_t plane = sizeof(uint16_t) * size_t(d.Lx) * d.Ly;
    const unsigned char* const in = reinterpret_cast<const unsigned char*>(odd ? d.buf1 : d.buf0);
    unsigned char* const out = reinterpret_cast<unsigned char*>(odd ? d.buf0 : d.buf1);
#pragma unroll
    for (int i = 0; i < 5; ++i) {
      from[i] = in + (i == 0 || !d.flip ? i : (i & 1 ? i + 1 : i - 1)) * plane;
      to[i] = out + i * plane;
    }
  }
};

// One step of a block's share of a D2Q5 lattice.  TABLES: see collide_warp (and the binomial
// sampler).  Returns whether a node of the lane overflowed.  A byte's place in a plane has 32
// bits (a request's sides are at most 32768).
template <bool TABLES>
__device__ __forceinline__ bool step_share(const StepArgs& a, const volatile ShareDesc& sd, uint32_t sub,
                                           const uint32_t* s, unsigned char* ring) {
  constexpr int Q = 5;
  const Alias4 to = Alias4::of(s, 0), tr = Alias4::of(s, 1);
  const uint32_t Lx = sd.d.Lx, Ly = sd.d.Ly, nodes = Lx * Ly, run1 = sd.w.run1;
  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t run0 = sd.w.run0 + (threadIdx.x >> 5);
  constexpr uint32_t kStride = kMultiThreads;  // nodes
  const uint32_t stride_y = kStride / Lx, stride_x = kStride - stride_y * Lx;
  uint32_t node = run0 * kMultiRun + lane;
  uint32_t y = node / Lx, x = node - y * Lx;
  bool bad = false;
  for (uint32_t r = run0; r < run1; r += kMultiThreads / 32, node += kStride) {
    const bool active = node < nodes;
    const uint32_t off = node * 2;
    uint32_t m[Q], post[Q];
    // (through L2 only: another SM may have written these lines in the step before)
#pragma unroll
    for (int i = 0; i < Q; ++i) m[i] = active ? __ldcg(reinterpret_cast<const uint16_t*>(sd.from[i] + off)) : 0u;
    if (!TABLES && a.particle) collide_particle<Q>(a, s, node, sd.d.t0 + sub, m, post);
    else collide_warp<Q, 4 * kMultiThreads, kMultiRing, TABLES>(a, sd.keys, to, tr, tr, ring, 4 * threadIdx.x, node, m, post);
    if (active) {
      uint32_t high = 0;
#pragma unroll
      for (int i = 0; i < Q; ++i) high |= post[i];
      bad |= high > 65535u;
      const auto put = [&](int i, uint32_t at) { *reinterpret_cast<uint16_t*>(sd.to[i] + at) = uint16_t(post[i]); };
      // (offsets modulo 2^32: row y starts at node - x)
      const uint32_t row = Lx * 2, rows = nodes * 2;
      put(0, off);
      put(1, off + (x + 1 == Lx ? 2 - row : 2));
      put(2, off + (x == 0 ? row - 2 : ~1u));
      put(3, y + 1 == Ly ? off + row - rows : off + row);
      put(4, y == 0 ? off + rows - row : off - row);
    }
    x += stride_x;
    y += stride_y;
    if (x >= Lx) {
      x -= Lx;
      y += 1;
    }
  }
  return bad;
}

__global__ void __launch_bounds__(kMultiThreads, 1)
    multi_round_kernel(const __grid_constant__ MultiArgs ma, const __grid_constant__ StepArgs common) {
  extern __shared__ uint4 smem4[];
  uint32_t* const tables = reinterpret_cast<uint32_t*>(smem4);  // kMultiTables slots
  unsigned char* const ring = reinterpret_cast<unsigned char*>(tables + kMultiTables * kDevTableWords4);
  __shared__ ShareDesc descs[kMultiDescs];  // from the last on, shares take turns in it
  __shared__ int stop, failed;
  const uint32_t first = ma.first[blockIdx.x], n = ma.first[blockIdx.x + 1] - first;
  const auto load = [&](uint32_t k, uint32_t sub) {
    ShareDesc& sd = descs[min(k, kMultiDescs - 1)];
    sd.w = ma.shares[first + k];
    sd.d = ma.lat[sd.w.lattice];
    sd.prepare(common, sub);
  };
  if (threadIdx.x == 0) stop = failed = 0;
  if (threadIdx.x < min(n, kMultiDescs)) load(threadIdx.x, 0);
  __syncthreads();
  // the first shares' tables; from the last slot on, shares take turns in it
  const uint32_t held = min(n, kMultiTables);
  for (uint32_t k = 0; k < held; ++k)
    stage_tables4(descs[k].d.tables, tables + k * kDevTableWords4, descs[k].d.particle != 0);
  uint32_t in_last = held - 1;  // the share whose tables are in the last slot
  __syncthreads();
  unsigned long long busy = 0;
  for (uint32_t sub = 0;; ++sub) {
    const uint32_t begin = uint32_t(clock());
    for (uint32_t k = 0; k < n; ++k) {
      if (k >= kMultiDescs - 1 && n > kMultiDescs) {
        __syncthreads();
        if (threadIdx.x == 0) load(k, sub);
        __syncthreads();
      }
      const ShareDesc& sd = descs[min(k, kMultiDescs - 1)];
      const LatDesc& d = sd.d;
      // done for this round, or stopped by an overflow in an earlier step
      if (sub >= d.steps || (failed && *reinterpret_cast<volatile uint32_t*>(ma.fail + sd.w.lattice) < sub)) continue;
      const uint32_t slot = min(k, kMultiTables - 1);
      uint32_t* const s = tables + slot * kDevTableWords4;
      if (slot == kMultiTables - 1 && in_last != k) {
        __syncthreads();
        stage_tables4(d.tables, s, d.particle != 0);
        in_last = k;
        __syncthreads();
      }
      StepArgs a = common;
      a.omega_mode = d.omega_mode;
      a.rest_mode = d.rest_mode;
      a.replica = d.replica;
      a.particle = d.particle;
      const bool plain = !d.particle && d.omega_mode == kTable && d.rest_mode == kTable;
      const bool bad = plain ? step_share<true>(a, sd, sub, s, ring) : step_share<false>(a, sd, sub, s, ring);
      if (bad) {
        atomicMin(ma.fail + sd.w.lattice, sub);
        __threadfence();
        atomicOr(ma.sync, kRunMark);
      }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      busy += uint32_t(clock()) - begin;
      if (sub + 1 < ma.steps) {
        const unsigned long long v = run_barrier(ma.sync, (sub + 1) * gridDim.x);
        if (v == ~0ull) {
          atomicExch(ma.gave_up, 1u);
          stop = 1;
        } else if (v >= kRunMark) {
          failed = 1;  // some lattice, in this step or (a faster block's) the next: fail[] says
        }
      }
    }
    if (sub + 1 >= ma.steps) break;
    // meanwhile
    if (threadIdx.x >= 32 && threadIdx.x - 32 < min(n, kMultiDescs)) descs[threadIdx.x - 32].prepare(common, sub + 1);
    __syncthreads();
    if (stop) break;
  }
  if (threadIdx.x == 0) ma.cycles[blockIdx.x] = busy;
}

}  // namespace

size_t multi_smem_bytes() {
  return sizeof(uint32_t) * (kMultiTables * kDevTableWords4 + size_t(kMultiRing) * kMultiThreads);
}

cudaError_t prepare_multi_kernel() {
  return cudaFuncSetAttribute(multi_round_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, int(multi_smem_bytes()));
}

cudaError_t launch_multi_round(const MultiArgs& ma, const StepArgs& common, int blocks, cudaStream_t s) {
  MultiArgs m = ma;
  StepArgs c = common;
  void* p[] = {&m, &c};
  return cudaLaunchCooperativeKernel(reinterpret_cast<const void*>(multi_round_kernel), dim3(uint32_t(blocks)),
                                     dim3(kMultiThreads), p, multi_smem_bytes(), s);
}

}  // namespace ilg
