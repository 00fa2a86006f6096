// Multi-lattice steps: one cooperative launch advances every resident lattice of a server by
// the steps of a round.  The lattices' nodes, laid end to end and weighted by what a node of
// each costs, are cut into one equal share per block (one block per SM); a share holds parts
// of few lattices, so a block keeps their alias tables in shared memory for the whole round,
// and a barrier of all blocks separates the steps.  Each lattice keeps its own step counter,
// replica word and two buffers, so its result is the one it would have had alone.
// Bound: integer issue (see collide_warp; 70 % of it while many lattices run).  24 requests of
// 64 to 1024 a side at 5 to 100 per velocity: 55.3 ms in these launches.  Shares of a lattice
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

// One step of a block's share of a D2Q5 lattice.  TABLES: see collide_warp (and the binomial
// sampler).  Returns whether a node of the lane overflowed.
template <bool TABLES>
__device__ __forceinline__ bool step_share(const StepArgs& a, const LatDesc& d, const WorkShare& w, uint32_t sub,
                                           const uint32_t* s, unsigned char* ring) {
  constexpr int Q = 5;
  const Alias4 to = Alias4::of(s, 0), tr = Alias4::of(s, 1);
  const uint32_t Lx = d.Lx, Ly = d.Ly, nodes = Lx * Ly, t = d.t0 + sub;
  const size_t plane = nodes;
  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t run0 = w.run0 + (threadIdx.x >> 5);
  constexpr uint32_t kStride = kMultiThreads;  // nodes
  const uint32_t stride_y = kStride / Lx, stride_x = kStride - stride_y * Lx;
  uint32_t node = run0 * kMultiRun + lane;
  uint32_t y = node / Lx, x = node - y * Lx;
  const bool odd = ((sub + d.phase) & 1u) != 0;
  const uint16_t* const in = odd ? d.buf1 : d.buf0;
  uint16_t* const out = odd ? d.buf0 : d.buf1;
  // the flip F_i(n) = n_{-i}: velocity i of the collision reads plane -i
  const uint16_t* from[Q];
#pragma unroll
  for (int i = 0; i < Q; ++i) from[i] = in + (i == 0 || !d.flip ? i : (i & 1 ? i + 1 : i - 1)) * plane;
  const WordKeys keys = word_keys(a, t);
  bool bad = false;
  for (uint32_t r = run0; r < w.run1; r += kMultiThreads / 32, node += kStride) {
    const bool active = node < nodes;
    uint32_t m[Q], post[Q];
    // (through L2 only: another SM may have written these lines in the step before)
#pragma unroll
    for (int i = 0; i < Q; ++i) m[i] = active ? __ldcg(from[i] + node) : 0u;
    if (!TABLES && a.particle) collide_particle<Q>(a, s, node, t, m, post);
    else collide_warp<Q, 4 * kMultiThreads, kMultiRing, TABLES>(a, keys, to, tr, tr, ring, 4 * threadIdx.x, node, m, post);
    if (active) {
      uint32_t high = 0;
#pragma unroll
      for (int i = 0; i < Q; ++i) high |= post[i];
      bad |= high > 65535u;
      uint16_t* const o = out + node;  // row y starts at node - x
      o[0] = uint16_t(post[0]);
      (o + plane)[x + 1 == Lx ? -int32_t(x) : 1] = uint16_t(post[1]);
      (o + 2 * plane)[x == 0 ? int32_t(Lx) - 1 : -1] = uint16_t(post[2]);
      const uint32_t yp = y + 1 == Ly ? 0 : y + 1;
      const uint32_t ym = y == 0 ? Ly - 1 : y - 1;
      out[3 * plane + size_t(yp) * Lx + x] = uint16_t(post[3]);
      out[4 * plane + size_t(ym) * Lx + x] = uint16_t(post[4]);
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
  __shared__ LatDesc descs[kMultiDescs];
  __shared__ WorkShare shares[kMultiDescs];
  __shared__ int stop, failed;
  const uint32_t first = ma.first[blockIdx.x], n = ma.first[blockIdx.x + 1] - first;
  if (threadIdx.x == 0) stop = failed = 0;
  if (threadIdx.x < min(n, kMultiDescs)) {
    const WorkShare w = ma.shares[first + threadIdx.x];
    shares[threadIdx.x] = w;
    descs[threadIdx.x] = ma.lat[w.lattice];
  }
  __syncthreads();
  // the first shares' tables; from the last slot on, shares take turns in it
  const uint32_t held = min(n, kMultiTables);
  for (uint32_t k = 0; k < held; ++k)
    stage_tables4(descs[k].tables, tables + k * kDevTableWords4, descs[k].particle != 0);
  uint32_t in_last = held - 1;  // the share whose tables are in the last slot
  __syncthreads();
  unsigned long long busy = 0;
  for (uint32_t sub = 0;; ++sub) {
    const uint32_t begin = uint32_t(clock());
    for (uint32_t k = 0; k < n; ++k) {
      const WorkShare w = k < kMultiDescs ? shares[k] : ma.shares[first + k];
      const LatDesc d = k < kMultiDescs ? descs[k] : ma.lat[w.lattice];
      // done for this round, or stopped by an overflow in an earlier step
      if (sub >= d.steps || (failed && *reinterpret_cast<volatile uint32_t*>(ma.fail + w.lattice) < sub)) continue;
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
      const bool bad = plain ? step_share<true>(a, d, w, sub, s, ring) : step_share<false>(a, d, w, sub, s, ring);
      if (bad) {
        atomicMin(ma.fail + w.lattice, sub);
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
