// Kernels of the lattice-gas path: the fused flip + collision + streaming step,
// the Poisson initial state, the integer sums and the double-precision
// projections of the observables, and a Philox probe.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>

#include "ilg_collide.cuh"
#include "ilg_device.cuh"
#include "ilg_fixed.cuh"
#include "ilg_launch.h"
#include "ilg_sync.cuh"

namespace ilg {

// --------------------------------------------------------------------------
// steps, node-parallel: any extent, any occupations.  Each lane loads the Q occupations
// of its node, flips, collides with its warp (collide_warp) and scatters n'_i to the neighbour
// x + v_i (periodic).  One launch takes T steps: the alias tables are staged in shared
// memory once, and a barrier of all blocks (a cooperative launch) separates the steps,
// instead of a launch, a staging pass and an idle tail per step.
// Bound: integer issue (65 % of it over all, about 75 % between the barriers; some 650 warp
// instructions per 32 nodes at 50 per velocity and omega* = 0.5) on large lattices; the
// barrier and the latency of one node (1 to 2 us a step) on small ones.  One block of 1024 threads per SM holds the tables
// once, in the 64-bit form whose draw takes two instructions fewer than the packed one
// (29.1 against 31.0 us per step for two blocks of 512, 33 with packed tables).  Us per
// step against one launch per step with a collision that loops per lane: 1024^2 at 50 per
// velocity 24.0 / 37.3 (omega* 0.5), 15.0 / 26.8 (0.1); 1501 x 777 at 100 per velocity
// 41.8 / 66; 1024^2 at 200 per velocity, omega* = 1, 80.5 / 241; 96 x 40 1.6 / 18.7.
// --------------------------------------------------------------------------
constexpr uint32_t kStepRing = 16;  // extension words per lane

__host__ __device__ constexpr uint32_t run_table_words(int Q) { return Q == 9 ? kDevBlockWords9 : kDevStagedWords; }

// sync[0]: the barrier word, sync[1]: set to 1 when a wait gave up.  TABLES: the binomial
// sampler with both probabilities strictly between 0 and 1; false: anything else.  Off: type
// of a byte's place in a plane, 32 bits where that is enough (an add each for the five loads
// and stores instead of two: 1024^2 at 50 per velocity 24.0 / 24.3 us per step, 15.0 / 15.25
// at omega* = 0.1).
template <int Q, int THREADS, bool TABLES, class Off>
__global__ void __launch_bounds__(THREADS, 1)
    step_run_kernel(const __grid_constant__ StepArgs a, uint16_t* buf0, uint16_t* buf1, uint32_t t0, uint32_t T,
                    unsigned long long* fail, unsigned long long* sync) {
  extern __shared__ uint4 smem4[];
  __shared__ int stop;
  uint32_t* s = reinterpret_cast<uint32_t*>(smem4);
  // a step before this launch overflowed (one of its own stops it at the barriers: a block that
  // started late must not leave the others waiting there)
  if (threadIdx.x == 0) stop = *reinterpret_cast<volatile unsigned long long*>(fail) < t0;
  constexpr uint32_t kTables = run_table_words(Q);
  // the block's first words: the alias tables, or the particle sampler's boundaries (all
  // copies in flight at once, the first node's words made meanwhile)
  for (uint32_t i = threadIdx.x; i < kTables / 4; i += THREADS)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(uint32_t(__cvta_generic_to_shared(smem4 + i))),
                 "l"(reinterpret_cast<const uint4*>(a.tables) + i)
                 : "memory");
  unsigned char* const ring = reinterpret_cast<unsigned char*>(smem4) + 4 * kTables;
  const Alias8 to = Alias8::of(s, 0), tr = Alias8::of(s, 1), ta = Alias8::of(s, Q == 9 ? 2 : 1);

  const uint32_t nodes = a.Lx * a.Ly;
  const size_t plane = nodes;
  const uint32_t stride = gridDim.x * THREADS;
  const uint32_t stride_y = stride / a.Lx, stride_x = stride - stride_y * a.Lx;
  const uint32_t lane = threadIdx.x & 31u;
  // the warp's first node: runs of 32 go to the blocks in turn, so that what is left for the
  // last pass lies on all SMs and not on some with all their warps (1501 x 777 at 100 per velocity
  // 42.2 instead of 44.5 us per step, 2^20 nodes of D1Q3 23.7 / 25.3).  Four warps in a row take
  // theirs in another order than the four before: with the same one a sub-partition meets the
  // same part of a row each time, the crowded one of a sine (1024^2 at 50 +- 20, omega* = 0.5:
  // 24.8 us per step, here 24.0; 15.6, here 15.3 at 0.1; 1024 nodes in a row per block 24.85, 16.0)
  const uint32_t warp = threadIdx.x >> 5, place = (warp & ~3u) | ((warp + (warp >> 2)) & 3u);
  const uint32_t base0 = (place * gridDim.x + blockIdx.x) * 32;
  const uint32_t y0 = (base0 + lane) / a.Lx, x0 = base0 + lane - y0 * a.Lx;
  // the launch-wide Philox rounds of a step, and the first node's words: made for the next
  // step between a block's arrival at the barrier and its wait there (1024^2 at 50 per
  // velocity 25.0 instead of 25.5 us per step, 15.7 instead of 16.2 at omega* = 0.1).  D2Q9
  // has no registers for sixteen more words (768^2 at 10 per velocity 15.5 instead of 13.0)
  constexpr int NB = Q == 9 ? 4 : 2;
  constexpr bool kAhead = Q != 9;
  NodeKeys<NB> keys = word_keys<NB>(a, t0);
  SlotWords<NB> first;
  if (kAhead && (TABLES || !a.particle)) first.make(keys, a.rk, base0 + lane);
  asm volatile("cp.async.wait_all;\n" ::: "memory");
  __syncthreads();
  if (stop) return;
  for (uint32_t step = 0;; ++step) {
    const uint32_t t = t0 + step;
    const uint16_t* const in = (step & 1) ? buf1 : buf0;
    uint16_t* const out = (step & 1) ? buf0 : buf1;
    bool bad = false;
    // (x, y) of the lane's node, advanced by the grid stride (stride_y rows and stride_x
    // nodes) with a carry instead of a division per node
    uint32_t base = base0, x = x0, y = y0;
    // the flip F_i(n) = n_{-i}: velocity i of the collision reads plane -i
    const unsigned char* from[Q];
    unsigned char* to_plane[Q];
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      from[i] = reinterpret_cast<const unsigned char*>(in + (i == 0 || !a.flip ? i : (i & 1 ? i + 1 : i - 1)) * plane);
      to_plane[i] = reinterpret_cast<unsigned char*>(out + i * plane);
    }
    while (base < nodes) {
      const uint32_t node = base + lane;
      const bool active = node < nodes && node >= base;
      const Off off = Off(node) * 2;
      uint32_t m[Q], post[Q];
      // (through L2 only: another SM wrote these lines in the step before)
#pragma unroll
      for (int i = 0; i < Q; ++i) m[i] = active ? __ldcg(reinterpret_cast<const uint16_t*>(from[i] + off)) : 0u;
      if (!TABLES && a.particle) collide_particle<Q>(a, s, node, t, m, post);
      else if constexpr (kAhead) {
        SlotWords<NB> w = first;
        if (base != base0) w.make(keys, a.rk, node);
        collide_warp<Q, 4 * THREADS, kStepRing, TABLES>(a, keys, to, tr, ta, ring, 4 * threadIdx.x, node, m, post, &w);
      } else {
        collide_warp<Q, 4 * THREADS, kStepRing, TABLES>(a, keys, to, tr, ta, ring, 4 * threadIdx.x, node, m, post);
      }
      if (active) {
        uint32_t high = 0;
#pragma unroll
        for (int i = 0; i < Q; ++i) high |= post[i];
        bad |= high > 65535u;
        const auto put = [&](int i, Off at) { *reinterpret_cast<uint16_t*>(to_plane[i] + at) = uint16_t(post[i]); };
        // (offsets modulo 2^32: row y starts at node - x)
        const Off right = x + 1 == a.Lx ? Off(2) - Off(a.Lx) * 2 : Off(2), left = x == 0 ? Off(a.Lx) * 2 - 2 : Off(0) - 2;
        put(0, off);
        put(1, off + right);
        put(2, off + left);
        if constexpr (Q >= 5) {
          const Off row = Off(a.Lx) * 2, rows = Off(nodes) * 2;
          const Off up = y + 1 == a.Ly ? off + row - rows : off + row, down = y == 0 ? off + rows - row : off - row;
          put(3, up);
          put(4, down);
          if constexpr (Q == 9) {
            put(5, up + right);
            put(6, down + left);
            put(7, down + right);
            put(8, up + left);
          }
        }
      }
      x += stride_x;
      y += stride_y;
      if (x >= a.Lx) {
        x -= a.Lx;
        y += 1;
      }
      if (nodes - base <= stride) break;  // (base + stride may pass 2^32)
      base += stride;
    }
    if (bad) {
      note_overflow(a, fail, t);
      __threadfence();
      atomicOr(sync, kRunMark);
    }
    if (step + 1 == T) break;
    __syncthreads();
    if (threadIdx.x == 0) run_arrive(sync);
    // while the other blocks finish: the next step's words that need nothing of theirs
    keys = word_keys<NB>(a, t + 1);
    if (kAhead && (TABLES || !a.particle)) first.make(keys, a.rk, base0 + lane);
    if (threadIdx.x == 0) {
      const unsigned long long v = run_wait(sync, (step + 1) * gridDim.x);
      if (v == ~0ull) {
        note_gave_up(a, sync + 1);
        stop = 1;
      } else if (v >= kRunMark) {
        // a step overflowed: this one, or already the next one (a faster block's)
        stop = *reinterpret_cast<volatile unsigned long long*>(fail) <= t;
      }
    }
    __syncthreads();
    if (stop) break;
  }
}

constexpr size_t run_smem(int Q, int threads) {
  return sizeof(uint32_t) * (run_table_words(Q) + size_t(kStepRing) * threads);
}

// Shapes: one block per SM of as few threads (128, 512, 1024) as give every node a lane of
// its own; beyond that 1024 (D2Q9: 512, a node's nine planes need the registers).
struct RunShape {
  const void* fn;
  int threads;
};

template <int Q, int THREADS>
static const void* run_of(bool tables, bool far) {
  if constexpr (THREADS == (Q == 9 ? 512 : 1024)) {
    if (far) return tables ? reinterpret_cast<const void*>(step_run_kernel<Q, THREADS, true, uint64_t>)
                           : reinterpret_cast<const void*>(step_run_kernel<Q, THREADS, false, uint64_t>);
  }
  return tables ? reinterpret_cast<const void*>(step_run_kernel<Q, THREADS, true, uint32_t>)
                : reinterpret_cast<const void*>(step_run_kernel<Q, THREADS, false, uint32_t>);
}

// far: planes of more than 2^32 bytes (the largest blocks only).
template <int THREADS>
static const void* run_fn(int Q, bool tables, bool far = false) {
  if (Q == 3) return run_of<3, THREADS>(tables, far);
  if (Q == 5) return run_of<5, THREADS>(tables, far);
  if constexpr (THREADS <= 512) return run_of<9, THREADS>(tables, far);
  return nullptr;
}

// --------------------------------------------------------------------------
// several steps of a lattice that one cluster of blocks holds in its shared memory, a lane per
// node: block r keeps THREADS nodes' planes (two buffers), a node's results go straight into
// the planes of whichever blocks hold its neighbours, and the hardware's cluster barrier
// separates the steps.  A node's destinations never change, so their addresses are made once.
// Bound: the latency of one node's collision and of the barrier; through buffers in L2 a step
// also waited for its stores and its loads there.  Us per step, buffers in L2 with the cluster's
// barrier (to 4096 nodes) or the grid's / here: D1Q3 256 nodes 1.54 / 0.77, 8192 2.06 / 1.10;
// D2Q5 96 x 40 1.72 / 0.86, 64^2 at 50 per velocity 2.37 / 1.47, 90^2 2.06 / 1.13, 90^2 at 100
// 3.24 / 2.99; D2Q9 64^2 2.03 / 1.23, 90^2 2.34 / 1.82.  Blocks of 1024 threads (to 16384 nodes)
// lose to all SMs with the grid barrier at 25 per velocity and more (128^2 at 50 3.45 / 2.62).
// --------------------------------------------------------------------------
constexpr uint32_t kClusterBlocks = 16;  // (beyond 8 a kernel opts in)

template <int Q, int THREADS>
__global__ void __launch_bounds__(THREADS, 1)
    step_cluster_kernel(const __grid_constant__ StepArgs a, uint16_t* buf0, uint16_t* buf1, uint32_t t0, uint32_t T,
                        unsigned long long* fail) {
  extern __shared__ uint4 smem4[];
  __shared__ int stop;
  __shared__ uint32_t mark;  // the first step of this launch that overflowed
  uint32_t* const s = reinterpret_cast<uint32_t*>(smem4);
  if (threadIdx.x == 0) {
    stop = *reinterpret_cast<volatile unsigned long long*>(fail) < t0;
    mark = ~0u;
  }
  constexpr uint32_t kTables = run_table_words(Q);
  for (uint32_t i = threadIdx.x; i < kTables / 4; i += THREADS)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(uint32_t(__cvta_generic_to_shared(smem4 + i))),
                 "l"(reinterpret_cast<const uint4*>(a.tables) + i)
                 : "memory");
  unsigned char* const ring = reinterpret_cast<unsigned char*>(smem4) + 4 * kTables;
  // planes of this block's nodes, [buffer][velocity][THREADS]
  uint16_t* const planes = reinterpret_cast<uint16_t*>(ring + kStepRing * 4 * THREADS);
  constexpr uint32_t kBuffer = Q * THREADS;
  const Alias8 to = Alias8::of(s, 0), tr = Alias8::of(s, 1), ta = Alias8::of(s, Q == 9 ? 2 : 1);
  const uint32_t nodes = a.Lx * a.Ly, tid = threadIdx.x, node = blockIdx.x * THREADS + tid;
  const bool active = node < nodes;
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    planes[i * THREADS + tid] = active ? __ldcg(buf0 + (size_t(i) * nodes + node)) : 0;
    if (!active) planes[kBuffer + i * THREADS + tid] = 0;  // nobody writes there
  }
  // where velocity i's results go in buffer 0 of the block that holds the neighbour
  uint32_t dest[Q];
  {
    const uint32_t y = node / a.Lx, x = node - y * a.Lx;
    const uint32_t xs[3] = {x == 0 ? a.Lx - 1 : x - 1, x, x + 1 == a.Lx ? 0 : x + 1};
    const uint32_t ys[3] = {y == 0 ? a.Ly - 1 : y - 1, y, y + 1 == a.Ly ? 0 : y + 1};
    // +x, -x, +y, -y, then D2Q9's (+1,+1), (-1,-1), (+1,-1), (-1,+1)
    constexpr int dx[9] = {0, 1, -1, 0, 0, 1, -1, 1, -1}, dy[9] = {0, 0, 0, 1, -1, 1, -1, -1, 1};
    const uint32_t own = uint32_t(__cvta_generic_to_shared(planes));
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      const uint32_t d = active ? ys[1 + dy[i]] * a.Lx + xs[1 + dx[i]] : node;
      asm("mapa.shared::cluster.u32 %0, %1, %2;\n" : "=r"(dest[i]) : "r"(own + 2 * (i * THREADS + d % THREADS)), "r"(d / THREADS));
    }
  }
  constexpr int NB = Q == 9 ? 4 : 2;
  NodeKeys<NB> keys = word_keys<NB>(a, t0);
  SlotWords<NB> words;
  words.make(keys, a.rk, node);
  asm volatile("cp.async.wait_all;\n" ::: "memory");
  __syncthreads();
  if (stop) return;
  // every block has started: its planes are written by other blocks from here on
  cluster_arrive();
  cluster_wait();
  uint32_t step = 0;
  for (;; ++step) {
    const uint32_t t = t0 + step, in = (step & 1) * kBuffer, out = 2 * (kBuffer - in);
    uint32_t m[Q], post[Q];
    // the flip F_i(n) = n_{-i}: velocity i of the collision reads plane -i
#pragma unroll
    for (int i = 0; i < Q; ++i) m[i] = planes[in + (i == 0 || !a.flip ? i : (i & 1 ? i + 1 : i - 1)) * THREADS + tid];
    collide_warp<Q, 4 * THREADS, kStepRing, true>(a, keys, to, tr, ta, ring, 4 * tid, node, m, post, &words);
    if (active) {
      uint32_t high = 0;
#pragma unroll
      for (int i = 0; i < Q; ++i) {
        high |= post[i];
        asm volatile("st.shared::cluster.u16 [%0], %1;\n" ::"r"(dest[i] + out), "h"(uint16_t(post[i])) : "memory");
      }
      if (high > 65535u) {
        note_overflow(a, fail, t);
        cluster_mark(&mark, step, gridDim.x);
      }
    }
    __syncwarp();
    cluster_arrive();
    if (step + 1 < T) {
      // while the others finish: the next step's words
      keys = word_keys<NB>(a, t + 1);
      words.make(keys, a.rk, node);
    }
    cluster_wait();
    // (a faster block may already have marked the next step)
    if (*reinterpret_cast<volatile uint32_t*>(&mark) <= step) break;
    if (step + 1 == T) {
      ++step;
      break;
    }
  }
  // the state after `step` steps, into the buffer that many single steps would have left it in
  if (active) {
    uint16_t* const to_state = (step & 1) ? buf1 : buf0;
#pragma unroll
    for (int i = 0; i < Q; ++i) to_state[size_t(i) * nodes + node] = planes[(step & 1) * kBuffer + i * THREADS + tid];
  }
}

constexpr size_t cluster_smem(int Q, int threads) { return run_smem(Q, threads) + size_t(2) * Q * threads * sizeof(uint16_t); }

template <int THREADS>
static const void* cluster_fn(int Q) {
  return Q == 3   ? reinterpret_cast<const void*>(step_cluster_kernel<3, THREADS>)
         : Q == 5 ? reinterpret_cast<const void*>(step_cluster_kernel<5, THREADS>)
                  : reinterpret_cast<const void*>(step_cluster_kernel<9, THREADS>);
}

static const void* cluster_fn(int Q, int threads) {
  return threads == 128 ? cluster_fn<128>(Q) : threads == 256 ? cluster_fn<256>(Q) : cluster_fn<512>(Q);
}

// Sixteen blocks of as few threads as hold the lattice; 0: none does.
static int cluster_threads(bool tables, uint64_t nodes) {
  if (!tables) return 0;
  for (int threads : {128, 256, 512})
    if (nodes <= kClusterBlocks * uint64_t(threads)) return threads;
  return 0;
}

static bool run_tables(int Q, const StepArgs& a) {
  return !a.particle && a.omega_mode == kTable && a.rest_mode == kTable && (Q != 9 || a.axis_mode == kTable);
}

// --------------------------------------------------------------------------
// several steps of a lattice whose planes all SMs together hold in shared memory: block b keeps
// an equal share of the nodes' runs of 32 (row-major), and a result for a node of another share
// goes there as a word of a mailbox in L2 that carries the step's tag beside the value; whoever
// needs it polls that word, so no barrier of all blocks and no fence stands between the steps.
// Runs whose neighbours lie in other shares come first in a step: their words are on the way
// while the rest collides.  A mailbox word of one parity is written again only by a node that
// has had, as an input, a result of the node that read it.
// buf0 is only read: should a step overflow, the caller takes the steps before it again from
// there, since the shares may be steps apart by then.
// Bound: integer issue; with few nodes per SM a word's way to L2 and back.  Us per step, buffers
// in L2 and a barrier of all blocks / here: D2Q5 100^2 at 12 per velocity 2.09 / 1.43, 301 x 200
// 2.58 / 1.78, 400^2 at 50 8.01 / 5.61, 512^2 at 50 8.13 / 7.00, 850^2 at 50 18.3 / 17.5; D1Q3
// 65000 nodes at 30 2.46 / 1.46, 2^18 4.75 / 3.50, 2^20 13.3 / 12.0; D2Q9 200^2 3.15 / 2.43.
// Packed tables and shorter rings of extension words, which would let the planes of 1024^2 fit,
// cost there what the barrier takes (at 50 per velocity 24.9 / 25.7).  A pause between polls costs
// more than the polls (301 x 200 at 50 per velocity 2.79, 3.9 with 20 ns).
// --------------------------------------------------------------------------
struct ResidentArgs {
  uint32_t* mail;        // [parity][velocity - 1][node]: tag << 16 | value
  uint32_t tag;          // of the first step's results; below 2^16 for all steps
  uint32_t stride;       // nodes of the largest share
  unsigned long long* gave_up;  // set to 1 when a poll gave up
};
constexpr uint32_t kMailPolls = 1u << 21;  // seconds

__device__ __forceinline__ uint32_t mail_load(const uint32_t* p) {
  uint32_t v;
  asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];\n" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void mail_store(uint32_t* p, uint32_t v) {
  asm volatile("st.relaxed.gpu.global.u32 [%0], %1;\n" ::"l"(p), "r"(v) : "memory");
}

template <int Q, int THREADS>
__global__ void __launch_bounds__(THREADS, 1)
    step_resident_kernel(const __grid_constant__ StepArgs a, const uint16_t* buf0, uint16_t* buf1, uint32_t t0, uint32_t T,
                         unsigned long long* fail, const __grid_constant__ ResidentArgs ra) {
  constexpr uint32_t kTables = run_table_words(Q);
  extern __shared__ uint4 smem4[];
  __shared__ int stop;
  uint32_t* const s = reinterpret_cast<uint32_t*>(smem4);
  if (threadIdx.x == 0) stop = *reinterpret_cast<volatile unsigned long long*>(fail) < t0;
  for (uint32_t i = threadIdx.x; i < kTables / 4; i += blockDim.x)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(uint32_t(__cvta_generic_to_shared(smem4 + i))),
                 "l"(reinterpret_cast<const uint4*>(a.tables) + i)
                 : "memory");
  unsigned char* const words = reinterpret_cast<unsigned char*>(smem4) + 4 * kTables;
  uint16_t* const planes = reinterpret_cast<uint16_t*>(words + kStepRing * 4 * THREADS);  // [buffer][velocity][stride]
  const Alias8 to = Alias8::of(s, 0), tr = Alias8::of(s, 1), ta = Alias8::of(s, Q == 9 ? 2 : 1);

  const uint32_t nodes = a.Lx * a.Ly, lane = threadIdx.x & 31u, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
  const uint32_t runs = (nodes + 31) >> 5;
  // runs [r0, r0 + n) of the lattice, nodes [a0, a0 + P)
  const uint32_t r0 = uint32_t(uint64_t(blockIdx.x) * runs / gridDim.x);
  const uint32_t n = uint32_t(uint64_t(blockIdx.x + 1) * runs / gridDim.x) - r0;
  const uint32_t a0 = r0 * 32, P = min(n * 32, nodes - a0);
  // how far a node's neighbours lie, wraps from the last row to the first aside (D2Q9: up to
  // two rows from a row's ends)
  const uint32_t near = Q == 3 ? 1 : (Q == 5 ? a.Lx : a.Lx + 1);
  const uint32_t edge = min((near + 31) / 32 + 1, (n + 1) / 2);  // runs at either end that come first
  const uint32_t stride = ra.stride, buffer = Q * stride;
  for (uint32_t l = threadIdx.x; l < P; l += blockDim.x)
#pragma unroll
    for (int i = 0; i < Q; ++i) planes[i * stride + l] = __ldcg(buf0 + (size_t(i) * nodes + a0 + l));
  uint32_t* const xs = reinterpret_cast<uint32_t*>(planes + 2 * buffer);  // x of each run's first node
  for (uint32_t r = threadIdx.x; r < n; r += blockDim.x) xs[r] = (a0 + 32 * r) % a.Lx;
  constexpr int NB = Q == 9 ? 4 : 2;
  asm volatile("cp.async.wait_all;\n" ::: "memory");
  __syncthreads();
  if (stop) return;

  // the j-th run of a step: the ends of the share first
  const auto run_of = [&](uint32_t j) { return j >= 2 * edge ? j - edge : (j & 1 ? n - 1 - j / 2 : j / 2); };
  // a node's neighbours in its row and beside it (wrapped), and whether they lie in this share
  struct Around {
    uint32_t right, left, dy_up, dy_down;  // (what to add to a node to move a row up / down)
  };
  const auto around = [&](uint32_t node, uint32_t x) {
    Around o;
    o.right = x + 1 == a.Lx ? node + 1 - a.Lx : node + 1;
    o.left = x == 0 ? node + a.Lx - 1 : node - 1;
    o.dy_up = node + a.Lx >= nodes ? a.Lx - nodes : a.Lx;
    o.dy_down = node < a.Lx ? nodes - a.Lx : 0u - a.Lx;
    return o;
  };
  // neighbour of velocity i (+x, -x, +y, -y, then D2Q9's (+1,+1), (-1,-1), (+1,-1), (-1,+1))
  const auto neighbour = [&](const Around& o, uint32_t node, int i) {
    constexpr int dx[9] = {0, 1, -1, 0, 0, 1, -1, 1, -1}, dy[9] = {0, 0, 0, 1, -1, 1, -1, -1, 1};
    const uint32_t in_row = dx[i] > 0 ? o.right : (dx[i] < 0 ? o.left : node);
    return dy[i] > 0 ? in_row + o.dy_up : (dy[i] < 0 ? in_row + o.dy_down : in_row);
  };
  const auto opposite = [](int i) { return i == 0 ? 0 : (i & 1 ? i + 1 : i - 1); };
  // the words of plane p for this share's nodes whose plane-p value comes from elsewhere, of the
  // state that tag stands for (parity: of its step)
  const auto take_mail = [&](const Around& o, uint32_t node, bool active, uint32_t tag, uint32_t parity, uint32_t (&v)[Q]) {
    const uint32_t* const box = ra.mail + size_t(parity) * (Q - 1) * nodes + node;
    uint32_t w[Q];
    bool cross[Q];
    bool missing = false;
#pragma unroll
    for (int p = 1; p < Q; ++p) {
      cross[p] = active && neighbour(o, node, opposite(p)) - a0 >= P;
      w[p] = cross[p] ? mail_load(box + size_t(p - 1) * nodes) : 0u;
    }
#pragma unroll
    for (int p = 1; p < Q; ++p) missing |= cross[p] && (w[p] >> 16) != tag;
    for (uint32_t polls = 0; missing; ++polls) {
      if (polls == kMailPolls || *reinterpret_cast<volatile int*>(&stop)) {
        note_gave_up(a, ra.gave_up);
        *reinterpret_cast<volatile int*>(&stop) = 1;
        break;
      }
      missing = false;
#pragma unroll
      for (int p = 1; p < Q; ++p)
        if (cross[p] && (w[p] >> 16) != tag) {
          w[p] = mail_load(box + size_t(p - 1) * nodes);
          missing |= (w[p] >> 16) != tag;
        }
    }
#pragma unroll
    for (int p = 1; p < Q; ++p)
      if (cross[p]) v[p] = w[p] & 0xFFFFu;
  };

  // A step's launch-wide Philox words: shares of several runs per warp (or nearly so) read them
  // from shared memory, made there by one thread a step ahead, and have the registers for the
  // collision (us per step: 513 x 512 at 12 per velocity 4.30 / 4.54 in registers, 768^2 at 10
  // 7.4 / 7.8, 850^2 at 50 17.5 / 17.9); where a step is one node's chain they stay in registers
  // (100^2 1.44 / 1.38; D2Q9 200^2 2.50 / 2.44).
  constexpr bool kSharedWords = THREADS >= 512 && Q != 9;
  __shared__ NodeKeys<NB> step_words[2];
  NodeKeys<NB> held = word_keys<NB>(a, t0);
  const bool maker = kSharedWords && threadIdx.x == blockDim.x - 1;
  if (maker) step_words[0] = held;
  if (kSharedWords) __syncthreads();
  for (uint32_t step = 0;; ++step) {
    const uint32_t t = t0 + step, in = (step & 1) * buffer, out = buffer - in;
    if (maker) step_words[(step + 1) & 1] = word_keys<NB>(a, t + 1);
    bool bad = false;
    for (uint32_t j = warp; j < n; j += warps) {
      const uint32_t r = run_of(j), l = 32 * r + lane, node = a0 + l;
      const bool active = l < P;
      const uint32_t x0 = xs[r];
      uint32_t x = x0 + lane;
      if (x >= a.Lx) x -= a.Lx;
      const uint32_t reach = Q == 9 && (x0 == 0 || x0 + 32 >= a.Lx) ? 2 * a.Lx : near;
      // every neighbour of the run's nodes in this share
      const bool inner = 32 * r >= reach && 32 * r + 31 + reach < P && 32 * r + a0 >= reach && 32 * r + a0 + 31 + reach < nodes;
      uint32_t v[Q], m[Q], post[Q];
#pragma unroll
      for (int i = 0; i < Q; ++i) v[i] = active ? planes[in + i * stride + l] : 0u;
      Around o = around(node, x);
      if (!inner && step > 0) take_mail(o, node, active, ra.tag + step - 1, step & 1, v);
      // the flip F_i(n) = n_{-i}: velocity i of the collision reads plane -i
#pragma unroll
      for (int i = 0; i < Q; ++i) m[i] = a.flip ? v[opposite(i)] : v[i];
      if constexpr (kSharedWords) {
        const volatile NodeKeys<NB>& shared = step_words[step & 1];
        collide_warp<Q, 4 * THREADS, kStepRing, true>(a, shared, to, tr, ta, words, 4 * threadIdx.x, node, m, post);
      } else {
        collide_warp<Q, 4 * THREADS, kStepRing, true>(a, held, to, tr, ta, words, 4 * threadIdx.x, node, m, post);
      }
      if (active) {
        uint32_t high = 0;
#pragma unroll
        for (int i = 0; i < Q; ++i) high |= post[i];
        bad |= high > 65535u;
        planes[out + l] = uint16_t(post[0]);
        if (inner) {
#pragma unroll
          for (int i = 1; i < Q; ++i) planes[out + i * stride + (neighbour(o, node, i) - a0)] = uint16_t(post[i]);
        } else {
          uint32_t* const box = ra.mail + size_t((step + 1) & 1) * (Q - 1) * nodes;
          const uint32_t tag = (ra.tag + step) << 16;
#pragma unroll
          for (int i = 1; i < Q; ++i) {
            const uint32_t d = neighbour(o, node, i);
            if (d - a0 < P) planes[out + i * stride + (d - a0)] = uint16_t(post[i]);
            else mail_store(box + (size_t(i - 1) * nodes + d), tag | (post[i] & 0xFFFFu));
          }
        }
      }
    }
    if (bad) note_overflow(a, fail, t);
    if (!kSharedWords) held = word_keys<NB>(a, t + 1);
    __syncthreads();
    if (stop || step + 1 == T) break;
  }
  if (stop) return;
  for (uint32_t r = warp; r < n; r += warps) {
    const uint32_t l = 32 * r + lane, node = a0 + l;
    const bool active = l < P;
    uint32_t x = xs[r] + lane, v[Q];
    if (x >= a.Lx) x -= a.Lx;
#pragma unroll
    for (int i = 0; i < Q; ++i) v[i] = active ? planes[(T & 1) * buffer + i * stride + l] : 0u;
    take_mail(around(node, x), node, active, ra.tag + T - 1, T & 1, v);
    if (active)
#pragma unroll
      for (int i = 0; i < Q; ++i) buf1[size_t(i) * nodes + node] = uint16_t(v[i]);
  }
}

static RunShape run_shape(int Q, const StepArgs& a, uint64_t nodes, uint32_t sms) {
  const bool tables = run_tables(Q, a);
  if (nodes <= uint64_t(sms) * 128) return {run_fn<128>(Q, tables), 128};
  const bool far = nodes > (uint64_t(1) << 31);
  if (Q == 9 || nodes <= uint64_t(sms) * 512) return {run_fn<512>(Q, tables, far), 512};
  return {run_fn<1024>(Q, tables, far), 1024};
}

template <int THREADS>
static const void* resident_fn(int Q) {
  if (Q == 3) return reinterpret_cast<const void*>(step_resident_kernel<3, THREADS>);
  if (Q == 5) return reinterpret_cast<const void*>(step_resident_kernel<5, THREADS>);
  if constexpr (THREADS <= 512) return reinterpret_cast<const void*>(step_resident_kernel<9, THREADS>);
  return nullptr;
}

struct ResidentShape {
  const void* fn;
  int threads;            // of the instantiation; a block has no more warps than runs
  uint32_t blocks, runs;  // runs of the largest share
  size_t smem;
};
constexpr size_t kResidentSmem = 227 * 1024 - 256;

// One share per SM, in blocks of as few threads as give every node a lane (as run_shape); false:
// the planes do not fit, the lattice is a cluster's, a run may span more than two rows, or a
// D2Q9 block would have more than one run per warp (its eight words per node then cost more than
// the barrier: 512^2 8.5 us per step / 7.5).
static bool resident_shape(int Q, uint32_t Lx, uint64_t nodes, uint32_t sms, ResidentShape* r) {
  if (Lx < 32 || nodes <= uint64_t(kClusterBlocks) * 512 || nodes >= (1u << 30)) return false;
  const uint32_t runs = uint32_t((nodes + 31) / 32);
  r->blocks = std::min(runs, sms);
  r->runs = (runs + r->blocks - 1) / r->blocks;
  if (Q == 9 && r->runs > 16) return false;
  r->threads = r->runs <= 4 ? 128 : (r->runs <= 16 ? 512 : 1024);
  r->fn = r->threads == 128 ? resident_fn<128>(Q) : r->threads == 512 ? resident_fn<512>(Q) : resident_fn<1024>(Q);
  r->smem = sizeof(uint32_t) * (run_table_words(Q) + size_t(kStepRing) * r->threads + r->runs) +
            sizeof(uint16_t) * 2 * Q * 32 * size_t(r->runs);
  return r->smem <= kResidentSmem;
}

size_t step_resident_mail_words(int Q, uint32_t Lx, uint64_t nodes, uint32_t sms) {
  ResidentShape r;
  return resident_shape(Q, Lx, nodes, sms, &r) ? 2 * size_t(Q - 1) * nodes : 0;
}

cudaError_t launch_step_resident(int Q, const StepArgs& a, const uint16_t* buf0, uint16_t* buf1, uint32_t t, uint32_t T,
                                 unsigned long long* fail, unsigned long long* sync, uint32_t* mail, uint32_t tag,
                                 uint32_t sms, cudaStream_t s) {
  ResidentShape r;
  if (!run_tables(Q, a) || !resident_shape(Q, a.Lx, uint64_t(a.Lx) * a.Ly, sms, &r)) return cudaErrorNotSupported;
  StepArgs args = a;
  ResidentArgs ra{mail, tag, 32 * r.runs, sync + 1};
  void* p[] = {&args, &buf0, &buf1, &t, &T, &fail, &ra};
  return cudaLaunchCooperativeKernel(r.fn, dim3(r.blocks), dim3(std::min<uint32_t>(r.threads, 32 * r.runs)), p, r.smem, s);
}

cudaError_t prepare_step_kernels(int Q) {
  cudaError_t e = cudaSuccess;
  auto set = [&](const void* f, int threads) {
    if (f && e == cudaSuccess)
      e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, int(run_smem(Q, threads)));
  };
  for (bool tables : {false, true}) {
    set(run_fn<128>(Q, tables), 128);
    set(run_fn<512>(Q, tables), 512);
    set(run_fn<1024>(Q, tables), 1024);
    set(Q == 9 ? run_fn<512>(Q, tables, true) : run_fn<1024>(Q, tables, true), Q == 9 ? 512 : 1024);
  }
  for (const void* f : {resident_fn<128>(Q), resident_fn<512>(Q), resident_fn<1024>(Q)})
    if (f && e == cudaSuccess)
      e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, int(kResidentSmem));
  for (int threads : {128, 256, 512}) {
    const void* f = cluster_fn(Q, threads);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, int(cluster_smem(Q, threads)));
    if (e == cudaSuccess) e = cudaFuncSetAttribute(f, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  }
  return e;
}

cudaError_t launch_step_run(int Q, const StepArgs& a, uint16_t* buf0, uint16_t* buf1, uint32_t t, uint32_t T,
                            unsigned long long* fail, unsigned long long* sync, uint32_t sms, cudaStream_t s) {
  const uint64_t nodes = uint64_t(a.Lx) * a.Ly;
  const int ct = T > 1 ? cluster_threads(run_tables(Q, a), nodes) : 0;
  if (ct) {
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr = {};
    uint32_t blocks = 1;
    while (uint64_t(blocks) * ct < nodes) blocks *= 2;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = blocks;
    attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3(ct);
    cfg.dynamicSmemBytes = cluster_smem(Q, ct);
    cfg.stream = s;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    StepArgs ca = a;
    void* p[] = {&ca, &buf0, &buf1, &t, &T, &fail};
    if (cudaLaunchKernelExC(&cfg, cluster_fn(Q, ct), p) == cudaSuccess) return cudaSuccess;
    cudaGetLastError();  // no room for a cluster (SMs reserved elsewhere): the grid barrier instead
  }
  const RunShape r = run_shape(Q, a, nodes, sms);
  const dim3 grid(uint32_t(std::min<uint64_t>((nodes + r.threads - 1) / r.threads, sms)));
  StepArgs args = a;
  void* p[] = {&args, &buf0, &buf1, &t, &T, &fail, &sync};
  if (T == 1) return cudaLaunchKernel(r.fn, grid, dim3(r.threads), p, run_smem(Q, r.threads), s);
  const cudaError_t e = cudaMemsetAsync(sync, 0, sizeof(unsigned long long), s);
  if (e != cudaSuccess) return e;
  return cudaLaunchCooperativeKernel(r.fn, grid, dim3(r.threads), p, run_smem(Q, r.threads), s);
}

// --------------------------------------------------------------------------
// initial state: n_i = number of table entries T[j], j < K-1, with u >= T[j]
// (binary search), u = word i of the init stream of the node.
// --------------------------------------------------------------------------
template <int Q>
__global__ void __launch_bounds__(256) init_kernel(InitArgs a, uint16_t* __restrict__ out) {
  const uint32_t nodes = a.Lx * a.Ly;
  const size_t plane = nodes;
  for (uint32_t node = blockIdx.x * blockDim.x + threadIdx.x; node < nodes;
       node += gridDim.x * blockDim.x) {
    const uint32_t y = node / a.Lx;
    const uint32_t x = node - y * a.Lx;
    uint32_t r = 0;
    if (a.axis == 1) r = uint32_t((uint64_t(a.mode) * x) % a.period);
    else if (a.axis == 2) r = uint32_t((uint64_t(a.mode) * y) % a.period);
    uint32_t W[(Q + 3) / 4 * 4];
#pragma unroll
    for (int b = 0; b < (Q + 3) / 4; ++b) {
      const uint4 w = philox(counter(node, 0u, a.replica, kDevTagInit | uint32_t(b)), a.key0, a.key1);
      W[4 * b] = w.x;
      W[4 * b + 1] = w.y;
      W[4 * b + 2] = w.z;
      W[4 * b + 3] = w.w;
    }
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      // weight class of the velocity: rest, moving (D2Q9: axis, diagonal)
      const uint32_t cls = !a.weighted || i == 0 ? 0u : (Q == 9 && i > 4 ? 2u : 1u);
      const uint32_t idx = cls * a.period + r;
      const uint32_t* T = a.table + a.offset[idx];
      const uint32_t K = a.count[idx];
      const uint32_t u = W[i];
      // first j in [0, K-1) with T[j] > u, i.e. the count of entries <= u
      uint32_t lo = 0, hi = K - 1;
      while (lo < hi) {
        const uint32_t mid = (lo + hi) >> 1;
        if (u >= T[mid]) lo = mid + 1;
        else hi = mid;
      }
      out[i * plane + node] = uint16_t(lo);
    }
  }
}

// The same where every node has the same mean (one table per weight class) and there are
// enough nodes to pay for it: the inversion starts from a guide in shared memory, whose
// entry for the draw's top bits holds the first outcome j whose table entry lies above the
// bucket's start, and that entry: below it the outcome is j, else the search goes on upward
// (about one draw in eighty at a mean of 10).  Four nodes per lane (D2Q9: two) where the
// lattice has a multiple of four (8-byte stores).
// Bound: integer issue, two Philox blocks per D2Q5 node.  16384^2 D2Q5 5.3 -> 1.7 ms,
// 4096^2 D2Q9 0.59 -> 0.20 ms; on 600^2 the two are equal.
constexpr uint32_t kGuideBits = 10;
constexpr uint32_t kGuide = 1u << kGuideBits;
constexpr int kInitThreads = 512;
constexpr size_t kInitUniformSmem = 96 * 1024;        // guides and tables, two blocks per SM
constexpr uint64_t kInitUniformNodesPerSm = 4096;     // below: the guides cost more than they save

struct RoundKeys {
  uint32_t k[20];
};

template <int Q, int NPT>
__global__ void __launch_bounds__(kInitThreads, 2) init_uniform_kernel(const __grid_constant__ InitArgs a, uint32_t classes,
                                                                       const __grid_constant__ RoundKeys rk,
                                                                       uint16_t* __restrict__ out) {
  extern __shared__ uint4 smem4[];
  uint2* guide = reinterpret_cast<uint2*>(smem4);                             // kGuide per class: {T[j], j}
  uint32_t* table = reinterpret_cast<uint32_t*>(guide + classes * kGuide);    // the classes' tables, as offset[] says
  const uint32_t words = a.offset[classes - 1] + a.count[classes - 1] - a.offset[0];
  for (uint32_t i = threadIdx.x; i < words; i += kInitThreads) table[i] = a.table[a.offset[0] + i];
  __syncthreads();
  for (uint32_t i = threadIdx.x; i < classes * kGuide; i += kInitThreads) {
    const uint32_t c = i >> kGuideBits, u = (i & (kGuide - 1)) << (32 - kGuideBits);
    const uint32_t* T = table + (a.offset[c] - a.offset[0]);
    uint32_t lo = 0, hi = a.count[c] - 1;
    while (lo < hi) {
      const uint32_t mid = (lo + hi) >> 1;
      if (u >= T[mid]) lo = mid + 1;
      else hi = mid;
    }
    guide[i] = make_uint2(T[lo], lo);
  }
  __syncthreads();
  const uint32_t nodes = a.Lx * a.Ly;
  const size_t plane = nodes;
  constexpr int NB = (Q + 3) / 4;
  // the launch-wide Philox rounds, as step_keys makes them (t = 0, the init tag)
  const StepKeys<NB> keys = stream_keys<NB>(rk.k, 0u, a.replica, kDevTagInit);
  for (uint64_t v = uint64_t(blockIdx.x) * kInitThreads + threadIdx.x; v * NPT < nodes; v += uint64_t(gridDim.x) * kInitThreads) {
    const uint32_t node0 = uint32_t(v) * NPT;
    uint32_t n[Q][NPT];
#pragma unroll
    for (int k = 0; k < NPT; ++k) {
      uint32_t W[4 * NB];
      step_blocks<NB>(keys, rk.k, node0 + k, W);
#pragma unroll
      for (int i = 0; i < Q; ++i) {
        const uint32_t c = !a.weighted || i == 0 ? 0u : (Q == 9 && i > 4 ? 2u : 1u);
        const uint32_t u = W[i];
        const uint2 g = guide[c * kGuide + (u >> (32 - kGuideBits))];
        uint32_t j = g.y;
        if (u >= g.x) {
          const uint32_t* T = table + (a.offset[c] - a.offset[0]);
          const uint32_t last = a.count[c] - 1;
          while (j < last && u >= T[j]) ++j;
        }
        n[i][k] = j;
      }
    }
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      uint16_t* const p = out + (i * plane + node0);
      if constexpr (NPT == 4)
        *reinterpret_cast<uint2*>(p) = make_uint2(n[i][0] | (n[i][1] << 16), n[i][2] | (n[i][3] << 16));
      else if constexpr (NPT == 2)
        *reinterpret_cast<uint32_t*>(p) = n[i][0] | (n[i][1] << 16);
      else
        *p = uint16_t(n[i][0]);
    }
  }
}

template <int Q>
static cudaError_t init_uniform_launch(const InitArgs& a, uint32_t classes, uint32_t words, uint16_t* out, uint32_t sms,
                                       cudaStream_t s) {
  const size_t smem = sizeof(uint2) * classes * kGuide + sizeof(uint32_t) * words;
  const uint32_t nodes = a.Lx * a.Ly;
  RoundKeys rk;
  for (int r = 0; r < 10; ++r) {
    rk.k[2 * r] = a.key0 + uint32_t(r) * 0x9E3779B9u;
    rk.k[2 * r + 1] = a.key1 + uint32_t(r) * 0xBB67AE85u;
  }
  auto go = [&](auto kernel) -> cudaError_t {
    const cudaError_t e =
        cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, int(kInitUniformSmem));
    if (e != cudaSuccess) return e;
    kernel<<<2 * sms, kInitThreads, smem, s>>>(a, classes, rk, out);
    return cudaGetLastError();
  };
  constexpr int kNpt = Q == 9 ? 2 : 4;  // (four nodes of nine velocities spill)
  return nodes % 4 == 0 && reinterpret_cast<uintptr_t>(out) % 8 == 0 ? go(init_uniform_kernel<Q, kNpt>)
                                                                     : go(init_uniform_kernel<Q, 1>);
}

cudaError_t launch_init(int Q, const InitArgs& a, uint32_t words, uint16_t* out, uint32_t sms, cudaStream_t s) {
  const uint64_t nodes = uint64_t(a.Lx) * a.Ly;
  const uint32_t classes = a.weighted ? (Q == 9 ? 3u : 2u) : 1u;
  if (a.period == 1 && nodes >= uint64_t(sms) * kInitUniformNodesPerSm &&
      sizeof(uint2) * classes * kGuide + sizeof(uint32_t) * size_t(words) <= kInitUniformSmem) {
    if (Q == 3) return init_uniform_launch<3>(a, classes, words, out, sms, s);
    if (Q == 5) return init_uniform_launch<5>(a, classes, words, out, sms, s);
    return init_uniform_launch<9>(a, classes, words, out, sms, s);
  }
  const int grid = int(std::min<uint64_t>((nodes + 255) / 256, uint64_t(sms) * 4));
  if (Q == 3) init_kernel<3><<<grid, 256, 0, s>>>(a, out);
  else if (Q == 5) init_kernel<5><<<grid, 256, 0, s>>>(a, out);
  else init_kernel<9><<<grid, 256, 0, s>>>(a, out);
  return cudaGetLastError();
}

// --------------------------------------------------------------------------
// integer sums: N(x,y) = sum_i n_i; column sums C(x), row sums R(y) and the mass.  A block
// takes 32 vectors of VEC nodes (16-byte loads where rows are a multiple of 8 and the
// state is aligned) by 8 R rows, adds its eight row groups in shared memory and issues one
// 64-bit atomic per column; row sums by warp shuffles, one atomic per warp and row.
// Bound: HBM for states beyond L2 (16384^2 D2Q5: 0.39 ms, 0.98 of the measured copy rate),
// the latency of a thread's R dependent rows for small ones: R is as small as still gives
// every SM four blocks (1024^2: 4 us where 64 rows in one thread took 45).
// --------------------------------------------------------------------------
constexpr uint32_t kSumGroups = 8;    // row groups (warps) of a block
constexpr uint32_t kSumMaxRows = 64;  // rows per thread at most

template <int Q, int VEC>
__global__ void __launch_bounds__(32 * kSumGroups) sums_kernel(const uint16_t* __restrict__ in, uint32_t Lx, uint32_t Ly,
                                                               uint32_t R, unsigned long long* __restrict__ col,
                                                               unsigned long long* __restrict__ row,
                                                               unsigned long long* __restrict__ mass, int want_rows) {
  __shared__ uint32_t red[kSumGroups][32 * VEC];
  __shared__ unsigned long long total[kSumGroups];
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");  // (they wait for this kernel's end themselves)
  const uint32_t tx = threadIdx.x & 31u, ty = threadIdx.x >> 5;
  const uint64_t x = (uint64_t(blockIdx.x) * 32 + tx) * VEC;
  const size_t plane = size_t(Lx) * Ly;
  const uint32_t chunks = (Ly + kSumGroups * R - 1) / (kSumGroups * R);
  // a block that has the lattice to itself writes its sums over what was there
  const bool alone = gridDim.x == 1 && gridDim.y == 1;
  unsigned long long sum = 0;
  for (uint32_t chunk = blockIdx.y; chunk < chunks; chunk += gridDim.y) {
    const uint32_t y0 = chunk * kSumGroups * R;
    uint32_t acc[VEC];  // at most 64 rows of 9 x 65535
#pragma unroll
    for (int j = 0; j < VEC; ++j) acc[j] = 0;
#pragma unroll 2
    for (uint32_t k = 0; k < R; ++k) {
      const uint32_t y = y0 + ty + kSumGroups * k;
      if (y >= Ly || y < y0) break;
      uint32_t n[VEC];
#pragma unroll
      for (int j = 0; j < VEC; ++j) n[j] = 0;
      if (x < Lx) {
        const uint16_t* p = in + (size_t(y) * Lx + x);
#pragma unroll
        for (int i = 0; i < Q; ++i) {
          if constexpr (VEC == 8) {
            const uint4 w = __ldg(reinterpret_cast<const uint4*>(p + i * plane));
            n[0] += w.x & 0xFFFFu;
            n[1] += w.x >> 16;
            n[2] += w.y & 0xFFFFu;
            n[3] += w.y >> 16;
            n[4] += w.z & 0xFFFFu;
            n[5] += w.z >> 16;
            n[6] += w.w & 0xFFFFu;
            n[7] += w.w >> 16;
          } else {
            n[0] += p[i * plane];
          }
        }
      }
      uint32_t N = 0;
#pragma unroll
      for (int j = 0; j < VEC; ++j) {
        acc[j] += n[j];
        N += n[j];
      }
      if (want_rows) {
        N = __reduce_add_sync(0xFFFFFFFFu, N);  // at most 256 nodes of 9 x 65535
        if (tx == 0) {
          if (alone) row[y] = N;
          else if (N) atomicAdd(row + y, static_cast<unsigned long long>(N));
        }
      }
    }
#pragma unroll
    for (int j = 0; j < VEC; ++j) red[ty][tx * VEC + j] = acc[j];
    __syncthreads();
    const uint64_t c = uint64_t(blockIdx.x) * 32 * VEC + threadIdx.x;
    if (threadIdx.x < 32 * VEC && c < Lx) {
      unsigned long long C = 0;
#pragma unroll
      for (uint32_t g = 0; g < kSumGroups; ++g) C += red[g][threadIdx.x];
      if (alone) col[c] = C;
      else if (C) atomicAdd(col + c, C);
      sum += C;
    }
    __syncthreads();
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) sum += __shfl_down_sync(0xFFFFFFFFu, sum, o);
  if (tx == 0) total[ty] = sum;
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned long long M = 0;
    for (uint32_t g = 0; g < kSumGroups; ++g) M += total[g];
    if (alone) *mass = M;
    else if (M) atomicAdd(mass, M);
  }
}

template <int Q>
static cudaError_t sums_launch(const uint16_t* in, uint32_t Lx, uint32_t Ly, unsigned long long* col,
                               unsigned long long* row, unsigned long long* mass, int want_rows, uint32_t sms,
                               cudaStream_t s) {
  const bool wide = Lx % 8 == 0 && reinterpret_cast<uintptr_t>(in) % 16 == 0;
  const uint32_t width = wide ? 256 : 32;
  const uint32_t gx = uint32_t((uint64_t(Lx) + width - 1) / width);
  const uint64_t groups = (uint64_t(Ly) + kSumGroups - 1) / kSumGroups;  // rows per thread if one block took all
  const uint32_t want = std::max<uint32_t>(1, 4 * sms / gx);            // blocks along y
  const uint32_t R = uint32_t(std::min<uint64_t>(kSumMaxRows, std::max<uint64_t>(1, groups / want)));
  const dim3 grid(gx, uint32_t(std::min<uint64_t>(65535, (groups + R - 1) / R)));
  if (grid.x > 1 || grid.y > 1) {  // (one block: nothing to clear; giving it 40 rows instead of 8 took longer than that)
    const bool together = want_rows && row == col + Lx;
    cudaError_t e = cudaMemsetAsync(mass, 0, sizeof(unsigned long long) * (1 + size_t(Lx) + (together ? Ly : 0)), s);
    if (e == cudaSuccess && want_rows && !together) e = cudaMemsetAsync(row, 0, sizeof(unsigned long long) * Ly, s);
    if (e != cudaSuccess) return e;
  }
  if (wide) sums_kernel<Q, 8><<<grid, 32 * kSumGroups, 0, s>>>(in, Lx, Ly, R, col, row, mass, want_rows);
  else sums_kernel<Q, 1><<<grid, 32 * kSumGroups, 0, s>>>(in, Lx, Ly, R, col, row, mass, want_rows);
  return cudaGetLastError();
}

cudaError_t launch_sums(int Q, const uint16_t* in, uint32_t Lx, uint32_t Ly, unsigned long long* col,
                        unsigned long long* row, unsigned long long* mass, int want_rows, uint32_t sms, cudaStream_t s) {
  if (Q == 9) return sums_launch<9>(in, Lx, Ly, col, row, mass, want_rows, sms, s);
  if (Q == 3) return sums_launch<3>(in, Lx, Ly, col, row, mass, want_rows, sms, s);
  return sums_launch<5>(in, Lx, Ly, col, row, mass, want_rows, sms, s);
}

// --------------------------------------------------------------------------
// projections: the entries of a mode cut into chunks, one block each.  D(x) = L*S(x) - M
// in exact int64, times cos and sin of 2 pi r / L, r = (m*x) mod L; the block that finishes
// last adds the chunks' sums (the same result every time).
// Bound: the fp64 pipe: a warp's double instruction takes 64 cycles of its sub-partition,
// whatever lanes are active, so a mode is spread over as many SMs as its length feeds and
// the products are summed in 128-bit integers (FixedSums): the sine and cosine, some 70
// double instructions, are all that is left.  Against compensated double sums (DoubleSums,
// still taken where 128 bits might not do), whose trees took most of a short mode's time:
// mass and one mode of a ring of 256 nodes 27 / 35 us, of 1024^2 31 / 39, 64 modes of 16384^2
// 482 / 556, two modes of 2^22 nodes 707 / 1011; on the states tried the results are the same to the
// last bit (sines below 2^-9 have fewer than 53 bits here: see FixedSums).
// --------------------------------------------------------------------------
__device__ __forceinline__ void two_sum(double a, double b, double& s, double& e) {
  s = a + b;
  const double bb = s - a;
  e = (a - (s - bb)) + (b - bb);
}

struct Dot2 {
  double s, c;
  __device__ void add_product(double a, double b) {
    const double p = a * b;
    const double pe = fma(a, b, -p);
    double q;
    two_sum(s, p, s, q);
    c += q + pe;
  }
  __device__ void merge(double os, double oc) {
    double q;
    two_sum(s, os, s, q);
    c += oc + q;
  }
};

constexpr int kProjThreads = 64;
constexpr int kProjWarps = kProjThreads / 32;
constexpr int kProjWords = 4;  // 8-byte words of a chunk's sums

struct ProjArgs {
  const unsigned long long* colsum;
  const unsigned long long* rowsum;
  const unsigned long long* mass_in;
  uint32_t Lx, Ly;
  uint32_t nmodes;
  unsigned long long* part;  // kProjWords per chunk and mode
  unsigned int* ticket;      // per mode, 0 between launches
  double* res;               // 4 per mode (device or mapped host memory)
  unsigned long long* mass_out;
  uint32_t modes[kProjModes];  // modulo the side's length
  uint32_t along_y[kProjModes / 32];
};

// The two sums as 128-bit integers, the trigonometric values rounded to 2^-62 (those of
// 2^-9 and more are that already): exact while 2 L M 2^62 < 2^127.
struct FixedSums {
  __int128 re = 0, im = 0;
  __device__ void add(double cs, double sn, long long D) {
    re += __int128(fixed62(cs)) * D;
    im += __int128(fixed62(sn)) * D;
  }
  __device__ void pack(unsigned long long (&w)[kProjWords]) const {
    w[0] = (unsigned long long)re;
    w[1] = (unsigned long long)(re >> 64);
    w[2] = (unsigned long long)im;
    w[3] = (unsigned long long)(im >> 64);
  }
  __device__ void merge(const unsigned long long (&w)[kProjWords]) {
    re += (__int128(static_cast<long long>(w[1])) << 64) + w[0];
    im += (__int128(static_cast<long long>(w[3])) << 64) + w[2];
  }
  // of a part as packed
  __device__ static double value(unsigned long long lo, unsigned long long hi) {
    return i128_to_double_2m62(I128{lo, (long long)hi});
  }
};

// The two sums compensated in double precision (Ogita, Rump & Oishi 2005: error-free
// TwoProduct by FMA, TwoSum), for any L and M.
struct DoubleSums {
  Dot2 re{0.0, 0.0}, im{0.0, 0.0};
  __device__ void add(double cs, double sn, long long D) {
    re.add_product(cs, double(D));
    im.add_product(sn, double(D));
  }
  __device__ void pack(unsigned long long (&w)[kProjWords]) const {
    w[0] = (unsigned long long)__double_as_longlong(re.s);
    w[1] = (unsigned long long)__double_as_longlong(re.c);
    w[2] = (unsigned long long)__double_as_longlong(im.s);
    w[3] = (unsigned long long)__double_as_longlong(im.c);
  }
  __device__ void merge(const unsigned long long (&w)[kProjWords]) {
    re.merge(__longlong_as_double((long long)w[0]), __longlong_as_double((long long)w[1]));
    im.merge(__longlong_as_double((long long)w[2]), __longlong_as_double((long long)w[3]));
  }
  __device__ static double value(unsigned long long s, unsigned long long c) {
    return __longlong_as_double((long long)s) + __longlong_as_double((long long)c);
  }
};

// fixed tree over the block's threads: warp shuffles, then the warps' sums (in thread 0)
template <class Sums>
__device__ __forceinline__ void block_sums(Sums& v, unsigned long long (*sw)[kProjWords]) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  unsigned long long w[kProjWords];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    v.pack(w);
#pragma unroll
    for (int i = 0; i < kProjWords; ++i) w[i] = __shfl_down_sync(0xFFFFFFFFu, w[i], o);
    v.merge(w);
  }
  v.pack(w);
  __syncthreads();
  if (lane == 0) {
#pragma unroll
    for (int i = 0; i < kProjWords; ++i) sw[warp][i] = w[i];
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int k = 1; k < kProjWarps; ++k) {
#pragma unroll
      for (int i = 0; i < kProjWords; ++i) w[i] = sw[k][i];
      v.merge(w);
    }
  }
}

// Cosine and sine of 2 pi m x / L.
__device__ __forceinline__ void mode_at(uint32_t L, uint32_t m, uint64_t x, double& cs, double& sn) {
  // (m, x < L)
  const uint32_t r = L <= 65536u ? (m * uint32_t(x)) % L : uint32_t((uint64_t(m) * x) % L);
  sincospi(2.0 * double(r) / double(L), &sn, &cs);
}

// One warp: a mode's results from its sums (in lane 0).  Lane 0 takes the real part, lane 1 the
// imaginary one: two divisions one after the other, not four.
template <class Sums>
__device__ __forceinline__ void write_mode(const ProjArgs& a, uint32_t mi, uint32_t L, const Sums& v) {
  unsigned long long w[kProjWords];
  v.pack(w);
#pragma unroll
  for (int i = 0; i < kProjWords; ++i) w[i] = __shfl_sync(0xFFFFFFFFu, w[i], 0);
  const bool first = threadIdx.x == 0;
  const double q = Sums::value(first ? w[0] : w[2], first ? w[1] : w[3]) / double(L);
  const double re = __shfl_sync(0xFFFFFFFFu, q, 0), im = __shfl_sync(0xFFFFFFFFu, q, 1);
  const double K = double(a.Lx) * double(a.Ly);
  const double p = (first ? re * re + im * im : im) / (first ? K : K / 2.0);
  if (threadIdx.x < 2) {
    a.res[4 * mi + threadIdx.x] = q;
    a.res[4 * mi + 3 - threadIdx.x] = p;  // S(k), amplitude
  }
}

// cs, sn: the first entry's of this thread
template <class Sums>
__device__ __forceinline__ void project_chunk(const ProjArgs& a, const unsigned long long* S, uint32_t L, uint32_t m,
                                              long long M, double cs, double sn, unsigned long long (*sw)[kProjWords],
                                              bool* last) {
  const uint32_t mi = blockIdx.y, P = gridDim.x;
  const uint32_t x0 = uint32_t(uint64_t(L) * blockIdx.x / P), x1 = uint32_t(uint64_t(L) * (blockIdx.x + 1) / P);
  Sums v;
  for (uint64_t x = uint64_t(x0) + threadIdx.x; x < x1;) {
    v.add(cs, sn, static_cast<long long>(L) * static_cast<long long>(S[x]) - M);
    x += kProjThreads;
    if (x < x1) mode_at(L, m, x, cs, sn);
  }
  block_sums(v, sw);
  if (P > 1) {
    volatile unsigned long long* const part = a.part + size_t(mi) * P * kProjWords;
    unsigned long long w[kProjWords];
    if (threadIdx.x == 0) {
      v.pack(w);
#pragma unroll
      for (int i = 0; i < kProjWords; ++i) part[size_t(kProjWords) * blockIdx.x + i] = w[i];
      __threadfence();
      *last = atomicAdd(a.ticket + mi, 1u) == P - 1;
    }
    __syncthreads();
    if (!*last) return;
    __threadfence();
    v = Sums{};
    for (uint32_t k = threadIdx.x; k < P; k += kProjThreads) {
#pragma unroll
      for (int i = 0; i < kProjWords; ++i) w[i] = part[size_t(kProjWords) * k + i];
      v.merge(w);
    }
    block_sums(v, sw);
  }
  if (threadIdx.x < 32) {
    write_mode(a, mi, L, v);
    if (threadIdx.x == 0) {
      if (P > 1) a.ticket[mi] = 0;
      if (mi == 0) *a.mass_out = static_cast<unsigned long long>(M);
    }
  }
}

__global__ void __launch_bounds__(kProjThreads) project_kernel(const __grid_constant__ ProjArgs a) {
  __shared__ unsigned long long sw[kProjWarps][kProjWords];
  __shared__ bool last;
  const bool along_x = !((a.along_y[blockIdx.y / 32] >> (blockIdx.y % 32)) & 1u);
  const unsigned long long* S = along_x ? a.colsum : a.rowsum;
  const uint32_t L = along_x ? a.Lx : a.Ly, m = a.modes[blockIdx.y];
  double cs, sn;
  mode_at(L, m, min(uint64_t(L) * blockIdx.x / gridDim.x + threadIdx.x, uint64_t(L) - 1), cs, sn);
  // (launched while the sums' kernel runs: from here on what it wrote is there)
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const long long M = static_cast<long long>(*a.mass_in);
  // sum |D| <= 2 L M
  if (__umul64hi(L, (unsigned long long)M) == 0) project_chunk<FixedSums>(a, S, L, m, M, cs, sn, sw, &last);
  else project_chunk<DoubleSums>(a, S, L, m, M, cs, sn, sw, &last);
}

// A launch's modes, modulo their sides' lengths; returns the longest side among them.
static uint32_t set_modes(ProjArgs& a, const int32_t* modes) {
  std::memset(a.along_y, 0, sizeof a.along_y);
  uint32_t L = 0;
  for (uint32_t j = 0; j < a.nmodes; ++j) {
    const int32_t mx = modes[2 * j], my = modes[2 * j + 1];
    const int64_t side = my == 0 ? a.Lx : a.Ly, m = my == 0 ? mx : my;
    a.modes[j] = uint32_t((m % side + side) % side);
    if (my != 0) a.along_y[j / 32] |= 1u << (j % 32);
    L = std::max(L, uint32_t(side));
  }
  return L;
}

// --------------------------------------------------------------------------
// a small lattice's mass and projections in one launch: a cluster of eight blocks per mode, each
// with an eighth of the mode's side.  A block adds its nodes up in shared memory while its first
// sines are made; with D(x) = L N(x) - M, the sums of c D are L S - M C (S = sum c N, C = sum c,
// exact as the other form's), so the mass has to be known only in the end.
// Bound: latency (a launch, the sines' double precision, a reduction, two divisions): a call
// takes 23.0 us for 256 nodes where the two launches took 24.8 to 25.6.
// --------------------------------------------------------------------------
constexpr uint32_t kSmallProjBlocks = 8, kSmallProjThreads = 256, kSmallProjNodes = 16384, kSmallProjModes = 32;
constexpr uint32_t kSmallProjSide = kSmallProjBlocks * kSmallProjThreads;  // at most one entry per thread

struct SmallSums {
  unsigned long long w[9];  // S, C (real, imaginary: low, high word each), mass
  __device__ void add(const SmallSums& o) {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const unsigned __int128 v = ((unsigned __int128)w[2 * k + 1] << 64 | w[2 * k]) +
                                  ((unsigned __int128)o.w[2 * k + 1] << 64 | o.w[2 * k]);
      w[2 * k] = (unsigned long long)v;
      w[2 * k + 1] = (unsigned long long)(v >> 64);
    }
    w[8] += o.w[8];
  }
  __device__ void warp_sum() {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      SmallSums other;
#pragma unroll
      for (int i = 0; i < 9; ++i) other.w[i] = __shfl_down_sync(0xFFFFFFFFu, w[i], o);
      add(other);
    }
  }
  __device__ __int128 value(int k) const { return (__int128)((unsigned __int128)w[2 * k + 1] << 64 | w[2 * k]); }
};

template <int Q>
__global__ void __launch_bounds__(kSmallProjThreads) small_project_kernel(const __grid_constant__ ProjArgs a,
                                                                          const uint16_t* __restrict__ state) {
  constexpr uint32_t kWarps = kSmallProjThreads / 32;
  __shared__ uint32_t count[kSmallProjThreads];  // (at most 2048 nodes of a column: below 2^32)
  __shared__ SmallSums parts[kSmallProjBlocks * kWarps];              // the first block's: all warps' sums
  const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5, mi = blockIdx.y, rank = blockIdx.x;
  cluster_arrive();
  const bool along_x = !((a.along_y[mi / 32] >> (mi % 32)) & 1u);
  const uint32_t L = along_x ? a.Lx : a.Ly, m = a.modes[mi], nodes = a.Lx * a.Ly;
  const uint32_t x0 = L * rank / kSmallProjBlocks, n = L * (rank + 1) / kSmallProjBlocks - x0;
  count[tid] = 0;
  // an entry's sine is made by the last threads first: other warps load meanwhile (23.0 / 23.9 us)
  const uint32_t e0 = kSmallProjThreads - 1 - tid;
  __syncthreads();
  double cs = 0.0, sn = 0.0;
  if (e0 < n) mode_at(L, m, x0 + e0, cs, sn);
  const uint32_t items = along_x ? n * a.Ly : n * a.Lx;
  for (uint32_t j = tid; j < items; j += kSmallProjThreads) {
    const uint32_t row = j / (along_x ? n : a.Lx), at = j - row * (along_x ? n : a.Lx);
    const uint32_t node = along_x ? row * a.Lx + x0 + at : x0 * a.Lx + j;
    uint32_t v = 0;
#pragma unroll
    for (int i = 0; i < Q; ++i) v += __ldcg(state + size_t(i) * nodes + node);
    atomicAdd(&count[along_x ? at : row], v);
  }
  __syncthreads();
  SmallSums v{};
  const uint32_t N = e0 < n ? count[e0] : 0;
  const long long c = fixed62(cs), sine = fixed62(sn);
  v.w[8] = N;
  const __int128 sums[4] = {__int128(c) * N, __int128(sine) * N, c, sine};
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    v.w[2 * k] = (unsigned long long)sums[k];
    v.w[2 * k + 1] = (unsigned long long)(sums[k] >> 64);
  }
  v.warp_sum();
  cluster_wait();  // the first block has started
  {
    uint32_t at;
    asm("mapa.shared::cluster.u32 %0, %1, 0;\n" : "=r"(at) : "r"(uint32_t(__cvta_generic_to_shared(&parts[rank * kWarps + warp]))));
    if (lane == 0)
#pragma unroll
      for (int i = 0; i < 9; ++i) asm volatile("st.shared::cluster.u64 [%0], %1;\n" ::"r"(at + 8 * i), "l"(v.w[i]) : "memory");
  }
  __syncwarp();
  cluster_arrive();
  cluster_wait();
  if (rank != 0 || warp != 0) return;
  v = parts[lane];
  for (uint32_t k = lane + 32; k < kSmallProjBlocks * kWarps; k += 32) v.add(parts[k]);
  v.warp_sum();
  const __int128 M = (__int128)v.w[8];
  FixedSums r;
  r.re = v.value(0) * L - v.value(2) * M;
  r.im = v.value(1) * L - v.value(3) * M;
  write_mode(a, mi, L, r);
  if (lane == 0 && mi == 0) *a.mass_out = v.w[8];
}

// (us per call, one launch / two: 256 nodes and one mode 23.0 / 24.8, 96 x 40 23.2 / 26.1, 128^2
// 24.2 / 26.0, 16 modes 27.1 / 28.9, 60 35.5 / 35.6, 200 67 / 57; a side of 2000 25.2 / 28.0, of
// 4096 28.4 / 27.4, of 5400 31.0 / 28.3)
bool takes_small_project(uint32_t Lx, uint32_t Ly, uint32_t nmodes) {
  return std::max(Lx, Ly) <= kSmallProjSide && uint64_t(Lx) * Ly <= kSmallProjNodes && nmodes <= kSmallProjModes;
}

cudaError_t launch_small_project(int Q, const uint16_t* state, uint32_t Lx, uint32_t Ly, const int32_t* modes,
                                 uint32_t nmodes, double* res, unsigned long long* mass, cudaStream_t s) {
  ProjArgs a{};
  a.Lx = Lx;
  a.Ly = Ly;
  a.mass_out = mass;
  const void* fn = Q == 3   ? reinterpret_cast<const void*>(small_project_kernel<3>)
                   : Q == 5 ? reinterpret_cast<const void*>(small_project_kernel<5>)
                            : reinterpret_cast<const void*>(small_project_kernel<9>);
  a.nmodes = nmodes;
  a.res = res;
  set_modes(a, modes);
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeClusterDimension;
  attr.val.clusterDim.x = kSmallProjBlocks;
  attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(kSmallProjBlocks, nmodes);
  cfg.blockDim = dim3(kSmallProjThreads);
  cfg.stream = s;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  void* p[] = {&a, &state};
  return cudaLaunchKernelExC(&cfg, fn, p);
}

cudaError_t launch_project(const ProjWork& w, uint32_t Lx, uint32_t Ly, const int32_t* modes, uint32_t nmodes,
                           double* res, unsigned long long* mass, cudaStream_t s) {
  ProjArgs a{};
  a.colsum = w.col;
  a.rowsum = w.row;
  a.mass_in = w.mass;
  a.Lx = Lx;
  a.Ly = Ly;
  a.part = w.scratch;
  a.ticket = reinterpret_cast<unsigned int*>(w.scratch + 4 * (kProjBlocks + kProjModes));
  a.mass_out = mass;
  for (uint32_t k = 0; k < nmodes; k += kProjModes) {
    a.nmodes = std::min(nmodes - k, kProjModes);
    a.res = res + size_t(4) * k;
    const uint32_t L = set_modes(a, modes + 2 * size_t(k));
    const uint32_t P = uint32_t(std::min<uint64_t>(std::max<uint32_t>(1, kProjBlocks / a.nmodes),
                                                   (uint64_t(L) + kProjThreads - 1) / kProjThreads));
    // the first launch begins, and makes its first sines and cosines, while the sums' kernel runs
    // (us per call of the observables: 1024^2 33.6 -> 28.7, 256 nodes 27.6 -> 25.6)
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr = {};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cfg.gridDim = dim3(P, a.nmodes);
    cfg.blockDim = dim3(kProjThreads);
    cfg.stream = s;
    cfg.attrs = &attr;
    cfg.numAttrs = k == 0 ? 1 : 0;
    if (const cudaError_t e = cudaLaunchKernelEx(&cfg, project_kernel, a); e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

// --------------------------------------------------------------------------
// Philox probe
// --------------------------------------------------------------------------
__global__ void philox_kernel(const uint4* __restrict__ ctr, uint32_t k0, uint32_t k1, uint4* __restrict__ out,
                              size_t n) {
  for (size_t i = blockIdx.x * size_t(blockDim.x) + threadIdx.x; i < n; i += size_t(gridDim.x) * blockDim.x)
    out[i] = philox(ctr[i], k0, k1);
}

cudaError_t launch_philox(const uint32_t* ctr, uint32_t k0, uint32_t k1, uint32_t* out, size_t n,
                          cudaStream_t s) {
  const int grid = int(n < 65536 * 256 ? (n + 255) / 256 : 65536);
  philox_kernel<<<grid > 0 ? grid : 1, 256, 0, s>>>(reinterpret_cast<const uint4*>(ctr), k0, k1,
                                                     reinterpret_cast<uint4*>(out), n);
  return cudaGetLastError();
}

}  // namespace ilg
