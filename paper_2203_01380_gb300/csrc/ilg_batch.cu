// Batched D1Q3 replicas: one persistent launch advances every ring of a batch by T
// steps.  Blocks pull replicas from a queue ordered by decreasing ring length
// (longest processing time first); a block copies its replica's ring and alias
// tables into shared memory, runs all T steps there (flip, collision, streaming,
// two buffers, one barrier per step) and writes the ring back.  Random numbers are
// keyed by the replica's own id, so a replica's result does not depend on which
// block ran it or on the other replicas of the batch.
#include <cuda_runtime.h>

#include <algorithm>
#include <functional>
#include <type_traits>

#include "ilg_batch.h"
#include "ilg_collide.cuh"
#include "ilg_device.cuh"
#include "ilg_fixed.cuh"
#include "ilg_sync.cuh"

namespace ilg {

namespace {

// Compensated double-precision sum (Ogita, Rump & Oishi 2005), per thread and
// merged across the block.
__device__ __forceinline__ void two_sum_b(double a, double b, double& s, double& e) {
  s = a + b;
  const double bb = s - a;
  e = (a - (s - bb)) + (b - bb);
}

template <int THREADS>
__device__ double block_dot2(double s, double c, double* red) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const double os = __shfl_down_sync(0xFFFFFFFFu, s, o);
    const double oc = __shfl_down_sync(0xFFFFFFFFu, c, o);
    double q;
    two_sum_b(s, os, s, q);
    c += oc + q;
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (lane == 0) {
    red[2 * warp] = s;
    red[2 * warp + 1] = c;
  }
  __syncthreads();
  double r = 0.0;
  if (threadIdx.x == 0) {
    double S = red[0], C = red[1];
    for (int w = 1; w < THREADS / 32; ++w) {
      double q;
      two_sum_b(S, red[2 * w], S, q);
      C += red[2 * w + 1] + q;
    }
    r = S + C;
  }
  return r;  // valid in thread 0
}

// Fixed-point (2^-62) cosine and sine of 2 pi r / L.
__device__ __forceinline__ longlong2 trig_fixed(uint32_t r, uint32_t L) {
  double sn, cs;
  sincospi(2.0 * double(r) / double(L), &sn, &cs);
  return make_longlong2(fixed62(cs), fixed62(sn));
}

// Complex amplitude of axis mode m of a ring: with D(x) = L N(x) - M and r = (m x) mod L,
//   re = sum_x cos(2 pi r / L) D(x) / L,  im = sum_x sin(2 pi r / L) D(x) / L.
// The trigonometric values enter as 2^-62 fixed-point integers and the sums are exact, so
// they do not depend on the summation order.  A step adds only
//   sum_x c(x) N(x),  c = c1 2^32 + c0:  N c0 < 3 65535 2^32 and |N c1| < 2^48 per node, below
// 2^63 over the longest ring (four wide multiply-adds per node, against two 64 x 64 -> 128
// products);
// the factor L and the M sum_x c(x) term, the same for every step, join when a state's
// sums are written out (write_sums).
static_assert((uint64_t(3 * 65535) << 32) * kBatchMaxL / kBatchMaxL == uint64_t(3 * 65535) << 32 &&
                  (uint64_t(3 * 65535) << 32) * kBatchMaxL < uint64_t(1) << 63,
              "a ring's sums of low parts");
struct ModeSums {
  long long v[4];  // cos low, cos high, sin low, sin high
  __device__ __forceinline__ void clear() { v[0] = v[1] = v[2] = v[3] = 0; }
  __device__ __forceinline__ void add(const longlong2& cs, uint32_t N) {
    v[0] += (long long)(uint64_t(uint32_t(cs.x)) * N);
    v[1] += (long long)(int32_t(cs.x >> 32)) * (long long)(int32_t(N));
    v[2] += (long long)(uint64_t(uint32_t(cs.y)) * N);
    v[3] += (long long)(int32_t(cs.y >> 32)) * (long long)(int32_t(N));
  }
  // Sums over the warp: lane 8 k returns the sum of v[k] (k = 0..3).  The first two
  // exchanges halve the values a lane keeps: 6 exchanges instead of 20.
  __device__ __forceinline__ long long warp_sum(uint32_t lane) const {
    const bool hi = (lane & 16) != 0;
    long long a = hi ? v[2] : v[0], b = hi ? v[3] : v[1];
    a += __shfl_xor_sync(kFullWarp, hi ? v[0] : v[2], 16);
    b += __shfl_xor_sync(kFullWarp, hi ? v[1] : v[3], 16);
    const bool odd = (lane & 8) != 0;
    long long c = odd ? b : a;
    c += __shfl_xor_sync(kFullWarp, odd ? a : b, 8);
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) c += __shfl_xor_sync(kFullWarp, c, o);
    return c;
  }
};

// One warp: the 128-bit sums (L 2^62 re, L 2^62 im) of `count` <= 8 states, each as two (lo,
// hi) pairs in out[4 i .. 4 i + 3], from the partial sums red(i)[4 j + k] of R warps and the
// ring's c[k] = sum_x of the parts of its trigonometric values.  Lane 4 i + k adds up part k
// of state i.
template <uint32_t R, class Red>
__device__ __forceinline__ void write_sums(const Red& red, uint32_t count, const long long* c, uint32_t L, uint64_t mass,
                                           long long* out) {
  const uint32_t lane = threadIdx.x & 31u, i = lane >> 2, k = lane & 3u;
  long long v = 0;
  if (i < count) {
#pragma unroll
    for (uint32_t j = 0; j < R; ++j) v += red(i)[4 * j + k];
  }
  const long long high = __shfl_down_sync(kFullWarp, v, 1);  // even lanes: the high part beside the low one
  if (i < count && (k & 1u) == 0) {
    const __int128 S = (__int128(high) << 32) + v;
    const __int128 C = (__int128(c[k + 1]) << 32) + c[k];
    const __int128 r = S * __int128(L) - C * __int128((long long)mass);
    out[lane] = (long long)(unsigned long long)r;
    out[lane + 1] = (long long)(r >> 64);
  }
}

// What the slot and extension blocks of one step share (StepKeys, WordKeys) without the
// words that depend on the ring alone, as two 16-byte shared loads.
struct __align__(16) BatchStepKeys {
  uint32_t G, H0, I0, J0, H1, I1, J1, ext_c;
};

// Lane j of a warp: the launch-wide words of step s0 + j (s0 a multiple of 32) of a ring
// whose step counter is t0.
__device__ __forceinline__ void make_step_keys(const StepArgs& a, uint32_t t0, uint32_t s0, BatchStepKeys (&keys)[2][32]) {
  const uint32_t j = threadIdx.x & 31u;
  const WordKeys k = word_keys(a, t0 + s0 + j);
  keys[(s0 >> 5) & 1][j] = BatchStepKeys{k.slot.G,    k.slot.H[0], k.slot.I[0], k.slot.J[0],
                                         k.slot.H[1], k.slot.I[1], k.slot.J[1], k.ext_c};
}
__device__ __forceinline__ void make_step_keys(const StepArgs& a, uint32_t t0, uint32_t s0, WordKeys (&keys)[2][32]) {
  const uint32_t j = threadIdx.x & 31u;
  keys[(s0 >> 5) & 1][j] = word_keys(a, t0 + s0 + j);
}

// The words a node is collided with: those in shared memory, or those held in registers.
__device__ __forceinline__ const volatile WordKeys& step_words(const WordKeys& shared, const WordKeys&) { return shared; }
__device__ __forceinline__ const WordKeys& step_words(const BatchStepKeys&, const WordKeys& held) { return held; }

// Rings of a block: shared memory, the block's threads and how its words are kept.  Bound:
// integer issue for long rings (see collide_warp), the latency of a step (its node's
// Philox rounds, two dependent table draws and a barrier) for short ones.  A block holds
// the alias tables in 64-bit form where one block per SM is resident (1024 threads; a
// draw takes two instructions fewer), packed where several share an SM.  Measured
// against per-lane loops and one 128-bit projection per node and step: 2048 rings of 64 to
// 8192 nodes x 2000 steps 190 ms / 249 ms; 512 rings of 320 nodes x 2000 steps with
// statistics 6.2 / 10.6 ms; one ring of 256 nodes with its records 1.0 / 2.06 us per step.
template <int THREADS>
struct BatchShape {
  static constexpr int kPerSm = 1024 / THREADS;
  static constexpr bool kPairs = THREADS == 1024;
  static constexpr uint32_t kTableWords = kPairs ? kDevStagedWords : kDevTableWords4;
  static constexpr uint32_t kRing = kBatchExtWords;
  // Warps that only record (the mode's sums, the states), beside those that collide: a
  // state's sums are taken while the next one is made, off the step's chain of waits, and
  // added up across these few warps instead of all.  Bound by the loads of the
  // trigonometric values (16 bytes per node; 131 KB for 8192 nodes come from L2), hence
  // their number: with one to three, rings of 8192 nodes at 10 per velocity took 19.7 us
  // per step.  Against colliding warps that record as well, per step: one ring of 256 nodes
  // 1.01 / 1.28 us, with its states 1.07 / 1.41; 512 rings of 320 nodes 3.51 / 3.91; 152
  // rings of 8192 nodes at 10 per velocity 10.5 / 11.6, at 100 25.6 / 25.4.
  static constexpr uint32_t kRecorders = THREADS == 1024 ? 8 : (THREADS == 512 ? 4 : 2);
  // most threads of a block: the recording warps come on top where a 256-thread block has
  // an SM to itself
  static constexpr int kMost = THREADS + (THREADS == 256 ? 64 : 0);
};

// The shared memory of a batch block beside its dynamic part.  ALONE: a 256-thread block that
// has an SM to itself (no more rings than SMs).  A step's launch-wide words are then read where
// they are used: with few warps that is off the step's chain (one ring of 64 nodes with its
// states 0.77 instead of 0.81 us per step, of 128 0.86 / 0.90); where warps keep the issue busy
// the loads cost more than the registers (512 rings of 320 nodes 6.40 / 6.20 ms, 152 rings of
// 8192 at 100 per velocity 22.8 / 21.7 us per step).
template <int THREADS, bool ALONE>
struct BatchShared {
  // states whose partial sums are written out together, and room for as many again
  static constexpr uint32_t kGroup = 8, kSlots = 2 * kGroup;
  uint32_t task;
  uint32_t fail;  // first step that would overflow
  unsigned long long mass;
  long long c[4];  // sums of the mode's trigonometric values
  long long red[kSlots][4 * BatchShape<THREADS>::kRecorders];  // partial sums of the last states
  std::conditional_t<ALONE, WordKeys, BatchStepKeys> keys[2][32];  // of 64 steps
};

// All steps of one ring that lies in src (3 planes of L; dst: the other buffer): the first
// `colliders` warps of the block collide, the recording warps (REC: the mode's sums at every
// state; STATES: every state to b.states) follow them and see a state's planes in the step
// that reads them.  TABLES: see collide_warp (and the binomial sampler).  Returns the steps
// done; src is the buffer that holds the state.
template <int THREADS, bool ALONE, bool REC, bool STATES, bool TABLES, class Tab>
__device__ __forceinline__ uint32_t run_ring(const BatchArgs& b, const StepArgs& a, const ReplicaDesc& d, uint32_t r,
                                             const uint32_t* tables, const Tab& to, const Tab& tr, unsigned char* words,
                                             BatchShared<THREADS, ALONE>& sh, uint16_t*& src, uint16_t* dst, uint32_t colliders) {
  constexpr uint32_t S = 4 * THREADS;
  constexpr uint32_t R = REC || STATES ? BatchShape<THREADS>::kRecorders : 0;
  constexpr uint32_t kGroup = BatchShared<THREADS, ALONE>::kGroup, kSlots = BatchShared<THREADS, ALONE>::kSlots;
  const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5;
  const uint32_t L = d.L, T = b.T;
  const uint64_t mass = sh.mass;
  // no occupation can pass 65535 while the whole ring holds no more than that
  const bool safe = mass <= 65535ull;
  const auto bar = [&]() { asm volatile("bar.sync 1, %0;" ::"r"((colliders + R) * 32) : "memory"); };
  // (a faster warp may already have marked the next step)
  const auto stopped = [&](uint32_t s) { return !safe && *reinterpret_cast<volatile uint32_t*>(&sh.fail) <= s; };
  // the flip F_i(n) = n_{-i}: velocity i of the collision reads plane -i
  const uint32_t p1 = d.flip ? 2 * L : L, p2 = d.flip ? L : 2 * L;
  uint32_t s = 0;
  if constexpr (R != 0) {
    if (warp >= colliders) {
      const uint32_t j = warp - colliders;
      const longlong2* trig = REC ? b.trig + d.state_off / 3 : nullptr;  // this ring's values
      const auto red = [&](uint32_t st) { return sh.red[st % kSlots]; };
      const auto write_group = [&](uint32_t s0, uint32_t count) {
        write_sums<R>([&](uint32_t i) { return red(s0 + i); }, count, sh.c, L, mass,
                      b.record + (size_t(r) * (T + 1) + s0) * 4);
      };
      for (;; ++s) {
        ModeSums ms;
        if constexpr (REC) ms.clear();
        // the state after step s - 1, planes rest, +1, -1
        uint16_t* const rs = STATES && s > 0 ? b.states + d.state_off * T + size_t(s - 1) * 3 * L : nullptr;
#pragma unroll 4
        for (uint32_t x = 32 * j + lane; x < L; x += 32 * R) {
          const uint32_t m0 = src[x], m1 = src[L + x], m2 = src[2 * L + x];
          if constexpr (REC) ms.add(trig[x], m0 + m1 + m2);
          if constexpr (STATES) {
            if (s > 0) {
              rs[x] = uint16_t(m0);
              rs[L + x] = uint16_t(m1);
              rs[2 * L + x] = uint16_t(m2);
            }
          }
        }
        if constexpr (REC) {
          const long long v = ms.warp_sum(lane);
          if ((lane & 7) == 0) red(s)[4 * j + (lane >> 3)] = v;
        }
        if (s == T) break;
        bar();
        if (stopped(s)) break;  // src still holds the state
        uint16_t* tmp = src;
        src = dst;
        dst = tmp;
        if (REC && (s % kGroup) == kGroup - 1 && j == 0) write_group(s - (kGroup - 1), kGroup);
      }
      bar();
      if constexpr (REC) {
        // the states since the last group (s: the last state whose sums exist)
        if (j == 0) write_group(s / kGroup * kGroup, s % kGroup + 1);
      }
      return s;
    }
  }
  WordKeys held;
  held.slot.A = uint32_t((uint64_t(0xCD9E8D57u) * a.replica) >> 32) ^ a.rk[0];
  held.ext_e = uint32_t(uint64_t(0xCD9E8D57u) * a.replica) ^ a.rk[2];
  for (; s < T; ++s) {
    if constexpr (!ALONE) {
      const uint4* q = reinterpret_cast<const uint4*>(&sh.keys[(s >> 5) & 1][s & 31]);
      const uint4 k0 = q[0], k1 = q[1];
      held.slot.G = k0.x;
      held.slot.H[0] = k0.y;
      held.slot.I[0] = k0.z;
      held.slot.J[0] = k0.w;
      held.slot.H[1] = k1.x;
      held.slot.I[1] = k1.y;
      held.slot.J[1] = k1.z;
      held.ext_c = k1.w;
    }
    const auto& k = step_words(sh.keys[(s >> 5) & 1][s & 31], held);
    bool bad = false;
    for (uint32_t x0 = warp * 32; x0 < L; x0 += colliders * 32) {
      const uint32_t x = x0 + lane;
      const bool active = x < L;
      uint32_t m[3], post[3];
      m[0] = active ? src[x] : 0u;
      m[1] = active ? src[p1 + x] : 0u;
      m[2] = active ? src[p2 + x] : 0u;
      if (!TABLES && a.particle) collide_particle<3>(a, tables, x, d.t + s, m, post);
      else collide_warp<3, S, BatchShape<THREADS>::kRing, TABLES>(a, k, to, tr, tr, words, 4 * tid, x, m, post);
      if (active) {
        bad |= (post[0] | post[1] | post[2]) > 65535u;
        dst[x] = uint16_t(post[0]);
        dst[L + (x + 1 == L ? 0 : x + 1)] = uint16_t(post[1]);
        dst[2 * L + (x == 0 ? L - 1 : x - 1)] = uint16_t(post[2]);
      }
    }
    if (bad) atomicMin(&sh.fail, s);
    bar();
    if (stopped(s)) break;  // src still holds the state
    // the steps' launch-wide Philox words, over those of the 32 steps just done
    if (warp == 0 && (s & 31) == 31) make_step_keys(a, d.t, s + 33, sh.keys);
    uint16_t* tmp = src;
    src = dst;
    dst = tmp;
  }
  bar();
  return s;
}

template <int THREADS, bool REC, bool STATES, bool ALONE = false>
__global__ void __launch_bounds__(REC || STATES ? BatchShape<THREADS>::kMost : THREADS,
                                  REC || STATES ? 65536 / (64 * BatchShape<THREADS>::kMost) : BatchShape<THREADS>::kPerSm)
    batch_d1q3_kernel(const __grid_constant__ BatchArgs b, const __grid_constant__ StepArgs common) {
  using Shape = BatchShape<THREADS>;
  using Tab = std::conditional_t<Shape::kPairs, Alias8, Alias4>;
  extern __shared__ uint4 smem4[];
  uint32_t* tables = reinterpret_cast<uint32_t*>(smem4);
  unsigned char* const words = reinterpret_cast<unsigned char*>(tables + Shape::kTableWords);
  uint16_t* ring = reinterpret_cast<uint16_t*>(words + Shape::kRing * 4 * THREADS);  // 2 x 3 x Lmax
  __shared__ BatchShared<THREADS, ALONE> sh;
  const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5;
  const uint32_t threads = blockDim.x;

  for (;;) {
    if (tid == 0) {
      sh.task = atomicAdd(b.counter, 1u);
      sh.fail = ~0u;
      sh.mass = 0ull;
      sh.c[0] = sh.c[1] = sh.c[2] = sh.c[3] = 0;
    }
    __syncthreads();
    const uint32_t task = sh.task;
    if (task >= b.n) break;
    const uint32_t r = b.order[task];
    const ReplicaDesc d = b.desc[r];
    const uint32_t L = d.L;
    StepArgs a = common;
    a.omega_mode = d.omega_mode;
    a.rest_mode = d.rest_mode;
    a.replica = d.replica;
    a.particle = d.particle;

    // tables (the particle sampler's boundaries as they are) and ring into shared memory
    if constexpr (Shape::kPairs) {
      const uint4* g4 = reinterpret_cast<const uint4*>(b.tables + size_t(r) * kDevBlockWords);
#pragma unroll 8
      for (uint32_t i = tid; i < kDevStagedWords / 4; i += threads) smem4[i] = g4[i];
    } else {
      stage_tables4(b.tables + size_t(r) * kDevBlockWords, tables, a.particle != 0);
    }
    const Tab to = Tab::of(tables, 0), tr = Tab::of(tables, 1);
    uint16_t* const gs = b.state + d.state_off;
    unsigned long long part = 0;
    for (uint32_t i = tid; i < 3 * L; i += threads) {
      ring[i] = gs[i];
      part += gs[i];
    }
    // the ring's mass, and the sums of the recorded mode's trigonometric values
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) part += __shfl_down_sync(kFullWarp, part, o);
    if (lane == 0 && part) atomicAdd(&sh.mass, part);
    if constexpr (REC) {
      const longlong2* trig = b.trig + d.state_off / 3;
      ModeSums ms;
      ms.clear();
      for (uint32_t x0 = warp * 32; x0 < L; x0 += threads)
        if (x0 + lane < L) ms.add(trig[x0 + lane], 1u);
      const long long v = ms.warp_sum(lane);
      if ((lane & 7) == 0) atomicAdd(reinterpret_cast<unsigned long long*>(&sh.c[lane >> 3]), (unsigned long long)v);
    }
    if (warp == 0) {
      make_step_keys(a, d.t, 0, sh.keys);
      make_step_keys(a, d.t, 32, sh.keys);
    }
    __syncthreads();
    // the ring's colliding warps, and those that record it; the others have nothing to do
    constexpr uint32_t R = REC || STATES ? Shape::kRecorders : 0;
    const uint32_t colliders = min((L + 31) >> 5, threads / 32 - R);
    if (warp < colliders + R) {
      uint16_t* src = ring;
      const bool plain = !a.particle && a.omega_mode == kTable && a.rest_mode == kTable;
      const uint32_t done =
          plain ? run_ring<THREADS, ALONE, REC, STATES, true>(b, a, d, r, tables, to, tr, words, sh, src, ring + 3 * L, colliders)
                : run_ring<THREADS, ALONE, REC, STATES, false>(b, a, d, r, tables, to, tr, words, sh, src, ring + 3 * L, colliders);
      // ring back to global memory; the replica's step counter moves on
      for (uint32_t i = tid; i < 3 * L; i += (colliders + R) * 32) gs[i] = src[i];
      if (tid == 0) {
        b.desc[r].t = d.t + done;
        if (sh.fail != ~0u) b.failed[r] = 1u;
      }
    }
    __syncthreads();
  }
}

// --- a ring split between the blocks of a cluster ----------------------------
//
// Where a ring per block would leave SMs idle (few rings, or rings of unlike length), a ring's
// nodes are split between the blocks of a cluster, one block per SM.  A block keeps its own
// nodes and a halo of 8 to 23 nodes on both sides, which it advances as well (a node's random
// words depend on the node and the step alone); with every step the outermost nodes of the halo
// lapse, and when it is used up the neighbours' nodes come through the cluster's shared memory.
// So the blocks meet once in 8 to 23 steps and not in each: occupations sent to the neighbour in
// every step, as words with the step's tag, cost 0.4 us per step (rings of 64 nodes 1.09 us per
// step instead of 0.69).
// Bound as before by integer issue for long shares and a node's chain of draws for short
// ones.  Us per step, one block per ring / split: one ring of 8192 nodes at 50 per velocity
// 15.1 / 1.75, 18 rings of up to 8192 15.1 / 2.5, 38 of 4000 6.2 / 2.9, 76 of 1000 1.9 / 1.4;
// with statistics 12 rings of 1000 2.58 / 1.11, 70 of 320 1.03 / 0.91; one ring of 256 with
// its states 1.01 / 0.88.  Rings below 256 nodes gain nothing (128: 0.90 / 0.92, 64: 0.81 /
// 0.89) and stay in one block.

constexpr uint32_t kSplitFrom = 256;  // nodes of the batch's longest ring
constexpr uint32_t kMostHalo = 24;

struct ShareShared {
  uint32_t fail;  // first step that would overflow
  unsigned long long mass;
  long long c[4];                        // sums of the mode's trigonometric values
  // nodes that came from the left, from the right neighbour, by the exchange's parity: a
  // neighbour writes one again after the next exchange, which all reach behind their reading
  uint16_t mail[2][2][3 * kMostHalo];
  WordKeys keys[2][32];
};

__device__ __forceinline__ uint32_t mapa(const void* p, uint32_t rank) {
  uint32_t at;
  asm("mapa.shared::cluster.u32 %0, %1, %2;\n" : "=r"(at) : "r"(uint32_t(__cvta_generic_to_shared(p))), "r"(rank));
  return at;
}

// A block's part of a ring: its own nodes lo .. lo + n - 1 and `halo` nodes on both sides,
// local nodes 0 .. n + 2 halo - 1 of planes of `stride` nodes.
struct Share {
  uint32_t lo, n, halo, stride;
  uint32_t left, right;  // the neighbours' ranks
};

// The neighbours' nodes beside the block's own.
// (threads: those that work on the share; none in a block without nodes)
__device__ __forceinline__ void exchange(const Share& h, uint16_t* src, ShareShared& sh, uint32_t parity, uint32_t threads) {
  const uint32_t H = h.halo, items = threadIdx.x < threads ? 6 * H : 0;
  for (uint32_t j = threadIdx.x; j < items; j += threads) {
    const uint32_t side = j >= 3 * H, q = j - side * 3 * H, v = q / H, c = q - v * H;  // first nodes left, last right
    const uint32_t at = mapa(&sh.mail[parity][side ^ 1][q], side ? h.right : h.left);
    asm volatile("st.shared::cluster.u16 [%0], %1;\n" ::"r"(at), "h"(src[v * h.stride + c + (side ? h.n : H)]) : "memory");
  }
  cluster_arrive();
  cluster_wait();
  for (uint32_t j = threadIdx.x; j < items; j += threads) {
    const uint32_t side = j >= 3 * H, q = j - side * 3 * H, v = q / H, c = q - v * H;
    src[v * h.stride + c + (side ? H + h.n : 0)] = sh.mail[parity][side][q];
  }
  __syncthreads();
}

// T steps of a share (see run_ring); src holds the state of its own nodes afterwards.  A
// step that would overflow is marked and the share goes on with occupations cut to 16 bits:
// the ring's blocks then start again and stop before that step.  The recording warps add
// their sums of a state to the record in memory (parts as in ModeSums; zero at the start).
template <bool REC, bool STATES, bool TABLES, class Tab>
__device__ __forceinline__ void run_share(const BatchArgs& b, const StepArgs& a, const ReplicaDesc& d, uint32_t r,
                                          const Share& h, uint32_t T, const uint32_t* tables, const Tab& to, const Tab& tr,
                                          unsigned char* words, ShareShared& sh, uint16_t*& src, uint16_t* dst,
                                          uint32_t colliders, uint32_t recorders) {
  constexpr uint32_t S = 4 * 1024;
  const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5;
  const uint32_t H = h.halo, n = h.n, P = h.stride, N = n + 2 * H, L = d.L;
  const auto bar = [&]() { asm volatile("bar.sync 1, %0;" ::"r"((colliders + recorders) * 32) : "memory"); };
  uint32_t s = 0, since = 0, parity = 0;  // steps since the last exchange
  const auto meet = [&]() {
    if (since == H && H) {
      exchange(h, src, sh, parity, (colliders + recorders) * 32);
      parity ^= 1;
      since = 0;
    }
  };
  const auto turn = [&]() {
    uint16_t* tmp = src;
    src = dst;
    dst = tmp;
    since += 1;
  };
  if (warp >= colliders + recorders) {
    // nothing to do but the exchanges
    for (; s < T; ++s) {
      meet();
      turn();
    }
    return;
  }
  if constexpr (REC || STATES) {
    if (warp >= colliders) {
      const longlong2* trig = REC ? b.trig + d.state_off / 3 + h.lo : nullptr;
      unsigned long long* const rec =
          REC ? reinterpret_cast<unsigned long long*>(b.record) + size_t(r) * (size_t(b.T) + 1) * 4 : nullptr;
      for (;; ++s) {
        if (s < T) meet();
        ModeSums ms;
        if constexpr (REC) ms.clear();
        uint16_t* const rs = STATES && s > 0 ? b.states + d.state_off * b.T + size_t(s - 1) * 3 * L + h.lo : nullptr;
#pragma unroll 4
        for (uint32_t i = 32 * (warp - colliders) + lane; i < n; i += 32 * recorders) {
          const uint32_t m0 = src[H + i], m1 = src[P + H + i], m2 = src[2 * P + H + i];
          if constexpr (REC) ms.add(trig[i], m0 + m1 + m2);
          if constexpr (STATES) {
            if (s > 0) {
              rs[i] = uint16_t(m0);
              rs[L + i] = uint16_t(m1);
              rs[2 * L + i] = uint16_t(m2);
            }
          }
        }
        if constexpr (REC) {
          const long long v = ms.warp_sum(lane);
          if ((lane & 7) == 0) atomicAdd(rec + 4 * size_t(s) + (lane >> 3), (unsigned long long)v);
        }
        if (s == T) return;
        bar();
        turn();
      }
    }
  }
  // the flip F_i(n) = n_{-i}: velocity i of the collision reads plane -i
  const uint32_t p1 = d.flip ? 2 * P : P, p2 = d.flip ? P : 2 * P;
  const uint32_t past = H ? P - 1 : 0, before = H ? P - 1 : N - 1;  // a spare node, or the ring's other end
  for (; s < T; ++s) {
    meet();
    // (read where they are used: 0.93 instead of 0.98 us per step for 5 rings of 3000; in run_ring,
    // whose shares keep the issue busy, 22.8 instead of 21.7 for 152 rings of 8192)
    const volatile WordKeys& k = sh.keys[(s >> 5) & 1][s & 31];
    bool bad = false;
    // without the `since` outermost nodes, whose neighbours' particles have not come
    const uint32_t valid = H ? N - 2 * since : N;
    for (uint32_t i0 = warp * 32; i0 < N; i0 += colliders * 32) {
      const uint32_t i = i0 + lane;
      const bool active = i - (H ? since : 0u) < valid;
      uint32_t x = h.lo + i + (i < H && h.lo + i < H ? L : 0) - H;  // modulo L
      x -= x >= L ? L : 0;
      uint32_t m[3], post[3];
      m[0] = active ? src[i] : 0u;
      m[1] = active ? src[p1 + i] : 0u;
      m[2] = active ? src[p2 + i] : 0u;
      if (!TABLES && a.particle) collide_particle<3>(a, tables, x, d.t + s, m, post);
      else collide_warp<3, S, kBatchExtWords, TABLES>(a, k, to, tr, tr, words, 4 * tid, x, m, post);
      if (active) {
        bad |= (post[0] | post[1] | post[2]) > 65535u && i - H < n;
        dst[i] = uint16_t(post[0]);
        dst[P + (i + 1 == N ? past : i + 1)] = uint16_t(post[1]);
        dst[2 * P + (i == 0 ? before : i - 1)] = uint16_t(post[2]);
      }
    }
    if (bad) atomicMin(&sh.fail, s);
    bar();
    if (warp == 0 && (s & 31) == 31) make_step_keys(a, d.t, s + 33, sh.keys);
    turn();
  }
}

// How a ring of L nodes lies in a cluster: parts of at least 32 nodes, and as many nodes
// beside them as fill the last warp (8 to 23).  One part: no halo.
struct RingSplit {
  uint32_t parts, most, halo, tiles;
};
__host__ __device__ constexpr RingSplit ring_split(uint32_t L, uint32_t blocks) {
  RingSplit q{L / 32 < blocks ? L / 32 : blocks, 0, 0, 0};
  if (q.parts < 2) q.parts = 1;
  q.most = (L + q.parts - 1) / q.parts;
  q.tiles = (q.most + (q.parts > 1 ? 16 : 0) + 31) / 32;
  q.halo = q.parts > 1 ? (32 * q.tiles - q.most) / 2 : 0;
  return q;
}

// One ring by `blocks` blocks of a cluster, of which this is number `rank`; ALONE: by one block
// where blocks = 1.
template <bool REC, bool STATES, bool ALONE>
__device__ __forceinline__ void run_split(const BatchArgs& b, const StepArgs& common, uint32_t r, uint32_t blocks,
                                          uint32_t rank, uint32_t recorders, uint4* smem4, ShareShared& sh) {
  uint32_t* tables = reinterpret_cast<uint32_t*>(smem4);
  unsigned char* const words = reinterpret_cast<unsigned char*>(tables + kDevStagedWords);
  uint16_t* const ring = reinterpret_cast<uint16_t*>(words + kBatchExtWords * 4 * 1024);  // 2 x 3 x stride
  const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5, threads = blockDim.x;
  const auto meet = [&] {
    if (ALONE && blocks == 1) {
      __syncthreads();
    } else {
      cluster_arrive();
      cluster_wait();
    }
  };
  const ReplicaDesc d = b.desc[r];
  const uint32_t L = d.L;
  StepArgs a = common;
  a.omega_mode = d.omega_mode;
  a.rest_mode = d.rest_mode;
  a.replica = d.replica;
  a.particle = d.particle;
  const RingSplit q = ring_split(L, blocks);
  Share h;
  h.halo = q.halo;
  h.stride = q.most + 2 * q.halo + 1;
  h.lo = min(rank, q.parts) * L / q.parts;
  h.n = min(rank + 1, q.parts) * L / q.parts - h.lo;
  h.right = rank + 1 >= q.parts ? 0 : rank + 1;
  h.left = rank == 0 ? q.parts - 1 : rank - 1;
  const uint32_t N = h.n ? h.n + 2 * h.halo : 0;
  if (tid == 0) {
    sh.mass = 0ull;
    sh.c[0] = sh.c[1] = sh.c[2] = sh.c[3] = 0;
  }
  {
    const uint4* g4 = reinterpret_cast<const uint4*>(b.tables + size_t(r) * kDevBlockWords);
#pragma unroll 8
    for (uint32_t i = tid; i < kDevStagedWords / 4; i += threads) smem4[i] = g4[i];
  }
  uint16_t* const gs = b.state + d.state_off;
  unsigned long long* const rec =
      REC ? reinterpret_cast<unsigned long long*>(b.record) + size_t(r) * (size_t(b.T) + 1) * 4 : nullptr;
  __syncthreads();
  if constexpr (REC) {
    // the whole ring's mass and the sums of the mode's values
    const longlong2* trig = b.trig + d.state_off / 3;
    unsigned long long part = 0;
    ModeSums ms;
    ms.clear();
    for (uint32_t x = tid; x < L; x += threads) {
      part += uint32_t(gs[x]) + gs[L + x] + gs[2 * L + x];
      ms.add(trig[x], 1u);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) part += __shfl_down_sync(kFullWarp, part, o);
    if (lane == 0 && part) atomicAdd(&sh.mass, part);
    const long long v = ms.warp_sum(lane);
    if ((lane & 7) == 0) atomicAdd(reinterpret_cast<unsigned long long*>(&sh.c[lane >> 3]), (unsigned long long)v);
  }
  const Alias8 to = Alias8::of(tables, 0), tr = Alias8::of(tables, 1);
  const uint32_t colliders = min((N + 31) >> 5, threads / 32 - recorders);
  uint32_t T = b.T;
  uint16_t* src;
  bool over = false;
  for (;;) {
    src = ring;
    for (uint32_t i = tid; i < N; i += threads) {
      const uint32_t x = (h.lo + i + L - h.halo) % L;
#pragma unroll
      for (uint32_t v = 0; v < 3; ++v) ring[v * h.stride + i] = gs[v * L + x];
    }
    if (tid == 0) sh.fail = ~0u;
    if (warp == 0) {
      make_step_keys(a, d.t, 0, sh.keys);
      make_step_keys(a, d.t, 32, sh.keys);
    }
    if constexpr (REC)
      for (size_t i = rank * threads + tid; i < (size_t(b.T) + 1) * 4; i += blocks * threads) rec[i] = 0ull;
    meet();
    const bool plain = !a.particle && a.omega_mode == kTable && a.rest_mode == kTable;
    const uint32_t R = h.n ? recorders : 0;
    uint16_t* const other = ring + 3 * h.stride;
    if (plain)
      run_share<REC, STATES, true>(b, a, d, r, h, T, tables, to, tr, words, sh, src, other, colliders, R);
    else
      run_share<REC, STATES, false>(b, a, d, r, h, T, tables, to, tr, words, sh, src, other, colliders, R);
    meet();
    uint32_t fail = ~0u;
    if (ALONE && blocks == 1) fail = sh.fail;
    else if (lane < blocks)
      asm volatile("ld.shared::cluster.u32 %0, [%1];\n" : "=r"(fail) : "r"(mapa(&sh.fail, lane)) : "memory");
    fail = __reduce_min_sync(kFullWarp, fail);
    if (fail == ~0u) break;
    // once more from the start, as far as the ring goes
    over = true;
    T = fail;
    meet();  // all have read `fail`
  }
  for (uint32_t i = tid; i < h.n; i += threads) {
#pragma unroll
    for (uint32_t v = 0; v < 3; ++v) gs[v * L + h.lo + i] = src[v * h.stride + h.halo + i];
  }
  if constexpr (REC) {
    // the parts' sums into the states' 128-bit sums, as write_sums
    const __int128 M = (long long)sh.mass;
    for (size_t i = rank * threads + tid; i < 2 * (size_t(T) + 1); i += blocks * threads) {
      const uint32_t k = 2 * (i & 1);
      const long long low = (long long)__ldcg(rec + 2 * i), high = (long long)__ldcg(rec + 2 * i + 1);
      const __int128 S = (__int128(high) << 32) + low, Z = (__int128(sh.c[k + 1]) << 32) + sh.c[k];
      const __int128 v = S * __int128(L) - Z * M;
      rec[2 * i] = (unsigned long long)v;
      rec[2 * i + 1] = (unsigned long long)(v >> 64);
    }
  }
  if (rank == 0 && tid == 0) {
    b.desc[r].t = d.t + T;
    if (over) b.failed[r] = 1u;
  }
}

// PULL: clusters of `blocks` pull the `split` longest rings one by one, then the others `blocks`
// at a time, one per block.  Else every ring has a cluster.
template <bool REC, bool STATES, bool PULL>
__global__ void __launch_bounds__(1024, 1)
    batch_cluster_kernel(const __grid_constant__ BatchArgs b, const __grid_constant__ StepArgs common, uint32_t blocks,
                         uint32_t recorders, uint32_t split) {
  extern __shared__ uint4 smem4[];
  __shared__ ShareShared sh;
  const uint32_t rank = blockIdx.x % blocks;
  const auto meet = [] {
    cluster_arrive();
    cluster_wait();
  };
  if constexpr (!PULL) {
    run_split<REC, STATES, false>(b, common, b.order[blockIdx.x / blocks], blocks, rank, recorders, smem4, sh);
    meet();  // no block leaves while another may read from it
  } else {
    __shared__ uint32_t tasks[2];
    meet();  // all blocks have started
    for (uint32_t turn = 0;; turn ^= 1) {
      if (rank == 0 && threadIdx.x < 32) {
        const uint32_t lane = threadIdx.x;
        uint32_t next = 0;
        if (lane == 0) next = atomicAdd(b.counter, 1u);
        next = __shfl_sync(kFullWarp, next, 0);
        if (lane < blocks)
          asm volatile("st.shared::cluster.u32 [%0], %1;\n" ::"r"(mapa(&tasks[turn], lane)), "r"(next) : "memory");
      }
      meet();  // (and all are done with the last task)
      const uint32_t task = tasks[turn];
      const bool alone = task >= split;
      const uint64_t first = alone ? split + uint64_t(task - split) * blocks : task, at = first + (alone ? rank : 0);
      if (first >= b.n) return;  // no block reads from another after this
      if (at < b.n)
        run_split<REC, STATES, true>(b, common, b.order[at], alone ? 1 : blocks, alone ? 0 : rank, recorders, smem4, sh);
    }
  }
}

// The instantiation for a shape and what it records.
const void* batch_fn(int threads, bool rec, bool states, bool alone) {
  auto pick = [&](auto shape, auto own) {
    constexpr int N = decltype(shape)::value;
    constexpr bool A = decltype(own)::value;
    if (rec) return states ? reinterpret_cast<const void*>(batch_d1q3_kernel<N, true, true, A>)
                           : reinterpret_cast<const void*>(batch_d1q3_kernel<N, true, false, A>);
    return states ? reinterpret_cast<const void*>(batch_d1q3_kernel<N, false, true, A>)
                  : reinterpret_cast<const void*>(batch_d1q3_kernel<N, false, false, A>);
  };
  if (threads == 256)
    return alone ? pick(std::integral_constant<int, 256>{}, std::true_type{})
                 : pick(std::integral_constant<int, 256>{}, std::false_type{});
  if (threads == 512) return pick(std::integral_constant<int, 512>{}, std::false_type{});
  return pick(std::integral_constant<int, 1024>{}, std::false_type{});
}

}  // namespace

// Default shape: 256-thread blocks, several per SM, for rings of at most kBatchSmallL nodes
// where there are more rings than SMs (or the rings need no more threads); else one
// 1024-thread block per SM.  The autotuner (ilg_batch_autotune) may pick 256, 512 or 1024
// threads instead.
constexpr uint32_t kBatchSmallL = 1024;

template <bool PULL>
static const void* share_fn(bool rec, bool states) {
  if (rec) return states ? reinterpret_cast<const void*>(batch_cluster_kernel<true, true, PULL>)
                         : reinterpret_cast<const void*>(batch_cluster_kernel<true, false, PULL>);
  return states ? reinterpret_cast<const void*>(batch_cluster_kernel<false, true, PULL>)
                : reinterpret_cast<const void*>(batch_cluster_kernel<false, false, PULL>);
}

size_t batch_smem_bytes(uint32_t Lmax, int threads) {
  const uint32_t table = threads == 1024 ? BatchShape<1024>::kTableWords : BatchShape<256>::kTableWords;
  return sizeof(uint32_t) * (table + size_t(kBatchExtWords) * threads) + sizeof(uint16_t) * 2 * 3 * size_t(Lmax);
}

// largest dynamic shared memory a shape may ask for (the 227 KB a block may opt into,
// less room for the kernel's static shared memory)
constexpr size_t kBatchSmemCap = 220 * 1024;

bool batch_shape_fits(uint32_t Lmax, int threads) { return batch_smem_bytes(Lmax, threads) <= kBatchSmemCap; }

uint32_t batch_default_threads(uint32_t Lmax, uint32_t n, uint32_t sms) {
  return Lmax <= 256 || (Lmax <= kBatchSmallL && n > sms) ? 256 : 1024;
}

// The same limit for every batch of the process, whatever its rings' length.
cudaError_t prepare_batch_kernel(uint32_t Lmax, int threads) {
  if (!batch_shape_fits(Lmax, threads)) return cudaErrorInvalidValue;
  for (bool rec : {false, true})
    for (bool states : {false, true}) {
      for (bool alone : {false, true}) {
        const cudaError_t e = cudaFuncSetAttribute(batch_fn(threads, rec, states, alone),
                                                   cudaFuncAttributeMaxDynamicSharedMemorySize, int(kBatchSmemCap));
        if (e != cudaSuccess) return e;
      }
      for (const void* fn : {share_fn<false>(rec, states), share_fn<true>(rec, states)}) {
        cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, int(kBatchSmemCap));
        if (e == cudaSuccess) e = cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        if (e != cudaSuccess) return e;
      }
    }
  return cudaSuccess;
}

// (more than half of an SM's: a block has an SM to itself)
static size_t share_smem(uint32_t Lmax, uint32_t blocks) {
  const size_t n = sizeof(uint32_t) * (kDevStagedWords + size_t(kBatchExtWords) * 1024) +
                   2 * 3 * sizeof(uint16_t) * std::max(ring_split(Lmax, blocks).most + 2 * kMostHalo + 1, kSplitFrom);
  return std::max<size_t>(n, 116 * 1024);
}

// What a step costs, in us at 30 per velocity: a ring of one block, a part of a ring.
static double ring_cost(double nodes) { return std::max(0.65 + 0.7e-3 * nodes, 0.4 + 1.45e-3 * nodes); }
static double part_cost(double nodes) { return std::max(0.72 + 0.8e-3 * nodes, 0.55 + 1.6e-3 * nodes); }

// When pieces of work, the longest first, are done by workers that pull them: at the earliest
// (all busy to the end), and one piece after the other.
template <class Cost>
static double work_bound(uint32_t pieces, uint32_t workers, const Cost& cost) {
  double sum = 0;
  for (uint32_t i = 0; i < pieces; ++i) sum += cost(i);
  return std::max(cost(0), sum / workers);
}
template <class Cost>
static double makespan(uint32_t pieces, uint32_t workers, const Cost& cost) {
  constexpr uint32_t kMost = 512;
  if (pieces <= workers) return cost(0);
  if (workers > kMost) return work_bound(pieces, workers, cost);
  double free_at[kMost], end = 0;  // a heap, the earliest first
  for (uint32_t i = 0; i < pieces; ++i) {
    double t = cost(i);
    uint32_t held = i;
    if (i >= workers) {
      std::pop_heap(free_at, free_at + workers, std::greater<double>());
      held = workers - 1;
      t += free_at[held];
    }
    free_at[held] = t;
    std::push_heap(free_at, free_at + held + 1, std::greater<double>());
    end = std::max(end, t);
  }
  return end;
}

// The split form, where it is expected to be faster than a ring per block: the size of cluster
// with which the rings are done first (a tenth allowed for what pulling costs).  Us per step, a
// ring per block / split: 100 rings of 64 to 8192 nodes at 30 per velocity 11.9 / 4.3, 200 12.0 /
// 6.5, 400 at 50 15.2 / 13.2; 150 of 64 to 2000 3.3 / 2.2.  At least 256 threads (they stage the
// tables); one recording warp for four colliding ones, at most 8: 9 rings of up to 1000 nodes with
// states 1.52 us per step, with twice as many 1.53, with all 1.58.
static bool launch_split(const BatchArgs& b, const uint32_t* lengths, const StepArgs& common, int sms, cudaStream_t s) {
  const uint32_t N = uint32_t(sms), n = b.n;
  // more than eight rings per SM keep all SMs busy to the end
  if (b.Lmax < kSplitFrom || n > 8 * N) return false;
  const bool rec = b.record || b.states;
  const auto is_long = [](uint32_t L) { return L >= kSplitFrom; };
  const uint32_t split = uint32_t(std::partition_point(lengths, lengths + n, is_long) - lengths);
  // (rings of up to kBatchSmallL nodes in larger numbers: several blocks on an SM)
  const bool several = b.Lmax <= kBatchSmallL && n > N;
  double nodes = 0;
  for (uint32_t i = 0; i < n; ++i) nodes += lengths[i];
  const auto whole = [&](uint32_t i) { return ring_cost(lengths[i]); };
  double least = several ? std::max(whole(0), 1.45e-3 * nodes / N) : makespan(n, N, whole);
  uint32_t best = 0, clusters = 0;
  bool pull = false;
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeClusterDimension;
  attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg{};
  cfg.stream = s;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  uint32_t recorders = 0;
  const auto shape = [&](uint32_t blocks) {
    const uint32_t tiles = std::max(ring_split(b.Lmax, blocks).tiles, split < n ? kSplitFrom / 32 : 1u);
    recorders = rec ? std::clamp((tiles + 1) / 4, 1u, 8u) : 0u;
    const uint32_t rounds = (tiles + 31 - recorders) / (32 - recorders);
    attr.val.clusterDim.x = blocks;
    cfg.blockDim = dim3(std::max(256u, ((tiles + rounds - 1) / rounds + recorders) * 32));
    cfg.dynamicSmemBytes = share_smem(b.Lmax, blocks);
    cfg.gridDim = dim3(blocks);
  };
  for (uint32_t blocks = std::min(16u, b.Lmax / 32); blocks >= 2; --blocks) {
    const uint32_t pieces = split + (n - split + blocks - 1) / blocks;
    const auto piece = [&](uint32_t i) {
      return i < split ? part_cost(double(lengths[i]) / blocks) : ring_cost(lengths[split + (i - split) * blocks]);
    };
    const bool own = n <= N / blocks;  // perhaps a cluster for every ring
    const double longest = part_cost(double(b.Lmax) / blocks);
    if ((own ? longest : 1.1 * work_bound(pieces, N / blocks, piece)) >= least) continue;
    shape(blocks);
    int fit = 0;
    const void* fn = share_fn<true>(b.record != nullptr, b.states != nullptr);
    if (cudaOccupancyMaxActiveClusters(&fit, fn, &cfg) != cudaSuccess || fit < 1) {
      cudaGetLastError();
      continue;
    }
    const double t = n <= uint32_t(fit) ? longest : 1.1 * makespan(pieces, uint32_t(fit), piece);
    if (t >= least) continue;
    least = t;
    best = blocks;
    pull = n > uint32_t(fit);
    clusters = pull ? std::min(pieces, uint32_t(fit)) : n;
  }
  if (!best) return false;
  shape(best);
  cfg.gridDim = dim3(clusters * best);
  BatchArgs ba = b;
  StepArgs ca = common;
  uint32_t whole_from = split;
  void* p[] = {&ba, &ca, &best, &recorders, &whole_from};
  const void* fn = pull ? share_fn<true>(b.record != nullptr, b.states != nullptr)
                        : share_fn<false>(b.record != nullptr, b.states != nullptr);
  if (cudaLaunchKernelExC(&cfg, fn, p) == cudaSuccess) return true;
  cudaGetLastError();
  return false;
}

// Persistent grid: as many blocks as fit on every SM (shared memory and registers
// decide), at most one per ring.  A block has as many of its shape's threads as the longest
// ring keeps equally busy (320 nodes on the 256-thread shape: 160 threads, two nodes each),
// and the recording warps.
cudaError_t launch_batch(const BatchArgs& b, const uint32_t* lengths, const StepArgs& common, int sms, cudaStream_t s,
                         int shape) {
  if (launch_split(b, lengths, common, sms, s)) return cudaSuccess;
  const size_t smem = batch_smem_bytes(b.Lmax, shape);
  const bool rec = b.record != nullptr || b.states != nullptr;
  const uint32_t most = uint32_t(shape) / 32, tiles = (b.Lmax + 31) / 32;
  const uint32_t recorders = !rec ? 0u : shape == 1024 ? BatchShape<1024>::kRecorders
                                      : shape == 512   ? BatchShape<512>::kRecorders
                                                       : BatchShape<256>::kRecorders;
  // all of the shape's warps collide where a block has an SM to itself
  const uint32_t room = shape == 256 && b.n <= uint32_t(sms) ? most : most - recorders;
  const uint32_t rounds = (tiles + room - 1) / room;
  const int threads = int(((tiles + rounds - 1) / rounds + recorders) * 32);
  const void* fn = batch_fn(shape, b.record != nullptr, b.states != nullptr, b.n <= uint32_t(sms));
  int per_sm = 1;
  const cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, threads, smem);
  if (e != cudaSuccess) return e;
  if (per_sm < 1) per_sm = 1;
  const uint32_t cap = uint32_t(per_sm) * uint32_t(sms);
  BatchArgs ba = b;
  StepArgs ca = common;
  void* p[] = {&ba, &ca};
  return cudaLaunchKernel(fn, dim3(b.n < cap ? b.n : cap), dim3(threads), p, smem, s);
}

}  // namespace ilg

namespace ilg {
namespace {

// Per replica: mass and the amplitude A^LG of one mode (one block per replica).
__global__ void __launch_bounds__(256) batch_obs_kernel(const ReplicaDesc* __restrict__ desc,
                                                        const uint16_t* __restrict__ state, int32_t mode,
                                                        unsigned long long* __restrict__ mass_out,
                                                        double* __restrict__ amp_out) {
  __shared__ unsigned long long s_mass;
  __shared__ double s_red[2 * 8];
  const ReplicaDesc d = desc[blockIdx.x];
  const uint32_t L = d.L;
  const uint16_t* s = state + d.state_off;
  if (threadIdx.x == 0) s_mass = 0ull;
  __syncthreads();
  unsigned long long part = 0;
  for (uint32_t x = threadIdx.x; x < L; x += blockDim.x) part += (unsigned long long)s[x] + s[L + x] + s[2 * L + x];
  if (part) atomicAdd(&s_mass, part);
  __syncthreads();
  const long long M = (long long)s_mass;
  const uint32_t m = uint32_t(((int64_t(mode) % int64_t(L)) + L) % L);
  double ps = 0.0, pc = 0.0;
  for (uint32_t x = threadIdx.x; x < L; x += blockDim.x) {
    const long long N = (long long)s[x] + s[L + x] + s[2 * L + x];
    const long long D = (long long)L * N - M;
    const uint32_t rr = uint32_t((uint64_t(m) * x) % L);
    double sn, cs;
    sincospi(2.0 * double(rr) / double(L), &sn, &cs);
    const double p = sn * double(D);
    const double pe = fma(sn, double(D), -p);
    double q;
    two_sum_b(ps, p, ps, q);
    pc += q + pe;
  }
  const double im = block_dot2<256>(ps, pc, s_red) / double(L);
  if (threadIdx.x == 0) {
    mass_out[blockIdx.x] = (unsigned long long)M;
    amp_out[blockIdx.x] = im / (double(L) / 2.0);
  }
}

// ring r's trig[state_off_r / 3 + x] = fixed-point (cos, sin) of 2 pi ((m_r x) mod L_r) / L_r,
// m_r the mode reduced modulo L_r
__global__ void batch_trig_rings_kernel(const ReplicaDesc* __restrict__ desc, uint32_t n, int32_t mode,
                                        longlong2* __restrict__ trig) {
  for (uint32_t r = blockIdx.x; r < n; r += gridDim.x) {
    const uint32_t L = desc[r].L;
    const uint32_t m = uint32_t(((int64_t(mode) % int64_t(L)) + L) % L);
    longlong2* out = trig + desc[r].state_off / 3;
    for (uint32_t x = threadIdx.x; x < L; x += blockDim.x) out[x] = trig_fixed(uint32_t((uint64_t(m) * x) % L), L);
  }
}

// Raw 128-bit sums (L 2^62 re, L 2^62 im) -> (re, im) in double, rounded once and
// divided by L.
__global__ void batch_convert_kernel(const ReplicaDesc* __restrict__ desc, const long long* __restrict__ raw,
                                     uint32_t n, uint32_t T, double* __restrict__ rec) {
  const size_t total = size_t(n) * (T + 1);
  for (size_t i = size_t(blockIdx.x) * blockDim.x + threadIdx.x; i < total; i += size_t(gridDim.x) * blockDim.x) {
    const double L = double(desc[i / (T + 1)].L);
    const long long* v = raw + 4 * i;
    I128 re, im;
    re.lo = (unsigned long long)v[0];
    re.hi = v[1];
    im.lo = (unsigned long long)v[2];
    im.hi = v[3];
    rec[2 * i] = i128_to_double_2m62(re) / L;
    rec[2 * i + 1] = i128_to_double_2m62(im) / L;
  }
}

// amp[r T + s] = im / (L_r / 2) of the record entry after step s.
__global__ void batch_amp_kernel(const ReplicaDesc* __restrict__ desc, const double* __restrict__ record,
                                 uint32_t n, uint32_t T, double* __restrict__ amp) {
  const size_t total = size_t(n) * T;
  for (size_t i = size_t(blockIdx.x) * blockDim.x + threadIdx.x; i < total; i += size_t(gridDim.x) * blockDim.x) {
    const size_t r = i / T, s = i - r * T;
    amp[i] = record[(r * (T + 1) + s + 1) * 2 + 1] / (double(desc[r].L) / 2.0);
  }
}

// Ensemble statistics over the n rings of the record, one block per time index t:
// means of re and im, sample variances (divisor n - 1) and the connected
// correlation with t = 0 of a = re + i im:  cov = sum (a(t) - <a(t)>) conj(a(0) - <a(0)>) / (n - 1).
// Fixed-order sums (deterministic); two passes (means, then deviations).
__global__ void __launch_bounds__(256) batch_ensemble_kernel(const double* __restrict__ record, uint32_t n,
                                                             uint32_t T, double* __restrict__ out) {
  __shared__ double red[4][256];
  const uint32_t t = blockIdx.x;
  const size_t stride = size_t(T + 1) * 2;
  double v[4] = {0.0, 0.0, 0.0, 0.0};
  for (uint32_t r = threadIdx.x; r < n; r += blockDim.x) {
    const double* o = record + r * stride;
    v[0] += o[2 * t];
    v[1] += o[2 * t + 1];
    v[2] += o[0];
    v[3] += o[1];
  }
  auto reduce4 = [&](double (&w)[4]) {
    for (int k = 0; k < 4; ++k) red[k][threadIdx.x] = w[k];
    __syncthreads();
    for (int h = 128; h > 0; h >>= 1) {
      if (int(threadIdx.x) < h)
        for (int k = 0; k < 4; ++k) red[k][threadIdx.x] += red[k][threadIdx.x + h];
      __syncthreads();
    }
    for (int k = 0; k < 4; ++k) w[k] = red[k][0];
    __syncthreads();
  };
  reduce4(v);
  const double mre = v[0] / n, mim = v[1] / n, m0re = v[2] / n, m0im = v[3] / n;
  double w[4] = {0.0, 0.0, 0.0, 0.0};
  for (uint32_t r = threadIdx.x; r < n; r += blockDim.x) {
    const double* o = record + r * stride;
    const double dre = o[2 * t] - mre, dim = o[2 * t + 1] - mim;
    const double d0re = o[0] - m0re, d0im = o[1] - m0im;
    w[0] += dre * dre;
    w[1] += dim * dim;
    w[2] += dre * d0re + dim * d0im;
    w[3] += dim * d0re - dre * d0im;
  }
  reduce4(w);
  if (threadIdx.x == 0) {
    const size_t P = T + 1;
    const double dn = double(n) - 1.0;
    out[0 * P + t] = mre;
    out[1 * P + t] = mim;
    out[2 * P + t] = w[0] / dn;
    out[3 * P + t] = w[1] / dn;
    out[4 * P + t] = w[2] / dn;
    out[5 * P + t] = w[3] / dn;
  }
}

}  // namespace

cudaError_t launch_batch_obs(const ReplicaDesc* desc, const uint16_t* state, uint32_t n, int32_t mode,
                             unsigned long long* mass, double* amp, cudaStream_t s) {
  batch_obs_kernel<<<n, 256, 0, s>>>(desc, state, mode, mass, amp);
  return cudaGetLastError();
}

cudaError_t launch_batch_amp(const ReplicaDesc* desc, const double* record, uint32_t n, uint32_t T, double* amp,
                             cudaStream_t s) {
  const size_t total = size_t(n) * T;
  const int grid = int(total / 256 + 1 < 4096 ? total / 256 + 1 : 4096);
  batch_amp_kernel<<<grid, 256, 0, s>>>(desc, record, n, T, amp);
  return cudaGetLastError();
}

cudaError_t launch_batch_convert(const ReplicaDesc* desc, const long long* raw, uint32_t n, uint32_t T, double* rec,
                                 cudaStream_t s) {
  const size_t total = size_t(n) * (T + 1);
  const int grid = int(total / 256 + 1 < 4096 ? total / 256 + 1 : 4096);
  batch_convert_kernel<<<grid, 256, 0, s>>>(desc, raw, n, T, rec);
  return cudaGetLastError();
}

cudaError_t launch_batch_trig_rings(const ReplicaDesc* desc, uint32_t n, int32_t mode, longlong2* trig, cudaStream_t s) {
  batch_trig_rings_kernel<<<n < 1024u ? n : 1024u, 256, 0, s>>>(desc, n, mode, trig);
  return cudaGetLastError();
}

cudaError_t launch_batch_ensemble(const double* record, uint32_t n, uint32_t T, double* out, cudaStream_t s) {
  batch_ensemble_kernel<<<T + 1, 256, 0, s>>>(record, n, T, out);
  return cudaGetLastError();
}

}  // namespace ilg
