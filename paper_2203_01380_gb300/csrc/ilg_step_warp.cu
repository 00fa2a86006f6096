// Warp-segment fused step with 8- or 4-node vectors, shaped for integer issue.
//
// The step's time goes to the integer work of its random numbers (two Philox
// blocks and six alias draws per node), so this kernel spends its registers on the
// independent work of wide vectors in few warps rather than on data in flight:
//  - each lane owns a vector of NPT consecutive nodes (16- or 8-byte accesses; a
//    warp covers 32 NPT nodes of a row per tile); the next tile's occupations are
//    copied into the warp's shared-memory buffer by cp.async while the current tile
//    collides, so the copy holds no registers;
//  - the flip is a compile-time choice of which plane of the buffer is read as which
//    velocity, so it costs nothing;
//  - the fast collision runs branch-free on every node of a vector whose
//    occupations are all below ROWS (64: the rows of the alias tables, staged in
//    shared memory once per SM); the rare node outside that domain is redone by the
//    general collision, out of line (its registers do not weigh on the fast path);
//  - warp w takes the w-th of equal shares of the row-major sequence of all tiles (32
//    vectors of a row) and walks it tile by tile, as segments that end at row ends; neighbouring lanes trade
//    edge values by shuffles, and the two values that cross a segment's ends are
//    written as single 16-bit stores by the warp that computes them, so no node is
//    computed twice and no warp waits for another;
//  - a lane's vector and its results stay in registers, and it collides two nodes at a
//    time (fast_pair), so that sums and results are formed for both at once.
// Every random number is keyed by node and step, so the bits equal those of every
// other step kernel.
#include <cuda_runtime.h>

#include <algorithm>

#include "ilg_d2q9.cuh"
#include "ilg_device.cuh"
#include "ilg_launch.h"
#include "ilg_sync.cuh"

namespace ilg {
namespace {

// NPT consecutive nodes of one plane: node k in the low (k even) or high (k odd)
// half of word k / 2
template <int NPT>
struct __align__(2 * NPT < 16 ? 2 * NPT : 16) VN {
  static_assert(NPT == 4 || NPT == 8 || NPT == 16, "vectors of 4, 8 or 16 nodes (8-byte or 16-byte copies)");
  uint32_t w[NPT / 2];
};

template <int NPT>
__device__ __forceinline__ void stv(uint16_t* p, const uint32_t (&w)[NPT / 2]) {
  if constexpr (NPT >= 8) {
#pragma unroll
    for (int j = 0; j < NPT / 8; ++j)
      reinterpret_cast<uint4*>(p)[j] = make_uint4(w[4 * j], w[4 * j + 1], w[4 * j + 2], w[4 * j + 3]);
  } else {
    *reinterpret_cast<uint2*>(p) = make_uint2(w[0], w[1]);
  }
}
template <int NPT>
__device__ __forceinline__ uint32_t node_of(const VN<NPT>& v, int k) {
  return (k & 1) ? (v.w[k >> 1] >> 16) : (v.w[k >> 1] & 0xFFFFu);
}

// asynchronous copy of BYTES (8 or 16) global -> shared (zero-filled when !valid: no
// global read)
template <int BYTES>
__device__ __forceinline__ void cp_async(void* dst, const void* src, bool valid) {
  const uint32_t s = static_cast<uint32_t>(__cvta_generic_to_shared(dst));
  if constexpr (BYTES == 16)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(s), "l"(src), "r"(valid ? 16 : 0) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;\n" ::"r"(s), "l"(src), "r"(valid ? 8 : 0) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
// all but the most recent group of this thread's copies have landed
__device__ __forceinline__ void cp_async_wait_prior() { asm volatile("cp.async.wait_group 1;\n" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

// the flip F_i(n) = n_{-i}: velocity i of the collision reads plane -i
template <bool FLIP>
__device__ __forceinline__ constexpr int source_plane(int i) {
  return !FLIP || i == 0 ? i : (i & 1 ? i + 1 : i - 1);
}

// a b + c on the FMA pipe
__device__ __forceinline__ uint32_t mad(uint32_t a, uint32_t b, uint32_t c) {
  uint32_t d;
  asm("mad.lo.u32 %0, %1, %2, %3;\n" : "=r"(d) : "r"(a), "r"(b), "r"(c));
  return d;
}

// Binomial(n, P) for n < 64 with one draw u through the alias table at shared address
// `table` (rows of 64 columns, column u >> 26): the column's own outcome below its
// threshold, else its alias.
__device__ __forceinline__ uint32_t draw(uint32_t table, uint32_t n, uint32_t u) {
  const uint32_t j = u >> 26;
  uint32_t thr, r;
  asm("ld.shared.v2.u32 {%0, %1}, [%2];\n" : "=r"(thr), "=r"(r) : "r"(mad(j, 8, mad(n, 512, table))));
  return u < thr ? j : r;
}

// Shared addresses of the staged tables: thinning, rest, D2Q9's axis share.
struct FastTables {
  uint32_t to, tr, ta;
};

// Axis bit A (0: x, 1: y) and sign bit B (0: +, 1: -) of the first `c` <= 32 particles:
// how many have A set, both, B alone.
__device__ __forceinline__ void count3(uint32_t c, uint32_t A, uint32_t B, uint32_t& a, uint32_t& both, uint32_t& b) {
  const uint32_t mask = __funnelshift_lc(0xFFFFFFFFu, 0u, c);  // (1 << c) - 1, c <= 32
  a = __popc(A & mask);
  both = __popc(A & B & mask);
  b = __popc(~A & B & mask);
}

// What bounds it: the ALU and FMA-heavy pipes.  Each takes two cycles per warp instruction and
// sub-partition; a 32 x 32 -> 64 product takes four of the FMA-heavy pipe and, measured beside
// 3-input logic, two of the ALU pipe as well, so a node's 30 products fill 120 and 60 cycles
// before anything else, and the two pipes are as full as they get (collisions alone, D2Q5: 220
// cycles per 32 nodes, 208 of them the ALU pipe's, 165 the FMA-heavy pipe's).  Hence: what can be a
// multiply-add is one (table addresses, halves packed and parted), and sums, differences, limits
// and the checks on them are made once for the two nodes, in 16-bit halves.  GNUPS against one node
// at a time, 16384^2 D2Q5 165 / 159; 8192^2 4-node vectors 149 / 138; 8192^2 D2Q9 77.4 / 72.7 (there
// one pair at a time from the tile buffer).  Not faster: the table's outcome selected by a
// predicated multiply-add instead of on the ALU pipe (D2Q5 166 for some of the draws, 159 for all).
//
// Fast collision of two neighbouring nodes whose occupations (w: the even node's in the low
// halves) are all below 64, branch-free: node0 the even node, p their results packed alike.
// Returns bits 12 and 28: the even / the odd node needs the general collision (more than 63
// removed, or more than 32 moving particles of a kind); its half of p is then garbage in
// [0, 126], but every table index stayed inside the staged rows.
template <int Q>
__device__ __forceinline__ uint32_t fast_pair(const FastTables& T, const StepKeys<Q == 9 ? 4 : 2>& keys,
                                              const uint32_t (&rk)[20], uint32_t node0, const uint32_t (&w)[Q],
                                              uint32_t (&p)[Q]) {
  constexpr int NB = Q == 9 ? 4 : 2;
  uint32_t W[2][4 * NB], r[Q], D[Q];
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    step_blocks<NB>(keys, rk, node0 + h, W[h]);
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      const uint32_t high = w[i] >> 16;
      const uint32_t m = h ? high : mad(high, 0xFFFF0000u, w[i]);
      const uint32_t x = draw(T.to, m, W[h][i]);
      if (h) D[i] = mad(x, 65536u, r[i]);
      else r[i] = x;
    }
  }
  uint32_t removed = D[0];
#pragma unroll
  for (int i = 1; i < Q; ++i) removed += D[i];
  const uint32_t rr = __vminu2(removed, 0x003F003Fu);
  const uint32_t rr1 = rr >> 16, rr0 = mad(rr1, 0xFFFF0000u, rr);
  const uint32_t rest0 = draw(T.tr, rr0, W[0][Q]), rest1 = draw(T.tr, rr1, W[1][Q]);
  const uint32_t rest = mad(rest1, 65536u, rest0);
  const uint32_t mv = rr - rest, mv1 = rr1 - rest1, mv0 = rr0 - rest0;
  p[0] = w[0] - D[0] + rest;
  // 4096 - 64 + removed and 4096 - 33 + moving reach bit 12 beyond the limits
  uint32_t over = removed + 0x0FC00FC0u;
  if constexpr (Q == 3) {
    over |= mv + 0x0FDF0FDFu;
    const uint32_t k0 = __popc(W[0][Q + 1] & __funnelshift_lc(0xFFFFFFFFu, 0u, mv0));
    const uint32_t k1 = __popc(W[1][Q + 1] & __funnelshift_lc(0xFFFFFFFFu, 0u, mv1));
    const uint32_t minus = mad(k1, 65536u, k0);
    p[1] = w[1] - D[1] + (mv - minus);
    p[2] = w[2] - D[2] + minus;
  } else {
    uint32_t ax = mv, ax0 = mv0, ax1 = mv1;
    if constexpr (Q == 9) {
      ax0 = draw(T.ta, mv0, W[0][10]);
      ax1 = draw(T.ta, mv1, W[1][10]);
      ax = mad(ax1, 65536u, ax0);
    }
    over |= ax + 0x0FDF0FDFu;
    constexpr int A = Q == 9 ? 11 : Q + 1;
    uint32_t a[2], both[2], b[2];
    count3(ax0, W[0][A], W[0][A + 1], a[0], both[0], b[0]);
    count3(ax1, W[1][A], W[1][A + 1], a[1], both[1], b[1]);
    const uint32_t ny = mad(a[1], 65536u, a[0]), nmy = mad(both[1], 65536u, both[0]), nmx = mad(b[1], 65536u, b[0]);
    p[1] = (w[1] - D[1] + ax) - ny - nmx;
    p[2] = w[2] - D[2] + nmx;
    p[3] = w[3] - D[3] + (ny - nmy);
    p[4] = w[4] - D[4] + nmy;
    if constexpr (Q == 9) {
      // diagonal particles: x-sign bit X, y-sign bit Y (0: +, 1: -)
      const uint32_t dg = mv - ax;
      over |= dg + 0x0FDF0FDFu;
      count3(mv0 - ax0, W[0][13], W[0][14], a[0], both[0], b[0]);
      count3(mv1 - ax1, W[1][13], W[1][14], a[1], both[1], b[1]);
      const uint32_t x = mad(a[1], 65536u, a[0]), xy = mad(both[1], 65536u, both[0]), yo = mad(b[1], 65536u, b[0]);
      p[5] = (w[5] - D[5] + dg) - x - yo;
      p[6] = w[6] - D[6] + xy;
      p[7] = w[7] - D[7] + yo;
      p[8] = w[8] - D[8] + (x - xy);
    }
  }
  return over & 0x10001000u;
}

// The general collision of the nodes of a vector marked in `slow`, out of line.  N:
// the lane's slot of the current tile buffer in shared memory (plane i at N[32 i], before
// the flip); velocity i's result of node k replaces half-word k of N[32 i].  In shared memory
// so that no register array of the caller has its address taken (which would keep it in local
// memory on every tile).
// st: the staged tables (all rows of each, laid out as the table block; from global memory a
// node's dozen dependent draws would keep its warp ten times longer).  Returns true when a
// result exceeds 65535.
template <int Q, bool FLIP, int NPT>
__device__ __noinline__ bool slow_nodes(const StepArgs& a, const uint32_t* st, uint32_t node0, uint32_t t,
                                        VN<NPT>* N, uint32_t slow) {
  bool bad = false;
  while (slow) {
    const int k = __ffs(slow) - 1;
    slow &= slow - 1;
    uint32_t m[Q], o[Q];
#pragma unroll
    for (int i = 0; i < Q; ++i) m[i] = node_of(N[32 * source_plane<FLIP>(i)], k);
    if constexpr (Q == 9) collide9_general(a, st, node0 + k, t, m, o);
    else collide<Q>(a, st, node0 + k, t, m, o);
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      bad |= o[i] > 65535u;
      reinterpret_cast<uint16_t*>(&N[32 * i])[k] = uint16_t(o[i]);
    }
  }
  return bad;
}

// Collide the NPT nodes of one vector (first node `node0`) into the packed post-collision
// planes P.  N holds the vector's occupations with the flip already applied; slot is where
// they came from in the tile buffer (for the out-of-line general collision, which leaves its
// results there); keys: the launch-wide part of every node's slot blocks.
template <int Q, bool FLIP, int ROWS, int NPT>
__device__ __forceinline__ void collide_vec(const StepArgs& a, const StepKeys<Q == 9 ? 4 : 2>& keys, const uint32_t* tables,
                                            const FastTables& T, uint32_t node0, uint32_t t,
                                            VN<NPT> (&N)[Q], VN<NPT> (&P)[Q], VN<NPT>* slot, bool& bad) {
  static_assert(ROWS == 64 && NPT <= 8, "six-bit rows; the pairs' marks stay in their halves");
  constexpr uint32_t kHigh = 0xFFC0FFC0u;  // bits of values >= ROWS
  uint32_t any = 0;
#pragma unroll
  for (int i = 0; i < Q; ++i)
#pragma unroll
    for (int j = 0; j < NPT / 2; ++j) any |= N[i].w[j];
  uint32_t slow = 0;
  if (any & kHigh) {
    // nodes beyond the fast collision's rows: marked for the general one, and their values
    // cut to six bits so that they pass through the fast one without harm
    constexpr uint32_t kLow = ~kHigh;
#pragma unroll
    for (int j = 0; j < NPT / 2; ++j) {
      uint32_t w = 0;
#pragma unroll
      for (int i = 0; i < Q; ++i) {
        w |= N[i].w[j];
        N[i].w[j] &= kLow;
      }
      w &= kHigh;
      slow |= ((w & 0xFFFFu) ? 1u : 0u) << (2 * j) | ((w >> 16) ? 2u : 0u) << (2 * j);
    }
  }
  uint32_t over = 0;  // pair j's bits end at 12 + H - 1 - j and 28 + H - 1 - j
#pragma unroll
  for (int j = 0; j < NPT / 2; ++j) {
    uint32_t w[Q], p[Q];
#pragma unroll
    for (int i = 0; i < Q; ++i) w[i] = N[i].w[j];
    const uint32_t e = fast_pair<Q>(T, keys, a.rk, node0 + 2 * j, w, p);
    over = j == 0 ? e : mad(over, 2u, e);
#pragma unroll
    for (int i = 0; i < Q; ++i) P[i].w[j] = p[i];
  }
  if (over) {
#pragma unroll
    for (int j = 0; j < NPT / 2; ++j) {
      const uint32_t e = over >> (NPT / 2 - 1 - j);
      slow |= ((e >> 12) & 1u) << (2 * j) | ((e >> 28) & 1u) << (2 * j + 1);
    }
  }
  if (slow) {
    bad |= slow_nodes<Q, FLIP, NPT>(a, tables, node0, t, slot, slow);
    // take the general collision's half-words for the nodes it redid
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      const VN<NPT> r = slot[32 * i];
#pragma unroll
      for (int j = 0; j < NPT / 2; ++j) {
        const uint32_t mask = ((slow >> (2 * j)) & 1u ? 0x0000FFFFu : 0u) | ((slow >> (2 * j + 1)) & 1u ? 0xFFFF0000u : 0u);
        P[i].w[j] = (P[i].w[j] & ~mask) | (r.w[j] & mask);
      }
    }
  }
}

// The segment that starts at vector g of the row-major sequence of all vectors
// (vpr per row) and ends at the end of its row or at end, whichever comes first:
// row y, vectors [v0, v1) of that row.
__device__ __forceinline__ void segment_at(uint32_t g, uint32_t end, uint32_t vpr, uint32_t& y, uint32_t& v0,
                                           uint32_t& v1) {
  y = g / vpr;
  v0 = g - y * vpr;
  v1 = min(vpr, v0 + (end - g));
}

// Queue the copies of one lane's vector (tile row rowoff, vector v) into its slots of
// the warp's tile buffer tb (Q planes of 32 vectors).
template <int Q, int NPT>
__device__ __forceinline__ void stage_tile(VN<NPT>* tb, const uint16_t* __restrict__ in, size_t plane, size_t rowoff,
                                           uint32_t v, bool active, uint32_t lane) {
  static_assert(2 * NPT <= 16, "one copy per vector");
#pragma unroll
  for (int i = 0; i < Q; ++i)
    cp_async<2 * NPT>(tb + i * 32 + lane, active ? in + i * plane + rowoff + size_t(v) * NPT : in, active);
  cp_async_commit();
}

// Velocity i's displacement (dx, dy) in the storage order of each lattice.
template <int Q>
__device__ __forceinline__ constexpr int vel_dx(int i) {
  return Q == 9 ? ((i == 1 || i == 5 || i == 7) ? 1 : ((i == 2 || i == 6 || i == 8) ? -1 : 0))
                : (i == 1 ? 1 : (i == 2 ? -1 : 0));
}
template <int Q>
__device__ __forceinline__ constexpr int vel_dy(int i) {
  return Q == 9 ? ((i == 3 || i == 5 || i == 8) ? 1 : ((i == 4 || i == 6 || i == 7) ? -1 : 0))
                : (Q == 5 ? (i == 3 ? 1 : (i == 4 ? -1 : 0)) : 0);
}

// T steps from t0, the state in buf0, a barrier of all blocks between them (a cooperative
// launch) that alternate the buffers; !RUN: one step (the loop costs 0.5 % of a step's time,
// more than a launch does on lattices of 2^26 nodes and beyond).  sync: as launch_step_run.
template <int Q, bool FLIP, int ROWS, int NPT, int THREADS, bool RUN>
__global__ void __launch_bounds__(THREADS, 1)
    step_warp_kernel(const __grid_constant__ StepArgs a, uint16_t* buf0, uint16_t* buf1, uint32_t t0, uint32_t T,
                     unsigned long long* fail, unsigned long long* sync) {
  extern __shared__ uint4 smem4[];
  __shared__ int stop;
  // a step before this launch overflowed (one of its own stops it at the barriers: a block that
  // started late must not leave the others waiting there)
  if (threadIdx.x == 0) stop = *reinterpret_cast<const volatile unsigned long long*>(fail) < t0;
  constexpr uint32_t kTables = Q == 9 ? 3 : 2;           // thinning, rest (D2Q9: and the axis share)
  constexpr uint32_t kRow4 = ROWS * kDevAliasCols / 2;  // uint4 per staged table
  {
    // rows 0..ROWS-1 of each alias table (uint2 entries, two per uint4)
    const uint4* g4 = reinterpret_cast<const uint4*>(a.tables);
    constexpr uint32_t kTab4 = kDevAliasEntries / 2;  // uint4 per full table
#pragma unroll 8
    for (uint32_t i = threadIdx.x; i < kTables * kRow4; i += THREADS)
      smem4[i] = g4[(i / kRow4) * kTab4 + (i % kRow4)];
  }
  __syncthreads();
  if (stop) return;
  const uint32_t* const tables = reinterpret_cast<const uint32_t*>(smem4);
  const uint32_t base = static_cast<uint32_t>(__cvta_generic_to_shared(smem4));
  const FastTables tab{base, base + ROWS * kDevAliasCols * 8, base + 2 * ROWS * kDevAliasCols * 8};

  constexpr unsigned kFull = 0xFFFFFFFFu;
  constexpr int H = NPT / 2;  // words per vector
  const uint32_t Lx = a.Lx, Ly = a.Ly;
  const size_t plane = size_t(Lx) * Ly;
  const uint32_t vpr = Lx / NPT;
  const uint32_t lane = threadIdx.x & 31u;
  // this warp's two tile buffers (Q planes of 32 vectors each) after the tables
  VN<NPT>* tbuf = reinterpret_cast<VN<NPT>*>(smem4 + kTables * kRow4) + (threadIdx.x >> 5) * (2 * Q * 32);
  for (uint32_t step = 0;; ++step) {
  const uint32_t t = t0 + step;
  const uint16_t* const __restrict__ in = RUN && (step & 1) ? buf1 : buf0;
  uint16_t* const __restrict__ out = RUN && (step & 1) ? buf0 : buf1;
  bool bad = false;
  // this warp's share of the row-major sequence of all vectors, [g, end): an equal share of
  // the tiles (a row's vectors, 32 at a time; one that is not full costs as much as one that
  // is), worked out anew each step to keep its registers free meanwhile
  uint32_t w = (blockIdx.x * THREADS + threadIdx.x) >> 5;
  asm volatile("" : "+r"(w));
  const uint32_t tpr = (vpr + 31) >> 5, nwarps = gridDim.x * (THREADS / 32);
  const uint64_t tiles = uint64_t(tpr) * Ly;
  auto vector_of = [&](uint64_t tile) {
    const uint32_t ty = uint32_t(tile / tpr);
    return ty * vpr + (uint32_t(tile) - ty * tpr) * 32;
  };
  uint32_t g = vector_of(w * tiles / nwarps);
  const uint32_t end = vector_of((w + 1) * tiles / nwarps);
  if (g < end) {
  const StepKeys<Q == 9 ? 4 : 2> keys = step_keys<Q == 9 ? 4 : 2>(a, t);  // the launch-uniform Philox rounds

  uint32_t y, v0, v1;
  segment_at(g, end, vpr, y, v0, v1);
  uint32_t vb = v0;
  int buf = 0;
  stage_tile<Q, NPT>(tbuf, in, plane, size_t(y) * Lx, vb + lane, vb + lane < v1, lane);
  uint32_t carry[Q];   // +x planes: the value of the previous tile's lane 31
  VN<NPT> held[Q];     // -x planes, lane 31: the vector waiting for the next tile's first node
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    carry[i] = 0;
    held[i] = VN<NPT>{};
  }
  // [p1 .. p_{NPT-1}, r]: a -x vector with r for its last slot
  auto shift_down = [](const VN<NPT>& p, uint32_t r) {
    VN<NPT> o;
#pragma unroll
    for (int j = 0; j < H - 1; ++j) o.w[j] = __byte_perm(p.w[j], p.w[j + 1], 0x5432);
    o.w[H - 1] = __byte_perm(p.w[H - 1], r, 0x5432);
    return o;
  };
  while (true) {
    // the next tile: of this segment, or the first of the segment that follows it;
    // its copies are queued before this tile collides
    const uint32_t g_next = g + (v1 - v0);  // first vector after this segment
    const bool same = vb + 32 < v1;
    const bool more = same || g_next < end;
    uint32_t ny = y, nv0 = v0, nv1 = v1, nvb = vb + 32;
    if (!same && more) {
      segment_at(g_next, end, vpr, ny, nv0, nv1);
      nvb = nv0;
    }
    stage_tile<Q, NPT>(tbuf + (buf ^ 1) * (Q * 32), in, plane, size_t(ny) * Lx, nvb + lane, more && nvb + lane < nv1, lane);
    cp_async_wait_prior();
    VN<NPT>* const slot = tbuf + buf * (Q * 32) + lane;
    const uint32_t v = vb + lane;
    const bool active = v < v1;
    const uint32_t x0 = v * NPT;
    VN<NPT> P[Q];
    VN<NPT> cur[Q];
#pragma unroll
    for (int i = 0; i < Q; ++i) cur[i] = slot[32 * source_plane<FLIP>(i)];
    collide_vec<Q, FLIP, ROWS, NPT>(a, keys, tables, tab, uint32_t(size_t(y) * Lx) + x0, t, cur, P, slot, bad);
    const uint32_t yp = y + 1 == Ly ? 0 : y + 1;
    const uint32_t ym = y == 0 ? Ly - 1 : y - 1;
    // streaming: velocity i lands in row y + dy of its plane, shifted by dx within it
    auto row_of = [&](int i) {
      const int dy = vel_dy<Q>(i);
      return out + i * plane + size_t(dy == 0 ? y : (dy > 0 ? yp : ym)) * Lx;
    };
    if (active) {
#pragma unroll
      for (int i = 0; i < Q; ++i)
        if (vel_dx<Q>(i) == 0) stv<NPT>(row_of(i) + x0, P[i].w);
    }
    // +x planes: each node's value moves one node right (the left neighbour's last
    // node); -x planes: one node left (the right neighbour's first node)
    uint32_t left[Q], right[Q], tile_first[Q];
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      if (vel_dx<Q>(i) > 0) {
        const uint32_t last = P[i].w[H - 1] >> 16;
        left[i] = __shfl_up_sync(kFull, last, 1);
        if (lane == 0) left[i] = carry[i];
        carry[i] = __shfl_sync(kFull, last, 31);
      } else if (vel_dx<Q>(i) < 0) {
        const uint32_t first = P[i].w[0] & 0xFFFFu;
        right[i] = __shfl_down_sync(kFull, first, 1);
        tile_first[i] = __shfl_sync(kFull, first, 0);
      }
    }
    if (lane == 31 && vb > v0) {
#pragma unroll
      for (int i = 0; i < Q; ++i)
        if (vel_dx<Q>(i) < 0) stv<NPT>(row_of(i) + (vb - 1) * NPT, shift_down(held[i], tile_first[i]).w);
    }
    if (active) {
      const bool seg_first = v == v0, seg_last = v + 1 == v1;
      if (!seg_first) {
#pragma unroll
        for (int i = 0; i < Q; ++i) {
          if (vel_dx<Q>(i) > 0) {
            // [l, p0 .. p_{NPT-2}]
            uint32_t o[H];
            o[0] = __byte_perm(left[i], P[i].w[0], 0x5410);
#pragma unroll
            for (int j = 1; j < H; ++j) o[j] = __byte_perm(P[i].w[j - 1], P[i].w[j], 0x5432);
            stv<NPT>(row_of(i) + x0, o);
          }
        }
      } else {
#pragma unroll
        for (int i = 0; i < Q; ++i) {
          uint16_t* const row = row_of(i);
          if (vel_dx<Q>(i) > 0) {
            // the segment's first +x slot belongs to the node left of the segment
            row[x0 + 1] = uint16_t(P[i].w[0]);
#pragma unroll
            for (int j = 1; j < H; ++j)
              *reinterpret_cast<uint32_t*>(row + x0 + 2 * j) = __byte_perm(P[i].w[j - 1], P[i].w[j], 0x5432);
          } else if (vel_dx<Q>(i) < 0) {
            // and this node's -x value belongs to that node's slot
            row[x0 == 0 ? Lx - 1 : x0 - 1] = uint16_t(P[i].w[0]);
          }
        }
      }
      if (seg_last) {
#pragma unroll
        for (int i = 0; i < Q; ++i) {
          uint16_t* const row = row_of(i);
          if (vel_dx<Q>(i) > 0) {
            // the segment's last +x value belongs to the first slot of the next segment
            row[x0 + NPT == Lx ? 0 : x0 + NPT] = uint16_t(P[i].w[H - 1] >> 16);
          } else if (vel_dx<Q>(i) < 0) {
            // [p1 .. p_{NPT-1}]: the last -x slot belongs to the node right of the segment
#pragma unroll
            for (int j = 0; j < H - 1; ++j)
              *reinterpret_cast<uint32_t*>(row + x0 + 2 * j) = __byte_perm(P[i].w[j], P[i].w[j + 1], 0x5432);
            row[x0 + NPT - 2] = uint16_t(P[i].w[H - 1] >> 16);
          }
        }
      } else if (lane < 31) {
#pragma unroll
        for (int i = 0; i < Q; ++i)
          if (vel_dx<Q>(i) < 0) stv<NPT>(row_of(i) + x0, shift_down(P[i], right[i]).w);
      } else {
#pragma unroll
        for (int i = 0; i < Q; ++i)
          if (vel_dx<Q>(i) < 0) held[i] = P[i];
      }
    }
    if (!more) break;
    if (!same) {
#pragma unroll
      for (int i = 0; i < Q; ++i) carry[i] = 0;
      g = g_next;
      y = ny;
      v0 = nv0;
      v1 = nv1;
    }
    vb = nvb;
    buf ^= 1;
  }
  cp_async_wait_all();  // the last (empty) group: nothing lands after the warp exits
  }
  if (bad) {
    note_overflow(a, fail, t);
    __threadfence();
    atomicOr(sync, kRunMark);
  }
  if (!RUN || step + 1 == T) break;
  __syncthreads();
  if (threadIdx.x == 0) {
    const unsigned long long v = run_barrier(sync, (step + 1) * gridDim.x);
    if (v == ~0ull) {
      note_gave_up(a, sync + 1);
      stop = 1;
    } else if (v >= kRunMark) {
      // a step overflowed: this one, or already the next one (a faster block's)
      stop = *reinterpret_cast<const volatile unsigned long long*>(fail) <= t;
    }
  }
  __syncthreads();
  if (stop) break;
  }
}

// Shapes (the autotuner's two candidates): one block per SM, so the 64 staged table
// rows exist once per SM; kNpt nodes per lane, kThreads threads, a multiple of 128 so
// that the four sub-partitions of an SM hold equally many warps.  Few warps with room
// for all their registers (16384^2 D2Q5, 8 nodes per lane, G node updates/s: 12 warps at up
// to 168 registers 162, 16 at 128 158.7, 20 at 96 157.2, all without spills; the pipes are as
// full in each, and more warps stage and stream beside one another).
constexpr int kRows = 64;
template <int SHAPE>
struct WarpShape;
template <>
struct WarpShape<0> {
  static constexpr int kNpt = 8;
  static constexpr int kThreads = 384;
};
template <>
struct WarpShape<1> {
  static constexpr int kNpt = 4;
  static constexpr int kThreads = 640;
};

// D2Q9 (nine planes, four Philox blocks and eleven draws per node): 4 nodes per lane, 384 or
// 512 threads (8192^2: 77.4 and 77.0 G node updates/s; 640, at 96 registers, spill: 59; 8 nodes
// per lane in 384 threads 70)
template <int Q, int SHAPE>
struct WarpShapeQ : WarpShape<SHAPE> {};
template <>
struct WarpShapeQ<9, 0> {
  static constexpr int kNpt = 4;
  static constexpr int kThreads = 384;
};
template <>
struct WarpShapeQ<9, 1> {
  static constexpr int kNpt = 4;
  static constexpr int kThreads = 512;
};

// tables, then two tile buffers of Q planes x 32 vectors per warp
template <int Q, int SHAPE>
constexpr size_t warp_smem() {
  using S = WarpShapeQ<Q, SHAPE>;
  return sizeof(uint2) * (Q == 9 ? 3 : 2) * kRows * kDevAliasCols +
         size_t(S::kThreads / 32) * 2 * Q * 32 * (2 * S::kNpt);
}

template <int Q, bool FLIP, int SHAPE, bool RUN>
const void* warp_kernel() {
  using S = WarpShapeQ<Q, SHAPE>;
  return reinterpret_cast<const void*>(step_warp_kernel<Q, FLIP, kRows, S::kNpt, S::kThreads, RUN>);
}

template <int Q, int SHAPE>
const void* warp_fn(bool flip, bool run) {
  if (run) return flip ? warp_kernel<Q, true, SHAPE, true>() : warp_kernel<Q, false, SHAPE, true>();
  return flip ? warp_kernel<Q, true, SHAPE, false>() : warp_kernel<Q, false, SHAPE, false>();
}

template <int Q, int SHAPE>
cudaError_t warp_attr() {
  cudaError_t e = cudaSuccess;
  for (bool flip : {false, true})
    for (bool run : {false, true})
      if (e == cudaSuccess)
        e = cudaFuncSetAttribute(warp_fn<Q, SHAPE>(flip, run), cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 int(warp_smem<Q, SHAPE>()));
  return e;
}

template <int Q, int SHAPE>
cudaError_t warp_launch(const StepArgs& a, uint16_t* buf0, uint16_t* buf1, uint32_t t, uint32_t T,
                        unsigned long long* fail, unsigned long long* sync, int grid, cudaStream_t s) {
  const void* fn = warp_fn<Q, SHAPE>(a.flip != 0, T > 1);
  StepArgs args = a;
  void* p[] = {&args, &buf0, &buf1, &t, &T, &fail, &sync};
  const dim3 threads(WarpShapeQ<Q, SHAPE>::kThreads);
  if (T == 1) return cudaLaunchKernel(fn, dim3(grid), threads, p, warp_smem<Q, SHAPE>(), s);
  const cudaError_t e = cudaMemsetAsync(sync, 0, sizeof(unsigned long long), s);
  if (e != cudaSuccess) return e;
  return cudaLaunchCooperativeKernel(fn, dim3(grid), threads, p, warp_smem<Q, SHAPE>(), s);
}

template <int Q>
void shape_of(int shape, uint32_t* npt, uint32_t* threads) {
  if (shape == 1) {
    *npt = WarpShapeQ<Q, 1>::kNpt;
    *threads = WarpShapeQ<Q, 1>::kThreads;
  } else {
    *npt = WarpShapeQ<Q, 0>::kNpt;
    *threads = WarpShapeQ<Q, 0>::kThreads;
  }
}

void shape_of(int Q, int shape, uint32_t* npt, uint32_t* threads) {
  if (Q == 9) shape_of<9>(shape, npt, threads);
  else shape_of<5>(shape, npt, threads);
}

}  // namespace

template <int Q>
static cudaError_t warp_attrs() {
  const cudaError_t e = warp_attr<Q, 0>();
  return e == cudaSuccess ? warp_attr<Q, 1>() : e;
}

cudaError_t prepare_step_warp_kernels(int Q) {
  return Q == 3 ? warp_attrs<3>() : Q == 5 ? warp_attrs<5>() : warp_attrs<9>();
}

uint32_t step_warp_width(int Q, int shape) {
  uint32_t npt, threads;
  shape_of(Q, shape, &npt, &threads);
  return npt;
}

// Blocks of a launch: one per SM, or fewer on lattices too small to give each warp a tile.
static uint32_t step_warp_grid(int Q, uint32_t Lx, uint32_t Ly, uint32_t sms, int shape) {
  uint32_t npt, threads;
  shape_of(Q, shape, &npt, &threads);
  const uint64_t cap = sms;
  const uint64_t warps = std::max<uint64_t>(1, uint64_t(Lx / npt) * Ly / 32);
  return uint32_t(std::min<uint64_t>(cap, (warps + threads / 32 - 1) / (threads / 32)));
}

cudaError_t launch_step_warp(int Q, int shape, const StepArgs& a, uint16_t* buf0, uint16_t* buf1, uint32_t t, uint32_t T,
                             unsigned long long* fail, unsigned long long* sync, uint32_t sms, cudaStream_t s) {
  const int grid = int(step_warp_grid(Q, a.Lx, a.Ly, sms, shape));
  if (Q == 3)
    return shape == 1 ? warp_launch<3, 1>(a, buf0, buf1, t, T, fail, sync, grid, s)
                      : warp_launch<3, 0>(a, buf0, buf1, t, T, fail, sync, grid, s);
  if (Q == 5)
    return shape == 1 ? warp_launch<5, 1>(a, buf0, buf1, t, T, fail, sync, grid, s)
                      : warp_launch<5, 0>(a, buf0, buf1, t, T, fail, sync, grid, s);
  return shape == 1 ? warp_launch<9, 1>(a, buf0, buf1, t, T, fail, sync, grid, s)
                    : warp_launch<9, 0>(a, buf0, buf1, t, T, fail, sync, grid, s);
}

}  // namespace ilg
