// The collision of one node per lane by a whole warp (any occupations):
// the node-parallel kernels' collision, where many nodes need more random words than
// the slot words.
//
// What bounds it: the ALU pipe (two cycles per warp instruction and sub-partition),
// then the wide products of Philox on the FMA-heavy pipe.  Per-lane loops over chunks
// and groups spend most of their issue slots on divergence and on branches per lane,
// so here every loop runs as often as the warp's neediest lane asks (a vote), and a
// lane that is done draws from row 0 of the table or masks its bits away: the same
// result without a branch.  The words beyond the slot words wait in a ring of K words
// per lane in shared memory (lane-interleaved, so no access conflicts), filled one
// Philox block at a time by all lanes together when one of them runs short.
//
// A vote costs some 40 cycles of latency and three issue slots, so few stand in a node's
// chain: one asks whether any occupation exceeds a chunk; behind it three are asked at once,
// the first block is made without asking, and the rest velocity (which holds the most in
// equilibrium) takes its further chunks by itself.  Against a vote for every block and a
// second chunk drawn for all velocities, us per step: D2Q5 1024^2 at 50 per velocity 25.5 /
// 27.5 (omega* = 0.5), 16.2 / 18.4 (0.1), 1501 x 777 at 100 44.8 / 52.2; D2Q9 1024^2 at 50
// 49.6 / 56.0; where nothing exceeds a chunk it is the same (D2Q5 768^2 at 10: 8.25) up to
// 5 % slower (rings of 8192 nodes at 10: 8.56 / 8.13).
#pragma once

#include <cstdint>

#include "ilg_device.cuh"

namespace ilg {

constexpr unsigned kFullWarp = 0xFFFFFFFFu;

// What is the same for every node of a launch (or of a lattice and step) in the first
// three Philox rounds (see StepKeys), and the two words an extension block's own part
// of them starts from.
template <int NB>
struct NodeKeys {
  StepKeys<NB> slot;
  uint32_t ext_c;  // round 2's x2 of extension block 0, without the block index
  uint32_t ext_e;  // round 3's x0 without the block's product
};

using WordKeys = NodeKeys<2>;  // D1Q3, D2Q5 (two slot blocks; D2Q9: four)

template <int NB = 2>
__device__ __forceinline__ NodeKeys<NB> word_keys(const StepArgs& a, uint32_t t) {
  constexpr uint32_t M0 = 0xD2511F53u, M1 = 0xCD9E8D57u;
  NodeKeys<NB> k;
  k.slot = step_keys<NB>(a, t);
  k.ext_c = uint32_t((uint64_t(M0) * t) >> 32) ^ kDevTagExt ^ a.rk[1];
  k.ext_e = uint32_t(uint64_t(M1) * a.replica) ^ a.rk[2];
  return k;
}

// Rounds 4..10 of a block whose words after round 3 are c.
__device__ __forceinline__ uint4 philox_tail(uint4 c, const uint32_t (&rk)[20]) {
#pragma unroll
  for (int r = 3; r < 10; ++r) {
    const uint64_t p0 = uint64_t(0xD2511F53u) * c.x;
    const uint64_t p1 = uint64_t(0xCD9E8D57u) * c.z;
    c = make_uint4(uint32_t(p1 >> 32) ^ c.y ^ rk[2 * r], uint32_t(p1), uint32_t(p0 >> 32) ^ c.w ^ rk[2 * r + 1],
                   uint32_t(p0));
  }
  return c;
}

// A node's slot words at a step, and its part of rounds 1-3.  They depend on the node and
// the step alone: a kernel that waits for the step before makes its first node's meanwhile.
template <int NB>
struct SlotWords {
  uint32_t W[4 * NB], r2h, r2l, p1l;
  template <class Keys>
  __device__ __forceinline__ void make(const Keys& k, const uint32_t (&rk)[20], uint32_t node) {
    const uint64_t P1 = uint64_t(0xD2511F53u) * (node ^ k.slot.A);
    const uint64_t R2 = uint64_t(0xCD9E8D57u) * (uint32_t(P1 >> 32) ^ k.slot.G);
    r2h = uint32_t(R2 >> 32);
    r2l = uint32_t(R2);
    p1l = uint32_t(P1);
#pragma unroll
    for (int b = 0; b < NB; ++b) {
      const uint4 v = philox_tail(make_uint4(r2h ^ k.slot.H[b], r2l, p1l ^ k.slot.I[b], k.slot.J[b]), rk);
      W[4 * b] = v.x;
      W[4 * b + 1] = v.y;
      W[4 * b + 2] = v.z;
      W[4 * b + 3] = v.w;
    }
  }
};

// The words of one node and step.  S: bytes between a lane's consecutive words in the
// ring (4 x the threads that share it), K: words per lane (a power of two).
template <uint32_t S, uint32_t K>
struct NodeWords {
  static_assert((K & (K - 1)) == 0 && (S & (S - 1)) == 0 && K >= 8, "a ring of whole blocks");
  static constexpr uint32_t kWrap = S * K - 1;
  unsigned char* ring;     // shared memory
  uint32_t rd, wr;         // byte positions of the next word to take and to write (unwrapped)
  uint32_t r2h, r2l, p1l;  // the node's part of rounds 1-3
  uint32_t blk;            // next extension block

  template <class Keys>
  __device__ __forceinline__ void begin(const Keys& k, unsigned char* ring_, uint32_t lane_off, uint32_t node) {
    const uint64_t P1 = uint64_t(0xD2511F53u) * (node ^ k.slot.A);
    const uint64_t R2 = uint64_t(0xCD9E8D57u) * (uint32_t(P1 >> 32) ^ k.slot.G);
    r2h = uint32_t(R2 >> 32);
    r2l = uint32_t(R2);
    p1l = uint32_t(P1);
    ring = ring_;
    rd = wr = lane_off;
    blk = 0;
  }
  template <class Keys>
  __device__ __forceinline__ uint4 slot(const Keys& k, const uint32_t (&rk)[20], int b) const {
    return philox_tail(make_uint4(r2h ^ k.slot.H[b], r2l, p1l ^ k.slot.I[b], k.slot.J[b]), rk);
  }
  template <int NB>
  __device__ __forceinline__ void begin(const SlotWords<NB>& w, unsigned char* ring_, uint32_t lane_off) {
    r2h = w.r2h;
    r2l = w.r2l;
    p1l = w.p1l;
    ring = ring_;
    rd = wr = lane_off;
    blk = 0;
  }
  // the next extension block into the ring
  template <class Keys>
  __device__ __forceinline__ void fill(const Keys& k, const uint32_t (&rk)[20]) {
    const uint64_t R1 = uint64_t(0xCD9E8D57u) * (k.ext_c ^ blk);
    const uint64_t P2 = uint64_t(0xD2511F53u) * (uint32_t(R1 >> 32) ^ k.ext_e);
    const uint4 b = philox_tail(make_uint4(r2h ^ uint32_t(R1) ^ rk[4], r2l, p1l ^ uint32_t(P2 >> 32) ^ rk[5], uint32_t(P2)), rk);
    uint32_t* p = reinterpret_cast<uint32_t*>(ring + (wr & kWrap));  // whole blocks: the four words do not wrap
    p[0] = b.x;
    p[S / 4] = b.y;
    p[2 * (S / 4)] = b.z;
    p[3 * (S / 4)] = b.w;
    wr += 4 * S;
    blk += 1;
  }
  // every lane has at least `bytes` of words afterwards (at most MAX words, MAX <= K - 4);
  // lanes with room fill together.  A lane without room has more than K - 8 words, so one
  // block is enough for four words in a ring of more than 8; in a ring of 8 the single test
  // gained nothing (rings of 256 nodes 0.85 instead of 0.83 us per step).
  template <uint32_t MAX, class Keys>
  __device__ __forceinline__ void ensure(const Keys& k, const uint32_t (&rk)[20], uint32_t bytes) {
    static_assert(MAX <= K - 4, "whole blocks must fit beside what is asked for");
    if constexpr (MAX <= 4 && K > 8) {
      if (__any_sync(kFullWarp, wr - rd < bytes)) {
        if (wr - rd <= (K - 4) * S) fill(k, rk);
      }
    } else {
      while (__any_sync(kFullWarp, wr - rd < bytes)) {
        if (wr - rd <= (K - 4) * S) fill(k, rk);
      }
    }
  }
  // the word `ahead` places after the next one
  __device__ __forceinline__ uint32_t peek(uint32_t ahead = 0) const {
    return *reinterpret_cast<const uint32_t*>(ring + ((rd + ahead * S) & kWrap));
  }
};

// Binomial(x, P) beyond its first chunk: chunks of 63 trials, each with the lane's next
// extension word; left = x - 63 (negative or zero: none).  A lane that is done draws from
// row 0: nothing.  Two chunks per pass; in a ring of 8 words (batches, whose occupations run
// up to 200 per velocity) four at a time while some lane has more than two left: 152 rings of
// 8192 nodes at 100 per velocity 21.7 instead of 22.1 us per step, at 10 8.43 / 8.55.  In the
// rings of 16 of the other kernels that gains beyond 100 per velocity only (D2Q5 1024^2 at 200
// 80.3 / 83.2) and costs 1 % at 50.
template <uint32_t S, uint32_t K, class Keys, class Tab>
__device__ __forceinline__ uint32_t more_chunks(NodeWords<S, K>& e, const Keys& k, const uint32_t (&rk)[20],
                                                const Tab& A, int32_t left) {
  uint32_t r = 0;
  if constexpr (K > 8) {
    while (__any_sync(kFullWarp, left > 0)) {
      e.template ensure<2>(k, rk, left > int32_t(kDevNmax) ? 2 * S : (left > 0 ? S : 0u));
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        r += A(uint32_t(__vimin_s32_relu(left, int32_t(kDevNmax))), e.peek());
        if (left > 0) e.rd += S;
        left -= int32_t(kDevNmax);
      }
    }
  } else {
    constexpr int32_t kN = int32_t(kDevNmax);
    const auto chunk = [&]() {
      r += A(uint32_t(__vimin_s32_relu(left, kN)), e.peek());
      if (left > 0) e.rd += S;
      left -= kN;
    };
    bool some = __any_sync(kFullWarp, left > 0);
    if (!some) return 0;
    while (__any_sync(kFullWarp, left > 2 * kN)) {
      e.template ensure<4>(k, rk, left > 2 * kN ? (left > 3 * kN ? 4 * S : 3 * S) : (left > kN ? 2 * S : (left > 0 ? S : 0u)));
#pragma unroll
      for (int u = 0; u < 4; ++u) chunk();
      some = __any_sync(kFullWarp, left > 0);
    }
    if (some) {
      e.template ensure<2>(k, rk, left > kN ? 2 * S : (left > 0 ? S : 0u));
      chunk();
      chunk();
    }
  }
  return r;
}

// Bits of c particles' two direction words, 32 particles at a time: the first words A, B,
// every further group the lane's next two extension words (a mask of no bits once a lane is
// done).  Returns the numbers of particles with A set, with both set, and with B alone.
struct BitCounts {
  uint32_t a, both, b;
};
template <uint32_t S, uint32_t K, class Keys>
__device__ __forceinline__ BitCounts count_bits(NodeWords<S, K>& e, const Keys& k, const uint32_t (&rk)[20], uint32_t c,
                                                uint32_t A, uint32_t B) {
  constexpr uint32_t kPass = 2;  // groups whose words (one block) are asked for at once
  int32_t left = int32_t(c);
  uint32_t mask = __funnelshift_lc(kFullWarp, 0u, uint32_t(left));
  left = max(left - 32, 0);
  A &= mask;
  B &= mask;
  BitCounts n{uint32_t(__popc(A)), uint32_t(__popc(A & B)), uint32_t(__popc(B & ~A))};
  const auto group = [&]() {
    mask = __funnelshift_lc(kFullWarp, 0u, uint32_t(left));
    A = e.peek() & mask;
    B = e.peek(1) & mask;
    n.a += __popc(A);
    n.both += __popc(A & B);
    n.b += __popc(B & ~A);
    if (left > 0) e.rd += 2 * S;
    left = max(left - 32, 0);
  };
  while (__any_sync(kFullWarp, left > 0)) {
    e.template ensure<2 * kPass>(k, rk, min(uint32_t(left + 31) >> 5, kPass) * (2 * S));
    group();
    for (uint32_t u = 1; u < kPass && __any_sync(kFullWarp, left > 0); ++u) group();
  }
  return n;
}

// The collision of one node per lane (m: its occupations after the flip, all zero for a
// lane without a node); all 32 lanes call it together.  The same words and results as
// collide() (D2Q9: collide9_general()).  ring: the block's ring of K words per thread in
// shared memory, lane_off: 4 x the thread's index; ta: D2Q9's axis-share table (others: any);
// made: the node's slot words, if they are there already.
// TABLES: every probability lies strictly between 0 and 1 and is drawn through its table
// (known outside the loop over nodes: the tests for the other cases would be made for every
// node).
template <int Q, uint32_t S, uint32_t K, bool TABLES, class Keys, class Tab>
__device__ __forceinline__ void collide_warp(const StepArgs& a, const Keys& k, const Tab& to, const Tab& tr, const Tab& ta,
                                             unsigned char* ring, uint32_t lane_off, uint32_t node,
                                             const uint32_t (&m)[Q], uint32_t (&out)[Q],
                                             const SlotWords<Q == 9 ? 4 : 2>* made = nullptr) {
  static_assert(K >= 4 + uint32_t(Q), "a word for each velocity beside the block being written");
  constexpr int NB = Q == 9 ? 4 : 2;
  constexpr int32_t kN = int32_t(kDevNmax);
  NodeWords<S, K> e;
  uint32_t W[4 * NB];
  if (made) {
    e.begin(*made, ring, lane_off);
#pragma unroll
    for (int i = 0; i < 4 * NB; ++i) W[i] = made->W[i];
  } else {
    e.begin(k, ring, lane_off, node);
#pragma unroll
    for (int b = 0; b < NB; ++b) {
      const uint4 v = e.slot(k, a.rk, b);
      W[4 * b] = v.x;
      W[4 * b + 1] = v.y;
      W[4 * b + 2] = v.z;
      W[4 * b + 3] = v.w;
    }
  }

  // thinning
  uint32_t r[Q], removed = 0;
  if (TABLES || a.omega_mode == kTable) {
    uint32_t most = m[1];
#pragma unroll
    for (int i = 2; i < Q; ++i) most = max(most, m[i]);
#pragma unroll
    for (int i = 0; i < Q; ++i) r[i] = to(min(m[i], kDevNmax), W[i]);
    if (__any_sync(kFullWarp, max(most, m[0]) > uint32_t(kN))) {
      const bool rest1 = __any_sync(kFullWarp, m[0] > uint32_t(kN)), move1 = __any_sync(kFullWarp, most > uint32_t(kN)),
                 move2 = __any_sync(kFullWarp, most > uint32_t(2 * kN));
      e.fill(k, a.rk);  // no lane has a word yet
      if (rest1) {
        // the rest velocity by itself: it holds the most in equilibrium, often alone
        const int32_t left = int32_t(m[0]) - kN;
        const bool two = __any_sync(kFullWarp, left > kN);
        r[0] += to(uint32_t(__vimin_s32_relu(left, kN)), e.peek());
        if (left > 0) e.rd += S;
        if (two) r[0] += more_chunks(e, k, a.rk, to, left - kN);
      }
      if (move1) {
        if (!move2) {
          // one more chunk at most: no loop
          uint32_t need = 0;
#pragma unroll
          for (int i = 1; i < Q; ++i) need += m[i] > uint32_t(kN) ? S : 0u;
          e.template ensure<Q - 1>(k, a.rk, need);
#pragma unroll
          for (int i = 1; i < Q; ++i) {
            r[i] += to(uint32_t(max(int32_t(m[i]) - kN, 0)), e.peek());
            if (m[i] > uint32_t(kN)) e.rd += S;
          }
        } else {
#pragma unroll
          for (int i = 1; i < Q; ++i) r[i] += more_chunks(e, k, a.rk, to, int32_t(m[i]) - kN);
        }
      }
    }
  } else {
#pragma unroll
    for (int i = 0; i < Q; ++i) r[i] = a.omega_mode == kAlways ? m[i] : 0u;
  }
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    out[i] = m[i] - r[i];
    removed += r[i];
  }

  // a share of x through a table: the first chunk with its slot word, then extension words
  auto share = [&](uint32_t mode, const Tab& A, uint32_t x, uint32_t slot) -> uint32_t {
    if (TABLES || mode == kTable) {
      const uint32_t s = A(min(x, kDevNmax), slot);
      return s + more_chunks(e, k, a.rk, A, int32_t(x) - kN);
    }
    return mode == kAlways ? x : 0u;
  };
  // share sent to rest
  const uint32_t to_rest = share(a.rest_mode, tr, removed, W[Q]);
  out[0] += to_rest;

  // directions of the moving particles, 32 at a time
  const uint32_t moving = removed - to_rest;
  if constexpr (Q == 3) {
    // one sign word per group
    constexpr uint32_t kPass = 4;
    int32_t left = int32_t(moving);
    uint32_t mask = __funnelshift_lc(kFullWarp, 0u, uint32_t(left));
    uint32_t minus = __popc(W[Q + 1] & mask);
    left = max(left - 32, 0);
    while (__any_sync(kFullWarp, left > 0)) {
      e.template ensure<kPass>(k, a.rk, min(uint32_t(left + 31) >> 5, kPass) * S);
      for (uint32_t u = 0; u < kPass && __any_sync(kFullWarp, left > 0); ++u) {
        mask = __funnelshift_lc(kFullWarp, 0u, uint32_t(left));
        minus += __popc(e.peek() & mask);
        if (left > 0) e.rd += S;
        left = max(left - 32, 0);
      }
    }
    out[1] += moving - minus;
    out[2] += minus;
  } else {
    // axis bit (0: x, 1: y), sign bit (0: +, 1: -); on D2Q9 of the axis particles
    const uint32_t axis = Q == 9 ? share(a.axis_mode, ta, moving, W[10]) : moving;
    const BitCounts n = count_bits(e, k, a.rk, axis, W[Q == 9 ? 11 : Q + 1], W[Q == 9 ? 12 : Q + 2]);
    out[1] += axis - n.a - n.b;
    out[2] += n.b;
    out[3] += n.a - n.both;
    out[4] += n.both;
    if constexpr (Q == 9) {
      // diagonal particles: x-sign bit, y-sign bit
      const uint32_t diag = moving - axis;
      const BitCounts d = count_bits(e, k, a.rk, diag, W[13], W[14]);
      out[5] += diag - d.a - d.b;
      out[6] += d.both;
      out[7] += d.b;
      out[8] += d.a - d.both;
    }
  }
}

}  // namespace ilg
