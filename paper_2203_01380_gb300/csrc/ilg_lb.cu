// Lattice Boltzmann comparator (Sec. IV, Eq. MRTLB) in double precision.
//
// With one rate omega^j for the odd (current) moments and one rate omega for the
// even non-conserved ones, the moment-space update splits by parity: the part of
// f - f^0 that is odd under v -> -v is exactly its projection on the odd moments,
// the even part its projection on the even ones (the transform matrix is
// orthonormal under the symmetric weights and every moment has a definite parity).
// So, per opposite pair (i, -i) with weight w_m and per rest velocity,
//   post_i  = omega w_m rho + a1 f_i + a2 f_-i,  a1,2 = ((1 - omega) +- (1 - omega^j)) / 2
//   post_0  = omega w_0 rho + (1 - omega) f_0
// then push-streaming to x + v_i.  It is computed in 64-bit integers (relax_fixed), where a
// node's values are of like size, and in double precision elsewhere.  No moment matrix appears;
// the oracle uses the matrix.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <string>
#include <vector>

#include "ilg_internal.h"
#include "ilg_sync.cuh"

namespace {

constexpr int kLbThreads = 256;
// threads of a step kernel's block: four blocks per SM, or (wide) one, whose loads run ahead and
// need the registers (D2Q5 1024^2, us per step: 1024 threads 13.3, 768 12.4, 512 12.6)
__host__ __device__ constexpr int lb_run_threads(int Q, bool wide) { return !wide ? 256 : (Q == 9 ? 512 : 768); }
constexpr uint32_t kLbMaxModes = 256;
constexpr int kLbModeThreads = 64;     // of a projection's blocks
constexpr int kLbClusterBlocks = 16;  // (beyond 8 a kernel opts in)
constexpr uint32_t kLbCols = 32;       // columns of a block of their sums (or kLbThreads)
constexpr uint32_t kLbFewRows = 8;
constexpr uint32_t kLbFirstModes = 64; // passed as a kernel argument
constexpr uint32_t kLbRowChunk = 64;   // rows per partial column sum
constexpr uint32_t kLbChunk = 4096;    // entries per partial of a projection

// The kernels read the planes of a pair (i, -i) exchanged where swap is set (1 - omega^j < 0):
// with the signs of a1's and a2's odd parts the odd part of f - f^0 then relaxes with
// |1 - omega^j|.
struct LbCoef {
  double cr;   // omega w_0
  double cm;   // omega w_m (moving, D2Q9: axis)
  double cd;   // D2Q9: omega w_diagonal
  double l2;   // 1 - omega
  double a1;   // ((1 - omega) + |1 - omega^j|) / 2
  double a2;   // ((1 - omega) - |1 - omega^j|) / 2
  // times 2^64: omega w_0 / 2, omega w_m, omega w_diagonal, |1 - omega| / 2, |1 - omega^j| / 2
  unsigned long long hr, hm, hd, he, ho;
  // what relax_fixed adds to the products with rho, and takes from those with a pair's difference
  unsigned long long more, less;
  int minus;   // 1 - omega < 0
  int swap;    // 1 - omega^j < 0
};

// ---- the relaxation on the integer pipes ----
// An SM has two fp64 lanes: a warp's fp64 operation takes 64 cycles of its sub-partition, and
// a D2Q5 node has 15 of them (9 with the density and its products in integers).  A 64-bit
// integer sum takes two instructions and the upper half of a 64-bit product five, so the
// whole node is relaxed in fixed point: the values shifted to the largest one's exponent
// (exact), sums exact, products to two units of 2^-61 of the largest value, and each result
// rounded once to 53 bits (the fp64 form rounds it three times).  A D2Q5 node takes 278 warp
// instructions per 32 nodes.  Us per step against nine fp64 operations per node with the
// density's sums and products in integers: D2Q5 1024^2 12.3 / 22.0 (the barrier, the loads'
// latency and the ALU pipe), 4096^2 215 / 317 (0.92 of the measured copy bandwidth), 16384^2
// 3.57 / 4.94 ms (0.88); D2Q9 1024^2 25.5 / 40.5.  Error after 200 steps of a sine against
// extended precision: D2Q5 5e-16 / 1.2e-14 of a value at the rates (1.8, 0.2).

// The upper half of a 128-bit product less 0 to 2 units, 1.25 on average.
__device__ __forceinline__ unsigned long long upper_product(unsigned long long a, unsigned long long b) {
  const uint32_t a0 = uint32_t(a), a1 = uint32_t(a >> 32), b0 = uint32_t(b), b1 = uint32_t(b >> 32);
  return static_cast<unsigned long long>(a1) * b1 + __umulhi(a0, b1) + __umulhi(a1, b0);
}

// False (and nothing else) unless all values are positive, of ordinary size and within 2^kRoom
// of one another, and the results between some 2^-5 of the largest value and four times it.
// MINUS: 1 - omega < 0.
template <int Q, bool MINUS>
__device__ __forceinline__ bool relax_fixed(const LbCoef& k, const double (&f)[Q], double (&post)[Q]) {
  using u64 = unsigned long long;
  constexpr int kRoom = Q == 3 ? 9 : (Q == 5 ? 8 : 7);  // Q 2^(53 + kRoom) < 2^64
  constexpr uint32_t kLeast = Q == 9 ? 1u << 22 : 1u << 24;  // times 2^32: a result's least size
  int e[Q], top = 0, low = 1 << 20;
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    e[i] = int(uint32_t(__double2hiint(f[i])) >> 20);  // with the sign bit: a negative value is above any limit
    top = max(top, e[i]);
    low = min(low, e[i]);
  }
  if (low < 64 || top > 1980 || top - low > kRoom) return false;
  u64 F[Q], rho = 0, V[Q];
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    const uint32_t hi = (uint32_t(__double2hiint(f[i])) & 0xFFFFFu) | 0x100000u;
    F[i] = ((u64(hi) << 32) | uint32_t(__double2loint(f[i]))) << (kRoom - top + e[i]);
    rho += F[i];
  }
  const auto even = [&](u64 c, u64 s) { return MINUS ? c - s : c + s; };
  const u64 half = even(upper_product(rho, k.hr) + k.more, upper_product(F[0], k.he));
  V[0] = 2 * half;
  u64 c = upper_product(rho, k.hm) + k.more;
#pragma unroll
  for (int i = 1; i < Q; i += 2) {
    if (Q == 9 && i == 5) c = upper_product(rho, k.hd) + k.more;
    const u64 B = even(c, upper_product(F[i] + F[i + 1], k.he));
    // (f_i - f_-i) |1 - omega^j| / 2 from the difference plus 2^62
    const u64 t = upper_product(F[i] - F[i + 1] + (1ull << 62), k.ho) - k.less;
    V[i] = B + t;
    V[i + 1] = B - t;
  }
  // (no sum reaches 2^64 but twice `half`; a negative result passes any limit)
  uint32_t least = uint32_t(V[0] >> 32), most = 0;
#pragma unroll
  for (int i = 1; i < Q; ++i) {
    least = min(least, uint32_t(V[i] >> 32));
    most = max(most, uint32_t(V[i] >> 32));
  }
  if (least < kLeast || most >= (1u << 31) || uint32_t(half >> 32) >= (1u << 30)) return false;
  const uint32_t scale = uint32_t(top - kRoom - 1) << 20;
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    // p >= 2 bits dropped, half a unit rounded up
    const uint32_t p = 11 - __clz(int(V[i] >> 32));
    const u64 r = V[i] + (1u << (p - 1));
    const uint32_t lo = __funnelshift_r(uint32_t(r), uint32_t(r >> 32), p);
    const uint32_t hi = (uint32_t(r >> 32) >> p) + scale + (p << 20);
    post[i] = __hiloint2double(int(hi), int(lo));
  }
  return true;
}

template <int Q>
__device__ __forceinline__ void relax(const LbCoef& k, const double (&f)[Q], double (&post)[Q]) {
  if (k.minus ? relax_fixed<Q, true>(k, f, post) : relax_fixed<Q, false>(k, f, post)) return;
  double rho = f[0] + f[1] + f[2];
  if constexpr (Q >= 5) rho = rho + f[3] + f[4];
  if constexpr (Q == 9) rho = rho + f[5] + f[6] + f[7] + f[8];
  post[0] = fma(k.l2, f[0], k.cr * rho);
#pragma unroll
  for (int i = 1; i < Q; i += 2) {
    const double c = (Q == 9 && i >= 5 ? k.cd : k.cm) * rho;
    post[i] = fma(k.a1, f[i], fma(k.a2, f[i + 1], c));
    post[i + 1] = fma(k.a1, f[i + 1], fma(k.a2, f[i], c));
  }
}

// T steps, one node per thread: load the Q planes, relax, push.  f0 holds the state, the
// steps alternate the buffers; a barrier of all blocks (a cooperative launch) separates them.
// sync[0]: barrier word, sync[1]: 1 once a wait gave up.
template <int Q, bool WIDE>
__global__ void __launch_bounds__(lb_run_threads(Q, WIDE), WIDE ? 1 : 4)
    lb_run_kernel(const __grid_constant__ LbCoef k, double* f0, double* f1, uint32_t Lx, uint32_t Ly, uint32_t T,
                  unsigned long long* sync) {
  __shared__ int stop;
  if (threadIdx.x == 0) stop = 0;
  const uint32_t nodes = Lx * Ly;
  const size_t plane = nodes;
  constexpr uint32_t threads = lb_run_threads(Q, WIDE);
  const uint32_t stride = gridDim.x * threads, stride_y = stride / Lx, stride_x = stride - stride_y * Lx;
  // Runs of 32 nodes go to the blocks in turn (wide blocks): what is left for the last pass then
  // lies on all SMs (700^2 7.0 instead of 7.7 us per step, 1024^2 12.2 / 12.3; D2Q9 500^2 6.8 /
  // 7.5).  With several narrow blocks on an SM it lies there anyway (300 x 200 2.68 / 2.63).
  const uint32_t lane = threadIdx.x & 31u, run = WIDE ? (threadIdx.x >> 5) * gridDim.x + blockIdx.x : (blockIdx.x * threads + threadIdx.x) >> 5;
  const uint32_t first = run * 32 + lane;
  const uint32_t y0 = first / Lx, x0 = first - y0 * Lx;
  for (uint32_t step = 0;; ++step) {
    const double* const in = (step & 1) ? f1 : f0;
    double* const out = (step & 1) ? f0 : f1;
    uint32_t x = x0, y = y0, node = first;
    const double* from[Q];
#pragma unroll
    for (int i = 0; i < Q; ++i) from[i] = in + (i == 0 || !k.swap ? i : (i & 1 ? i + 1 : i - 1)) * plane;
    // (through L2 only: another SM wrote these lines in the step before)
    double next[Q];
    const auto load = [&](uint32_t at) {
#pragma unroll
      for (int i = 0; i < Q; ++i) next[i] = __ldcg(from[i] + at);
    };
    if (WIDE && node < nodes) load(node);
    while (node < nodes) {
      double f[Q], post[Q];
      if (!WIDE) load(node);
#pragma unroll
      for (int i = 0; i < Q; ++i) f[i] = next[i];
      if (WIDE && nodes - node > stride) load(node + stride);
      relax<Q>(k, f, post);
      const uint32_t yp = y + 1 == Ly ? 0 : y + 1;
      const uint32_t ym = y == 0 ? Ly - 1 : y - 1;
      double* const o = out + node;  // row y starts at node - x
      const int64_t right = x + 1 == Lx ? -int64_t(x) : 1, left = x == 0 ? int64_t(Lx) - 1 : -1;
      o[0] = post[0];
      o[int64_t(plane) + right] = post[1];
      o[int64_t(2 * plane) + left] = post[2];
      if constexpr (Q >= 5) {
        double* const up = out + (size_t(yp) * Lx + x);
        double* const down = out + (size_t(ym) * Lx + x);
        up[3 * plane] = post[3];
        down[4 * plane] = post[4];
        if constexpr (Q == 9) {
          // diagonal pairs (+1,+1)/(-1,-1) and (+1,-1)/(-1,+1)
          up[int64_t(5 * plane) + right] = post[5];
          down[int64_t(6 * plane) + left] = post[6];
          down[int64_t(7 * plane) + right] = post[7];
          up[int64_t(8 * plane) + left] = post[8];
        }
      }
      if (nodes - node <= stride) break;  // (node + stride may pass 2^32)
      node += stride;
      x += stride_x;
      y += stride_y;
      if (x >= Lx) {
        x -= Lx;
        y += 1;
      }
    }
    if (step + 1 == T) break;
    __syncthreads();
    if (threadIdx.x == 0 && ilg::run_barrier(sync, (step + 1) * gridDim.x) == ~0ull) {
      atomicExch(sync + 1, 1ull);
      stop = 1;
    }
    __syncthreads();
    if (stop) break;
  }
}

// Several steps of a lattice that one cluster holds in its shared memory, a node per thread:
// block r keeps blockDim.x nodes' planes (two buffers; a power of two), a node's results go
// straight into the planes of the blocks that hold its neighbours, and the cluster's barrier
// separates the steps.  Bound: the latency of a node's relaxation and of the barrier.  Us per
// step, buffers in L2 with the cluster's barrier (to 4096 nodes) or the grid's / here: D1Q3 500
// nodes 1.16 / 0.48, 16384 1.90 / 1.27; D2Q5 64^2 1.55 / 0.73, 128^2 2.10 / 1.73; D2Q9 56 x 66
// 2.23 / 1.13, 90^2 2.61 / 1.66 (in blocks of 1024 threads 128^2 would take 3.30, on all SMs
// 2.59).
template <int Q, int MOST>
__global__ void __launch_bounds__(MOST, 1)
    lb_cluster_kernel(const __grid_constant__ LbCoef k, double* f0, double* f1, uint32_t Lx, uint32_t Ly, uint32_t T) {
  extern __shared__ double planes[];  // [buffer][velocity][thread]
  const uint32_t nodes = Lx * Ly, threads = blockDim.x, tid = threadIdx.x, node = blockIdx.x * threads + tid;
  const uint32_t buffer = Q * threads;
  const bool active = node < nodes;
  uint32_t dest[Q];  // where velocity i's results go in buffer 0
  {
    const uint32_t y = node / Lx, x = node - y * Lx;
    const uint32_t xs[3] = {x == 0 ? Lx - 1 : x - 1, x, x + 1 == Lx ? 0 : x + 1};
    const uint32_t ys[3] = {y == 0 ? Ly - 1 : y - 1, y, y + 1 == Ly ? 0 : y + 1};
    constexpr int dx[9] = {0, 1, -1, 0, 0, 1, -1, 1, -1}, dy[9] = {0, 0, 0, 1, -1, 1, -1, -1, 1};
    const uint32_t own = uint32_t(__cvta_generic_to_shared(planes)), log = 31 - __clz(int(threads));
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      if (active) planes[i * threads + tid] = __ldcg(f0 + (size_t(i) * nodes + node));
      const uint32_t d = active ? ys[1 + dy[i]] * Lx + xs[1 + dx[i]] : node;
      asm("mapa.shared::cluster.u32 %0, %1, %2;\n"
          : "=r"(dest[i])
          : "r"(own + 8 * (i * threads + (d & (threads - 1)))), "r"(d >> log));
    }
  }
  // every block has started: its planes are written by other blocks from here on
  ilg::cluster_arrive();
  ilg::cluster_wait();
  for (uint32_t step = 0; step < T; ++step) {
    const uint32_t in = (step & 1) * buffer, out = 8 * (buffer - in);
    if (active) {
      double f[Q], post[Q];
#pragma unroll
      for (int i = 0; i < Q; ++i) f[i] = planes[in + (i == 0 || !k.swap ? i : (i & 1 ? i + 1 : i - 1)) * threads + tid];
      relax<Q>(k, f, post);
#pragma unroll
      for (int i = 0; i < Q; ++i)
        asm volatile("st.shared::cluster.f64 [%0], %1;\n" ::"r"(dest[i] + out), "d"(post[i]) : "memory");
    }
    __syncwarp();
    ilg::cluster_arrive();
    ilg::cluster_wait();
  }
  double* const state = (T & 1) ? f1 : f0;
  if (active) {
#pragma unroll
    for (int i = 0; i < Q; ++i) state[size_t(i) * nodes + node] = planes[(T & 1) * buffer + i * threads + tid];
  }
}

// f_i(x, y) = lambda[cls_i * period + r], r the phase residue of the node.
template <int Q>
__global__ void __launch_bounds__(kLbThreads) lb_init_kernel(const double* __restrict__ lam, uint32_t period,
                                                            int axis, uint32_t mode, int weighted,
                                                            double* __restrict__ out, uint32_t Lx, uint32_t Ly) {
  const size_t plane = size_t(Lx) * Ly;
  for (size_t node = size_t(blockIdx.x) * blockDim.x + threadIdx.x; node < plane;
       node += size_t(gridDim.x) * blockDim.x) {
    const uint32_t y = uint32_t(node / Lx);
    const uint32_t x = uint32_t(node - size_t(y) * Lx);
    uint32_t r = 0;
    if (axis == 1) r = uint32_t((uint64_t(mode) * x) % period);
    else if (axis == 2) r = uint32_t((uint64_t(mode) * y) % period);
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      const uint32_t cls = !weighted || i == 0 ? 0u : (Q == 9 && i > 4 ? 2u : 1u);
      out[i * plane + node] = lam[cls * period + r];
    }
  }
}

// Row sums of rho: one block per row, strided accumulation, fixed tree.
template <int Q>
__global__ void __launch_bounds__(kLbThreads) lb_rowsum_kernel(const double* __restrict__ f, uint32_t Lx,
                                                              uint32_t Ly, double* __restrict__ row) {
  __shared__ double red[kLbThreads];
  const size_t plane = size_t(Lx) * Ly;
  for (uint32_t y = blockIdx.x; y < Ly; y += gridDim.x) {
    double s = 0.0;
    for (uint32_t x = threadIdx.x; x < Lx; x += blockDim.x) {
      const size_t at = size_t(y) * Lx + x;
      double n = f[at];
#pragma unroll
      for (int i = 1; i < Q; ++i) n += f[i * plane + at];
      s += n;
    }
    red[threadIdx.x] = s;
    __syncthreads();
    for (int h = kLbThreads / 2; h > 0; h >>= 1) {
      if (int(threadIdx.x) < h) red[threadIdx.x] += red[threadIdx.x + h];
      __syncthreads();
    }
    if (threadIdx.x == 0) row[y] = red[0];
    __syncthreads();
  }
}

// Compensated accumulator: value s plus error term e (Knuth's two-sum; exact
// product errors through fma).  Round-to-nearest intrinsics keep the compiler from
// contracting the error-free transformations.
struct Acc {
  double s = 0.0, e = 0.0;
  __device__ void add(double v) {
    const double t = __dadd_rn(s, v);
    const double bp = __dsub_rn(t, s);
    e = __dadd_rn(e, __dadd_rn(__dsub_rn(s, __dsub_rn(t, bp)), __dsub_rn(v, bp)));
    s = t;
  }
  __device__ void add_product(double a, double b) {
    const double p = __dmul_rn(a, b);
    add(p);
    e = __dadd_rn(e, fma(a, b, -p));
  }
  __device__ void merge(const Acc& o) {
    add(o.s);
    e = __dadd_rn(e, o.e);
  }
};

// Fixed-order block reduction of the threads' accumulators (the same tree for
// every launch shape with N threads).
template <int N>
__device__ Acc block_acc(Acc a, double* ss, double* se) {
  ss[threadIdx.x] = a.s;
  se[threadIdx.x] = a.e;
  __syncthreads();
  for (int h = N / 2; h > 0; h >>= 1) {
    if (int(threadIdx.x) < h) {
      a.merge(Acc{ss[threadIdx.x + h], se[threadIdx.x + h]});
      ss[threadIdx.x] = a.s;
      se[threadIdx.x] = a.e;
    }
    __syncthreads();
  }
  const Acc r{ss[0], se[0]};
  __syncthreads();
  return r;
}

// True in every thread of the last of `blocks` blocks to come here (which sees what the
// others wrote, through L2); it leaves the counter at zero for the next launch.
__device__ bool last_block(uint32_t* counter, uint32_t blocks) {
  __shared__ bool last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) {
    last = atomicAdd(counter, 1u) == blocks - 1;
    if (last) *counter = 0;
  }
  __syncthreads();
  __threadfence();
  return last;
}

// Column sums of rho: a block adds kLbRowChunk rows of COLS columns, every kLbThreads / COLS-th
// part of the rows in other warps (one thread for all 64 rows waited 43 us for its loads on
// a 64 x 64 lattice, with its mass and one mode 95 us, here 58), the last block of the
// columns adds those partial sums, in a fixed order each, and, with mass != NULL (at most
// kLbChunk columns), the last block of all the columns: one launch instead of four.  Bound
// on small lattices: the launch and the loads' latency; on large ones the state's bytes.
template <int Q, uint32_t COLS>
__global__ void __launch_bounds__(kLbThreads) lb_col_kernel(const double* __restrict__ f, uint32_t Lx, uint32_t Ly,
                                                           double* __restrict__ part, double* __restrict__ col,
                                                           uint32_t* __restrict__ count, double* __restrict__ mass) {
  constexpr uint32_t kGroups = kLbThreads / COLS, kRows = kLbRowChunk / kGroups;
  __shared__ double ss[kLbThreads], se[kLbThreads];
  const uint32_t c = threadIdx.x % COLS, g = threadIdx.x / COLS;
  const uint32_t x = blockIdx.x * COLS + c;
  const size_t plane = size_t(Lx) * Ly;
  const auto groups_sum = [&](double v) {  // (valid in the first group)
    if constexpr (kGroups > 1) {
      ss[threadIdx.x] = v;
      __syncthreads();
#pragma unroll
      for (uint32_t i = 1; i < kGroups; ++i) v += ss[(threadIdx.x + i * COLS) % kLbThreads];
      __syncthreads();
    }
    return v;
  };
  double s = 0.0;
  const uint32_t y0 = blockIdx.y * kLbRowChunk + g * kRows;
  if (x < Lx) {
#pragma unroll 8
    for (uint32_t y = y0; y < min(y0 + kRows, Ly); ++y) {
      const double* const p = f + (size_t(y) * Lx + x);
      double n = p[0];
#pragma unroll
      for (int i = 1; i < Q; ++i) n += p[i * plane];
      s += n;
    }
  }
  s = groups_sum(s);
  if (gridDim.y > 1) {
    if (g == 0 && x < Lx) part[size_t(blockIdx.y) * Lx + x] = s;
    if (!last_block(count + blockIdx.x, gridDim.y)) return;
    s = 0.0;
    if (x < Lx) {
#pragma unroll 4
      for (uint32_t i = g; i < gridDim.y; i += kGroups) s += __ldcg(part + size_t(i) * Lx + x);
    }
    s = groups_sum(s);
  }
  if (g == 0 && x < Lx) col[x] = s;
  if (!mass || !last_block(count + gridDim.x, gridDim.x)) return;
  Acc a;
  for (uint32_t i = threadIdx.x; i < Lx; i += kLbThreads) a.add(__ldcg(col + i));
  const Acc r = block_acc<kLbThreads>(a, ss, se);
  if (threadIdx.x == 0) *mass = r.s + r.e;
}

// Partial sums over chunks of kLbChunk consecutive entries; part[c] = (s, e).
__global__ void __launch_bounds__(kLbThreads) lb_mass_partial_kernel(const double* __restrict__ col, uint32_t Lx,
                                                                    double2* __restrict__ part) {
  __shared__ double ss[kLbThreads], se[kLbThreads];
  const uint32_t x0 = blockIdx.x * kLbChunk;
  const uint32_t x1 = x0 + kLbChunk < Lx ? x0 + kLbChunk : Lx;
  Acc a;
  for (uint32_t x = x0 + threadIdx.x; x < x1; x += kLbThreads) a.add(col[x]);
  const Acc r = block_acc<kLbThreads>(a, ss, se);
  if (threadIdx.x == 0) part[blockIdx.x] = make_double2(r.s, r.e);
}

// The first modes of a call travel with the launch, without a copy of their own.
struct LbModes {
  int32_t m[2 * kLbFirstModes];
};

// Entries per block of a projection: one per thread while that makes at most 256 blocks (the
// sines and cosines in double precision bound it: 1024 entries in one block of 256 threads
// took 20 us), at most kLbChunk.
__host__ __device__ inline uint32_t lb_mode_chunk(uint32_t L) {
  if (L > 256u * kLbChunk) return kLbChunk;
  return ((L + 255) / 256 + kLbModeThreads - 1) / kLbModeThreads * kLbModeThreads;
}

// Blocks of a projection along any side of at most maxL entries (a side just past a multiple
// of 256 kLbModeThreads has fewer than a somewhat shorter one).
inline uint32_t lb_mode_blocks(uint32_t maxL) {
  return maxL > 256u * kLbChunk ? (maxL + kLbChunk - 1) / kLbChunk
                                : std::min((maxL + kLbModeThreads - 1) / kLbModeThreads, 256u);
}

// Block (c, j): chunk c of mode j; part[(2j) P + c] = re, part[(2j+1) P + c] = im, and
// the last block of a mode adds its P <= gridDim.x partials in a fixed order into
// out[1 + 2 j], out[2 + 2 j].  The mean M / L comes from out[0] (the mass).  modes: NULL for
// those in `first`.
__global__ void __launch_bounds__(kLbModeThreads) lb_mode_kernel(const double* __restrict__ col, const double* __restrict__ row,
                                                            uint32_t Lx, uint32_t Ly, const __grid_constant__ LbModes first,
                                                            const int32_t* __restrict__ modes, double* __restrict__ out,
                                                            double2* __restrict__ part, uint32_t* __restrict__ count) {
  __shared__ double ss[kLbModeThreads], se[kLbModeThreads];
  const uint32_t j = blockIdx.y;
  const int32_t mx = modes ? modes[2 * j] : first.m[2 * j], my = modes ? modes[2 * j + 1] : first.m[2 * j + 1];
  const bool along_x = mx != 0;
  const uint32_t L = along_x ? Lx : Ly;
  const uint32_t chunk = lb_mode_chunk(L), P = (L + chunk - 1) / chunk;
  if (blockIdx.x >= P) return;
  const double* C = along_x ? col : row;
  const int64_t mr = along_x ? mx : my;
  const uint64_t mode = uint64_t(((mr % int64_t(L)) + int64_t(L)) % int64_t(L));
  const double mean = out[0] / double(L);
  const uint32_t x0 = blockIdx.x * chunk;
  const uint32_t x1 = x0 + chunk < L ? x0 + chunk : L;
  Acc re, im;
  for (uint32_t x = x0 + threadIdx.x; x < x1; x += kLbModeThreads) {
    const uint64_t r = (mode * x) % L;
    double sn, cs;
    sincospi(2.0 * double(r) / double(L), &sn, &cs);
    const double d = C[x] - mean;
    re.add_product(cs, d);
    im.add_product(sn, d);
  }
  Acc a = block_acc<kLbModeThreads>(re, ss, se);
  Acc b = block_acc<kLbModeThreads>(im, ss, se);
  if (P > 1) {
    double2* const pr = part + size_t(2 * j) * gridDim.x;
    double2* const pi = pr + gridDim.x;
    if (threadIdx.x == 0) {
      pr[blockIdx.x] = make_double2(a.s, a.e);
      pi[blockIdx.x] = make_double2(b.s, b.e);
    }
    if (!last_block(count + j, P)) return;
    re = im = Acc{};
    for (uint32_t c = threadIdx.x; c < P; c += kLbModeThreads) {
      const double2 u = __ldcg(pr + c), v = __ldcg(pi + c);
      re.merge(Acc{u.x, u.y});
      im.merge(Acc{v.x, v.y});
    }
    a = block_acc<kLbModeThreads>(re, ss, se);
    b = block_acc<kLbModeThreads>(im, ss, se);
  }
  if (threadIdx.x == 0) {
    out[1 + 2 * j] = a.s + a.e;
    out[2 + 2 * j] = b.s + b.e;
  }
}

// Combines part[0 .. P) in a fixed order into *out (one block).
__global__ void __launch_bounds__(kLbThreads) lb_combine_kernel(const double2* __restrict__ part, uint32_t P,
                                                               double* __restrict__ out) {
  __shared__ double ss[kLbThreads], se[kLbThreads];
  Acc a;
  for (uint32_t c = threadIdx.x; c < P; c += kLbThreads) {
    const double2 v = part[c];
    a.merge(Acc{v.x, v.y});
  }
  const Acc r = block_acc<kLbThreads>(a, ss, se);
  if (threadIdx.x == 0) *out = r.s + r.e;
}

}  // namespace

struct ilg_lb {
  ilg_lb_params p{};
  int Q = 3;
  uint32_t Ly = 1;
  size_t nodes = 0;
  cudaStream_t stream = nullptr;
  int sms = 1;
  double* f[2] = {nullptr, nullptr};
  int cur = 0;
  uint64_t t = 0;
  bool has_state = false;
  LbCoef coef{};
  uint32_t chunks = 1;
  double2* d_red = nullptr;              // projection partials, 2 kLbMaxModes x chunks
  // one allocation: [0] barrier word of a several-step launch, [1] a wait gave up, then these
  unsigned long long* d_sync = nullptr;
  double* d_out = nullptr;               // mass, then re and im of each mode
  uint32_t* d_count = nullptr;           // arrivals: kLbMaxModes, then the column blocks and one; zero between launches
  int32_t* d_modes = nullptr;            // 2 kLbMaxModes
  double* d_col = nullptr;               // Lx
  double* d_row = nullptr;               // Ly
  double* d_part = nullptr;              // chunks x Lx partial column sums
  unsigned long long h_sync = 0;         // sync[1] as read back with the last results
  bool waits = false;                    // several-step launches since sync[1] was read
  int run_blocks = 0;                    // resident blocks of the step kernel
  std::string err;
};

namespace {

ilg_status lb_fail(ilg_lb* b, ilg_status s, const std::string& msg) {
  if (b) b->err = msg;
  else ilg::set_context_free_error(msg);
  return s;
}

ilg_status lb_cuda_fail(ilg_lb* b, cudaError_t e, const char* what) {
  return lb_fail(b, e == cudaErrorMemoryAllocation ? ILG_E_OOM : ILG_E_CUDA,
                 std::string(what) + ": " + cudaGetErrorString(e));
}

#define LB_CUDA(b, call, what)                             \
  do {                                                     \
    cudaError_t e_ = (call);                               \
    if (e_ != cudaSuccess) return lb_cuda_fail(b, e_, what); \
  } while (0)

// The gas's parameters that define the same lattice and initial means.
ilg_params as_gas(const ilg_lb_params& p) {
  ilg_params g{};
  g.lattice = p.lattice;
  g.Lx = p.Lx;
  g.Ly = p.Ly;
  g.mode_mx = p.mode_mx;
  g.mode_my = p.mode_my;
  g.init_weighted = p.init_weighted;
  g.n0 = p.n0;
  g.amp = p.amp;
  g.omega_eff = 1.0;
  g.theta = p.theta;
  return g;
}

int lb_grid(const ilg_lb* b) {
  const size_t blocks = (b->nodes + kLbThreads - 1) / kLbThreads;
  const size_t cap = size_t(b->sms) * (2048 / kLbThreads);
  return int(blocks < cap ? blocks : cap);
}

template <bool WIDE>
const void* lb_run_of(int Q) {
  return Q == 3   ? reinterpret_cast<const void*>(lb_run_kernel<3, WIDE>)
         : Q == 5 ? reinterpret_cast<const void*>(lb_run_kernel<5, WIDE>)
                  : reinterpret_cast<const void*>(lb_run_kernel<9, WIDE>);
}

// most threads of a cluster's block
int lb_cluster_threads(int Q) { return Q == 9 ? 512 : 1024; }

const void* lb_cluster_fn(int Q, int threads) {
  if (threads > 512)
    return Q == 3 ? reinterpret_cast<const void*>(lb_cluster_kernel<3, 1024>)
                  : reinterpret_cast<const void*>(lb_cluster_kernel<5, 1024>);
  return Q == 3   ? reinterpret_cast<const void*>(lb_cluster_kernel<3, 512>)
         : Q == 5 ? reinterpret_cast<const void*>(lb_cluster_kernel<5, 512>)
                  : reinterpret_cast<const void*>(lb_cluster_kernel<9, 512>);
}
size_t lb_cluster_smem(int Q, int threads) { return sizeof(double) * 2 * Q * threads; }

// Lattices of more nodes than this per SM: one wide block per SM, its threads' next values
// loaded while the present ones relax.  Us per step, narrow / wide: D2Q5 350^2 3.85 / 4.09,
// 400^2 5.08 / 4.25, 700^2 8.57 / 7.71, 1024^2 13.9 / 12.3; D1Q3 2^20 9.80 / 8.33; D2Q9 700^2
// 13.6 / 11.5.
constexpr size_t kLbWideNodesPerSm = 1024;
bool lb_wide(const ilg_lb* b) { return b->nodes > kLbWideNodesPerSm * b->sms; }
int lb_threads(const ilg_lb* b) { return lb_run_threads(b->Q, lb_wide(b)); }
const void* lb_run_fn(const ilg_lb* b) { return lb_wide(b) ? lb_run_of<true>(b->Q) : lb_run_of<false>(b->Q); }

bool lb_fits_cluster(const ilg_lb* b) { return b->nodes <= size_t(kLbClusterBlocks) * lb_cluster_threads(b->Q); }

// Several steps as one cluster; false where there is no room for it (SMs reserved elsewhere).
bool lb_launch_cluster(const ilg_lb* b, void** args) {
  // many small blocks: as many SMs as there are
  uint32_t threads = 64, blocks = 1;
  while (size_t(kLbClusterBlocks) * threads < b->nodes) threads *= 2;
  while (size_t(blocks) * threads < b->nodes) blocks *= 2;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr = {};
  attr.id = cudaLaunchAttributeClusterDimension;
  attr.val.clusterDim.x = blocks;
  attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
  cfg.gridDim = dim3(blocks);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = lb_cluster_smem(b->Q, int(threads));
  cfg.stream = b->stream;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  if (cudaLaunchKernelExC(&cfg, lb_cluster_fn(b->Q, int(threads)), args) == cudaSuccess) return true;
  cudaGetLastError();
  return false;
}

const void* lb_col_fn(int Q, bool wide) {
  if (wide)
    return Q == 3   ? reinterpret_cast<const void*>(lb_col_kernel<3, kLbThreads>)
           : Q == 5 ? reinterpret_cast<const void*>(lb_col_kernel<5, kLbThreads>)
                    : reinterpret_cast<const void*>(lb_col_kernel<9, kLbThreads>);
  return Q == 3   ? reinterpret_cast<const void*>(lb_col_kernel<3, kLbCols>)
         : Q == 5 ? reinterpret_cast<const void*>(lb_col_kernel<5, kLbCols>)
                  : reinterpret_cast<const void*>(lb_col_kernel<9, kLbCols>);
}

// v 2^bits, v not negative and the result below 2^65: exact but for bits below 1
unsigned __int128 scaled(double v, int bits) { return static_cast<unsigned __int128>(std::ldexp(v, bits)); }

// A bounded wait between the blocks of a several-step launch gave up (read back with the
// results): the buffers hold parts of different steps.
ilg_status lb_gave_up(ilg_lb* b) {
  b->has_state = false;
  b->h_sync = 0;
  b->waits = false;
  cudaMemsetAsync(b->d_sync, 0, 2 * sizeof(unsigned long long), b->stream);
  cudaStreamSynchronize(b->stream);
  return lb_fail(b, ILG_E_TIMEOUT, "a wait between the blocks of a several-step launch gave up: the state is lost");
}

// A fresh state: a wait that gave up in earlier steps, not read back yet, does not concern it.
cudaError_t lb_forget_waits(ilg_lb* b) {
  b->h_sync = 0;
  if (!b->waits) return cudaSuccess;
  b->waits = false;
  return cudaMemsetAsync(b->d_sync, 0, 2 * sizeof(unsigned long long), b->stream);  // behind those steps
}

}  // namespace

extern "C" {

ilg_status ilg_lb_create(const ilg_lb_params* params, void* stream, ilg_lb** out) {
  if (!out) return lb_fail(nullptr, ILG_E_INVALID, "out is NULL");
  *out = nullptr;
  if (!params) return lb_fail(nullptr, ILG_E_INVALID, "params is NULL");
  const ilg_lb_params& p = *params;
  const std::string why = ilg::validate_params(as_gas(p));
  if (!why.empty()) return lb_fail(nullptr, ILG_E_INVALID, why);
  if (!(p.omega_j >= 0.0 && p.omega_j <= 2.0)) return lb_fail(nullptr, ILG_E_INVALID, "omega_j must lie in [0, 2]");
  if (!(p.omega >= 0.0 && p.omega <= 2.0)) return lb_fail(nullptr, ILG_E_INVALID, "omega must lie in [0, 2]");
  ilg_lb* b = new ilg_lb();
  b->p = p;
  b->Q = p.lattice == ILG_D1Q3 ? 3 : (p.lattice == ILG_D2Q5 ? 5 : 9);
  b->Ly = p.lattice == ILG_D1Q3 ? 1 : p.Ly;
  b->p.Ly = b->Ly;
  b->nodes = size_t(p.Lx) * b->Ly;
  b->stream = static_cast<cudaStream_t>(stream);
  double w[9];
  ilg::weights(p.lattice, p.theta, w);
  LbCoef& k = b->coef;
  k = LbCoef{};
  k.minus = p.omega > 1.0;
  k.swap = p.omega_j > 1.0;
  const double lj = k.swap ? p.omega_j - 1.0 : 1.0 - p.omega_j;
  k.cr = p.omega * w[0];
  k.cm = p.omega * w[1];
  k.cd = b->Q == 9 ? p.omega * w[5] : 0.0;
  k.l2 = 1.0 - p.omega;
  k.a1 = 0.5 * (k.l2 + lj);
  k.a2 = 0.5 * (k.l2 - lj);
  // the same weights and rates in fixed point, exact but for the last bit of the products
  using u128 = unsigned __int128;
  const u128 half = scaled(p.omega, 63), one = u128(1) << 63;
  k.hr = static_cast<unsigned long long>((half * scaled(w[0], 64)) >> 64);
  k.hm = static_cast<unsigned long long>((half * scaled(w[1], 64)) >> 63);
  k.hd = b->Q == 9 ? static_cast<unsigned long long>((half * scaled(w[5], 64)) >> 63) : 0ull;
  k.he = static_cast<unsigned long long>(k.minus ? half - one : one - half);
  const u128 hj = scaled(p.omega_j, 63);
  k.ho = static_cast<unsigned long long>(k.swap ? hj - one : one - hj) & ~3ull;  // its product with 2^62 is whole
  // a product with a factor lacks about one unit
  const unsigned long long lacks = k.he != 0, odd = k.ho != 0;
  k.more = (k.hm != 0) + (k.minus ? 0 - lacks : lacks);
  k.less = (k.ho >> 2) - odd;
  b->chunks = (b->Ly + kLbRowChunk - 1) / kLbRowChunk;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&b->sms, cudaDevAttrMultiProcessorCount, dev);
  const size_t bytes = sizeof(double) * b->Q * b->nodes;
  if (e == cudaSuccess) e = ilg::dev_alloc(&b->f[0], bytes);
  if (e == cudaSuccess) e = ilg::dev_alloc(&b->f[1], bytes);
  const uint32_t maxL = p.Lx > b->Ly ? p.Lx : b->Ly;
  if (e == cudaSuccess) e = ilg::dev_alloc(&b->d_red, sizeof(double2) * 2 * kLbMaxModes * lb_mode_blocks(maxL));
  // one allocation: what has to be zero, then the modes and the sums
  const size_t words = 2 + 1 + 2 * kLbMaxModes, counters = kLbMaxModes + (p.Lx + kLbCols - 1) / kLbCols + 1;
  const size_t clear = words + (counters + 1) / 2;
  const size_t all = clear + kLbMaxModes + p.Lx + size_t(b->Ly) + size_t(b->chunks) * p.Lx;
  if (e == cudaSuccess) e = ilg::dev_alloc(&b->d_sync, sizeof(unsigned long long) * all);
  if (e == cudaSuccess) {
    b->d_out = reinterpret_cast<double*>(b->d_sync + 2);
    b->d_count = reinterpret_cast<uint32_t*>(b->d_sync + words);
    b->d_modes = reinterpret_cast<int32_t*>(b->d_sync + clear);
    b->d_col = reinterpret_cast<double*>(b->d_sync + clear + kLbMaxModes);
    b->d_row = b->d_col + p.Lx;
    b->d_part = b->d_row + b->Ly;
    e = cudaMemsetAsync(b->d_sync, 0, sizeof(unsigned long long) * clear, b->stream);
  }
  int per_sm = 0;
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, lb_run_fn(b), lb_threads(b), 0);
  if (e == cudaSuccess && lb_fits_cluster(b)) {
    for (const int threads : {512, lb_cluster_threads(b->Q)}) {
      const void* f = lb_cluster_fn(b->Q, threads);
      if (e == cudaSuccess) e = cudaFuncSetAttribute(f, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
      if (e == cudaSuccess)
        e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, int(lb_cluster_smem(b->Q, threads)));
    }
  }
  if (e != cudaSuccess) {
    ilg_lb_destroy(b);
    return lb_cuda_fail(nullptr, e, "ilg_lb_create");
  }
  b->run_blocks = int(std::min<size_t>(size_t(per_sm) * b->sms, (b->nodes + lb_threads(b) - 1) / lb_threads(b)));
  *out = b;
  return ILG_OK;
}

ilg_status ilg_lb_destroy(ilg_lb* b) {
  if (!b) return ILG_E_INVALID;
  if (b->f[0] || b->f[1]) cudaStreamSynchronize(b->stream);
  cudaFree(b->f[0]);
  cudaFree(b->f[1]);
  cudaFree(b->d_red);
  cudaFree(b->d_sync);
  delete b;
  return ILG_OK;
}

const char* ilg_lb_last_error(const ilg_lb* b) { return b ? b->err.c_str() : ilg_last_error(nullptr); }

// Sec. IV, Eq. omegaj: with the flip (omega_eff > 1) the collision fraction is
// omega* = 2 - omega_eff; the current then relaxes with omega^j = 2 - omega* and the
// even moments with omega*.  Without the flip every non-conserved moment relaxes with
// omega_eff.
ilg_status ilg_lb_rates(double omega_eff, double* omega_j, double* omega) {
  if (!omega_j || !omega || !(omega_eff > 0.0 && omega_eff <= 2.0)) {
    ilg::set_context_free_error("ilg_lb_rates: omega_eff must lie in (0, 2] and the outputs be non-NULL");
    return ILG_E_INVALID;
  }
  *omega_j = omega_eff;
  *omega = omega_eff > 1.0 ? 2.0 - omega_eff : omega_eff;
  return ILG_OK;
}

ilg_status ilg_lb_init(ilg_lb* b) {
  if (!b) return ILG_E_INVALID;
  const ilg_params g = as_gas(b->p);
  const uint32_t period = ilg::initial_period(g);
  const int classes = b->p.init_weighted ? (b->Q == 9 ? 3 : 2) : 1;
  std::vector<double> lam(size_t(classes) * period);
  for (int c = 0; c < classes; ++c)
    for (uint32_t r = 0; r < period; ++r) {
      const double v = ilg::initial_mean(g, b->Q, c, r, period);
      if (!(v >= 0.0) || v > ilg::kMaxMean)
        return lb_fail(b, ILG_E_INVALID, "initial mean " + std::to_string(v) + " outside [0, 700]");
      lam[size_t(c) * period + r] = v;
    }
  int axis = 0;
  uint32_t mode = 0;
  if (period > 1) {
    const bool along_x = b->p.mode_mx != 0;
    const int64_t L = period, m = along_x ? b->p.mode_mx : b->p.mode_my;
    axis = along_x ? 1 : 2;
    mode = uint32_t(((m % L) + L) % L);
  }
  LB_CUDA(b, lb_forget_waits(b), "lattice Boltzmann init");
  double* d_lam = nullptr;
  LB_CUDA(b, ilg::dev_alloc(&d_lam, sizeof(double) * lam.size()), "cudaMalloc");
  cudaError_t e = cudaMemcpyAsync(d_lam, lam.data(), sizeof(double) * lam.size(), cudaMemcpyHostToDevice, b->stream);
  if (e == cudaSuccess) {
    if (b->Q == 3)
      lb_init_kernel<3><<<lb_grid(b), kLbThreads, 0, b->stream>>>(d_lam, period, axis, mode, b->p.init_weighted,
                                                                  b->f[b->cur], b->p.Lx, b->Ly);
    else if (b->Q == 5)
      lb_init_kernel<5><<<lb_grid(b), kLbThreads, 0, b->stream>>>(d_lam, period, axis, mode, b->p.init_weighted,
                                                                  b->f[b->cur], b->p.Lx, b->Ly);
    else
      lb_init_kernel<9><<<lb_grid(b), kLbThreads, 0, b->stream>>>(d_lam, period, axis, mode, b->p.init_weighted,
                                                                  b->f[b->cur], b->p.Lx, b->Ly);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaStreamSynchronize(b->stream);
  cudaFree(d_lam);
  if (e != cudaSuccess) return lb_cuda_fail(b, e, "lattice Boltzmann init");
  b->t = 0;
  b->has_state = true;
  return ILG_OK;
}

ilg_status ilg_lb_set_state(ilg_lb* b, const double* host, size_t n, uint64_t t) {
  if (!b) return ILG_E_INVALID;
  if (!host || n != size_t(b->Q) * b->nodes) return lb_fail(b, ILG_E_INVALID, "state must hold Q*Lx*Ly doubles");
  LB_CUDA(b, lb_forget_waits(b), "copy in");
  LB_CUDA(b, cudaMemcpyAsync(b->f[b->cur], host, sizeof(double) * n, cudaMemcpyHostToDevice, b->stream), "copy in");
  LB_CUDA(b, cudaStreamSynchronize(b->stream), "copy in");
  b->t = t;
  b->has_state = true;
  return ILG_OK;
}

ilg_status ilg_lb_get_state(ilg_lb* b, double* host, size_t n, uint64_t* t) {
  if (!b) return ILG_E_INVALID;
  if (!b->has_state) return lb_fail(b, ILG_E_STATE, "no state: call ilg_lb_init or ilg_lb_set_state first");
  if (!host || n != size_t(b->Q) * b->nodes) return lb_fail(b, ILG_E_INVALID, "state must hold Q*Lx*Ly doubles");
  LB_CUDA(b, cudaMemcpyAsync(host, b->f[b->cur], sizeof(double) * n, cudaMemcpyDeviceToHost, b->stream), "copy out");
  if (b->waits)
    LB_CUDA(b, cudaMemcpyAsync(&b->h_sync, b->d_sync + 1, sizeof(unsigned long long), cudaMemcpyDeviceToHost, b->stream),
            "copy out");
  LB_CUDA(b, cudaStreamSynchronize(b->stream), "copy out");
  b->waits = false;
  if (b->h_sync != 0) return lb_gave_up(b);
  if (t) *t = b->t;
  return ILG_OK;
}

ilg_status ilg_lb_step(ilg_lb* b, uint32_t T) {
  if (!b) return ILG_E_INVALID;
  if (!b->has_state) return lb_fail(b, ILG_E_STATE, "no state: call ilg_lb_init or ilg_lb_set_state first");
  constexpr uint32_t kRunSteps = 4096;  // per launch
  const void* fn = lb_run_fn(b);
  bool run = true;
  for (uint32_t k = 0; k < T;) {
    uint32_t n = run ? std::min(T - k, kRunSteps) : 1;
    double *f0 = b->f[b->cur], *f1 = b->f[b->cur ^ 1];
    void* args[] = {&b->coef, &f0, &f1, &b->p.Lx, &b->Ly, &n, &b->d_sync};
    if (n > 1 && lb_fits_cluster(b) && lb_launch_cluster(b, args)) {
      // (no wait that could give up)
    } else if (n > 1) {
      LB_CUDA(b, cudaMemsetAsync(b->d_sync, 0, sizeof(unsigned long long), b->stream), "lattice Boltzmann step");
      const cudaError_t e = cudaLaunchCooperativeKernel(fn, dim3(b->run_blocks), dim3(lb_threads(b)), args, 0, b->stream);
      if (e == cudaErrorCooperativeLaunchTooLarge) {
        // the device cannot hold all blocks at once (SMs reserved elsewhere): step by step
        cudaGetLastError();
        run = false;
        continue;
      }
      LB_CUDA(b, e, "lattice Boltzmann step");
      b->waits = true;
    } else {
      LB_CUDA(b, cudaLaunchKernel(fn, dim3(b->run_blocks), dim3(lb_threads(b)), args, 0, b->stream), "lattice Boltzmann step");
    }
    b->cur ^= int(n & 1u);
    b->t += n;
    k += n;
  }
  return ILG_OK;
}

ilg_status ilg_lb_observables(ilg_lb* b, const int32_t* modes, uint32_t nmodes, uint64_t* t, double* mass,
                              double* re, double* im, double* amp) {
  if (!b) return ILG_E_INVALID;
  if (!b->has_state) return lb_fail(b, ILG_E_STATE, "no state: call ilg_lb_init or ilg_lb_set_state first");
  if (nmodes > kLbMaxModes) return lb_fail(b, ILG_E_INVALID, "at most 256 modes");
  if (nmodes && !modes) return lb_fail(b, ILG_E_INVALID, "modes is NULL");
  bool any_y = false;
  for (uint32_t j = 0; j < nmodes; ++j) {
    const int32_t mx = modes[2 * j], my = modes[2 * j + 1];
    if ((mx == 0) == (my == 0)) return lb_fail(b, ILG_E_INVALID, "each mode must be an axis mode");
    if (b->p.lattice == ILG_D1Q3 && my != 0) return lb_fail(b, ILG_E_INVALID, "D1Q3 has no y mode");
    any_y |= my != 0;
  }
  const uint32_t Lx = b->p.Lx, Ly = b->Ly;
  const double* f = b->f[b->cur];
  const uint32_t Pm = (Lx + kLbChunk - 1) / kLbChunk;
  {
    double* f_ = b->f[b->cur];
    uint32_t* count = b->d_count + kLbMaxModes;
    double* whole = Pm == 1 ? b->d_out : nullptr;
    void* args[] = {&f_, &b->p.Lx, &b->Ly, &b->d_part, &b->d_col, &count, &whole};
    // a thread for all rows of a chunk where there are few, or where such blocks fill the
    // SMs' warps twice over (8192^2: 804 us, 833 with eight threads)
    const bool wide = Ly <= kLbFewRows ||
                      uint64_t((Lx + kLbThreads - 1) / kLbThreads) * b->chunks >= uint64_t(b->sms) * 2 * (2048 / kLbThreads);
    const uint32_t cols = wide ? uint32_t(kLbThreads) : kLbCols;
    LB_CUDA(b, cudaLaunchKernel(lb_col_fn(b->Q, wide), dim3((Lx + cols - 1) / cols, b->chunks), dim3(kLbThreads), args, 0,
                                b->stream),
            "column sums");
  }
  if (any_y) {
    const int rg = int(Ly < uint32_t(b->sms) * 8 ? Ly : uint32_t(b->sms) * 8);
    if (b->Q == 3) lb_rowsum_kernel<3><<<rg, kLbThreads, 0, b->stream>>>(f, Lx, Ly, b->d_row);
    else if (b->Q == 5) lb_rowsum_kernel<5><<<rg, kLbThreads, 0, b->stream>>>(f, Lx, Ly, b->d_row);
    else lb_rowsum_kernel<9><<<rg, kLbThreads, 0, b->stream>>>(f, Lx, Ly, b->d_row);
    LB_CUDA(b, cudaGetLastError(), "row sums");
  }
  if (Pm > 1) {
    lb_mass_partial_kernel<<<Pm, kLbThreads, 0, b->stream>>>(b->d_col, Lx, b->d_red);
    LB_CUDA(b, cudaGetLastError(), "mass");
    lb_combine_kernel<<<1, kLbThreads, 0, b->stream>>>(b->d_red, Pm, b->d_out);
    LB_CUDA(b, cudaGetLastError(), "mass");
  }
  if (nmodes) {
    LbModes first{};
    const bool few = nmodes <= kLbFirstModes;
    if (few) std::copy(modes, modes + 2 * nmodes, first.m);
    else
      LB_CUDA(b, cudaMemcpyAsync(b->d_modes, modes, sizeof(int32_t) * 2 * nmodes, cudaMemcpyHostToDevice, b->stream),
              "copy modes");
    lb_mode_kernel<<<dim3(lb_mode_blocks(Lx > Ly ? Lx : Ly), nmodes), kLbModeThreads, 0, b->stream>>>(
        b->d_col, b->d_row, Lx, Ly, first, few ? nullptr : b->d_modes, b->d_out, b->d_red, b->d_count);
    LB_CUDA(b, cudaGetLastError(), "projection");
  }
  // sync[1] lies before the results
  std::vector<double> got(2 + 2 * size_t(nmodes));
  LB_CUDA(b, cudaMemcpyAsync(got.data(), b->d_sync + 1, sizeof(double) * got.size(), cudaMemcpyDeviceToHost, b->stream),
          "copy observables");
  LB_CUDA(b, cudaStreamSynchronize(b->stream), "observables");
  std::memcpy(&b->h_sync, got.data(), sizeof b->h_sync);
  b->waits = false;
  if (b->h_sync != 0) return lb_gave_up(b);
  const double* const h = got.data() + 1;
  if (t) *t = b->t;
  if (mass) *mass = h[0];
  const double half = double(Lx) * double(Ly) / 2.0;
  for (uint32_t j = 0; j < nmodes; ++j) {
    if (re) re[j] = h[1 + 2 * j];
    if (im) im[j] = h[2 + 2 * j];
    if (amp) amp[j] = h[2 + 2 * j] / half;
  }
  return ILG_OK;
}

}  // extern "C"
