// Barrier between blocks of one cooperative launch that alternate two buffers step by step.
#pragma once

#include <cstdint>

namespace ilg {

// The barrier word counts arrivals in its low half; the high half is a mark that a step
// overflowed.  Zero it before the launch.
constexpr unsigned long long kRunMark = 1ull << 32;
constexpr uint32_t kRunPolls = 1u << 23;  // seconds; the blocks of a step differ by far less

// One thread per block, after the block's own barrier: arrive.
__device__ __forceinline__ void run_arrive(unsigned long long* word) {
  __threadfence();
  atomicAdd(word, 1ull);
}

// The same thread: wait until `target` arrivals.  Returns the word, or ~0 when the wait gave
// up (bounded: the kernel then returns and the host reports it).
__device__ __forceinline__ unsigned long long run_wait(unsigned long long* word, uint32_t target) {
  unsigned long long v = 0;
  for (uint32_t k = 0; k < kRunPolls; ++k) {
    asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(word) : "memory");
    if (uint32_t(v) >= target) return v;
  }
  return ~0ull;
}

__device__ __forceinline__ unsigned long long run_barrier(unsigned long long* word, uint32_t target) {
  run_arrive(word);
  return run_wait(word, target);
}

// The same between the blocks of one cluster (the whole launch): the hardware's cluster barrier,
// and an overflow's step marked in every block's shared memory.
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_mark(uint32_t* mark, uint32_t step, uint32_t blocks) {
  const uint32_t own = static_cast<uint32_t>(__cvta_generic_to_shared(mark));
  for (uint32_t r = 0; r < blocks; ++r)
    asm volatile(
        "{\n.reg .b32 at;\n"
        "mapa.shared::cluster.u32 at, %0, %1;\n"
        "red.relaxed.cluster.shared::cluster.min.u32 [at], %2;\n}"
        ::"r"(own), "r"(r), "r"(step)
        : "memory");
}

}  // namespace ilg
