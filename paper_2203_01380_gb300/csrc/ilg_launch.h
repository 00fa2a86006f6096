// Kernel launchers of libilg.so (implemented in ilg_kernels.cu).
#pragma once

#include <cuda_runtime.h>

#include <cstddef>
#include <cstdint>

#include "ilg_device.cuh"

namespace ilg {

struct InitArgs {
  uint32_t Lx, Ly;
  uint32_t axis;      // 0 no sine mode, 1 along x, 2 along y
  uint32_t mode;      // wave number reduced to [0, period)
  uint32_t period;    // Lx, Ly, or 1
  uint32_t weighted;  // 1: classes rest / moving (D2Q9: rest / axis / diagonal)
  uint32_t key0, key1, replica;
  const uint32_t* offset;  // [classes * period]
  const uint32_t* count;   // [classes * period]
  const uint32_t* table;
};

cudaError_t prepare_step_kernels(int Q);  // opt in to the table block's shared memory
// T node-parallel steps from step t in one launch (buf0 holds the state; the steps
// alternate the buffers).  sync: two words, zeroed sync[1] on entry; sync[1] becomes 1 if
// a wait between blocks gave up
cudaError_t launch_step_run(int Q, const StepArgs& a, uint16_t* buf0, uint16_t* buf1, uint32_t t, uint32_t T,
                            unsigned long long* fail, unsigned long long* sync, uint32_t sms, cudaStream_t s);
// The same where all SMs hold the lattice's planes in shared memory: T steps (2 at least) from
// step t, the state in buf0 (only read), the state after them in buf1, whatever T.  mail:
// step_resident_mail_words words (0: the lattice does not fit), zeroed, in which no tag of
// [tag, tag + T) stands yet; tag at least 1, tag + T at most 2^16.  sync as launch_step_run.
// Should a step overflow, *fail is the first that does and buf1 holds nothing.
size_t step_resident_mail_words(int Q, uint32_t Lx, uint64_t nodes, uint32_t sms);
cudaError_t launch_step_resident(int Q, const StepArgs& a, const uint16_t* buf0, uint16_t* buf1, uint32_t t, uint32_t T,
                                 unsigned long long* fail, unsigned long long* sync, uint32_t* mail, uint32_t tag,
                                 uint32_t sms, cudaStream_t s);
cudaError_t prepare_step_vec_kernels();
uint32_t step_vec_width();  // nodes per thread of the default row-tiled step (rows must be a multiple)
uint32_t step_vec_blocks_per_sm(int npt);
// npt: nodes per thread, 8 (default) or 4 (rows a multiple of npt)
cudaError_t launch_step_vec(int Q, const StepArgs& a, const uint16_t* in, uint16_t* out, uint32_t t,
                            unsigned long long* fail, int grid, cudaStream_t s, int npt = 8);
// warp-segment form of the 8-node row-tiled step (segments of 8192 nodes of a row,
// one warp each): step_seg_units = the number of segments of a lattice
uint64_t step_seg_units(uint32_t Lx, uint32_t Ly);
cudaError_t launch_step_seg(int Q, const StepArgs& a, const uint16_t* in, uint16_t* out, uint32_t t,
                            unsigned long long* fail, int grid, cudaStream_t s);
// warp segments of staged vectors (ilg_step_warp.cu): rows a multiple of the width,
// every probability drawn through its table; D1Q3 and D2Q5: shape 0 = 8 nodes per
// lane, one block of 384 threads per SM, shape 1 = 4 nodes per lane, 640 threads;
// D2Q9: 4 nodes per lane, 384 (shape 0) or 512 (shape 1) threads
cudaError_t prepare_step_warp_kernels(int Q);
uint32_t step_warp_width(int Q, int shape);  // nodes per lane (rows must be a multiple)
// T steps from step t in one launch, as launch_step_run
cudaError_t launch_step_warp(int Q, int shape, const StepArgs& a, uint16_t* buf0, uint16_t* buf1, uint32_t t, uint32_t T,
                             unsigned long long* fail, unsigned long long* sync, uint32_t sms, cudaStream_t s);
size_t step_tb_smem_bytes(uint32_t B, uint32_t Tb);
cudaError_t prepare_step_tb_kernel(uint32_t B, uint32_t Tb);
cudaError_t launch_step_tb(const StepArgs& a, const uint16_t* in, uint16_t* out, uint32_t t0, uint32_t Tb,
                           uint32_t B, unsigned long long* fail, int grid, cudaStream_t s);
// words: entries of a.table
cudaError_t launch_init(int Q, const InitArgs& a, uint32_t words, uint16_t* out, uint32_t sms, cudaStream_t s);
// col (Lx words, the ones after mass), row (Ly words; want_rows) and mass
cudaError_t launch_sums(int Q, const uint16_t* in, uint32_t Lx, uint32_t Ly, unsigned long long* col,
                        unsigned long long* row, unsigned long long* mass, int want_rows, uint32_t sms, cudaStream_t s);
constexpr uint32_t kProjModes = 256;    // modes of one launch
constexpr uint32_t kProjBlocks = 2048;  // blocks of one launch: chunks of a mode x modes
constexpr size_t kProjScratchWords = 4 * (kProjBlocks + kProjModes) + kProjModes / 2;
// the sums of a state, and kProjScratchWords 8-byte words whose last kProjModes / 2 (the
// tickets) are 0 between launches
struct ProjWork {
  const unsigned long long* col;
  const unsigned long long* row;
  const unsigned long long* mass;
  unsigned long long* scratch;
};
// modes: host, nmodes > 0 pairs; res (4 doubles per mode) and mass: device or mapped host memory
cudaError_t launch_project(const ProjWork& w, uint32_t Lx, uint32_t Ly, const int32_t* modes, uint32_t nmodes,
                           double* res, unsigned long long* mass, cudaStream_t s);
// the same with the sums in one launch, for small lattices
bool takes_small_project(uint32_t Lx, uint32_t Ly, uint32_t nmodes);  // nmodes > 0
cudaError_t launch_small_project(int Q, const uint16_t* state, uint32_t Lx, uint32_t Ly, const int32_t* modes,
                                 uint32_t nmodes, double* res, unsigned long long* mass, cudaStream_t s);
cudaError_t launch_philox(const uint32_t* ctr, uint32_t k0, uint32_t k1, uint32_t* out, size_t n,
                          cudaStream_t s);

}  // namespace ilg
