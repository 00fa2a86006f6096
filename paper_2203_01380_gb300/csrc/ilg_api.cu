// C ABI of libilg.so: contexts, validation, scheduling of the kernels.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <new>
#include <string>
#include <vector>

#include "ilg_internal.h"
#include "ilg_launch.h"

using namespace ilg;

struct ilg_ctx {
  ilg_params p{};
  int Q = 0;
  uint32_t flip = 0;
  uint64_t P_omega = 0, P_rest = 0, P_axis = 0;  // P_axis: D2Q9 axis share
  cudaStream_t stream = nullptr;
  int device = 0;
  int sms = 0;
  size_t nodes = 0;
  uint16_t* buf[2] = {nullptr, nullptr};
  int cur = 0;
  uint64_t t = 0;
  bool has_state = false;
  uint32_t* d_tables = nullptr;            // thinning table, rest table
  unsigned long long* d_fail = nullptr;    // [0] first failing step, ~0 if none; [1], [2] the
                                           // words of a several-step launch (launch_step_run)
  // sums of a state (mass | column sums, Lx | row sums, Ly) in one array, cleared at once
  unsigned long long* d_mass = nullptr;
  unsigned long long* d_col = nullptr;
  unsigned long long* d_row = nullptr;
  unsigned long long* d_proj = nullptr;    // scratch of the projections
  // mailbox of the steps that keep the planes in shared memory, and the last tag in it
  uint32_t* d_mail = nullptr;
  size_t mail_words = 0;
  uint32_t mail_tag = 0;
  // pinned, written by the projections: mass, 4 per mode; after the words of h_word for up
  // to kFirstModes modes, an allocation of its own for more
  unsigned long long* h_obs = nullptr;
  uint32_t mode_cap = 0;
  uint32_t tb_depth = 0;                   // temporal blocking: steps per launch (0: off)
  uint32_t general = 0;                    // too many nodes would fail the fast collision: general at once
  int kernel_choice = -1;                  // single-step kernel chosen by ilg_autotune (-1: default)
  double omega_star = 0;
  unsigned long long* h_word = nullptr;    // pinned readback, kFailWords words
  volatile uint32_t* h_mark = nullptr;     // pinned: StepArgs::mark
  uint32_t* d_init = nullptr;              // tables of the initial state
  size_t init_words = 0;
  std::string err;
};

namespace {

constexpr size_t kFailWords = 3;
constexpr uint32_t kFirstModes = 64;

thread_local std::string g_create_error;

ilg_status fail(ilg_ctx* c, ilg_status s, const std::string& msg) {
  if (c) c->err = msg;
  else g_create_error = msg;
  return s;
}

ilg_status cuda_fail(ilg_ctx* c, cudaError_t e, const char* what) {
  const ilg_status s = (e == cudaErrorMemoryAllocation) ? ILG_E_OOM : ILG_E_CUDA;
  return fail(c, s, std::string(what) + ": " + cudaGetErrorString(e));
}

#define ILG_CUDA(c, call, what)                        \
  do {                                                 \
    cudaError_t e_ = (call);                           \
    if (e_ != cudaSuccess) return cuda_fail(c, e_, what); \
  } while (0)

int num_vel(int lattice) { return lattice == ILG_D1Q3 ? 3 : (lattice == ILG_D2Q5 ? 5 : 9); }

uint32_t prob_mode(uint64_t P) {
  if (P == 0) return kNever;
  if (P == (uint64_t(1) << 32)) return kAlways;
  return kTable;
}

}  // namespace

namespace ilg {
std::string validate_params(const ilg_params& p) {
  if (p.lattice != ILG_D1Q3 && p.lattice != ILG_D2Q5 && p.lattice != ILG_D2Q9)
    return "lattice must be ILG_D1Q3, ILG_D2Q5 or ILG_D2Q9";
  if (p.sampler != ILG_SAMPLER_BINOMIAL && p.sampler != ILG_SAMPLER_PARTICLE)
    return "sampler must be ILG_SAMPLER_BINOMIAL or ILG_SAMPLER_PARTICLE";
  const uint64_t Ly = p.lattice == ILG_D1Q3 ? 1 : p.Ly;
  if (p.Lx < 3) return "Lx must be >= 3";
  if (p.lattice != ILG_D1Q3 && p.Ly < 3) return "Ly must be >= 3";
  if (uint64_t(p.Lx) * Ly >= (uint64_t(1) << 32)) return "Lx * Ly must be below 2^32";
  if (!(p.omega_eff > 0.0 && p.omega_eff <= 2.0)) return "omega_eff must lie in (0, 2]";
  if (p.lattice == ILG_D1Q3 && !(p.theta > 0.0 && p.theta < 1.0)) return "theta must lie in (0, 1) on D1Q3";
  if (p.lattice == ILG_D2Q5 && !(p.theta > 0.0 && p.theta <= 0.5)) return "theta must lie in (0, 1/2] on D2Q5";
  if (p.lattice == ILG_D2Q9 && !(p.theta > 0.0 && p.theta < 1.0)) return "theta must lie in (0, 1) on D2Q9";
  if (!(p.n0 >= 0.0) || !std::isfinite(p.n0)) return "n0 must be finite and >= 0";
  if (!std::isfinite(p.amp)) return "amp must be finite";
  if (p.mode_mx != 0 && p.mode_my != 0) return "the initial sine must be an axis mode";
  if (p.lattice == ILG_D1Q3 && p.mode_my != 0) return "D1Q3 has no y mode";
  return "";
}

void round_keys(uint64_t seed, uint32_t* rk) {
  uint32_t k0 = uint32_t(seed), k1 = uint32_t(seed >> 32);
  for (int r = 0; r < 10; ++r) {
    rk[2 * r] = k0;
    rk[2 * r + 1] = k1;
    k0 += 0x9E3779B9u;
    k1 += 0xBB67AE85u;
  }
}
}  // namespace ilg

namespace {
using ilg::validate_params;

// row-tiled step: one block per row at a time, per_sm blocks per SM
int vec_grid(const ilg_ctx* c, size_t per_sm) {
  const size_t rows = c->p.Ly;
  const size_t cap = size_t(c->sms) * per_sm;
  return int(rows < cap ? rows : cap);
}

StepArgs step_args(const ilg_ctx* c) {
  StepArgs a{};
  a.Lx = c->p.Lx;
  a.Ly = c->Q == 3 ? 1 : c->p.Ly;
  a.flip = c->flip;
  a.omega_mode = prob_mode(c->P_omega);
  a.rest_mode = prob_mode(c->P_rest);
  a.axis_mode = prob_mode(c->P_axis);
  a.particle = c->p.sampler == ILG_SAMPLER_PARTICLE ? 1u : 0u;
  a.general = c->general | a.particle;
  a.key0 = uint32_t(c->p.seed);
  a.key1 = uint32_t(c->p.seed >> 32);
  a.replica = c->p.replica;
  a.tables = c->d_tables;
  a.mark = const_cast<uint32_t*>(c->h_mark);
  ilg::round_keys(c->p.seed, a.rk);
  return a;
}

void free_ctx(ilg_ctx* c) {
  cudaFree(c->buf[0]);
  cudaFree(c->buf[1]);
  cudaFree(c->d_tables);
  cudaFree(c->d_fail);
  cudaFree(c->d_mass);
  cudaFree(c->d_proj);
  cudaFree(c->d_mail);
  cudaFree(c->d_init);
  if (c->mode_cap > kFirstModes) cudaFreeHost(c->h_obs);
  if (c->h_word) cudaFreeHost(c->h_word);
}

}  // namespace

namespace ilg {
// message for ilg_last_error(NULL), set by entry points that have no context
void set_context_free_error(const std::string& msg) { g_create_error = msg; }
}  // namespace ilg

extern "C" {

const char* ilg_last_error(const ilg_ctx* ctx) {
  return ctx ? ctx->err.c_str() : g_create_error.c_str();
}

ilg_status ilg_create(const ilg_params* params, void* stream, ilg_ctx** out) {
  if (!out) return fail(nullptr, ILG_E_INVALID, "out is NULL");
  *out = nullptr;
  if (!params) return fail(nullptr, ILG_E_INVALID, "params is NULL");
  const std::string bad = validate_params(*params);
  if (!bad.empty()) return fail(nullptr, ILG_E_INVALID, bad);
  ilg_ctx* c = new (std::nothrow) ilg_ctx();
  if (!c) return fail(nullptr, ILG_E_OOM, "host allocation failed");
  c->p = *params;
  if (c->p.lattice == ILG_D1Q3) c->p.Ly = 1;
  c->Q = num_vel(c->p.lattice);
  c->stream = static_cast<cudaStream_t>(stream);
  double w[9];
  weights(c->p.lattice, c->p.theta, w);
  double omega_star = c->p.omega_eff;
  if (c->p.omega_eff > 1.0) {
    c->flip = 1;
    omega_star = 2.0 - c->p.omega_eff;
  }
  c->omega_star = omega_star;
  c->P_omega = quantise_probability(omega_star);
  c->P_rest = quantise_probability(w[0]);
  c->P_axis = c->Q == 9 ? quantise_probability(axis_share(c->p.theta)) : 0;
  c->nodes = size_t(c->p.Lx) * c->p.Ly;

  auto bail = [&](cudaError_t e, const char* what) {
    cuda_fail(nullptr, e, what);
    free_ctx(c);
    delete c;
    return (e == cudaErrorMemoryAllocation) ? ILG_E_OOM : ILG_E_CUDA;
  };
  cudaError_t e = cudaGetDevice(&c->device);
  if (e != cudaSuccess) return bail(e, "cudaGetDevice");
  e = cudaDeviceGetAttribute(&c->sms, cudaDevAttrMultiProcessorCount, c->device);
  if (e != cudaSuccess) return bail(e, "cudaDeviceGetAttribute");
  const size_t state_bytes = sizeof(uint16_t) * c->nodes * c->Q;
  for (int b = 0; b < 2; ++b) {
    e = dev_alloc(&c->buf[b], state_bytes);
    if (e != cudaSuccess) return bail(e, "cudaMalloc state");
  }
  static_assert(kBlockWords == kDevBlockWords && kBlockWords9 == kDevBlockWords9, "table block layout");
  const size_t block_words = c->Q == 9 ? kBlockWords9 : kBlockWords;
  if ((e = dev_alloc(&c->d_tables, sizeof(uint32_t) * block_words)) != cudaSuccess) return bail(e, "cudaMalloc tables");
  if ((e = dev_alloc(&c->d_fail, sizeof(unsigned long long) * kFailWords)) != cudaSuccess) return bail(e, "cudaMalloc flag");
  if ((e = dev_alloc(&c->d_mass, sizeof(unsigned long long) * (1 + size_t(c->p.Lx) + c->p.Ly))) != cudaSuccess)
    return bail(e, "cudaMalloc sums");
  c->d_col = c->d_mass + 1;
  c->d_row = c->d_col + c->p.Lx;
  if ((e = dev_alloc(&c->d_proj, sizeof(unsigned long long) * kProjScratchWords)) != cudaSuccess)
    return bail(e, "cudaMalloc projections");
  c->mail_words = step_resident_mail_words(c->Q, c->p.Lx, c->nodes, uint32_t(c->sms));
  if (c->mail_words && (e = dev_alloc(&c->d_mail, sizeof(uint32_t) * c->mail_words)) != cudaSuccess)
    return bail(e, "cudaMalloc mailbox");
  // the words of a failed step | mass and modes | the mark
  const size_t host_words = kFailWords + 1 + 4 * kFirstModes;
  if ((e = cudaMallocHost(&c->h_word, sizeof(unsigned long long) * (host_words + 1))) != cudaSuccess)
    return bail(e, "cudaMallocHost");
  c->h_obs = c->h_word + kFailWords;
  c->h_mark = reinterpret_cast<uint32_t*>(c->h_word + host_words);
  *c->h_mark = 0;
  c->mode_cap = kFirstModes;

  std::vector<uint32_t> tables(block_words, 0u);
  build_table_block(c->Q, c->p.sampler, c->P_omega, c->P_rest, c->P_axis, tables.data());
  if ((e = prepare_step_kernels(c->Q)) != cudaSuccess) return bail(e, "cudaFuncSetAttribute");
  if (c->Q != 9 && (e = prepare_step_vec_kernels()) != cudaSuccess) return bail(e, "cudaFuncSetAttribute");
  if ((e = prepare_step_warp_kernels(c->Q)) != cudaSuccess) return bail(e, "cudaFuncSetAttribute");
  e = cudaMemcpyAsync(c->d_tables, tables.data(), sizeof(uint32_t) * tables.size(), cudaMemcpyHostToDevice, c->stream);
  if (e != cudaSuccess) return bail(e, "copy tables");
  e = cudaMemsetAsync(c->d_fail, 0xFF, sizeof(unsigned long long), c->stream);
  if (e == cudaSuccess) e = cudaMemsetAsync(c->d_fail + 1, 0, 2 * sizeof(unsigned long long), c->stream);
  if (e == cudaSuccess) e = cudaMemsetAsync(c->d_proj, 0, sizeof(unsigned long long) * kProjScratchWords, c->stream);
  if (e == cudaSuccess && c->d_mail) e = cudaMemsetAsync(c->d_mail, 0, sizeof(uint32_t) * c->mail_words, c->stream);
  if (e != cudaSuccess) return bail(e, "reset flag");
  e = cudaStreamSynchronize(c->stream);
  if (e != cudaSuccess) return bail(e, "cudaStreamSynchronize");
  *out = c;
  return ILG_OK;
}

ilg_status ilg_destroy(ilg_ctx* c) {
  if (!c) return ILG_OK;
  cudaStreamSynchronize(c->stream);
  free_ctx(c);
  delete c;
  return ILG_OK;
}

ilg_status ilg_init(ilg_ctx* c) {
  if (!c) return ILG_E_INVALID;
  InitTables it;
  std::string msg;
  if (!build_init_tables(c->p, c->Q, &it, &msg)) return fail(c, ILG_E_INVALID, msg);
  // offsets | counts | tables, in one array that the context keeps (its size follows from the
  // parameters) and one copy
  const size_t cells = it.offset.size();
  std::vector<uint32_t> all;
  all.reserve(2 * cells + it.table.size());
  all.insert(all.end(), it.offset.begin(), it.offset.end());
  all.insert(all.end(), it.count.begin(), it.count.end());
  all.insert(all.end(), it.table.begin(), it.table.end());
  cudaError_t e = cudaSuccess;
  if (c->init_words < all.size()) {
    cudaFree(c->d_init);
    c->d_init = nullptr;
    c->init_words = 0;
    if ((e = dev_alloc(&c->d_init, sizeof(uint32_t) * all.size())) != cudaSuccess)
      return cuda_fail(c, e, "cudaMalloc init tables");
    c->init_words = all.size();
  }
  const uint32_t *d_off = c->d_init, *d_cnt = d_off + cells, *d_tab = d_cnt + cells;
  if ((e = cudaMemcpyAsync(c->d_init, all.data(), sizeof(uint32_t) * all.size(), cudaMemcpyHostToDevice, c->stream)) != cudaSuccess)
    return cuda_fail(c, e, "copy init tables");
  InitArgs a{};
  a.Lx = c->p.Lx;
  a.Ly = c->p.Ly;
  a.period = it.period;
  a.axis = 0;
  a.mode = 0;
  if (it.period > 1) {
    const bool along_x = c->p.mode_mx != 0;
    const int64_t L = it.period;
    const int64_t mraw = along_x ? c->p.mode_mx : c->p.mode_my;
    a.axis = along_x ? 1 : 2;
    a.mode = uint32_t(((mraw % L) + L) % L);
  }
  a.weighted = c->p.init_weighted ? 1 : 0;
  a.key0 = uint32_t(c->p.seed);
  a.key1 = uint32_t(c->p.seed >> 32);
  a.replica = c->p.replica;
  a.offset = d_off;
  a.count = d_cnt;
  a.table = d_tab;
  if ((e = launch_init(c->Q, a, uint32_t(it.table.size()), c->buf[c->cur], uint32_t(c->sms), c->stream)) != cudaSuccess)
    return cuda_fail(c, e, "init kernel");
  e = cudaStreamSynchronize(c->stream);
  if (e != cudaSuccess) return cuda_fail(c, e, "init kernel");
  c->t = 0;
  c->has_state = true;
  c->general = general_path(c->p.lattice, c->p.theta, c->omega_star, c->p.n0);
  return ILG_OK;
}

// Sums of the current state into d_mass / d_col (and d_row).
static ilg_status queue_sums(ilg_ctx* c, bool want_rows) {
  const uint32_t Lx = c->p.Lx, Ly = c->p.Ly;
  ILG_CUDA(c, launch_sums(c->Q, c->buf[c->cur], Lx, Ly, c->d_col, c->d_row, c->d_mass, want_rows ? 1 : 0, uint32_t(c->sms),
                          c->stream),
           "sums kernel");
  return ILG_OK;
}

// mean occupation of the current state decides between the collision paths
static ilg_status update_path_choice(ilg_ctx* c) {
  const ilg_status st = queue_sums(c, false);
  if (st != ILG_OK) return st;
  ILG_CUDA(c, cudaMemcpyAsync(c->h_word, c->d_mass, sizeof(unsigned long long), cudaMemcpyDeviceToHost, c->stream),
           "read mass");
  ILG_CUDA(c, cudaStreamSynchronize(c->stream), "copy state in");
  c->general = general_path(c->p.lattice, c->p.theta, c->omega_star, double(*c->h_word) / (double(c->nodes) * c->Q));
  return ILG_OK;
}

static ilg_status set_state_impl(ilg_ctx* c, const uint16_t* src, size_t n, uint64_t t, cudaMemcpyKind kind) {
  if (!c || !src) return ILG_E_INVALID;
  if (n != c->nodes * c->Q) return fail(c, ILG_E_INVALID, "state size must be Q * Lx * Ly");
  if (t >= (uint64_t(1) << 32)) return fail(c, ILG_E_INVALID, "t must be below 2^32");
  ILG_CUDA(c, cudaMemcpyAsync(c->buf[c->cur], src, sizeof(uint16_t) * n, kind, c->stream), "copy state in");
  c->t = t;
  c->has_state = true;
  return update_path_choice(c);  // (waits for the copy too)
}

static ilg_status get_state_impl(ilg_ctx* c, uint16_t* dst, size_t n, uint64_t* t, cudaMemcpyKind kind) {
  if (!c || !dst) return ILG_E_INVALID;
  if (!c->has_state) return fail(c, ILG_E_STATE, "no state: call ilg_init or ilg_set_state first");
  if (n != c->nodes * c->Q) return fail(c, ILG_E_INVALID, "state size must be Q * Lx * Ly");
  ILG_CUDA(c, cudaMemcpyAsync(dst, c->buf[c->cur], sizeof(uint16_t) * n, kind, c->stream), "copy state out");
  ILG_CUDA(c, cudaStreamSynchronize(c->stream), "copy state out");
  if (t) *t = c->t;
  return ILG_OK;
}

ilg_status ilg_set_state(ilg_ctx* c, const uint16_t* host, size_t n, uint64_t t) {
  return set_state_impl(c, host, n, t, cudaMemcpyHostToDevice);
}
ilg_status ilg_set_state_device(ilg_ctx* c, const uint16_t* dev, size_t n, uint64_t t) {
  return set_state_impl(c, dev, n, t, cudaMemcpyDeviceToDevice);
}
ilg_status ilg_get_state(ilg_ctx* c, uint16_t* host, size_t n, uint64_t* t) {
  return get_state_impl(c, host, n, t, cudaMemcpyDeviceToHost);
}
ilg_status ilg_get_state_device(ilg_ctx* c, uint16_t* dev, size_t n, uint64_t* t) {
  return get_state_impl(c, dev, n, t, cudaMemcpyDeviceToDevice);
}

ilg_status ilg_set_temporal_blocking(ilg_ctx* c, uint32_t depth) {
  if (!c) return ILG_E_INVALID;
  if (depth > kMaxTbDepth) return fail(c, ILG_E_INVALID, "temporal blocking depth above 8");
  if (depth >= 2 && c->Q != 5) return fail(c, ILG_E_INVALID, "temporal blocking is for D2Q5 lattices");
  if (depth >= 2) ILG_CUDA(c, prepare_step_tb_kernel(tb_tile(depth), depth), "cudaFuncSetAttribute");
  c->tb_depth = depth >= 2 ? depth : 0;
  return ILG_OK;
}

namespace {

// Single-step kernels, numbered as the autotuner's candidates (3 and 4 are the
// temporal-blocking depths).
enum : int { kKernelVec8 = 0, kKernelVec4 = 1, kKernelNode = 2, kKernelSeg = 5, kKernelWarp8 = 6, kKernelWarp4 = 7 };
constexpr int kCandidates = 8;

bool is_single_step(int cand) { return cand <= kKernelNode || (cand >= kKernelSeg && cand < kCandidates); }

bool kernel_applies(const ilg_ctx* c, const StepArgs& a, int kind) {
  if (kind == kKernelNode) return true;
  if (a.general) return false;  // the general path runs node-parallel
  if (kind == kKernelWarp8 || kind == kKernelWarp4) {
    // whole vectors per row; the fast collision draws every probability through its
    // table (D2Q9: the axis share too)
    return c->p.Lx % step_warp_width(c->Q, kind == kKernelWarp4 ? 1 : 0) == 0 && a.omega_mode == kTable &&
           a.rest_mode == kTable && (c->Q != 9 || a.axis_mode == kTable);
  }
  if (c->Q == 9) return false;  // the row-tiled register kernels: D1Q3 and D2Q5 only
  return c->p.Lx % (kind == kKernelVec4 ? 4u : 8u) == 0;
}

// resident warps of the row-tiled kernels (3 blocks of 8 warps per SM)
uint64_t vec_warps(const ilg_ctx* c) { return uint64_t(c->sms) * 3 * 8; }

// Lattices of at most this many nodes per SM run node-parallel: a tile of the staged warp
// kernel (256 nodes of D2Q5, 128 of D2Q9, one after the other in a lane) lasts longer than
// their whole step.  Beyond, D1Q3 and D2Q5 take the smaller tiles while a warp has few of
// them.  Us per step, 10 per velocity, node-parallel / 4-node / 8-node vectors: D2Q5 512^2
// 5.4 / 5.3 / 5.7, 768^2 8.8 / 8.1 / 8.6, 1024^2 13.4 / 10.5 / 11.8, 1448^2 24.4 / 19.4 /
// 18.1, 2048^2 45 / 33 / 30; D2Q9 (4-node) 1024^2 21 / 31, 1448^2 39 / 50, 2048^2 84 / 75.
// With the planes in shared memory the node-parallel steps stay ahead for longer (10 per velocity,
// omega_eff 1.8 / 1.5, node-parallel / 4-node: 640^2 5.4 / 6.1, 5.4 / 7.6; 768^2 7.3 / 7.7,
// 7.4 / 9.5; 864^2 8.9 / 7.8; D1Q3 2^19 4.8 / 5.6, 2^20 8.9 / 8.3).
constexpr uint64_t kRunNodesPerSm = 2048, kResidentNodesPerSm = 4096, kRunNodesPerSm9 = 16384, kWarp4NodesPerSm = 10240;

// Node-parallel steps that all SMs take with the planes in shared memory.  A launch reads the
// planes in and writes them out again, which a few steps have to repay (us for 4 steps, buffers in
// L2 / shared memory: 100^2 23 / 23, 400^2 48 / 41, 850^2 87 / 98; for 8 850^2 161 / 162).
bool takes_resident(const ilg_ctx* c, const StepArgs& a, uint32_t n) {
  return c->d_mail && n >= (c->nodes > 1024 * size_t(c->sms) ? 8u : 4u) && !a.particle && a.omega_mode == kTable &&
         a.rest_mode == kTable && (c->Q != 9 || a.axis_mode == kTable);
}

// the kernel that n steps run: the tuned one while it applies to the current state, else
// the default: node-parallel on small lattices; the shared-memory-staged warp kernel
// with 4- or 8-node vectors where the rows and probabilities allow; else 8-node row tiles
// where the rows allow; node-parallel otherwise
int pick_kernel(const ilg_ctx* c, const StepArgs& a, uint32_t n) {
  if (c->kernel_choice >= 0 && kernel_applies(c, a, c->kernel_choice)) return c->kernel_choice;
  const uint64_t sms = uint64_t(c->sms);
  const uint64_t run = c->Q == 9 ? kRunNodesPerSm9 : (takes_resident(c, a, n) ? kResidentNodesPerSm : kRunNodesPerSm);
  if (c->nodes <= run * sms) return kKernelNode;
  const bool w4 = kernel_applies(c, a, kKernelWarp4);
  if (c->Q != 9 && w4 && c->nodes <= kWarp4NodesPerSm * sms) return kKernelWarp4;
  if (kernel_applies(c, a, kKernelWarp8)) return kKernelWarp8;
  if (w4) return kKernelWarp4;
  if (!kernel_applies(c, a, kKernelVec8)) return kKernelNode;
  return step_seg_units(c->p.Lx, c->p.Ly) >= 2 * vec_warps(c) ? kKernelSeg : kKernelVec8;
}

// kernels that take several steps per launch
bool takes_runs(int kind) { return kind == kKernelNode || kind == kKernelWarp8 || kind == kKernelWarp4; }

// T steps from step t (one, unless takes_runs), the state in b0
cudaError_t launch_steps(const ilg_ctx* c, int kind, const StepArgs& a, uint16_t* b0, uint16_t* b1, uint64_t t, uint32_t T,
                         unsigned long long* fail_word) {
  const uint32_t sms = uint32_t(c->sms);
  if (kind == kKernelVec8 || kind == kKernelVec4) {
    const int npt = kind == kKernelVec8 ? 8 : 4;
    return launch_step_vec(c->Q, a, b0, b1, uint32_t(t), fail_word, vec_grid(c, step_vec_blocks_per_sm(npt)), c->stream, npt);
  }
  if (kind == kKernelSeg) {
    const uint64_t blocks = (step_seg_units(c->p.Lx, c->p.Ly) + 7) / 8, cap = vec_warps(c) / 8;
    return launch_step_seg(c->Q, a, b0, b1, uint32_t(t), fail_word, int(blocks < cap ? blocks : cap), c->stream);
  }
  if (kind == kKernelWarp8 || kind == kKernelWarp4)
    return launch_step_warp(c->Q, kind == kKernelWarp4 ? 1 : 0, a, b0, b1, uint32_t(t), T, fail_word, fail_word + 1, sms,
                            c->stream);
  return launch_step_run(c->Q, a, b0, b1, uint32_t(t), T, fail_word, fail_word + 1, sms, c->stream);
}

// A launch of single steps: n from step t, the state in buffer cur.
struct StepLaunch {
  uint64_t t;
  uint32_t n;
  int cur;
  bool resident;  // leaves its input as it was and its result in the other buffer
};

// T single steps from step t (the state in bufs[cur]; cur: afterwards), in few launches of
// several steps each where the kernel takes them.  done (or NULL): what was launched.
cudaError_t launch_singles(ilg_ctx* c, int kind, const StepArgs& a, uint16_t* const* bufs, int& cur, uint64_t t, uint32_t T,
                           unsigned long long* fail_word, std::vector<StepLaunch>* done = nullptr) {
  constexpr uint32_t kRunSteps = 4096;         // per launch
  constexpr uint64_t kRunNodes = 1ull << 26;  // beyond: a step takes half a millisecond and more, a launch nothing of it
  constexpr uint32_t kTags = 1u << 16;
  bool run = takes_runs(kind) && (kind == kKernelNode || c->nodes < kRunNodes);
  for (uint32_t k = 0; k < T;) {
    const uint32_t n = run ? std::min(T - k, kRunSteps) : 1;
    const bool resident = run && kind == kKernelNode && takes_resident(c, a, n);
    cudaError_t e;
    if (resident) {
      if (c->mail_tag + n >= kTags) {
        if ((e = cudaMemsetAsync(c->d_mail, 0, sizeof(uint32_t) * c->mail_words, c->stream)) != cudaSuccess) return e;
        c->mail_tag = 0;
      }
      e = launch_step_resident(c->Q, a, bufs[cur], bufs[cur ^ 1], uint32_t(t + k), n, fail_word, fail_word + 1, c->d_mail,
                               c->mail_tag + 1, uint32_t(c->sms), c->stream);
      if (e == cudaSuccess) c->mail_tag += n;
    } else {
      e = launch_steps(c, kind, a, bufs[cur], bufs[cur ^ 1], t + k, n, fail_word);
    }
    if (e == cudaErrorCooperativeLaunchTooLarge && n > 1) {
      // the device cannot hold all blocks at once (SMs reserved elsewhere): step by step
      cudaGetLastError();
      run = false;
      continue;
    }
    if (e != cudaSuccess) return e;
    if (done) done->push_back({t + k, n, cur, resident});
    k += n;
    cur ^= resident ? 1 : int(n & 1u);
  }
  return cudaSuccess;
}

int tb_grid(const ilg_ctx* c, uint32_t depth) {
  const uint32_t B = tb_tile(depth);
  const size_t tiles = size_t((c->p.Lx + B - 1) / B) * ((c->p.Ly + B - 1) / B);
  return int(std::min<size_t>(tiles, size_t(c->sms) * 2));
}

}  // namespace

ilg_status ilg_step(ilg_ctx* c, uint32_t T) {
  if (!c) return ILG_E_INVALID;
  NvtxRange nvtx("ilg_step");
  if (!c->has_state) return fail(c, ILG_E_STATE, "no state: call ilg_init or ilg_set_state first");
  if (c->t + T >= (uint64_t(1) << 32)) return fail(c, ILG_E_INVALID, "step counter would reach 2^32");
  if (T == 0) return ILG_OK;
  const StepArgs a = step_args(c);
  // high occupations and the particle sampler go straight to the general collision
  // (node-parallel kernel)
  const int kind = pick_kernel(c, a, T);
  const int cur0 = c->cur;
  const uint64_t t0 = c->t;
  // blocks of tb_depth steps (temporal blocking), then single steps; a block or step k
  // reads buffer cur0 ^ (k & 1)
  int cur = cur0;
  uint64_t t = t0;
  const uint32_t tb = c->tb_depth;
  if (tb >= 2) {
    const int tgrid = tb_grid(c, tb);
    for (uint32_t k = 0; k + tb <= T; k += tb) {
      cudaError_t e = launch_step_tb(a, c->buf[cur], c->buf[cur ^ 1], uint32_t(t), tb, tb_tile(tb), c->d_fail, tgrid,
                                     c->stream);
      if (e != cudaSuccess) return cuda_fail(c, e, "temporal blocking kernel");
      t += tb;
      cur ^= 1;
    }
  }
  const uint64_t t_single = t;  // single steps from here
  std::vector<StepLaunch> singles;
  if (const uint32_t n = uint32_t(t0 + T - t)) {
    const cudaError_t e = launch_singles(c, kind, a, c->buf, cur, t, n, c->d_fail, &singles);
    if (e != cudaSuccess) return cuda_fail(c, e, "step kernel");
  }
  ILG_CUDA(c, cudaStreamSynchronize(c->stream), "step");
  if (*c->h_mark == 0) {
    c->cur = cur;
    c->t = t0 + T;
    return ILG_OK;
  }
  // a step overflowed, or a wait gave up
  *c->h_mark = 0;
  ILG_CUDA(c, cudaMemcpyAsync(c->h_word, c->d_fail, sizeof(unsigned long long) * kFailWords, cudaMemcpyDeviceToHost,
                              c->stream),
           "read overflow word");
  ILG_CUDA(c, cudaStreamSynchronize(c->stream), "step");
  const unsigned long long f = c->h_word[0];
  if (c->h_word[2] != 0) {
    // a bounded wait between the blocks of a several-step launch gave up: the buffers
    // hold parts of different steps
    c->has_state = false;
    ILG_CUDA(c, cudaMemsetAsync(c->d_fail, 0xFF, sizeof(unsigned long long), c->stream), "reset flag");
    ILG_CUDA(c, cudaMemsetAsync(c->d_fail + 1, 0, 2 * sizeof(unsigned long long), c->stream), "reset flag");
    ILG_CUDA(c, cudaStreamSynchronize(c->stream), "reset flag");
    return fail(c, ILG_E_TIMEOUT, "a wait between the blocks of a several-step launch gave up: the state is lost");
  }
  if (f != ~0ull) {
    ILG_CUDA(c, cudaMemsetAsync(c->d_fail, 0xFF, sizeof(unsigned long long), c->stream), "reset flag");
    if (f < t_single) {
      // the block that started at step f failed: its input buffer still holds the state at f
      c->cur = cur0 ^ int((f - t0) / tb & 1u);
    } else {
      // the launch that step f belongs to: its input buffer still holds the state at f, or, with
      // the planes in shared memory, the state that the launch started from
      size_t j = 0;
      while (j + 1 < singles.size() && singles[j + 1].t <= f) ++j;
      const StepLaunch& l = singles[j];
      const uint32_t ahead = uint32_t(f - l.t);
      if (l.resident && ahead)
        ILG_CUDA(c, launch_step_run(c->Q, a, c->buf[l.cur], c->buf[l.cur ^ 1], uint32_t(l.t), ahead, c->d_fail, c->d_fail + 1,
                                    uint32_t(c->sms), c->stream),
                 "steps before the overflow");
      c->cur = l.cur ^ int(ahead & 1u);
    }
    c->t = f;
    ILG_CUDA(c, cudaStreamSynchronize(c->stream), "reset flag");
    char buf[160];
    std::snprintf(buf, sizeof(buf), "occupation above 65535 in the launch from step %llu; state kept at t = %llu", f, f);
    return fail(c, ILG_E_OVERFLOW, buf);
  }
  c->cur = cur;
  c->t = t0 + T;
  return ILG_OK;
}

ilg_status ilg_set_step_kernel(ilg_ctx* c, int32_t candidate) {
  if (!c) return ILG_E_INVALID;
  if (candidate < -1 || (candidate >= 0 && !is_single_step(candidate)))
    return fail(c, ILG_E_INVALID, "candidate must be -1, 0, 1, 2, 5, 6 or 7");
  c->kernel_choice = candidate;
  return ILG_OK;
}

ilg_status ilg_autotune(ilg_ctx* c, uint32_t trial_steps, ilg_tuning* out) {
  if (!c) return ILG_E_INVALID;
  if (!c->has_state) return fail(c, ILG_E_STATE, "no state: call ilg_init or ilg_set_state first");
  if (trial_steps == 0) trial_steps = 20;
  if (trial_steps > 1000) return fail(c, ILG_E_INVALID, "at most 1000 trial steps");
  if (c->t + 2ull * trial_steps + 16 >= (uint64_t(1) << 32))
    return fail(c, ILG_E_INVALID, "step counter would reach 2^32 in the trials");
  const StepArgs a = step_args(c);
  // trials on a copy of the state (two scratch buffers and their own overflow word);
  // every candidate gives the same bits, only the time is kept
  const size_t bytes = sizeof(uint16_t) * c->nodes * c->Q;
  uint16_t* s[2] = {nullptr, nullptr};
  unsigned long long* fw = nullptr;
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  auto release = [&]() {
    cudaFree(s[0]);
    cudaFree(s[1]);
    cudaFree(fw);
    if (e0) cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
  };
  cudaError_t e = dev_alloc(&s[0], bytes);
  if (e == cudaSuccess) e = dev_alloc(&s[1], bytes);
  if (e == cudaSuccess) e = dev_alloc(&fw, sizeof(unsigned long long) * kFailWords);
  if (e == cudaSuccess) e = cudaEventCreate(&e0);
  if (e == cudaSuccess) e = cudaEventCreate(&e1);
  if (e == cudaSuccess) e = cudaMemcpyAsync(s[0], c->buf[c->cur], bytes, cudaMemcpyDeviceToDevice, c->stream);
  if (e != cudaSuccess) {
    release();
    return cuda_fail(c, e, "autotune scratch");
  }
  // candidates: 0 8-node vectors, 1 4-node vectors, 2 node-parallel, 3 / 4 temporal
  // blocking of depth 2 / 4 (D2Q5), 5 warp segments of 8-node vectors, 6 / 7 the
  // shared-memory-staged warp kernel with 8 / 4 nodes per lane
  ilg_tuning res{};
  res.n = kCandidates;
  for (int k = 0; k < 8; ++k) res.ms_per_step[k] = -1.0;
  auto trial = [&](int cand, double* ms_per_step) -> cudaError_t {
    const uint32_t depth = cand == 3 ? 2u : (cand == 4 ? 4u : 1u);
    const uint32_t launches = std::max<uint32_t>(1, trial_steps / depth);
    uint64_t t = c->t;
    int cur = 0;
    auto some = [&](uint32_t n) -> cudaError_t {  // n launches of `depth` steps
      cudaError_t r = cudaSuccess;
      if (depth == 1) {
        r = launch_singles(c, cand, a, s, cur, t, n, fw);
      } else {
        for (uint32_t k = 0; k < n && r == cudaSuccess; ++k) {
          r = launch_step_tb(a, s[cur], s[cur ^ 1], uint32_t(t) + k * depth, depth, tb_tile(depth), fw, tb_grid(c, depth),
                             c->stream);
          cur ^= 1;
        }
      }
      t += uint64_t(n) * depth;
      return r;
    };
    cudaError_t r = cudaMemsetAsync(fw, 0xFF, sizeof(unsigned long long), c->stream);
    if (r == cudaSuccess) r = cudaMemsetAsync(fw + 1, 0, 2 * sizeof(unsigned long long), c->stream);
    if (r == cudaSuccess) r = some(1);  // warm-up launch
    if (r == cudaSuccess) r = cudaEventRecord(e0, c->stream);
    if (r == cudaSuccess) r = some(launches);
    if (r == cudaSuccess) r = cudaEventRecord(e1, c->stream);
    if (r == cudaSuccess) r = cudaMemcpyAsync(c->h_word, fw, sizeof(unsigned long long), cudaMemcpyDeviceToHost, c->stream);
    if (r == cudaSuccess) r = cudaStreamSynchronize(c->stream);
    float ms = 0.f;
    if (r == cudaSuccess) r = cudaEventElapsedTime(&ms, e0, e1);
    // a trial that overflowed skipped work after the overflow: its time is not kept
    if (r == cudaSuccess && *c->h_word == ~0ull) *ms_per_step = double(ms) / (double(launches) * depth);
    return r;
  };
  for (int cand = 0; cand < kCandidates && e == cudaSuccess; ++cand) {
    if (is_single_step(cand) && !kernel_applies(c, a, cand)) continue;
    if (!is_single_step(cand)) {
      if (c->Q != 5) continue;
      const uint32_t depth = cand == 3 ? 2u : 4u;
      if ((e = prepare_step_tb_kernel(tb_tile(depth), depth)) != cudaSuccess) break;
    }
    e = trial(cand, &res.ms_per_step[cand]);
  }
  release();
  *c->h_mark = 0;  // (a trial may have overflowed)
  if (e != cudaSuccess) return cuda_fail(c, e, "autotune trial");
  int best = -1;
  for (int k = 0; k < kCandidates; ++k)
    if (res.ms_per_step[k] >= 0.0 && (best < 0 || res.ms_per_step[k] < res.ms_per_step[best])) best = k;
  if (best < 0) return fail(c, ILG_E_OVERFLOW, "every trial overflowed: no choice made");
  if (!is_single_step(best)) {
    // temporal blocking; the remaining single steps take the fastest single-step kernel
    int single = -1;
    for (int k = 0; k < kCandidates; ++k)
      if (is_single_step(k) && res.ms_per_step[k] >= 0.0 &&
          (single < 0 || res.ms_per_step[k] < res.ms_per_step[single]))
        single = k;
    c->kernel_choice = single;
    c->tb_depth = best == 3 ? 2u : 4u;
    ILG_CUDA(c, prepare_step_tb_kernel(tb_tile(c->tb_depth), c->tb_depth), "cudaFuncSetAttribute");
  } else {
    c->kernel_choice = best;
    c->tb_depth = 0;
  }
  res.choice = uint32_t(best);
  res.tb_depth = c->tb_depth;
  res.threads = 256;
  if (out) *out = res;
  return ILG_OK;
}

ilg_status ilg_observables(ilg_ctx* c, const int32_t* modes, uint32_t nmodes, uint64_t* t, uint64_t* mass,
                           double* re, double* im, double* amp, double* Sk, int64_t* col_sums,
                           int64_t* row_sums) {
  if (!c) return ILG_E_INVALID;
  NvtxRange nvtx("ilg_observables");
  if (!c->has_state) return fail(c, ILG_E_STATE, "no state: call ilg_init or ilg_set_state first");
  if (nmodes && !modes) return fail(c, ILG_E_INVALID, "modes is NULL");
  bool want_rows = row_sums != nullptr;
  for (uint32_t i = 0; i < nmodes; ++i) {
    const int32_t mx = modes[2 * i], my = modes[2 * i + 1];
    if ((mx == 0) == (my == 0)) return fail(c, ILG_E_INVALID, "each mode must have exactly one nonzero component");
    if (my != 0 && c->Q == 3) return fail(c, ILG_E_INVALID, "D1Q3 has no y modes");
    if (my != 0) want_rows = true;
  }
  if (nmodes > c->mode_cap) {
    unsigned long long* more = nullptr;
    ILG_CUDA(c, cudaMallocHost(&more, sizeof(unsigned long long) * (1 + 4 * size_t(nmodes))), "cudaMallocHost modes");
    if (c->mode_cap > kFirstModes) cudaFreeHost(c->h_obs);
    c->h_obs = more;
    c->mode_cap = nmodes;
  }
  const uint32_t Lx = c->p.Lx, Ly = c->p.Ly;
  const double* const res = reinterpret_cast<const double*>(c->h_obs + 1);
  const bool small = nmodes && !col_sums && !row_sums && takes_small_project(Lx, Ly, nmodes);
  if (!small) {
    const ilg_status st = queue_sums(c, want_rows);
    if (st != ILG_OK) return st;
  }
  if (small)
    ILG_CUDA(c, launch_small_project(c->Q, c->buf[c->cur], Lx, Ly, modes, nmodes, const_cast<double*>(res), c->h_obs, c->stream),
             "projection kernel");
  else if (nmodes)
    ILG_CUDA(c, launch_project(ProjWork{c->d_col, c->d_row, c->d_mass, c->d_proj}, Lx, Ly, modes, nmodes,
                               const_cast<double*>(res), c->h_obs, c->stream),
             "projection kernel");
  else
    ILG_CUDA(c, cudaMemcpyAsync(c->h_word, c->d_mass, sizeof(unsigned long long), cudaMemcpyDeviceToHost, c->stream),
             "copy mass");
  if (col_sums)
    ILG_CUDA(c, cudaMemcpyAsync(col_sums, c->d_col, sizeof(int64_t) * Lx, cudaMemcpyDeviceToHost, c->stream), "copy sums");
  if (row_sums)
    ILG_CUDA(c, cudaMemcpyAsync(row_sums, c->d_row, sizeof(int64_t) * Ly, cudaMemcpyDeviceToHost, c->stream), "copy sums");
  ILG_CUDA(c, cudaStreamSynchronize(c->stream), "observables");
  const unsigned long long M = nmodes ? c->h_obs[0] : *c->h_word;
  if (t) *t = c->t;
  if (mass) *mass = M;
  for (uint32_t i = 0; i < nmodes; ++i) {
    if (re) re[i] = res[4 * i + 0];
    if (im) im[i] = res[4 * i + 1];
    if (amp) amp[i] = res[4 * i + 2];
    if (Sk) Sk[i] = res[4 * i + 3];
  }
  return ILG_OK;
}

ilg_status ilg_philox(const uint32_t* ctr, uint64_t seed, uint32_t* out, size_t n, void* stream) {
  if (!ctr || !out) return fail(nullptr, ILG_E_INVALID, "NULL argument");
  if (n == 0) return ILG_OK;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  uint32_t *d_c = nullptr, *d_o = nullptr;
  cudaError_t e = dev_alloc(&d_c, sizeof(uint32_t) * 4 * n);
  if (e == cudaSuccess) e = dev_alloc(&d_o, sizeof(uint32_t) * 4 * n);
  if (e == cudaSuccess) e = cudaMemcpyAsync(d_c, ctr, sizeof(uint32_t) * 4 * n, cudaMemcpyHostToDevice, s);
  if (e == cudaSuccess) e = launch_philox(d_c, uint32_t(seed), uint32_t(seed >> 32), d_o, n, s);
  if (e == cudaSuccess) e = cudaMemcpyAsync(out, d_o, sizeof(uint32_t) * 4 * n, cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  cudaFree(d_c);
  cudaFree(d_o);
  if (e != cudaSuccess) return cuda_fail(nullptr, e, "philox probe");
  return ILG_OK;
}

ilg_status ilg_binomial_table(uint64_t P, uint32_t* out) {
  if (!out || P == 0 || P >= (uint64_t(1) << 32)) return fail(nullptr, ILG_E_INVALID, "P must lie in (0, 2^32)");
  build_binomial_table(P, out);
  return ILG_OK;
}

ilg_status ilg_alias_table(uint64_t P, uint32_t* thr, uint32_t* alias) {
  if (!thr || !alias || P == 0 || P >= (uint64_t(1) << 32)) return fail(nullptr, ILG_E_INVALID, "P must lie in (0, 2^32)");
  std::vector<AliasEntry> t(kAliasEntries);
  build_alias_table(P, t.data());
  for (uint32_t i = 0; i < kAliasEntries; ++i) {
    thr[i] = t[i].thr;
    alias[i] = t[i].alias;
  }
  return ILG_OK;
}

ilg_status ilg_poisson_table(double lambda, uint32_t* out, uint32_t cap, uint32_t* K) {
  if (!out || !K || !(lambda >= 0.0) || lambda > kMaxMean) return fail(nullptr, ILG_E_INVALID, "bad argument");
  std::vector<uint32_t> buf(kPoissonCap);
  const uint32_t k = build_poisson_table(lambda, buf.data(), kPoissonCap);
  if (k == 0 || k > cap) return fail(nullptr, ILG_E_INVALID, "table longer than cap");
  std::memcpy(out, buf.data(), sizeof(uint32_t) * k);
  *K = k;
  return ILG_OK;
}

}  // extern "C"
