// pdmcf_batch.cu — BatchEngine: many resident instances advanced together, and the
// synchronous batched solve mcf_solve_batch.
//
// Per iteration: an edge launch over the instances of each non-empty group of shapes, one node
// and (where some instance takes a stop test) one check launch over all instances, then one
// scalar launch with a block per instance. Instance scalars live on the device (BatchScalars), so
// a chunk of iterations is captured once as a CUDA graph and replayed whatever the mix; the host
// reads the scalar mirror once per chunk to retire finished instances and admit new ones between
// chunks.
#include <cuda_runtime.h>

#include <algorithm>
#include <chrono>
#include <cmath>
#include <cstring>
#include <map>
#include <mutex>
#include <string>
#include <vector>

#include <nvtx3/nvToolsExt.h>

#include "pdmcf_batch_engine.h"

namespace pdmcf {

// Solver-side helpers (pdmcf_solver.cu).
cudaMemPool_t state_pool(int device);
cudaError_t pool_alloc(void** p, size_t bytes, cudaMemPool_t pool, cudaStream_t st);
int batch_prepare_state(mcf_problem* p, const mcf_options* o, cudaStream_t st, bool* warm);
void batch_state_pointers(mcf_problem* p, BatchInst* bi, int* parity);
void batch_finish_state(mcf_problem* p, int parity, const DevScalars& s, cudaStream_t st);

// ------------------------------------------------------------------ scalar kernel

constexpr int SCALAR_BLOCK = 512;

struct BatchScalarArgs {
  const BatchInst* insts;
  const int* slots;
  const int* nslots;
};

// Sums of K consecutive fields over nb items of `stride` doubles by the block's threads, in a
// fixed order; thread 0 gets them. Thread t adds items t, t + 512, ..., all K fields of an item at
// once, several items in flight. (A contiguous segment per thread, field by field, took most of the
// 95 us of this kernel at a stop test of n = 3000, m = 24 000.)
template <int K>
__device__ __forceinline__ void block_sums(const double* __restrict__ base, int nb, size_t stride, double* out,
                                           double (&sh)[8][SCALAR_BLOCK / 32]) {
  constexpr int W = K > 4 ? 8 : K > 1 ? 4 : 1;   // warp_sums takes a power of two
  double s[W];
#pragma unroll
  for (int k = 0; k < W; ++k) s[k] = 0.0;
#pragma unroll 8
  for (int b = threadIdx.x; b < nb; b += SCALAR_BLOCK)
#pragma unroll
    for (int k = 0; k < K; ++k) s[k] += base[(size_t)b * stride + k];
  const double sum = warp_sums<W>(s);
  const int lane = threadIdx.x & 31, field = lane / (32 / W);
  if (lane % (32 / W) == 0) sh[field][threadIdx.x >> 5] = sum;
  __syncthreads();
  if (threadIdx.x == 0) {
#pragma unroll
    for (int k = 0; k < K; ++k) {
      double t = 0.0;
      for (int w = 0; w < SCALAR_BLOCK / 32; ++w) t += sh[k][w];
      out[k] = t;
    }
  }
  __syncthreads();
}

// One block per resident instance: fixed-order FP64 sums of its per-edge and per-piece
// parts, the shared scalar update, parity flip and the stop rule (Algorithm 2.1, step 1,
// evaluated on the instance's own check iterations).
__global__ void __launch_bounds__(SCALAR_BLOCK) batch_scalar_kernel(BatchScalarArgs a) {
  __shared__ double sh[8][SCALAR_BLOCK / 32];
  if ((int)blockIdx.x >= *a.nslots) return;
  const BatchInst& I = a.insts[a.slots[blockIdx.x]];
  BatchScalars* bs = I.sc;
  const bool active = bs->active != 0, check = batch_is_check(bs), reduce = batch_reduces(bs);
  __syncthreads();   // all threads have read the scalars: from here on thread 0 moves them
  if (!active) return;
  // without a use for the sums of this iteration only the counters move
  if (!reduce) {
    if (threadIdx.x != 0) return;
    DevScalars* s = &bs->s;
    s->alpha_last = s->alpha;
    s->beta_last = s->beta;
    s->k += 1;
    bs->parity ^= 1;
    if (s->numeric_error) {
      bs->done = 2;
      bs->active = 0;
    }
    return;
  }
  double dF2, nodep[NODE_PARTS], chk[CHECK_PARTS];
  block_sums<1>(I.pe, I.m, 1, &dF2, sh);
  if (check) {   // after a check phase a node's pieces are in its first one
    block_sums<NODE_PARTS>(I.pn, I.n, (size_t)I.per * NODE_PARTS, nodep, sh);
    block_sums<CHECK_PARTS>(I.pc, I.m, CHECK_PARTS, chk, sh);
  } else {
    block_sums<1>(I.pn, I.n * I.per, NODE_PARTS, nodep, sh);
  }
  const double dY2 = nodep[0];
  if (threadIdx.x != 0) return;
  DevScalars* s = &bs->s;
  scalar_update(s, dF2, dY2, nodep, chk, check);
  bs->parity ^= 1;
  bool stop = false;
  bool stall = false;
  if (check) {
    const double nm = (double)I.n * (double)I.m;
    if (bs->stop_mode == MCF_STOP_PAPER && s->r < nm * bs->eps) stop = true;
    if (bs->stop_mode == MCF_STOP_REL_KKT && s->rel_kkt < bs->eps) stop = true;
    const int frozen = (s->freeze >= 0 && s->freeze <= s->k) ? 1 : 0;
    if (frozen != bs->stall_frozen) {   // constant omega from here on: a new phase
      bs->stall_frozen = frozen;
      bs->stall_best = INFINITY;
      bs->stall_count = 0;
    }
    if (!stop && bs->stop_mode == MCF_STOP_REL_KKT && bs->stall_checks > 0 &&
        s->rel_kkt < 100.0 * bs->eps) {
      if (s->rel_kkt < 0.95 * bs->stall_best) { bs->stall_best = s->rel_kkt; bs->stall_count = 0; }
      else if (++bs->stall_count >= bs->stall_checks) { stall = true; bs->stalled = 1; }
    }
  }
  if (s->k >= bs->max_iters || s->numeric_error || stop || stall) {
    bs->done = stop ? 1 : 2;    // 1: stop rule held, 2: iteration cap or numeric error
    bs->active = 0;
  }
}

// ------------------------------------------------------------------ engine

int batch_admit_shape(const mcf_problem* p) {
  const int ld = (p->n + 7) / 8 * 8;
  return pick_shape(ld / 4);
}

static int node_pieces_per(int n) { return batch_pieces_per((n + 7) / 8 * 8); }

// The slot's sums, as they are allocated and as admission counts them: one set per edge and per piece
// (the pieces of a node's column add up to 1 % of the state).
int64_t BatchEngine::extra_bytes(const mcf_problem* p) {
  return (int64_t)sizeof(double) * ((int64_t)p->m * (1 + CHECK_PARTS) +
                                    (int64_t)p->n * node_pieces_per(p->n) * NODE_PARTS);
}

BatchEngine::BatchEngine(int device, int max_slots)
    : device_(device), max_slots_(max_slots), slots_(max_slots), h_insts_(max_slots) {}

BatchEngine::~BatchEngine() {
  cudaSetDevice(device_);
  for (int s = 0; s < max_slots_; ++s)
    if (slots_[s].used) release(s, false);
  if (stream_) cudaStreamSynchronize(stream_);
  destroy_graphs();
  void* bufs[] = {d_insts_, d_sc_, d_slot_list_, d_nslots_, d_cls_count_, d_cls_inst_,
                  d_cls_eoff_, d_cls_noff_};
  for (void* b : bufs)
    if (b) cudaFree(b);
  if (h_sc_) cudaFreeHost(h_sc_);
  if (stream_) cudaStreamDestroy(stream_);
}

#define BCK(call)                                                                       \
  do {                                                                                  \
    cudaError_t e_ = (call);                                                            \
    if (e_ != cudaSuccess) {                                                            \
      set_error(std::string("CUDA error ") + cudaGetErrorString(e_) + " in " #call);    \
      return MCF_ERR_CUDA;                                                              \
    }                                                                                   \
  } while (0)

int BatchEngine::init() {
  int ndev = 0;
  if (cudaGetDeviceCount(&ndev) != cudaSuccess || ndev == 0) {
    cudaGetLastError();
    set_error("no CUDA device available (the solver has no CPU path)");
    return MCF_ERR_CUDA;
  }
  BCK(cudaSetDevice(device_));
  BCK(cudaStreamCreateWithFlags(&stream_, cudaStreamNonBlocking));
  BCK(cudaDeviceGetAttribute(&sms_, cudaDevAttrMultiProcessorCount, device_));
  pool_ = state_pool(device_);
  const size_t S = max_slots_;
  BCK(cudaMalloc((void**)&d_insts_, S * sizeof(BatchInst)));
  BCK(cudaMalloc((void**)&d_sc_, S * sizeof(BatchScalars)));
  BCK(cudaMallocHost((void**)&h_sc_, S * sizeof(BatchScalars)));
  BCK(cudaMalloc((void**)&d_slot_list_, S * sizeof(int)));
  BCK(cudaMalloc((void**)&d_nslots_, sizeof(int)));
  BCK(cudaMalloc((void**)&d_cls_count_, NUM_LISTS * sizeof(int)));
  BCK(cudaMalloc((void**)&d_cls_inst_, NUM_LISTS * S * sizeof(int)));
  BCK(cudaMalloc((void**)&d_cls_eoff_, NUM_LISTS * (S + 1) * sizeof(long long)));
  BCK(cudaMalloc((void**)&d_cls_noff_, NUM_LISTS * (S + 1) * sizeof(long long)));
  std::memset(h_sc_, 0, S * sizeof(BatchScalars));
  BCK(cudaMemsetAsync(d_sc_, 0, S * sizeof(BatchScalars), stream_));
  BCK(cudaMemsetAsync(d_nslots_, 0, sizeof(int), stream_));
  BCK(cudaMemsetAsync(d_cls_count_, 0, NUM_LISTS * sizeof(int), stream_));
  const BatchTable& T = batch_table();
  auto grid = [&](BatchKernel k, int block, int* out) -> cudaError_t {
    int occ = 0;
    const cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, (const void*)k, block, 0);
    *out = std::max(1, occ) * sms_;
    return e;
  };
  for (int g = 0; g < NUM_GROUPS; ++g) BCK(grid(T.edge[g], T.block[g], &grid_edge_[g]));
  BCK(grid(T.node, 256, &grid_node_));
  BCK(grid(T.node_chk, 256, &grid_node_chk_));
  BCK(grid(T.check, 256, &grid_check_));
  BCK(cudaStreamSynchronize(stream_));
  return MCF_OK;
}

int BatchEngine::free_slots() const {
  int f = 0;
  for (const auto& s : slots_) f += s.used ? 0 : 1;
  return f;
}

int BatchEngine::active_count() const {
  int a = 0;
  for (const auto& s : slots_) a += (s.used && !s.finished) ? 1 : 0;
  return a;
}

int BatchEngine::add(mcf_problem* p, const mcf_options& o, void* tag, int* slot_out,
                     int cls_override) {
  int s = -1;
  for (int i = 0; i < max_slots_ && s < 0; ++i)
    if (!slots_[i].used) s = i;
  if (s < 0) {
    set_error("no free batch slot");
    return MCF_ERR_BUSY;
  }
  const int nchunks = ((p->n + 7) / 8 * 8) / 4;
  int cls = cls_override >= 0 ? cls_override : batch_admit_shape(p);
  if (cls < 0 || kShapes[cls].group * kShapes[cls].vpt < nchunks) {
    set_error("instance too large for the batched kernels or shape too small");
    return MCF_ERR_INVALID;
  }
  BCK(cudaSetDevice(device_));
  bool warm = false;
  int rc = batch_prepare_state(p, &o, stream_, &warm);
  if (rc != MCF_OK) return rc;
  BatchSlot& sl = slots_[s];
  sl = BatchSlot();
  sl.parts = alloc_parts((size_t)extra_bytes(p));
  if (!sl.parts) {
    cudaStreamSynchronize(stream_);   // the state's preparation
    sl = BatchSlot();
    set_error("device allocation failed");
    return MCF_ERR_OOM;
  }
  // from here on a failed call leaves the slot to release()
  sl.used = true;
  sl.p = p;
  sl.opts = o;
  sl.tag = tag;
  sl.cls = cls;
  sl.bytes = device_bytes(p, MCF_FP32) + extra_bytes(p);
  BatchInst bi{};
  int parity0 = 0;
  batch_state_pointers(p, &bi, &parity0);
  bi.rho = (float)o.rho;
  bi.per = node_pieces_per(p->n);
  bi.pe = sl.parts;
  bi.pn = bi.pe + p->m;
  bi.pc = bi.pn + (size_t)p->n * bi.per * NODE_PARTS;
  bi.sc = d_sc_ + s;
  h_insts_[s] = bi;
  BatchScalars& hs = h_sc_[s];
  std::memset(&hs, 0, sizeof(hs));
  DevScalars& d = hs.s;
  d.eta = p->eta;
  d.omega = p->omega;
  d.alpha = d.eta / d.omega;
  d.beta = d.eta * d.omega;
  d.alpha_last = d.alpha;
  d.beta_last = d.beta;
  d.theta = o.theta;
  d.tau = o.tau;
  d.k_adapt = o.k_adapt > 0 ? o.k_adapt : 1;
  d.freeze = o.omega_freeze_iter;
  d.guard = o.adapt_guard;
  d.guard_below = o.adapt_guard_below;
  d.omega_ref = 0.0;
  d.omega_arm = 0.0;
  d.best_kkt = INFINITY;
  d.r = INFINITY;
  d.rel_kkt = INFINITY;
  d.n = p->n;
  d.m = p->m;
  hs.parity = parity0;
  hs.active = 1;
  hs.done = 0;
  hs.stop_mode = o.stop_mode;
  hs.max_iters = o.max_iters;
  hs.k_check = std::max(1, o.k_check);
  hs.eps = o.eps;
  hs.stall_checks = o.stall_checks;
  hs.stall_best = INFINITY;
  hs.stall_frozen = 0;
  lists_dirty_ = true;
  // read before the next chunk's copy back writes the mirror: same stream
  BCK(cudaMemsetAsync(sl.parts, 0, (size_t)extra_bytes(p), stream_));
  BCK(cudaMemcpyAsync(d_insts_ + s, &h_insts_[s], sizeof(bi), cudaMemcpyHostToDevice, stream_));
  BCK(cudaMemcpyAsync(d_sc_ + s, &hs, sizeof(hs), cudaMemcpyHostToDevice, stream_));
  (void)warm;
  *slot_out = s;
  return MCF_OK;
}

// Work lists of the edge-phase groups and of all instances (in slot order) and the scalar
// kernel's slot list.
int BatchEngine::upload_lists() {
  const size_t S = max_slots_;
  std::vector<int> count(NUM_LISTS, 0), inst(NUM_LISTS * S, 0), slot_list;
  std::vector<long long> eoff(NUM_LISTS * (S + 1), 0), noff(NUM_LISTS * (S + 1), 0);
  unsigned mask = 0;
  for (int s = 0; s < max_slots_; ++s) {
    const BatchSlot& sl = slots_[s];
    if (!sl.used || sl.finished) continue;
    for (int c : {batch_group(sl.cls), NUM_GROUPS}) {
      const int k = count[c]++;
      inst[c * S + k] = s;
      eoff[c * (S + 1) + k + 1] = eoff[c * (S + 1) + k] + sl.p->m;
      noff[c * (S + 1) + k + 1] = noff[c * (S + 1) + k] + (long long)sl.p->n * h_insts_[s].per;
    }
    slot_list.push_back(s);
    mask |= 1u << batch_group(sl.cls);
  }
  const int ns = (int)slot_list.size();
  if (slot_list.empty()) slot_list.push_back(0);
  BCK(cudaMemcpyAsync(d_cls_count_, count.data(), NUM_LISTS * sizeof(int), cudaMemcpyHostToDevice, stream_));
  BCK(cudaMemcpyAsync(d_cls_inst_, inst.data(), inst.size() * sizeof(int), cudaMemcpyHostToDevice, stream_));
  BCK(cudaMemcpyAsync(d_cls_eoff_, eoff.data(), eoff.size() * sizeof(long long), cudaMemcpyHostToDevice, stream_));
  BCK(cudaMemcpyAsync(d_cls_noff_, noff.data(), noff.size() * sizeof(long long), cudaMemcpyHostToDevice, stream_));
  BCK(cudaMemcpyAsync(d_slot_list_, slot_list.data(), slot_list.size() * sizeof(int), cudaMemcpyHostToDevice, stream_));
  BCK(cudaMemcpyAsync(d_nslots_, &ns, sizeof(int), cudaMemcpyHostToDevice, stream_));
  BCK(cudaStreamSynchronize(stream_));   // host staging vectors die at return
  class_mask_ = mask;
  lists_dirty_ = false;
  return MCF_OK;
}

int BatchEngine::launch_iteration(cudaStream_t st, bool with_check) {
  const BatchTable& T = batch_table();
  const size_t S = max_slots_;
  const BatchInst* insts = d_insts_;
  auto launch = [&](BatchKernel k, int list, int grid, int block) -> cudaError_t {
    BatchClassDev cls{d_cls_count_ + list, d_cls_inst_ + list * S, d_cls_eoff_ + list * (S + 1),
                      d_cls_noff_ + list * (S + 1)};
    void* kargs[] = {(void*)&insts, &cls};
    return cudaLaunchKernel((const void*)k, dim3(grid), dim3(block), kargs, 0, st);
  };
  for (int g = 0; g < NUM_GROUPS; ++g)
    if (class_mask_ & (1u << g)) BCK(launch(T.edge[g], g, grid_edge_[g], T.block[g]));
  BCK(launch(with_check ? T.node_chk : T.node, NUM_GROUPS, with_check ? grid_node_chk_ : grid_node_, 256));
  if (with_check) BCK(launch(T.check, NUM_GROUPS, grid_check_, 256));
  BatchScalarArgs sa{d_insts_, d_slot_list_, d_nslots_};
  batch_scalar_kernel<<<max_slots_, SCALAR_BLOCK, 0, st>>>(sa);
  BCK(cudaGetLastError());
  return MCF_OK;
}

void BatchEngine::destroy_graphs() {
  for (auto& kv : graphs_) cudaGraphExecDestroy(kv.second);
  graphs_.clear();
}

int BatchEngine::step(int iters) {
  nvtxRangePushA("pdmcf batched chunk");
  const int rc = step_impl(iters);
  nvtxRangePop();
  return rc;
}

// Iterations i of the next chunk (bit i) in which some active instance takes a stop test
// (batch_is_check at its k = k0 + i): the check launch of the other iterations would find
// nothing to do for any instance, so it is left out. Chunks longer than 64 iterations keep it
// in every iteration.
uint64_t BatchEngine::check_iterations(int iters) const {
  if (iters > 64) return ~0ull;
  uint64_t mask = 0;
  for (int s = 0; s < max_slots_; ++s) {
    const BatchSlot& sl = slots_[s];
    const BatchScalars& h = h_sc_[s];
    if (!sl.used || sl.finished || !h.active) continue;
    const long long kc = std::max(1LL, h.k_check);
    for (int i = 0; i < iters; ++i) {
      const long long k1 = h.s.k + i + 1;
      if (k1 % kc == 0 || k1 >= h.max_iters) mask |= 1ull << i;
    }
  }
  return mask;
}

int BatchEngine::step_impl(int iters) {
  BCK(cudaSetDevice(device_));
  if (lists_dirty_) {
    int rc = upload_lists();
    if (rc != MCF_OK) return rc;
  }
  if (class_mask_ == 0) return MCF_OK;
  const uint64_t checks = check_iterations(iters);
  auto with_check = [&](int i) { return i >= 64 || ((checks >> i) & 1ull) != 0; };
  const auto key = std::make_tuple(class_mask_, iters, checks);
  auto it = graphs_.find(key);
  if (it == graphs_.end() && !graphs_broken_) {
    if (graphs_.size() >= 64) destroy_graphs();   // bound the cache
    cudaGraph_t g = nullptr;
    cudaGraphExec_t ge = nullptr;
    bool ok = cudaStreamBeginCapture(stream_, cudaStreamCaptureModeThreadLocal) == cudaSuccess;
    for (int i = 0; i < iters && ok; ++i) ok = launch_iteration(stream_, with_check(i)) == MCF_OK;
    const cudaError_t e = cudaStreamEndCapture(stream_, &g);
    ok = ok && e == cudaSuccess && g && cudaGraphInstantiate(&ge, g, 0) == cudaSuccess;
    if (g) cudaGraphDestroy(g);
    if (!ok) {
      cudaGetLastError();
      graphs_broken_ = true;
    } else {
      it = graphs_.emplace(key, ge).first;
    }
  }
  if (it != graphs_.end()) {
    BCK(cudaGraphLaunch(it->second, stream_));
  } else {
    for (int i = 0; i < iters; ++i) {
      int rc = launch_iteration(stream_, with_check(i));
      if (rc != MCF_OK) return rc;
    }
  }
  BCK(cudaMemcpyAsync(h_sc_, d_sc_, (size_t)max_slots_ * sizeof(BatchScalars), cudaMemcpyDeviceToHost, stream_));
  BCK(cudaStreamSynchronize(stream_));
  for (int s = 0; s < max_slots_; ++s) {
    BatchSlot& sl = slots_[s];
    if (!sl.used || sl.finished || h_sc_[s].active) continue;
    sl.finished = true;
    const DevScalars& d = h_sc_[s].s;
    if (d.numeric_error) sl.status = MCF_ERR_NUMERIC;
    else if (h_sc_[s].done == 1 || sl.opts.stop_mode == MCF_STOP_NONE) sl.status = MCF_OK;
    else sl.status = MCF_ERR_NOT_CONVERGED;
    finished_.push_back(s);
    lists_dirty_ = true;
  }
  return MCF_OK;
}

std::vector<int> BatchEngine::take_finished() {
  std::vector<int> out;
  out.swap(finished_);
  return out;
}

// The parts of one slot, one allocation from the pool of the problems' states in the engine's
// stream order: with three cudaMalloc and cudaFree and three synchronisations per slot instead, a
// batch of 64 small networks took 6.2 ms around one iteration, now 3.8.
double* BatchEngine::alloc_parts(size_t bytes) {
  double* ptr = nullptr;
  const cudaError_t e = pool_ ? pool_alloc((void**)&ptr, bytes, pool_, stream_) : cudaMalloc((void**)&ptr, bytes);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return nullptr;
  }
  return ptr;
}

void BatchEngine::release(int s, bool wait) {
  BatchSlot& sl = slots_[s];
  if (!sl.used) return;
  cudaSetDevice(device_);
  const DevScalars& d = h_sc_[s].s;
  mcf_result& r = sl.res;
  r.iters = d.k;
  r.feasible = d.feasible;
  r.utility = d.P;
  r.dual_bound = d.D;
  r.r = d.r;
  r.r_over_nm = d.r / ((double)sl.p->n * (double)sl.p->m);
  r.rel_gap = d.rel_gap;
  r.rel_cons = d.rel_cons;
  r.rel_stat = d.rel_stat;
  r.rel_kkt = d.rel_kkt;
  r.nonpos_frac = d.nonpos_frac;
  r.omega = d.omega;
  r.delta_f = d.dF;
  r.delta_y = d.dY;
  r.omega_frozen_at = (d.freeze >= 0 && d.freeze <= d.k) ? d.freeze : -1;
  r.stalled = h_sc_[s].stalled;
  r.status = sl.status;
  batch_finish_state(sl.p, h_sc_[s].parity, d, stream_);
  if (pool_) cudaFreeAsync(sl.parts, stream_);
  else cudaFree(sl.parts);
  if (wait) cudaStreamSynchronize(stream_);
  const mcf_result keep = sl.res;
  const int st = sl.status;
  sl = BatchSlot();
  sl.res = keep;
  sl.status = st;
  h_sc_[s].active = 0;
  lists_dirty_ = true;
}

// ------------------------------------------------------------------ autotuner
// For a default class c (the smallest shape covering the chunks), the candidates are every
// shape whose capacity covers the class's largest vector and is at most 4x the class
// capacity (warp groups with more chunks per lane, or CTA groups). Each candidate runs 3 + 10
// batched iterations of 16 synthetic instances (ring plus 7 random out-edges per node, the
// class's largest n, log utility) in a private engine; the fastest per iteration wins. The
// choice depends only on the class, so an instance's shape never depends on the mix.

namespace {
std::mutex g_tune_mu;
std::map<std::pair<int, int>, int> g_tuned;   // (device, default class) -> tuned class

uint64_t splitmix(uint64_t& x) {
  uint64_t z = (x += 0x9e3779b97f4a7c15ULL);
  z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ULL;
  z = (z ^ (z >> 27)) * 0x94d049bb133111ebULL;
  return z ^ (z >> 31);
}

mcf_problem* synthetic_problem(int n, uint64_t seed) {
  const int deg = std::min(8, n - 1);
  std::vector<int32_t> t, h;
  for (int i = 0; i < n; ++i) {
    std::vector<int32_t> used{i, (i + 1) % n};
    t.push_back(i);
    h.push_back((i + 1) % n);
    while ((int)used.size() < deg + 1) {
      const int j = (int)(splitmix(seed) % (uint64_t)n);
      if (std::find(used.begin(), used.end(), j) != used.end()) continue;
      used.push_back(j);
      t.push_back(i);
      h.push_back(j);
    }
  }
  const int m = (int)t.size();
  std::vector<double> cap(m), w((size_t)n * n, 1.0);
  for (int l = 0; l < m; ++l) cap[l] = 1.0 + 9.0 * (double)(splitmix(seed) >> 11) / 9007199254740992.0;
  for (auto& x : w) x = 0.5 + (double)(splitmix(seed) >> 11) / 9007199254740992.0;
  mcf_problem* p = nullptr;
  mcf_create_problem(n, m, t.data(), h.data(), cap.data(), MCF_LOG, w.data(), nullptr, 0, &p);
  return p;
}

int tune_class(int device, int c0) {
  const int cap0 = kShapes[c0].group * kShapes[c0].vpt;
  const int n = std::max(4, cap0 * 4 - 8);
  std::vector<int> cands;
  for (int s = 0; s < NUM_SHAPES; ++s) {
    const int cap = kShapes[s].group * kShapes[s].vpt;
    // (shapes of one group are one kernel)
    if (s != c0 && batch_group(s) == batch_group(c0)) continue;
    if (cap >= cap0 && cap <= 4 * cap0) cands.push_back(s);
  }
  constexpr int kCount = 16;
  std::vector<mcf_problem*> probs;
  for (int i = 0; i < kCount; ++i) probs.push_back(synthetic_problem(n, 1000003ULL * (i + 1)));
  mcf_options o;
  mcf_options_default(&o);
  o.stop_mode = MCF_STOP_NONE;
  o.max_iters = 1 << 30;
  o.device = device;
  int best = c0;
  double best_t = 1e300;
  for (int c : cands) {
    BatchEngine eng(device, kCount);
    if (eng.init() != MCF_OK) break;
    bool ok = true;
    for (int i = 0; i < kCount && ok; ++i) {
      int slot = 0;
      ok = probs[i] && eng.add(probs[i], o, nullptr, &slot, c) == MCF_OK;
    }
    if (!ok || eng.step(3) != MCF_OK) continue;
    const auto t0 = std::chrono::steady_clock::now();
    if (eng.step(10) != MCF_OK) continue;
    const double dt = std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count();
    if (dt < best_t) { best_t = dt; best = c; }
  }
  for (mcf_problem* p : probs) mcf_destroy_problem(p);
  return best;
}
}  // namespace

int batch_class_for(int device, int nchunks, bool autotune) {
  const int c0 = pick_shape(nchunks);
  if (c0 < 0 || !autotune) return c0;
  {
    std::lock_guard<std::mutex> g(g_tune_mu);
    auto it = g_tuned.find({device, c0});
    if (it != g_tuned.end()) return it->second;
  }
  const int c = tune_class(device, c0);
  std::lock_guard<std::mutex> g(g_tune_mu);
  g_tuned.emplace(std::make_pair(device, c0), c);
  return g_tuned[{device, c0}];
}

}  // namespace pdmcf

using namespace pdmcf;

// Solve `count` independent problems together (FP32; an edge launch per group of shapes and one
// launch of each other phase for all of them). results[i] receives problem i's scalars and, if
// its T/F/Y pointers are set, its outputs. Returns MCF_OK when every problem met its stop rule.
extern "C" int mcf_solve_batch(mcf_problem** probs, int count, const mcf_options* opts,
                               mcf_result* results) {
  if (count < 0 || (count > 0 && (!probs || !results))) {
    set_error("problems or results are NULL");
    return MCF_ERR_INVALID;
  }
  int rc = pdmcf::validate_options(opts);
  if (rc != MCF_OK) return rc;
  if (opts->precision != MCF_FP32) {
    set_error("batched solves run FP32 iterates");
    return MCF_ERR_INVALID;
  }
  if (count == 0) return MCF_OK;
  for (int i = 0; i < count; ++i)
    if (probs[i] && probs[i]->busy.load() > 0) {
      set_error("a problem in the batch has an outstanding ticket (collect it with mcf_poll or "
                "mcf_wait, or discard it with mcf_cancel)");
      return MCF_ERR_BUSY;
    }
  const auto t0 = std::chrono::steady_clock::now();
  std::vector<std::unique_lock<std::mutex>> locks;   // held until the engine is gone
  BatchEngine eng(opts->device, count);
  rc = eng.init();
  if (rc != MCF_OK) return rc;
  for (int i = 0; i < count; ++i) {
    if (!probs[i]) {
      set_error("NULL problem in batch");
      return MCF_ERR_INVALID;
    }
    for (int j = 0; j < i; ++j)
      if (probs[j] == probs[i]) {
        set_error("a problem appears twice in the batch");
        return MCF_ERR_INVALID;
      }
    locks.emplace_back(probs[i]->lock);
    int slot = 0;
    const int nchunks = ((probs[i]->n + 7) / 8 * 8) / 4;
    const int cls = opts->shape >= 0 && opts->shape < NUM_SHAPES
                        ? opts->shape
                        : batch_class_for(opts->device, nchunks, opts->autotune != 0);
    rc = eng.add(probs[i], *opts, nullptr, &slot, cls);
    if (rc != MCF_OK) return rc;
  }
  const int chunk = std::max(1, std::min(opts->k_check, 50));
  while (eng.active_count() > 0) {
    rc = eng.step(chunk);
    if (rc != MCF_OK) return rc;
    (void)eng.take_finished();
  }
  const double secs = std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count();
  int worst = MCF_OK;
  for (int i = 0; i < count; ++i) eng.release(i, i + 1 == count);
  for (int i = 0; i < count; ++i) {
    mcf_result& out = results[i];
    double *T = out.T, *F = out.F, *Y = out.Y;
    out = eng.slot(i).res;
    out.T = T;
    out.F = F;
    out.Y = Y;
    out.seconds = secs;
    if ((T || F || Y) && (out.status == MCF_OK || out.status == MCF_ERR_NOT_CONVERGED)) {
      // All on one stream: each call's staging buffer is the one that the call before gave back. On
      // 64 streams the pool had to find or map another one: 64 networks 36.5 instead of 28.2 ms.
      rc = device_copy_outputs(probs[i], &out, eng.stream());
      if (rc != MCF_OK) return rc;
    }
    if (out.status != MCF_OK && worst == MCF_OK) worst = out.status;
  }
  return worst;
}
