// pdmcf_batch_engine.h — host engine that advances many resident instances together.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>
#include <map>
#include <tuple>
#include <vector>

#include "pdmcf_batch.cuh"
#include "pdmcf_internal.h"
#include "pdmcf_kernels.h"

namespace pdmcf {

using BatchKernel = void (*)(const BatchInst*, BatchClassDev);
// Edge-phase launches: shapes with a warp per edge share one for rows of up to 512 entries and
// one for up to 1024, each longer shape has its own. Node phase and check serve all instances.
constexpr int NUM_GROUPS = 2 + NUM_SHAPES - 4;
constexpr int batch_group(int shape) { return shape < 3 ? 0 : shape == 3 ? 1 : shape - 2; }
static_assert(kShapes[3].group == 32 && kShapes[4].group > 32, "the first four shapes are warp shapes");
struct BatchTable {
  BatchKernel edge[NUM_GROUPS];
  int block[NUM_GROUPS];
  BatchKernel node, node_chk, check;   // 256 threads
};
const BatchTable& batch_table();

// Device buffers of one instance the engine owns besides the problem's DeviceState.
struct BatchSlot {
  bool used = false;
  mcf_problem* p = nullptr;
  mcf_options opts{};
  void* tag = nullptr;
  int cls = -1;
  double* parts = nullptr;   // pe, pn and pc of its BatchInst
  int64_t bytes = 0;
  bool finished = false;
  int status = MCF_PENDING;
  mcf_result res{};
};

// Advances every resident instance by one PDHG iteration per step with one launch per
// phase and shape class. Not thread-safe: one owner thread drives it.
class BatchEngine {
 public:
  BatchEngine(int device, int max_slots);
  ~BatchEngine();
  int init();                         // allocate the tables; MCF_OK or an error
  int device() const { return device_; }
  cudaStream_t stream() const { return stream_; }
  int free_slots() const;
  int active_count() const;
  // Admit an FP32 request: allocates/initialises the instance state (cold or warm).
  int add(mcf_problem* p, const mcf_options& o, void* tag, int* slot_out, int cls = -1);
  // Run `iters` batched iterations (graph-captured), then refresh the host scalar mirror
  // and mark instances whose stop rule fired as finished.
  int step(int iters);
  // Finished slots since the last call.
  std::vector<int> take_finished();
  // Copy the slot's final state back into its problem and free the slot. The state may be used
  // on other streams once the engine's has been waited for: by this call or a later one with wait.
  void release(int slot, bool wait = true);
  const BatchSlot& slot(int s) const { return slots_[s]; }
  static int64_t extra_bytes(const mcf_problem* p);   // engine buffers per instance

 private:
  double* alloc_parts(size_t bytes);
  int step_impl(int iters);
  int upload_lists();
  int launch_iteration(cudaStream_t st, bool with_check);
  uint64_t check_iterations(int iters) const;
  void destroy_graphs();

  int device_;
  int max_slots_;
  cudaStream_t stream_ = nullptr;
  cudaMemPool_t pool_ = nullptr;        // of the problems' states; nullptr: plain allocations
  int sms_ = 0;
  BatchInst* d_insts_ = nullptr;
  BatchScalars* d_sc_ = nullptr;
  BatchScalars* h_sc_ = nullptr;       // pinned mirror
  int* d_slot_list_ = nullptr;
  int* d_nslots_ = nullptr;
  // work lists of the edge-phase launches and, at NUM_GROUPS, of all instances
  int* d_cls_count_ = nullptr;          // [NUM_LISTS]
  int* d_cls_inst_ = nullptr;           // [NUM_LISTS * max_slots]
  long long* d_cls_eoff_ = nullptr;     // [NUM_LISTS * (max_slots + 1)]
  long long* d_cls_noff_ = nullptr;
  static constexpr int NUM_LISTS = NUM_GROUPS + 1;
  int grid_edge_[NUM_GROUPS] = {};
  int grid_node_ = 0, grid_node_chk_ = 0, grid_check_ = 0;
  std::vector<BatchSlot> slots_;
  std::vector<BatchInst> h_insts_;
  bool lists_dirty_ = true;
  unsigned class_mask_ = 0;
  // key: class mask, iterations per chunk, iterations of the chunk with a stop test
  std::map<std::tuple<unsigned, int, uint64_t>, cudaGraphExec_t> graphs_;
  bool graphs_broken_ = false;
  std::vector<int> finished_;
};

int batch_admit_shape(const mcf_problem* p);   // default shape class of an FP32 instance
// Shape class the batched engine uses for an instance with this many 16-byte chunks per
// vector: the default class, or the autotuned choice once tuning has run for it.
int batch_class_for(int device, int nchunks, bool autotune);

}  // namespace pdmcf
