// Internal declarations shared by the library's translation units.
#pragma once

#include <cuda_runtime.h>

#include <atomic>
#include <cstdint>
#include <deque>
#include <functional>
#include <memory>
#include <mutex>
#include <string>
#include <unordered_map>
#include <utility>
#include <vector>

#include "tp.h"

namespace tp {

// Device-side error codes written to an error word (Workspace::err).
enum DeviceError : int {
  kDevOk = 0,
  kDevTimeout = 1,     // a bounded wait ran out of iterations
  kDevBounds = 2,      // debug bounds check failed
  kDevRace = 3,        // checked launch: a tile claimed twice or off the program's map
};

void set_detail(const std::string& s);
tp_status fail(tp_status s, const std::string& detail);
tp_status cuda_fail(cudaError_t e, const char* what);

size_t dtype_size(int32_t dtype);
bool is_contiguous(const tp_tensor& t);
int64_t numel(const tp_tensor& t);
// Byte range [lo, hi) reachable through the view (lo == hi for empty views).
void byte_range(const tp_tensor& t, uintptr_t* lo, uintptr_t* hi);

}  // namespace tp

namespace tp {
// `count` in-flight holds of one partition by work queued on one stream.
struct Hold {
  tp_partition* p;
  cudaStream_t stream;
  int64_t count;
};
using HoldKey = std::pair<tp_partition*, cudaStream_t>;
struct HoldKeyHash {
  size_t operator()(const HoldKey& k) const {
    return std::hash<const void*>()(k.first) * 31u ^ std::hash<const void*>()(k.second);
  }
};

// What the kernels of an operation, an event's operations or a graph report to
// as long as any of them may run.
struct Workspace {
  // Error word (DeviceError) in pinned host memory that kernels write to
  // directly, and only when something failed: an operation that went well
  // moves nothing to report so.
  int* err = nullptr;
};
// Device memory, kept by what may still use it: the operation being launched,
// the event that it is recorded into, its graph.
using Partial = std::shared_ptr<float>;      // matrix-vector partial sums (kPartialFloats)
using Counter = std::shared_ptr<unsigned>;   // of a tile queue
struct Scratch {
  std::vector<Partial> partials;
  std::vector<Counter> counters;
};
// What one SYNC operation at a time has of these.
struct Lent {
  Workspace* ws = nullptr;
  Partial sums;
  Counter counter;
};

// Workspaces of a context: lent to SYNC operations, each for its call, to an event
// and to a graph until it is gone and the work recorded into it has ended. It
// grows by blocks as more are out at a time. The last holder (the context, its
// events, its graphs) frees the words, so that events and graphs may be
// destroyed after their context; buffers on the device go with the context.
class WorkspacePool : public std::enable_shared_from_this<WorkspacePool> {
 public:
  ~WorkspacePool();
  cudaError_t take(Workspace** out);
  void give(Workspace* w);
  cudaError_t get(Partial* out);
  cudaError_t get(Counter* out);
  void close();                     // the context goes, with no work in flight
  std::atomic<bool> closed{false};
  static constexpr int64_t kPartialFloats = int64_t(1) << 20;
 private:
  static constexpr int kBlock = 4096;
  std::mutex mu_;
  std::deque<Workspace> all_;       // (a deque: their addresses stay)
  std::vector<Workspace*> free_;
  std::vector<int*> blocks_;        // error words, kBlock each
  std::vector<float*> partials_;    // every buffer of partial sums, and the idle ones
  std::vector<float*> free_partials_;
  std::vector<unsigned*> counter_blocks_;  // kBlock each
  std::vector<unsigned*> free_counters_;
};
}  // namespace tp

struct tp_ctx {
  int32_t device = 0;
  int32_t sm_count = 0;
  int32_t cc_major = 0, cc_minor = 0;
  size_t smem_optin = 0;
  std::mutex mu;
  // in-flight holds: (partition, stream) -> count; work chained on one
  // stream adds to the entry's count
  std::unordered_map<tp::HoldKey, int64_t, tp::HoldKeyHash> busy;
  tp_graph* capturing = nullptr;    // graph being captured, if any
  std::shared_ptr<tp::WorkspacePool> pool;
  tp::Workspace* own = nullptr;     // of launches that no operation reports for
  std::vector<tp::Lent> idle;       // of SYNC operations that have ended (under mu)
  // Device workspace, allocated once at creation.
  float* d_scratch = nullptr;       // small float scratch (kScratchFloats)
  uint32_t* d_claims = nullptr;     // tile-claim bitmap of checked launches (kClaimBits), all clear
  unsigned* d_claim_done = nullptr; // CTAs of the running checked launch that finished
  static constexpr int kScratchFloats = 4096;
  static constexpr int64_t kClaimBits = int64_t(1) << 26;   // 8 MiB
};

struct tp_partition {
  tp_ctx* ctx = nullptr;
  tp_tensor t{};
  int32_t rank = 0;
  int64_t shape[3] = {1, 1, 1};
  int64_t tile[3] = {1, 1, 1};
  int64_t grid[3] = {1, 1, 1};
  int64_t num_tiles = 0;
  int64_t num_programs = 0;
  int32_t kind = TP_MAP_IDENTITY;
  uintptr_t lo = 0, hi = 0;  // output bytes
  std::atomic<int> busy{0};  // number of in-flight holds
};

namespace tp {
// What a replay needs: kept by the graph and by the events that its replays in
// flight were recorded into.
struct GraphRun {
  explicit GraphRun(std::shared_ptr<WorkspacePool> p) : pool(std::move(p)) {}
  ~GraphRun();
  std::shared_ptr<WorkspacePool> pool;
  Workspace* ws = nullptr;           // of the recorded operations
  cudaGraph_t graph = nullptr;
  cudaGraphExec_t exec = nullptr;
  bool check_err = false;
  Scratch scratch;
};
}  // namespace tp

struct tp_event {
  tp_ctx* ctx = nullptr;
  std::shared_ptr<tp::WorkspacePool> pool;
  cudaEvent_t ev = nullptr;
  bool recorded = false;
  bool check_err = false;
  cudaStream_t stream = nullptr;  // stream of the last record
  tp::Workspace* ws = nullptr;    // of the operations recorded into it
  tp::Scratch scratch;            // that their work in flight uses
  std::vector<std::shared_ptr<tp::GraphRun>> replays;  // graphs replayed into it
  std::vector<tp::Hold> held;   // holds released when the event completes (appended per op)
};

struct tp_graph {
  tp_ctx* ctx = nullptr;
  std::shared_ptr<tp::GraphRun> run;
  cudaStream_t stream = nullptr;
  bool ended = false;
  bool uses_partial = false;         // a recorded operation does
  std::vector<tp_partition*> parts;  // partitions written by recorded nodes
};

namespace tp {

// Makes the context's device current in the calling thread for one entry
// point: a thread that has not used CUDA yet gets the device's primary
// context bound (driver-API calls such as TMA descriptor encoding need a
// current context), and a caller whose current device differs gets it back
// when the guard goes out of scope.
struct DeviceGuard {
  int restore = -1;
  DeviceGuard() = default;
  explicit DeviceGuard(const tp_ctx* ctx) { bind(ctx); }
  DeviceGuard(const DeviceGuard&) = delete;
  DeviceGuard& operator=(const DeviceGuard&) = delete;
  void bind(const tp_ctx* ctx) {
    static thread_local bool bound = false;
    if (!ctx) return;
    int cur = -1;
    if (cudaGetDevice(&cur) != cudaSuccess) cur = -1;
    if (bound && cur == ctx->device) return;
    if (cudaSetDevice(ctx->device) == cudaSuccess) {
      if (bound && cur >= 0 && cur != ctx->device && restore < 0) restore = cur;
      bound = true;
    }
  }
  ~DeviceGuard() {
    if (restore >= 0) cudaSetDevice(restore);
  }
};

// Launch protocol shared by every operation (§3.2 / §3.3 semantics):
//   begin(): validate exec + aliasing + busy state, mark the output busy
//            (SYNC/ASYNC) or record it into the capturing graph (CAPTURE);
//   end():   after the kernel launches, synchronize + release (SYNC), record
//            the completion event (ASYNC), or nothing (CAPTURE).
struct Op {
  Op() = default;
  explicit Op(const char* op_name) : name(op_name) {}
  const char* name = "op";   // entry point, for the TP_LOG trace
  tp_ctx* ctx = nullptr;
  const tp_exec* ex = nullptr;
  cudaStream_t stream = nullptr;
  std::vector<tp_partition*> outs;
  bool check_err = false;   // kernel may write the error word
  int* err = nullptr;       // error word for this operation's kernels (set by begin)
  Lent lent;                // SYNC: the operation's workspace; and its device memory (partial(), queue())
  bool queued = false;      // the counter's reset is enqueued or recorded
  bool marked = false;
  bool allow_checked = false;  // the op implements TP_EXEC_CHECKED (set before begin)
  bool allow_inject = false;   // the op implements TP_EXEC_INJECT_TIMEOUT (set before begin)
  bool allow_static_weights = false;  // the op implements TP_EXEC_STATIC_WEIGHTS (set before begin)
  DeviceGuard device;          // the context's device is current while the op launches

  tp_status begin(tp_ctx* c, const tp_exec* e, std::initializer_list<tp_partition*> outputs,
                  std::initializer_list<const tp_tensor*> inputs);
  tp_status begin_lists(tp_ctx* c, const tp_exec* e, const std::vector<tp_partition*>& outputs,
                        const std::vector<tp_tensor>& inputs);
  tp_status begin_impl(tp_ctx* c, const tp_exec* e, const std::vector<tp_partition*>& outputs,
                       const std::vector<const tp_tensor*>& inputs);
  tp_status end(cudaError_t launch_err);
  tp_status end_impl(cudaError_t launch_err);
  // Undo begin() after a failure that launched nothing (keeps the detail).
  void abort();
  // A buffer of WorkspacePool::kPartialFloats that no work uses which may run
  // beside this operation's.
  tp_status partial(float** out);
  // Likewise a tile-queue counter, zeroed on the operation's stream.
  tp_status queue(unsigned** out);
  void keep_scratch();  // hands both to the event or graph (ctx->mu held)
  void release();       // ends the outputs' holds, returns a SYNC operation's workspace
  bool capturing() const { return ex->mode == TP_CAPTURE; }
};

// Status of the error in `word` (or, when it holds none, in the context's
// word), read after the work that may write it has completed; clears it.
tp_status take_error(tp_ctx* ctx, int* word);
// Dynamic shared memory a CTA may opt in to (sm_103).
constexpr int kSmemOptin = 232448;
// Lets launches of kernel K ask for up to `bytes` of dynamic shared memory.
// The limit is the process's, so `bytes` is a constant of the instance, the
// most that any launch of it needs: a launch that set its own size could lower
// the limit under another thread's launch. Set once per device.
template <auto K>
cudaError_t allow_smem(int bytes) {
  static std::atomic<uint64_t> done{0};  // a bit per device
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const uint64_t bit = dev < 64 ? uint64_t(1) << dev : 0;
  if (done.load(std::memory_order_acquire) & bit) return cudaSuccess;
  e = cudaFuncSetAttribute(K, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e == cudaSuccess) done.fetch_or(bit, std::memory_order_release);
  return e;
}

// An ASYNC launch may record `ev` on `stream`: OK when the event tracks no
// unfinished work on another stream (completed work is released first).
tp_status event_claim(tp_event* ev, cudaStream_t stream);
// The context's tile-claim bitmap for one checked launch (TP_EXEC_CHECKED)
// that may set up to `bits` bits; the launch's last CTA clears them again.
tp_status claims_for(tp_ctx* ctx, int64_t bits, uint32_t** claims, unsigned** done);

// Kernel launchers (defined in the kernel translation units).
enum MapOp : int { kMapAxpy = 0, kMapGeluMul = 1, kMapScale = 2, kMapAddAccum = 3 };
tp_status launch_map(tp_ctx* ctx, tp_partition* out, int op, float alpha, const tp_tensor* x,
                     const tp_tensor* y, const tp_exec* ex, cudaStream_t stream, unsigned* queue, int* err);
tp_status launch_gemm_simt(tp_ctx* ctx, tp_partition* c, const tp_tensor* a, const tp_tensor* b,
                           const tp_gemm_config* cfg, const tp_exec* ex, cudaStream_t stream,
                           unsigned* queue);
tp_status launch_gemm_tc(tp_ctx* ctx, tp_partition* c, const tp_tensor* a, const tp_tensor* b,
                         const tp_gemm_config* cfg, const tp_exec* ex, cudaStream_t stream, int* err);

// Programs of the tensor-core GEMM (CTA pairs for 256-row tiles, CTAs
// otherwise) that can be resident at once for `cfg`.
tp_status gemm_tc_resident(tp_ctx* ctx, const tp_gemm_config* cfg, int32_t* programs);
// Whether the autotuner tries config c of its space on an M x N x K problem
// of `dtype` (a config it does not try is never proposed for it either).
bool autotune_config_runs(const tp_ctx* ctx, int64_t M, int64_t N, int64_t K, int32_t dtype,
                          const tp_gemm_config& c);

tp_status launch_gemm_tc_impl(tp_ctx* ctx, tp_partition* c, const tp_tensor* a, const tp_tensor* b,
                              const tp_gemm_config* cfg, const tp_exec* ex, cudaStream_t stream, int esize,
                              const float* scale_a, const float* scale_b, int* err);

}  // namespace tp
