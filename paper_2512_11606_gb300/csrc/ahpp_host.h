// Host-side definitions shared by the library's translation units.
#pragma once

#include <cuda_runtime.h>

#include <atomic>
#include <memory>
#include <mutex>
#include <string>
#include <vector>

#include <nvtx3/nvToolsExt.h>

#include "../../include/ahpp.h"
#include "ahpp_internal.cuh"
#include "ahpp_query1.cuh"
#include "ahpp_batch.cuh"
#include "ahpp_cluster.cuh"
#include "ahpp_groups.h"
#include "ahpp_threads.h"

namespace ahpp {

// NVTX range over a host call (visible in a profiler's timeline; the calls
// do nothing unless a tool is attached).
struct NvtxRange {
  explicit NvtxRange(const char* name) { nvtxRangePushA(name); }
  ~NvtxRange() { nvtxRangePop(); }
  NvtxRange(const NvtxRange&) = delete;
  NvtxRange& operator=(const NvtxRange&) = delete;
};

void set_error(const std::string& msg);
int cuda_fail(cudaError_t e, const char* where);

#define AHPP_CUDA(call)                                   \
  do {                                                    \
    cudaError_t e_ = (call);                              \
    if (e_ != cudaSuccess) return ::ahpp::cuda_fail(e_, #call); \
  } while (0)

// f's status; AHPP_ENOMEM for what it throws (nothing throws across the ABI).
template <typename F>
int no_throw(const F& f) {
  try {
    return f();
  } catch (const std::exception& e) {
    set_error(std::string("host memory or threads: ") + e.what());
  } catch (...) {
    set_error("host code failed");
  }
  return AHPP_ENOMEM;
}

struct HostItems {
  std::vector<uint4> items;
  std::vector<uint32_t> split_nchunks;
};

// Work-item shapes.
struct ItemShape {
  uint32_t short_max;   // rows with at most this many neighbours are "short"
  uint32_t group_rows;  // short rows per item (single query: one per lane)
  uint32_t group_nnz;   // max neighbours per short item (batched)
  uint32_t chunk;       // neighbours per chunk of a long row
};

HostItems build_items(const std::vector<uint32_t>& deg, const ItemShape& shape);
// Device allocation tracked by the graph.
struct DevBuf {
  void* p = nullptr;
  size_t bytes = 0;
};

}  // namespace ahpp

namespace ahpp {
// Places in a single query's result block (the barrier, which blocks poll, has a
// line of its own).
constexpr size_t kOutBits = 128, kOutBar = 256, kOutTop = 384;
static_assert(sizeof(QCtl) <= kOutBits, "control block");
constexpr size_t kOutBytes = kOutTop + 8 * (size_t)AHPP_MAX_K;
}  // namespace ahpp

namespace ahpp {
// A pull layout: its device arrays and what the host keeps of it.  `kept`: a
// launch that a caller made or captured may hold its addresses.
struct Layout {
  ahpp_graph* g;
  std::vector<void*> bufs;
  uint64_t bytes = 0;
  bool kept = false;
  explicit Layout(ahpp_graph* graph) : g(graph) {}
  Layout(const Layout&) = delete;
  Layout& operator=(const Layout&) = delete;
  ~Layout();
  // Device memory of the layout, filled from src if given (nullptr on failure).
  void* put(size_t n, const void* src);
};
struct Q1Built : Layout {
  using Layout::Layout;
  Q1Layout q;
  // lanes of the shortest rows, blocks of the grid, shared memory per block
  uint32_t vw = 0, grid = 0, smem = 0;
};
struct TileBuilt : Layout {
  using Layout::Layout;
  TileLayout t;
  // the items' costs (running sums), first units and chunks, and the ranges cut so far
  struct Cost {
    std::vector<uint64_t> cost;
    std::vector<uint32_t> unit;
    uint32_t n_chunks = 0;
  } cost[2];
  struct Cut { uint32_t warps; const uint4* r[2]; };
  std::vector<Cut> cuts;
};
// Device memory that is freed with its scope.
struct ScratchBufs {
  std::vector<void*> bufs;
  ~ScratchBufs() { for (void* p : bufs) cudaFree(p); }
};
// The layouts of one kind that a graph has; `cur` is the one in use.
template <typename L>
struct Layouts {
  std::vector<std::unique_ptr<L>> all;
  L* cur = nullptr;
  // Frees those that nothing may refer to any more.
  void drop() {
    for (size_t i = all.size(); i-- > 0;)
      if (!all[i]->kept && all[i].get() != cur) all.erase(all.begin() + i);
  }
};
}  // namespace ahpp

struct ahpp_graph {
  ahpp_config cfg{};
  int device = 0;
  int sm_count = 0;
  cudaStream_t stream = nullptr;
  cudaStream_t upload_stream = nullptr;   // see ahpp::upload
  std::mutex mu;

  uint64_t n_u = 0, n_v = 0, n_a = 0, n_e = 0, n_ea = 0;
  double lambda = 1.0;
  uint32_t lambda_T = 0;
  bool bf16 = true;

  ahpp::DevGraph dg{};
  std::vector<ahpp::DevBuf> bufs;   // everything allocated for the graph
  size_t n_graph_bufs = 0;          // bufs[0, n_graph_bufs): the graph's own arrays (what a cache saves)
  uint64_t graph_bytes = 0;       // the graph's own arrays
  uint64_t layout_bytes = 0;      // what is built from them for the pull rounds

  // internal <-> caller id maps of U
  std::vector<uint32_t> h_u_old2new, h_u_new2old;
  uint32_t* d_u_new2old = nullptr;
  uint32_t* d_u_old2new = nullptr;

  // single-query state
  ahpp::Q1State q1{};
  ahpp::ClusterLayout cl{};       // small graphs: the layout of the cluster kernel, which then runs them
  ahpp::Layouts<ahpp::Q1Built> q1_layouts;   // single-query pull layouts (dg.q1: the current one's)
  uint32_t q1_max_blocks = 0;     // the most blocks of k_query1 that the device keeps resident
  uint32_t q1_dense_div = 32;     // pull rounds once the frontier covers > 1/dense_div of the edges
  std::string tune_log;           // the last autotune's measurements (JSON object)
  // what a single query leaves for the host, in one block that one copy fetches:
  // control, final maxima, barrier, then nodes and scores; host_out: its pinned copy
  char *d_out = nullptr, *host_out = nullptr;
  uint32_t n_split1 = 0;
  uint32_t n_long_u = 0;          // U rows of more than 2,048 entries
  uint64_t q1_bytes = 0;

  // batched state (allocated on first use, grown on demand)
  ahpp::BatchState bt{};
  uint32_t batch_tile = 32, batch_groups = 0;   // groups: 0 = by the graph's size and the batch's
  int bt_grid = 0;
  uint64_t tile_bytes = 0;
  ahpp::Layouts<ahpp::TileBuilt> tile_layouts;   // batched pull layouts (dg.tl: the current one's)

  // top-k scratch
  void* topk_scratch = nullptr;
  size_t topk_scratch_bytes = 0;

  // failure-detection self-test: the next launch's grid barriers start with
  // a counter that can never reach the block count (see reset_barrier)
  std::atomic<int> wait_trap{0};
  // and the allocation after this many more fails (< 0: none does)
  std::atomic<int64_t> alloc_trap{-1};

  cudaError_t dev_malloc(void** p, size_t bytes);   // every device allocation of the graph
  void* alloc(size_t bytes);          // the same, tracked (nullptr on failure)
  void release_all();
};

namespace ahpp {
// Lets this thread allocate while a stream is being captured (by it or, in the
// global mode, by any thread): what grows during a call lives as long as the
// graph, so a launch that is only recorded may hold it.
struct GrowInCapture {
  cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
  GrowInCapture() { cudaThreadExchangeStreamCaptureMode(&mode); }
  ~GrowInCapture() { cudaThreadExchangeStreamCaptureMode(&mode); }
  GrowInCapture(const GrowInCapture&) = delete;
  GrowInCapture& operator=(const GrowInCapture&) = delete;
};
// Host memory to the device, there when this returns: a plain cudaMemcpy from
// pageable memory may return before its copy has arrived, and the library's
// streams (and most callers') do not wait for the default stream it is on.
cudaError_t upload(ahpp_graph* g, void* dst, const void* src, size_t bytes);
// Clear n grid barriers before a persistent launch on `stream`.  When the
// graph's self-test trap is armed (ahpp_selftest_arm_wait_timeout) the
// counters are set far below any block count instead, so the launch's first
// barrier never fills and every block's bounded spin runs out; the trap is
// consumed by the first launch that sees it.
int reset_barriers(ahpp_graph* g, GridBarrier* bars, uint32_t n, cudaStream_t stream);
void set_batch_params(const ahpp_graph* g, BatchParams& p);
// Zero if the error words of n barriers are clear; kStatusWait if a wait gave
// up.  Synchronous (reads them from the device on `stream`).
int barrier_status(const GridBarrier* bars, uint32_t n, cudaStream_t stream, int* status);
int build_graph(const ahpp_graph_desc* desc, ahpp_graph* g);
// The kernels' algorithm id of an AHPP_* constant (-1 if none).
int kernel_algo(int algo);
// Makes the sliced layout of the single-query pull rounds with at least vec_width
// lanes per row (0: by the graph's size) the current one: one that the graph has,
// else a new one.  On failure the current one stays.
int use_q1_layout(ahpp_graph* g, uint32_t vec_width);
void use_q1_layout(ahpp_graph* g, Q1Built* b);
int build_cluster_layout(ahpp_graph* g);
// A single query's launch, on the cluster kernel where the graph has its layout.
int launch_single(const ahpp_graph* g, const Q1State& s, const Q1Params& p, cudaStream_t stream);
// Index into kChunkSizes of a configured chunk size (0: the default), -1 if
// it is not one of them.
int chunk_choice(uint32_t chunk);
// The same for the batched pull rounds, with chunks of kChunkSizes[choice] entries.
int use_tile_layout(ahpp_graph* g, uint32_t choice);
void use_tile_layout(ahpp_graph* g, TileBuilt* b);
// The current layouts are those that calls work on from here on; candidates that
// none did are freed.
void settle_layouts(ahpp_graph* g);
// The items' ranges for a tile on `warps` warps (made on first use; those of the
// whole grid's warps with the layout).
int tile_ranges(ahpp_graph* g, uint32_t warps, const uint4** t, const uint4** u);
// A launch's groups of `grid` blocks: *groups, or one where there is no memory for
// the ranges of so many; their blocks each and ranges.
int plan_groups(ahpp_graph* g, uint32_t grid, uint32_t* groups, uint32_t* per_group, BatchParams& p);
// Tiles that run at once, of n_tiles to be run (see groups_of).
uint32_t tile_groups(const ahpp_graph* g, uint32_t n_tiles, bool serving);
int alloc_query_state(ahpp_graph* g);
// Bytes of a single query's state as limits count them (ahpp_query_dense_noalloc's
// array, hbm_budget_bytes): its vectors and the sums of rows of more than 2,048
// entries, whatever the layout of the pull rounds adds to them.
size_t single_state_bytes(const ahpp_graph* g);
int run_lambda(ahpp_graph* g);
int topk_single(ahpp_graph* g, const float* d_score, uint32_t k, uint32_t* d_nodes,
                float* d_scores, uint32_t* d_n, cudaStream_t stream);
// The batched kernel's grid (computed once per graph).
int batch_plan(ahpp_graph* g);
int run_single_device(ahpp_graph* g, uint32_t q, double eps, uint32_t k, uint32_t* d_out_nodes,
                      float* d_out_scores, uint32_t* d_out_n, ahpp_stats* d_stats, cudaStream_t s);
}  // namespace ahpp
