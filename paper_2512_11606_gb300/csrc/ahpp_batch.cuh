// Batched multi-source push: state and launch parameters.
//
// A tile holds 32 (or 16) queries; every per-node state array of a tile is
// laid out [node][tile] (query-minor), so a warp that visits one neighbour
// reads or writes the tile's values of that neighbour as one 128-byte (or
// 64-byte) line.  Buffers are sized for the widest tile (kTile); the kernel
// instance of a launch's width indexes them with its own width.
// The graph is streamed once per round per tile, shared by all its queries.
// `groups` tiles run concurrently, each on its own slice of the persistent
// grid with its own barrier; a group walks its tiles one after another.  A
// tile's round on a small graph is a few latencies and two barriers long
// whatever its share of the chip: 2,000 nodes, 50 us a tile and round with one
// group, 7 with eight.
#pragma once
#include "../../include/ahpp.h"
#include "ahpp_internal.cuh"

namespace ahpp {

constexpr int kTile = 32;          // widest tile (queries per tile); serving uses this width
constexpr int kTileNarrow = 16;    // the other width of the batched kernel
constexpr int kRadixBits = 8;      // top-k digit width (per-lane histograms of 256 bins)
constexpr int kRadixBins = 1 << kRadixBits;
constexpr int kRadixPasses = 64 / kRadixBits;
// Block size of the batched kernel: one block per SM (80 registers a thread).
constexpr int kBThreads = 768;
constexpr int kBWarps = kBThreads / 32;
constexpr int kBMinBlocks = 1;
// Dynamic shared memory per block: each warp's ring of kTRing units, then a
// region that holds the rows most gathered during a phase, and between phases
// the block reductions, the top-k radix histograms and the sort buffer.
constexpr uint32_t kTRing = 2;
constexpr size_t kTRingBytes = (size_t)kBWarps * kTRing * 512;
constexpr uint32_t kTHubRows = 256;
constexpr size_t kBatchSmem = kTRingBytes + (size_t)kTHubRows * 128;

// A round's accumulators of one query.  Every block adds three words per
// query, 15,000 atomics to a tile's 32 records at 152 blocks: they go to
// kAccCopies copies, so that the L2 slices share them, and the two counts take
// one 64-bit add (the barrier after phase 2: 17,000 cycles with one copy of four
// words on a graph whose round is 230,000, 8,000 so).
constexpr uint32_t kAccCopies = 8;
struct alignas(32) TAcc {
  uint32_t max_r_bits;             // max_u r_U after the round (float bits)
  uint32_t np;                     // Algorithm 4's counter: active V rows and attributes
  unsigned long long marked_deg;   // nodes marked, above bit 32 the sum of their degrees
  uint32_t max_rel_bits, above;    // APP(S): see RAcc
};
constexpr size_t kTAccs = 3 * (size_t)kAccCopies * kTile;

// Buffers of one tile in flight.
struct alignas(64) TileBuf {
  float *r_u = nullptr, *pi = nullptr, *pic = nullptr;   // [n_u][kTile]
  float* t = nullptr;                                    // [n_v + 2 n_acc][kTile], see TileLayout
  float* split_acc = nullptr;                            // [n_split_u][kTile]
  uint32_t* split_cnt = nullptr;                         // [n_split_u]
  TAcc* tacc = nullptr;                                  // [3][kAccCopies][kTile], rounds in turn
  RAcc* racc = nullptr;                                  // [2][kTile]: final sums of residues, reserves
  unsigned int* hist = nullptr;                          // [kRadixPasses][kTile][kRadixBins]
  unsigned long long* cand = nullptr;                    // [kTile][kmax] selected keys
  uint32_t* cand_cnt = nullptr;                          // [kTile]
};

constexpr uint32_t kMaxBatchGroups = 8;    // the configuration's and the autotuner's most
constexpr uint32_t kMaxGroups = 64;        // most tiles in flight at once

struct BatchState {
  TileBuf tb[kMaxGroups];      // host copies
  TileBuf* d_tb = nullptr;     // the same on the device
  GridBarrier* bars = nullptr; // [kMaxGroups], one per group
  uint32_t n_groups = 0;       // buffers allocated
  uint32_t kmax_cap = 0;       // candidate capacity per lane
};

struct BatchParams {
  uint32_t n = 0;                          // queries
  const uint32_t* q = nullptr;             // caller ids (device)
  const double* eps = nullptr;             // (device)
  const uint32_t* k = nullptr;             // (device), may be null when kmax == 0
  uint32_t kmax = 0;                       // output stride per query
  uint32_t* out_nodes = nullptr;           // [n][kmax] caller ids
  float* out_scores = nullptr;             // [n][kmax]
  uint32_t* out_n = nullptr;               // [n]
  ahpp_stats* out_stats = nullptr;         // [n], nullable
  float* out_dense = nullptr;              // [n][n_u] caller order, nullable
  const uint32_t* u_old2new = nullptr;
  const uint32_t* u_new2old = nullptr;
  int algo = 2;
  int kahan = 1;
  int switch_rule = 0;
  double lambda = 1.0;
  double log_inv = 0.0;
  uint32_t e_tot = 0;
  uint32_t max_rounds = 0;
  uint32_t groups = 1;
  const TileBuf* tbufs = nullptr;          // [groups] (batched) or [tiles] (serving)
  GridBarrier* bars = nullptr;             // [groups]
  const uint4 *ranges_t = nullptr, *ranges_u = nullptr;   // of a group's warps, two each (tile_ranges)
  float switch_unit = 0.f, switch_log = 0.f;   // see switch_due (rule 1's log; rule 0's is each query's)
  uint32_t tile = kTile;                   // queries per tile of this launch (kTile or kTileNarrow)
};

// Per-query control of one batched lane (kept in shared memory while a tile
// runs, in the slot table between serving steps).
struct LaneCtl {
  double eps_f;
  unsigned long long n_p, pushes;
  uint32_t rounds, switch_round;
  int phase, status, active, valid;
  float th_async, log_eps;   // smallest float above eps_f; log(eps_f)
};

enum : uint32_t { kSlotFree = 0, kSlotNew = 1, kSlotRunning = 2, kSlotFinished = 3 };

// One serving slot (lane qi % kTile of tile qi / kTile).  The host writes
// eps_f, q_new, k and state = kSlotNew; the step kernel moves it to Running
// and Finished; the host frees Finished slots after reading the results.
struct SlotState {
  LaneCtl ctl;
  double eps_f;
  uint32_t q_new;          // internal id of the source
  uint32_t k;              // top-k size (already clamped)
  uint32_t state;
  uint32_t pad;
};

struct ServeParams {
  SlotState* slots = nullptr;        // [n_tiles * kTile]
  uint32_t* tile_round = nullptr;    // [n_tiles] rounds run by each tile (accumulator rotation)
  const uint32_t* live = nullptr;    // [n_live] tiles to advance this step
  uint32_t n_live = 0;
  uint32_t rounds_per_step = 1;
};

int launch_batch(const DevGraph& g, const BatchParams& p, int grid, cudaStream_t stream);
int launch_serve_step(const DevGraph& g, const BatchParams& p, const ServeParams& sv, int grid, cudaStream_t stream);
int batch_max_grid(int sm_count);

}  // namespace ahpp
