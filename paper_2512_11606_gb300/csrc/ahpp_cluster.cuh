// One query on one thread-block cluster, for graphs that its shared memory holds.
#pragma once
#include "ahpp_internal.cuh"
#include "ahpp_query1.cuh"

namespace ahpp {

constexpr int kClThreads = 1024;
constexpr int kClWarps = kClThreads / 32;
constexpr uint32_t kClBlocks = 16;        // blocks of a cluster
// Warps that walk; the last one of a block runs the round's control meanwhile.
constexpr int kClWalkers = kClWarps - 1;
// A step: four entries for each lane of a warp, 16-bit indices and FP32
// coefficients ([32] uint2, then [32] float4).
constexpr uint32_t kClStepBytes = 768;

// Dynamic shared memory of a block, at most (the kernel's own takes 3 KB of the 227).
constexpr uint32_t kClSmemMax = 223 * 1024;

// Rows of one phase, cut into one contiguous range per block (of a multiple of
// four rows): t, the rows of V and then of A, and u, the rows of U.  cta[b] =
// {first row, rows, first item, items}; steps[b] = {first step, steps}.  A block's
// rows have local places: row r - first in place r - first, the further chunks of
// long rows after the rows.  Items (slices of consecutive rows, or a chunk of a
// row), whose lanes walk `columns` entries each:
//   {first place | columns << 16, rows | lg lanes per row << 8}
// meta[first row + i] = {degree, first of the row's further chunks | their number
// << 16}.  ranges[b * kClWalkers + w]: warp w's {item begin, end, step begin, end},
// counted within the block.  (Choosing the order of a row's entries so that a
// column's lookups fall into different banks changed nothing.)
struct ClusterRows {
  const uint4* cta = nullptr;
  const uint2* steps = nullptr;
  const uint2* items = nullptr;
  const uint2* meta = nullptr;
  const uint4* ranges = nullptr;
  uint32_t rows_max = 0, items_max = 0, places_max = 0;   // of any block
};

struct ClusterLayout {
  uint32_t n_blocks = 0;                  // of the cluster (0: the graph has no such layout)
  uint32_t smem_bytes = 0;
  ClusterRows t, u;                       // u's indices: t's rows
  const uint4* steps = nullptr;           // t's, then u's
};

int launch_cluster(const DevGraph& g, const ClusterLayout& c, const Q1State& s, const Q1Params& p,
                   cudaStream_t stream);

}  // namespace ahpp
