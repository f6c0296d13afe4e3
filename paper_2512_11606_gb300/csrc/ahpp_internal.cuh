// Internal device structures and helpers of the AHPP push library (sm_103a).
//
// Graph layout in HBM (all ids relabeled internally: U, V and A are each
// sorted by degree, largest first, so that hub rows sit together and rows
// of similar length share a warp):
//   CSR_UV  rows u: off[n_u+1], idx v, w(u,v) raw (pull V->U), c_uv (push U->V)
//   CSR_VU  rows v: off[n_v+1], idx u, c_uv (pull U->V), w(u,v) raw (push V->U)
//   CSR_UA  rows u: off[n_u+1], idx a, w(u,a) raw (bf16 or f32)
//   CSC_AU  rows a: off[n_a+1], idx u, w(u,a) raw (bf16 or f32), au_pc (pull U->A)
//   c_uv(u,v) = (1-alpha)(1-beta) w(u,v) / (d(u) d(v))       (Eq. 1's two factors)
//   rnorm_u[u] = 1 / sum_a w(u,a),  cnorm_a[a] = 1 / sum_u w(u,a)   (Eq. 2)
// One round of Algorithm 3 maps the pushed residues p (marked U nodes) to
//   t_V[v] = sum_u c_uv(u,v) p_u                           = r(v) / d(v)
//   t_A[a] = (1-alpha) beta cnorm_a[a] sum_u w(u,a) rnorm_u[u] p_u = r(a) / W_col(a)
//   r_U'[j] = kept_j + sum_v w(j,v) t_V[v] + sum_a w(j,a) t_A[a]
// either as a pull (gather over the opposite direction, no atomics) or as a
// push (scatter with atomics from the frontier).
//
// Residue encoding: r_u[u] >= 0 is a residue; r_u[u] < 0 marks u as selected
// for the next U-push with residue -r_u[u].  The reserve update
// pi += alpha * p happens when the push is executed.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

namespace ahpp {

constexpr int kThreads = 256;          // threads per block of the top-k kernel
constexpr uint32_t kItemLong = 0x40000000u;   // item = one whole long row (warp-cooperative)
constexpr uint32_t kItemSplit = 0x80000000u;  // item = one chunk of a split row (| slot)
// Entries per chunk of a long row in the batched pull phases: the choices of
// the configuration and of ahpp_autotune.
constexpr int kChunkChoices = 3;
constexpr uint32_t kChunkSizes[kChunkChoices] = {128, 256, 512};
constexpr int kChunkDefault = 1;

// Work items of a push round's flush over one row space (split_nchunks, the chunks
// of each split row, is read by nothing but belongs to the graph cache's files).
//   x = first row; y = number of rows (short group, one row per lane) or a flag;
//   z, w = local neighbour range [z, w) for long / split rows.
struct ItemList {
  const uint4* items = nullptr;
  uint32_t n_items = 0;
  uint32_t n_split = 0;                 // split rows
  const uint32_t* split_nchunks = nullptr;
};

// Sliced rows of the single-query pull phases (built by ahpp_q1layout.cu).
// A step is 128 entries, four per lane of a warp; it is stored as units of
// 512 bytes, 16 per lane: an index unit (uint32) and a coefficient unit (FP32),
// or one compact unit of four uint16 indices and four bfloat16 weights per lane
// (attribute steps whose indices fit and whose weights are bfloat16).  An item
// is a slice of 32 / vw rows of similar length (rows are sorted by degree)
// with vw lanes on each row: entry k of a row sits in step k / (4 vw), lane
// (k / 4) % vw of the row, place k % 4; places past a row's end hold index 0
// and coefficient 0.  An item's V steps come before its attribute steps.  Rows
// too long for one warp are cut into chunk items (vw = 32, one row):
//   {first row, rows | lg vw << 8 | chunk << 31, V steps, attribute steps}
// Every warp of the grid owns one range of items, its chunks first, cut so that
// the warps' costs are about equal, and their units, which lie in the order in
// which it uses them: ranges[w] = {item begin, end, unit begin, end}.
struct Q1Rows {
  const uint4* items = nullptr;
  const uint4* ranges = nullptr;
  const uint4* units = nullptr;         // [units][32]
  const uint32_t* chunks_of = nullptr;  // chunks of each split row (rows [0, n_split))
  uint32_t n_split = 0;
};

// The attribute hop U -> A, cut by blocks of U rows: block b of rows (vb[b] =
// {first row, rows}) adds up its rows' share of every attribute it touches
// from a copy of their residues in shared memory, then one reduction per
// (block, attribute).  Items over (block, attribute) segments:
//   {first segment, segments | lg vw << 8, first unit, steps}
// with row indices local to the block; ranges[w] = {item begin, end, unit
// begin, end} of warp w % kQ1Warps of block w / kQ1Warps; meta[s] = {place in the
// copies of t_A, bits of the float scale of the sum} of segment s.
struct Q1Segs {
  const uint4* items = nullptr;
  const uint4* ranges = nullptr;
  const uint2* vb = nullptr;
  const uint2* meta = nullptr;
  const uint4* units = nullptr;
  uint32_t n_vb = 0, own_cap = 0;       // blocks of rows, and the most rows of one
};

constexpr uint32_t kTaCopies = 8;        // copies of t_A, at most

struct Q1Layout {
  Q1Rows v, u;
  Q1Segs s;
  const uint32_t *deg_u = nullptr, *deg_v = nullptr, *deg_a = nullptr;
  uint32_t n_warps = 0;                 // ranges per row space
  // copies of t_A that the blocks of the attribute hop add to in turn: with few
  // attributes their reductions meet in a few lines of L2 (at 2,000 attributes
  // 152 blocks' took 20,000 of the round's 75,000 cycles, and 3.31 ms a query
  // became 2.61 with four copies)
  uint32_t ta_copies = 1;
  uint32_t compact_a = 0, compact_s = 0;   // attribute steps of u / s in compact units
  // leading entries of p, t_A and t_V that the pull phases hold in shared memory
  uint32_t hub_u = 0, hub_a = 0, hub_v = 0;
};

// Sliced rows of the batched pull phases (built by ahpp_tilelayout.cu).  A warp
// walks four rows at once, eight lanes to a row.  An item is four consecutive
// rows (rows are sorted by degree), or four chunks of long rows:
//   {first row, or first chunk; rows | chunk << 31; entries of the longest;
//    first unit}
// The chunk items come first, then, up to `pool`, those that the warps share out
// beforehand (tile_ranges), then those that warps take `batch` at a time when they
// are done; a last item holds the number of units.
// Its entries lie in units of 512 bytes: 16 entries of each row, two to a
// lane's 16 bytes as {index, coefficient, index, coefficient}; pair j of row r
// is in place 8 r + (j + 2 r) % 8, so that the four rows' reads of a pair hit
// different banks.  Index kNoEntry: nothing.  chunk_row: a chunk's row.
constexpr uint32_t kNoEntry = 0xffffffffu;
struct TileRows {
  const uint4* items = nullptr;
  const uint4* units = nullptr;         // [units][32]
  const uint32_t* chunk_row = nullptr;
  uint32_t n_items = 0, pool = 0, batch = 1;   // items; first of the pool; items per grab
};

// Phase 1 (t) pulls the rows of V and of A from the residues into one table of
// 128-byte rows: row v of V in place v, or, where chunks add up their sums (V
// rows longer than a chunk, and every attribute), accumulated row j in place
// n_v + j, in one of two sets of n_acc places (rounds alternate; the other set
// is cleared meanwhile).  The split V rows come first among the accumulated
// ones, then the attributes.  Phase 2 (u) pulls the rows of U over both hops at
// once from that table; its indices are those of the first set.
struct TileLayout {
  TileRows t, u;
  const uint32_t* acc_deg = nullptr;    // degrees of the accumulated rows
  const uint32_t* chunks_of = nullptr;  // chunks of each split U row (rows [0, n_split_u))
  uint32_t n_acc = 0, n_split_u = 0;
  uint32_t acc_max = 0, split_u_max = 0;   // the most of any chunk choice (buffers are sized for them)
  uint32_t chunk = 0;                   // index into kChunkSizes
};

struct DevGraph {
  uint32_t n_u = 0, n_v = 0, n_a = 0;
  uint32_t n_e = 0, n_ea = 0;
  const uint32_t *uv_off = nullptr, *uv_idx = nullptr;
  const float *uv_w = nullptr, *uv_c = nullptr;
  const uint32_t *vu_off = nullptr, *vu_idx = nullptr;
  const float *vu_c = nullptr, *vu_w = nullptr;
  const uint32_t *ua_off = nullptr, *ua_idx = nullptr;
  const void* ua_w = nullptr;
  const uint32_t *au_off = nullptr, *au_idx = nullptr;
  const void* au_w = nullptr;
  const float* au_pc = nullptr;         // A->U: (1-alpha) beta w(u,a) / (sum_a' w(u,a') sum_u' w(u',a)) (FP32)
  const float* rnorm_u = nullptr;
  const float* cnorm_a = nullptr;
  float alpha = 0.f;
  float k_attr = 0.f;                   // (1 - alpha) * beta
  // single-query push rounds: work items of the V and attribute flush
  ItemList s1_v, s1_a;
  Q1Layout q1;                          // single-query pull rounds
  TileLayout tl;                        // batched pull rounds
};

template <typename WA>
__device__ __forceinline__ float wload(const void* p, uint32_t i) {
  return static_cast<float>(static_cast<const WA*>(p)[i]);
}
template <>
__device__ __forceinline__ float wload<__nv_bfloat16>(const void* p, uint32_t i) {
  return __bfloat162float(static_cast<const __nv_bfloat16*>(p)[i]);
}

// ---------------------------------------------------------------- control

enum : int { kPhaseAsync = 0, kPhaseSync = 1, kPhaseDone = 2 };
enum : int { kStatusOk = 0, kStatusCap = 1, kStatusWait = 2, kStatusBadArg = 3 };
// kAlgoAPPS: APP(S), APP's per-node thresholds with ASRP's synchronous switch
// (the ablation arm of Exp-2).
enum : int { kAlgoAPP = 1, kAlgoASRP = 2, kAlgoAPPS = 3 };

// Per-node thresholds r_max (|N(u)| + |A(u)|) in this phase (APP, and APP(S)
// before its switch), else one threshold for every node.
__device__ __forceinline__ bool per_node_threshold(int algo, int phase) {
  return algo == kAlgoAPP || (algo == kAlgoAPPS && phase != kPhaseSync);
}

// Per-query control block (global memory; written by one leader thread,
// mirrored in registers by every thread of a persistent kernel).
struct QCtl {
  double eps;
  double eps_f;        // ASRP: eps / lambda;  APP: r_max = eps / (|E| + |E_A|)
  double lambda;
  uint64_t n_p;        // Algorithm 4's counter
  uint64_t pushes;     // sum of frontier sizes
  uint32_t rounds;
  uint32_t switch_round;
  uint32_t dense_rounds;
  int phase;           // kPhaseAsync / kPhaseSync / kPhaseDone
  int status;          // kStatus*
  int dense;           // next round runs as a pull sweep
  uint32_t q;          // internal id of the source
  uint32_t pad;
  double resid_sum, reserve_sum, max_resid;   // final reductions
};

// Per-round accumulators of one query (triple-buffered by round index).
struct RAcc {
  unsigned int max_r_bits;   // max_u r_U after the round (float bits, values >= 0)
  uint32_t marked;           // nodes marked for the next U-push
  unsigned long long marked_deg;   // sum of |N(u)| + |A(u)| over marked nodes
  unsigned long long np_flush;     // sum of |N(v)| (r(v) > 0) + |A^-1(a)| (r(a) > 0)
  double sum_r;              // batched kernel: final sums
  uint32_t n_list_u;               // push rounds: marked list length
  uint32_t pad;
  // APP(S): max_u r(u) / (|N(u)| + |A(u)|) after the round (float bits) and
  // the nodes whose residue exceeds APP's threshold r_max (|N(u)| + |A(u)|)
  unsigned int max_rel_bits;
  uint32_t above;
};

__device__ __forceinline__ uint32_t smem_addr(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// Software grid barrier for persistent cooperative launches: blocks count up
// one word, which the host clears before the launch, and wait until it has
// reached the arrivals of all blocks at all barriers so far (`epoch`, kept by
// the caller).  One word instead of a counter and a generation saves the last
// block's two extra round trips to L2 on the path that every block waits for.
// Every spin is bounded; on expiry the barrier records an error and returns
// false, and the kernel unwinds instead of hanging.
struct alignas(16) GridBarrier {
  unsigned int count;
  unsigned int err;
  unsigned int taken[2];     // batched kernel: grabs from the pools of its two phases
};

constexpr unsigned int kSpinLimit = 1u << 20;   // polls of about a microsecond: about one second
constexpr unsigned int kSpinEager = 64;         // polls before the wait backs off

// Arrivals and error flag in one acquiring load, as two words: an acquire is
// ordered behind a release of the same width only, and blocks arrive with a
// 32-bit one.
struct BarrierWords {
  unsigned int count, err;
};
__device__ __forceinline__ BarrierWords ld_barrier(const GridBarrier* b) {
  BarrierWords v;
  asm volatile("ld.acquire.gpu.global.v2.u32 {%0, %1}, [%2];" : "=r"(v.count), "=r"(v.err) : "l"(b) : "memory");
  return v;
}

// Barrier over the blocks [0, nblocks) that share `b`; epoch starts at 0 with
// b->count cleared and is the same in every block.  then() runs in thread 0 of
// every block once all have arrived, before the block's other threads go on.
template <typename Then>
__device__ __forceinline__ bool grid_sync(GridBarrier* b, unsigned int nblocks, unsigned int& epoch, Then then) {
  __shared__ unsigned int s_ok;
  epoch += nblocks;
  __syncthreads();
  if (threadIdx.x == 0) {
    // the release covers the block's writes (ordered before it by the block
    // barrier), the acquire its later reads; a fence on either side instead
    // would add about 500 cycles each to the 2,500 that this takes
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(&b->count) : "memory");
    unsigned int spins = 0;
    BarrierWords w = ld_barrier(b);
    while (w.err == 0 && (int)(w.count - epoch) < 0) {
      if (++spins > kSpinLimit) { atomicOr(&b->err, 1u); w.err = 1u; break; }
      if (spins > kSpinEager) __nanosleep(40);
      w = ld_barrier(b);
    }
    s_ok = w.err == 0;
    if (s_ok) then();
  }
  __syncthreads();
  return s_ok != 0;
}
__device__ __forceinline__ bool grid_sync(GridBarrier* b, unsigned int nblocks, unsigned int& epoch) {
  return grid_sync(b, nblocks, epoch, [] {});
}

// ------------------------------------------------------------ reductions

// Radix-select step on a histogram in shared memory (bins a power of two >= 32):
// the largest digit d such that the keys in buckets above d plus hist[d]
// reach krem.  Warp-collective: lane L sums bins [L*bins/32, (L+1)*bins/32),
// a suffix sum over the lanes and a ballot find the lane holding the
// crossing, and that lane walks its own bins.  Every lane receives d, cum
// (keys in the buckets above d) and h = hist[d].
__device__ __forceinline__ void radix_pick(const unsigned int* hist, int bins, uint32_t krem, int* d_out,
                                           uint32_t* cum_out, uint32_t* h_out) {
  const int lane = threadIdx.x & 31;
  const int per = bins >> 5;
  const unsigned int* mine = hist + lane * per;
  uint32_t sum = 0;
  for (int j = 0; j < per; ++j) sum += mine[(j + lane) & (per - 1)];   // rotated: fewer bank conflicts
  uint32_t suf = sum;                                   // keys in lanes >= lane
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t t = __shfl_down_sync(0xffffffffu, suf, o);
    if (lane + o < 32) suf += t;
  }
  const unsigned int ball = __ballot_sync(0xffffffffu, suf >= krem);
  const int L = ball ? 31 - __clz(ball) : 0;
  int d = 0;
  uint32_t cum = 0, h = 0;
  if (lane == L) {
    cum = suf - sum;                                    // keys in the lanes above L
    int j = per - 1;
    for (; j >= 0; --j) {
      h = mine[j];
      if (cum + h >= krem || j == 0) break;
      cum += h;
    }
    d = L * per + j;
  }
  *d_out = __shfl_sync(0xffffffffu, d, L);
  *cum_out = __shfl_sync(0xffffffffu, cum, L);
  *h_out = __shfl_sync(0xffffffffu, h, L);
}

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ double warp_sum_d(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// FP64 runs at two lanes a cycle on an SM of this chip: one FP64 instruction
// of a full block of 1,024 threads takes a quarter of a microsecond, an FP64
// log in every thread 25.  So the per-round tests of the kernels are taken in
// FP32 where that decides them for certain, and in FP64 only in the band where
// rounding could; the outcome is the FP64 test's in every case.

// Smallest float f with (r > th) <=> (r >= f) for every float r: the mark
// test r > th of Algorithm 4 taken exactly against the FP64 threshold.
__host__ __device__ inline float threshold_up(double th) {
  float f = (float)th;
  if ((double)f <= th) f = nextafterf(f, INFINITY);
  return f;
}

// r > th * cnt (APP's per-node threshold), th_f = (float)th.
__device__ __forceinline__ bool above_node_threshold(float r, double th, float th_f, uint32_t cnt) {
  const float t = th_f * (float)cnt;                 // relative error below 3 * 2^-24
  if (t > 1e-30f) {
    if (r > t * 1.000001f) return true;
    if (r < t * 0.999999f) return false;
  }
  return (double)r > th * (double)cnt;
}

// The switch test of Algorithm 4, n_p >= 2 (|E| + |E_A|) max(0, log(M / eps_f)) / log_inv
// (rule 0), or with log(1 / (lambda M)) in the place of the log (rule 1, as
// printed); never for rule 2.
static __device__ __noinline__ bool switch_due_fp64(uint32_t e_tot, int rule, double eps_f, double lambda,
                                                    double log_inv, unsigned long long n_p, float m) {
  const double EE = (double)e_tot, M = (double)m;
  const double budget = rule == 1 ? 2.0 * EE * (log(1.0 / (lambda * M)) / log_inv)
                                  : 2.0 * EE * fmax(0.0, log(M / eps_f) / log_inv);
  return (double)n_p >= budget;
}

// log_ref: (float)log(eps_f) (rule 0) or (float)log(1 / lambda) (rule 1);
// unit: (float)(2 (|E| + |E_A|) / log_inv).  Both logs are off by less than
// 1e-5 for every float M and normal eps_f, so a margin of 1e-4 decides.
__device__ __forceinline__ bool switch_due(uint32_t e_tot, int rule, double eps_f, double lambda, double log_inv,
                                           float unit, float log_ref, unsigned long long n_p, float m) {
  if (rule == 2) return false;
  const float l = logf(m), d = rule == 1 ? log_ref - l : fmaxf(0.f, l - log_ref);
  const float have = (float)n_p;
  if (have > unit * (d + 1e-4f) * 1.00001f) return true;
  if (have < unit * (d - 1e-4f) * 0.99999f) return false;
  return switch_due_fp64(e_tot, rule, eps_f, lambda, log_inv, n_p, m);
}

// Kahan-compensated accumulation s += v with compensation c (FP32).
__device__ __forceinline__ void kahan_add(float& s, float& c, float v) {
  float y = v - c;
  float t = s + y;
  c = (t - s) - y;
  s = t;
}

}  // namespace ahpp
