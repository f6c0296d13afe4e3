// Single-query persistent push kernel: state and launch parameters.
#pragma once
#include "ahpp_internal.cuh"

namespace ahpp {

// Block size of the single-query kernel: one block of kQ1Threads per SM (64
// registers a thread).  On the medium graph 1,024 threads with rings of four
// units took 24.0 ms a query, 768 threads 24.5, 512 with rings of eight 31.3.
constexpr int kQ1Threads = 1024;
constexpr int kQ1Warps = kQ1Threads / 32;
constexpr int kQ1Blocks = 1;
// The most dynamic shared memory of a block.  What is left of the 256 KB is L1,
// whose lines hold the lookups in flight: 21.4 ms a query on the medium graph
// at 188 KB, 22.0 at 160, 21.8 at 128 (less of the tables copied), 36.5 at 204.
constexpr uint32_t kQ1SmemMax = 188 * 1024;
// Units (512 bytes) of each warp's ring in shared memory: its stream of graph
// entries is copied that far ahead of its use.
constexpr uint32_t kQ1Ring = 4;
constexpr uint32_t kQ1RingBytes = kQ1Warps * kQ1Ring * 512;

// Device state of one query (all arrays indexed by internal ids).
struct Q1State {
  float *r_u = nullptr, *pi = nullptr, *pic = nullptr;   // residues (sign = marked), reserves, Kahan
  float *t_v = nullptr, *t_a = nullptr;                  // r(v)/d(v), r(a)/W_col(a)
  float* t_a2 = nullptr;                                 // the other t_A buffer (pull rounds alternate)
  uint32_t* list_u = nullptr;                            // push rounds: the marked list
  float* split_acc = nullptr;                            // sums of split rows (see SplitAcc)
  uint32_t* split_cnt = nullptr;                         // finished chunks of split U rows
  QCtl* ctl = nullptr;
  RAcc* racc = nullptr;                                  // [3]
  GridBarrier* bar = nullptr;
  unsigned int* final_maxr_bits = nullptr;               // [2]: max |r_U|, max pi
};

struct Q1Params {
  uint32_t q = 0;              // internal id of the source
  int algo = kAlgoASRP;
  int kahan = 1;
  int switch_rule = 0;
  double eps_f = 0.0;          // ASRP: eps / lambda;  APP: r_max = eps / (|E| + |E_A|)
  double lambda = 1.0;
  double log_inv = 0.0;        // ln(1 / (1 - alpha))
  uint32_t e_tot = 0;          // |E| + |E_A|
  // FP32 forms of the tests above (see switch_due, above_node_threshold):
  // smallest floats above eps_f and 0, eps_f, 2 e_tot / log_inv, and the log of
  // the switch test's reference
  float th_async = 0.f, th_sync = 0.f, eps_f32 = 0.f, switch_unit = 0.f, switch_log = 0.f;
  uint32_t max_rounds = 0;
  uint32_t dense_div = 32;     // pull rounds once the frontier covers > 1/dense_div of the edges
  uint32_t n_split = 0;        // entries of split_acc
  uint32_t smem_bytes = 0;     // dynamic shared memory of a block (Q1Layout's tables)
  // Theorem 3 mode: start from r = 1 on every U node, run exactly max_rounds
  // synchronous rounds; the reserves are then pi_T and final_maxr_bits[1]
  // holds max_u pi_T(u).
  int lambda_mode = 0;
  // Algorithm 1 mode: start from r = e_q in the synchronous phase (every
  // positive residue pushed each round) and run exactly max_rounds rounds;
  // the output is then reserves + residues, Algorithm 1's iterate.
  int pi_mode = 0;
};

int launch_query1(const DevGraph& g, const Q1State& s, const Q1Params& p, bool bf16, int grid,
                  cudaStream_t stream);
// Persistent grid of the single-query kernel with smem_bytes of dynamic
// shared memory per block (-1 if it cannot be made resident).
int query1_max_grid(int sm_count, uint32_t smem_bytes);

}  // namespace ahpp
