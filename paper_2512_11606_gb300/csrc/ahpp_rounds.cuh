// The rounds of a single query, as both kernels that run one see them: a
// thread's sums over a round, and the control that follows from the totals.
#pragma once
#include "ahpp_internal.cuh"
#include "ahpp_query1.cuh"

namespace ahpp {
namespace {

// Per-round sums of a thread; every sum stays below |E| + |E_A| < 2^32.
struct Q1Part {
  float max_r = 0.f;
  uint32_t marked = 0, marked_deg = 0, np_flush = 0;
  float max_rel = 0.f;       // APP(S) statistics (see RAcc)
  uint32_t above = 0;
};

// APP(S)'s round statistics of a residue r of a node with cnt = |N(u)| + |A(u)|:
// the largest r / cnt, and whether r exceeds APP's threshold r_max cnt.
__device__ __forceinline__ void app_stats(const Q1Params& p, float r, uint32_t cnt, Q1Part& part) {
  if (cnt) part.max_rel = fmaxf(part.max_rel, r / (float)cnt);
  if (above_node_threshold(r, p.eps_f, p.eps_f32, cnt)) part.above += 1;
}

// The query's control, kept in shared memory by thread 0 of every block (all
// read the same totals after a barrier, so all blocks agree).
struct Q1Loop {
  unsigned long long n_p, pushes, marked_deg;
  uint32_t rounds, switch_round, dense_rounds, marked;
  int phase, status, dense, switched, per_node, go;
  float theta;
};

// Before a round over `marked` nodes: stop, or how it runs.
__device__ __forceinline__ void begin_round(const Q1Params& p, Q1Loop& L, uint32_t marked,
                                            unsigned long long marked_deg) {
  L.marked = marked;
  L.marked_deg = marked_deg;
  L.go = 0;
  if (L.phase == kPhaseDone || L.marked == 0) { L.phase = kPhaseDone; return; }
  if (L.rounds >= p.max_rounds) { L.status = kStatusCap; return; }
  L.go = 1;
  if (!L.dense && L.marked_deg * (unsigned long long)p.dense_div > (unsigned long long)p.e_tot) L.dense = 1;
  L.pushes += L.marked;
  L.per_node = per_node_threshold(p.algo, L.phase);
  L.theta = L.phase == kPhaseSync ? p.th_sync : p.th_async;
}

// After a round that left the largest residue M (and APP(S)'s Mrel, `above`)
// and flushed np entries: its counters, the termination and the switch test.
template <bool APPS>
__device__ __forceinline__ void end_round(const Q1Params& p, Q1Loop& L, float M, unsigned long long np, float Mrel,
                                          uint32_t above) {
  ++L.rounds;
  L.n_p += L.marked_deg + np;
  L.switched = 0;
  auto due_at = [&](float m) {
    return L.phase == kPhaseAsync &&
           switch_due(p.e_tot, p.switch_rule, p.eps_f, p.lambda, p.log_inv, p.switch_unit, p.switch_log, L.n_p, m);
  };
  bool due = false;
  if (APPS) {
    // APP's stopping test; the switch budget in units of APP's thresholds
    if (above == 0) L.phase = kPhaseDone;
    else due = due_at(Mrel);
  } else if (p.algo == kAlgoASRP) {
    if (M < p.th_async) L.phase = kPhaseDone;            // M <= eps_f
    else due = due_at(M);
  }
  if (due) {
    L.phase = kPhaseSync;
    L.switch_round = L.rounds + 1;
    L.switched = 1;
  }
  L.go = L.phase != kPhaseDone;
  // marking of the next frontier in a push round
  L.per_node = per_node_threshold(p.algo, L.phase);
  L.theta = L.phase == kPhaseSync ? p.th_sync : p.th_async;
}

}  // namespace
}  // namespace ahpp
