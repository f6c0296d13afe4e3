// Single-query push on the whole GPU: one persistent cooperative launch runs
// every round of APP (Algorithm 3) or ASRP (Algorithm 4) for one source.
//
// A round is either
//   * a push round (small frontier): U-push of the marked list with atomic
//     scatter into t_V / t_A (the U-push of Algorithm 3), then the flush of
//     every V node and attribute with a positive t value (its V and attribute
//     steps) into r_U, in the work items of the pull phase 1 (long rows split
//     into chunks over warps, so a hub's flush is spread over the grid), then
//     the selection of the next frontier (warp-ballot compaction) and the
//     clearing of t_V / t_A;
//   * a pull round (large frontier, the synchronous sweep of Algorithm 4):
//     phase 1 gathers t_V from the marked residues over V->U and adds up t_A by
//     blocks of U rows; phase 2 gathers r_U' over U->V and U->A, applies the
//     reserve update of the pushed nodes and marks the next frontier.
// Both forms compute the same linear map of one round.  Rounds switch from
// push to pull when the frontier covers more than 1/dense_div of the edges.
// All control (termination, the ASRP switch test, the push/pull choice) is
// decided on the device from the round accumulators.
//
// What bounds a pull round, and what the layout does about it (GB300, one
// query, 20M edges and 20M attribute entries; a round took 0.320 ms with
// rows of CSR walked by two lanes each, 0.190 ms now; 2M + 2M: 0.077, 0.028):
//   - looking up 4-byte values at random: an SM finds one L1 line a cycle, so a
//     warp's 32 lookups take 32 cycles from L2.  The entries most looked up
//     (degree order: the first ones) are copied to shared memory each phase,
//     4 to 5 cycles a warp; the attribute hops stay there altogether;
//   - the latency of a row's index, then value: each warp's share of the graph
//     lies in the order of its use (Q1Rows) and is copied ahead to a ring in
//     shared memory, across the barrier too;
//   - uneven shares: cut by measured cost at load (ahpp_q1layout.cu);
//   - FP64: see switch_due; a log in every thread was 25 us of every round.
//   - reductions that meet in a few lines: see Q1Layout::ta_copies.
// Two barriers a round take about 2,500 cycles each; a small graph's round is
// mostly those and the few L2 latencies between them (the smallest graphs run
// on one cluster instead: ahpp_cluster.cu).
#include <algorithm>
#include <type_traits>

#include "ahpp_internal.cuh"
#include "ahpp_query1.cuh"
#include "ahpp_rounds.cuh"

namespace ahpp {

namespace {

__device__ __forceinline__ uint32_t lane_id() { return threadIdx.x & 31; }

// Warp-aggregated append of `val` for the lanes where `pred` holds.
__device__ __forceinline__ void warp_append(bool pred, uint32_t val, uint32_t* list,
                                            uint32_t* counter) {
  unsigned m = __ballot_sync(0xffffffffu, pred);
  if (!m) return;
  uint32_t lane = lane_id();
  uint32_t leader = __ffs(m) - 1;
  uint32_t base = 0;
  if (lane == leader) base = atomicAdd(counter, (uint32_t)__popc(m));
  base = __shfl_sync(0xffffffffu, base, leader);
  if (pred) list[base + __popc(m & ((1u << lane) - 1u))] = val;
}

struct Ctx {
  const DevGraph& g;   // references into the kernel's __grid_constant__ parameters
  const Q1State& s;
  const Q1Params& p;
  uint32_t gw, nw;     // global warp id / count
  uint32_t gt, nt;     // global thread id / count
};

// -------------------------------------------------- partials of a block

// Block reduction of p into acc, one atomic per field and block: one redux
// per field in each warp (the floats are >= 0, so their bits order them),
// then one in warp 0.
template <bool APPS>
__device__ __forceinline__ void flush_part(Q1Part& p, RAcc* acc) {
  __shared__ unsigned int sh[6][kQ1Warps];
  const uint32_t lane = lane_id(), warp = threadIdx.x >> 5;
  const unsigned int m = __reduce_max_sync(0xffffffffu, __float_as_uint(p.max_r));
  const unsigned int mk = __reduce_add_sync(0xffffffffu, p.marked);
  const unsigned int dg = __reduce_add_sync(0xffffffffu, p.marked_deg);
  const unsigned int np = __reduce_add_sync(0xffffffffu, p.np_flush);
  const unsigned int rel = APPS ? __reduce_max_sync(0xffffffffu, __float_as_uint(p.max_rel)) : 0u;
  const unsigned int ab = APPS ? __reduce_add_sync(0xffffffffu, p.above) : 0u;
  if (lane == 0) {
    sh[0][warp] = m; sh[1][warp] = mk; sh[2][warp] = dg; sh[3][warp] = np;
    if (APPS) { sh[4][warp] = rel; sh[5][warp] = ab; }
  }
  __syncthreads();
  if (warp == 0) {
    static_assert(kQ1Warps <= 32, "one lane per warp of the block");
    auto of = [&](int f) { return lane < (uint32_t)kQ1Warps ? sh[f][lane] : 0u; };
    const unsigned int bm = __reduce_max_sync(0xffffffffu, of(0));
    const unsigned int bmk = __reduce_add_sync(0xffffffffu, of(1));
    const unsigned int bdg = __reduce_add_sync(0xffffffffu, of(2));
    const unsigned int bnp = __reduce_add_sync(0xffffffffu, of(3));
    if (lane == 0 && bm) atomicMax(&acc->max_r_bits, bm);
    if (lane == 0 && bmk) atomicAdd(&acc->marked, bmk);
    if (lane == 0 && bdg) atomicAdd(&acc->marked_deg, (unsigned long long)bdg);
    if (lane == 0 && bnp) atomicAdd(&acc->np_flush, (unsigned long long)bnp);
    if (APPS) {
      const unsigned int brel = __reduce_max_sync(0xffffffffu, of(4));
      const unsigned int bab = __reduce_add_sync(0xffffffffu, of(5));
      if (lane == 0 && brel) atomicMax(&acc->max_rel_bits, brel);
      if (lane == 0 && bab) atomicAdd(&acc->above, bab);
    }
  }
  p = Q1Part();
}

// ------------------------------------------------------- sliced pull walks

// A lane's ring: its 16 bytes of each of the warp's next kQ1Ring units, copied
// to shared memory ahead of their use (cp.async, past L1).  Every lane reads
// back only what it copied itself, so waiting for its own copies is enough.
// HBM needs about 45 KB in flight per SM, more than prefetching to registers
// holds at 64 registers a thread.
struct Ring {
  const uint4* src;            // the lane's place in unit 0
  uint32_t base;               // the lane's place in the ring
  uint32_t next, end;          // next unit to copy, end of the stream

  // no block ends while copies to its shared memory are in flight
  __device__ __forceinline__ ~Ring() { asm volatile("cp.async.wait_all;" ::: "memory"); }
  // the next N units (each its own group of copies, empty past the end)
  template <int N>
  __device__ __forceinline__ void refill() {
#pragma unroll
    for (int i = 0; i < N; ++i) {
      if (next < end)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(base + (next % kQ1Ring) * 512u),
                     "l"(src + (size_t)next * 32) : "memory");
      asm volatile("cp.async.commit_group;" ::: "memory");
      ++next;
    }
  }
  // the stream [b, e) of units; the ring's earlier copies need not be waited
  // for: they are of a stream that ended, or were used
  __device__ __forceinline__ void start(const uint4* units, uint32_t b, uint32_t e) {
    src = units + lane_id();
    next = b;
    end = e;
    refill<kQ1Ring>();
  }
  // waits for the N oldest copies
  template <int N>
  __device__ __forceinline__ void wait() const {
    asm volatile("cp.async.wait_group %0;" ::"n"((int)kQ1Ring - N) : "memory");
  }
  // unit k of the stream (waited for)
  __device__ __forceinline__ uint4 unit(uint32_t k) const {
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(base + (k % kQ1Ring) * 512u) : "memory");
    return v;
  }
};

// x[i], from the copy of the first `hub` entries in shared memory when i is
// one of them (degree order: the hubs most gathers hit), else from L2.  An SM
// looks up one L1 line a cycle, so a warp's 32 scattered 4-byte gathers take
// 32 cycles from global memory (294 G gathers/s on the chip) and 4 to 5 from
// shared memory (1,325).  The loads go past L1: a line that is used once only
// takes a place there.
__device__ __forceinline__ float gather(uint32_t i, uint32_t hub, uint32_t s_base, const float* x) {
  float v;
  asm volatile("{\n\t.reg .pred p;\n\t"
               "setp.lt.u32 p, %1, %2;\n\t"
               "@p ld.shared.f32 %0, [%3];\n\t"
               "@!p ld.relaxed.gpu.global.f32 %0, [%4];\n\t}"
               : "=f"(v) : "r"(i), "r"(hub), "r"(s_base + 4u * i), "l"(x + i) : "memory");
  return v;
}
__device__ __forceinline__ float4 gather4(uint4 i, uint32_t hub, uint32_t s_base, const float* x) {
  return make_float4(gather(i.x, hub, s_base, x), gather(i.y, hub, s_base, x), gather(i.z, hub, s_base, x),
                     gather(i.w, hub, s_base, x));
}
// The pushed part of four residues (marked nodes hold theirs negated).
__device__ __forceinline__ float4 pushed(float4 r) {
  return make_float4(fmaxf(-r.x, 0.f), fmaxf(-r.y, 0.f), fmaxf(-r.z, 0.f), fmaxf(-r.w, 0.f));
}
__device__ __forceinline__ float ld_shared(uint32_t a) {
  float v;
  asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(a) : "memory");
  return v;
}

// Indices and coefficients of a step at unit k (k advances); compact: one unit
// of uint16 indices and bfloat16 weights.  The caller refills the ring once it
// has used them.
struct Step {
  uint4 i;
  float4 c;
};
__device__ __forceinline__ Step wide_step(const Ring& r, uint32_t& k) {
  Step s;
  s.i = r.unit(k);
  const uint4 c = r.unit(k + 1);
  s.c = make_float4(__uint_as_float(c.x), __uint_as_float(c.y), __uint_as_float(c.z), __uint_as_float(c.w));
  k += 2;
  return s;
}
__device__ __forceinline__ Step compact_step(const Ring& r, uint32_t& k) {
  const uint4 b = r.unit(k);
  ++k;
  Step s;
  s.i = make_uint4(b.x & 0xffffu, b.x >> 16, b.y & 0xffffu, b.y >> 16);
  s.c = make_float4(__uint_as_float(b.z << 16), __uint_as_float(b.z & 0xffff0000u),
                    __uint_as_float(b.w << 16), __uint_as_float(b.w & 0xffff0000u));
  return s;
}

__device__ __forceinline__ float dot4(float4 c, float4 x, float s) {
  return fmaf(c.w, x.w, fmaf(c.z, x.z, fmaf(c.y, x.y, fmaf(c.x, x.x, s))));
}

// A reduction that returns nothing (an atomicAdd whose result is unused may
// still be issued as a returning atomic).
__device__ __forceinline__ void red_add(float* p, float v) {
  asm volatile("red.relaxed.gpu.global.add.f32 [%0], %1;" ::"l"(p), "f"(v) : "memory");
}

// Sum over the vw = 1 << lg lanes of a row (every lane of the warp calls it).
__device__ __forceinline__ float row_sum(float s, uint32_t lg) {
  for (uint32_t o = (1u << lg) >> 1; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  return s;
}

// The accumulators of split rows, in split_acc: one per split V row for either
// parity of the pull rounds, then one per split U row (split_cnt counts their
// finished chunks).
struct SplitAcc {
  float *v_cur, *v_next, *u;
};
__device__ __forceinline__ SplitAcc split_acc(const Q1State& s, const Q1Layout& Q, int sel) {
  const uint32_t n = Q.v.n_split;
  return SplitAcc{s.split_acc + (sel ? n : 0u), s.split_acc + (sel ? 0u : n), s.split_acc + 2 * n};
}

// ---------------------------------------------------------------- phase 1
// t_V[v] = sum_u c_uv p_u ;  t_A[a] = k_attr cnorm_a[a] sum_u (w(u,a) rnorm_u[u]) p_u
// t_V is pulled over the rows of V; the chunks of a split row add to its
// accumulator, which phase 2 reads in the row's place.  t_A is added up by
// blocks of U rows (Q1Segs): the rows' p lies in shared memory, so the |E_A|
// lookups never leave the SM, and a block gives each attribute it touches one
// reduction.

template <bool COMPACT>
__device__ __forceinline__ void attribute_hop(const Ctx& c, Ring& ra, uint4 r, uint32_t s_own, float* ta) {
  const Q1Segs& S = c.g.q1.s;
  const uint32_t lane = lane_id();
  uint32_t k = r.z;
  uint4 a = r.x < r.y ? S.items[r.x] : make_uint4(0, 0, 0, 0);
  for (uint32_t it = r.x; it < r.y; ++it) {
    const uint4 cur = a;
    if (it + 1 < r.y) a = S.items[it + 1];
    const uint32_t lg = (cur.y >> 8) & 7u, row = lane >> lg;
    const bool lead = row < (cur.y & 0xffu) && (lane & ((1u << lg) - 1u)) == 0;
    const uint2 meta = lead ? S.meta[cur.x + row] : make_uint2(0, 0);
    float s = 0.f;
#pragma unroll 1
    for (uint32_t j = 0; j < cur.w; ++j) {
      ra.wait<COMPACT ? 1 : 2>();
      const Step st = COMPACT ? compact_step(ra, k) : wide_step(ra, k);
      const float4 x = make_float4(ld_shared(s_own + 4 * st.i.x), ld_shared(s_own + 4 * st.i.y),
                                   ld_shared(s_own + 4 * st.i.z), ld_shared(s_own + 4 * st.i.w));
      ra.refill<COMPACT ? 1 : 2>();
      s = dot4(st.c, x, s);
    }
    s = row_sum(s, lg);
    if (lead && s != 0.f) red_add(&ta[meta.x], __uint_as_float(meta.y) * s);
  }
}

// rg: this warp's ranges of the attribute hop, the V rows and the U rows (in
// shared memory); `ring` holds the first units of the attribute hop's already,
// and of the U rows' on return.
template <bool COMPACT>
__device__ __forceinline__ void phase1(const Ctx& c, Q1Part& part, Ring& ring, const uint4* rg, float* ta,
                                       const SplitAcc& acc, float* smem) {
  const DevGraph& g = c.g;
  const Q1Layout& Q = g.q1;
  const uint32_t lane = lane_id(), hub = Q.hub_u;
  const float* r_u = c.s.r_u;
  float* s_own = smem + kQ1RingBytes / 4;
  float* s_hub = s_own + Q.s.own_cap;
  for (uint32_t i = threadIdx.x; i < hub / 4; i += kQ1Threads)
    reinterpret_cast<float4*>(s_hub)[i] = reinterpret_cast<const float4*>(r_u)[i];
  for (uint32_t b = blockIdx.x; b < Q.s.n_vb; b += gridDim.x) {
    const uint2 rows = Q.s.vb[b];
    for (uint32_t i = threadIdx.x; i < rows.y; i += kQ1Threads)
      s_own[i] = fmaxf(-r_u[rows.x + i], 0.f) * g.rnorm_u[rows.x + i];
    __syncthreads();
    uint4 r = rg[0];
    if (b != blockIdx.x) {
      r = Q.s.ranges[b * kQ1Warps + (threadIdx.x >> 5)];
      ring.start(Q.s.units, r.z, r.w);
    }
    attribute_hop<COMPACT>(c, ring, r, smem_addr(s_own), ta);
    if (b + gridDim.x < Q.s.n_vb) __syncthreads();
  }
  if (blockIdx.x >= Q.s.n_vb) __syncthreads();
  const uint32_t s_base = smem_addr(s_hub);
  const Q1Rows& L = Q.v;
  const uint4 r = rg[1];
  ring.start(L.units, r.z, r.w);
  uint32_t k = r.z;
  uint4 a = r.x < r.y ? L.items[r.x] : make_uint4(0, 0, 0, 0);
  for (uint32_t it = r.x; it < r.y; ++it) {
    const uint4 ca = a;
    if (it + 1 < r.y) a = L.items[it + 1];
    const uint32_t lg = (ca.y >> 8) & 7u, row = lane >> lg, v = ca.x + row;
    const bool lead = row < (ca.y & 0xffu) && (lane & ((1u << lg) - 1u)) == 0;
    const uint32_t deg = lead ? Q.deg_v[v] : 0u;
    float s = 0.f;
#pragma unroll 1
    for (uint32_t j = 0; j < ca.z; ++j) {
      ring.wait<2>();
      const Step st = wide_step(ring, k);
      const float4 x = gather4(st.i, hub, s_base, r_u);
      ring.refill<2>();
      s = dot4(st.c, pushed(x), s);
    }
    s = row_sum(s, lg);
    if (!lead) continue;
    if (ca.y >> 31) {
      if (s != 0.f) red_add(&acc.v_cur[v], s);
    } else {
      c.s.t_v[v] = s;
      if (s > 0.f) part.np_flush += deg;
    }
  }
  ring.start(Q.u.units, rg[2].z, rg[2].w);
}

// ---------------------------------------------------------------- phase 2
// r_U'[u] = kept_u + sum_v w(u,v) t_V[v] + sum_a w(u,a) t_A[a]; reserve update of
// the nodes pushed this round; marking of the next frontier with threshold th.

// Residue r_old (reserve pv, compensation pc) of row u takes in s.
template <bool APPS>
__device__ __forceinline__ void finish_row(const Ctx& c, uint32_t u, float s, float r_old, float pv, float pc,
                                           uint32_t cnt, float th, bool per_node, Q1Part& part) {
  float kept = r_old;
  if (r_old < 0.f) {
    const float add = c.g.alpha * (-r_old);
    if (c.p.kahan) {
      kahan_add(pv, pc, add);
      c.s.pic[u] = pc;
    } else {
      pv += add;
    }
    c.s.pi[u] = pv;
    kept = 0.f;
  }
  const float r_new = kept + s;
  part.max_r = fmaxf(part.max_r, r_new);
  if (APPS) app_stats(c.p, r_new, cnt, part);
  const bool mark = per_node ? above_node_threshold(r_new, c.p.eps_f, c.p.eps_f32, cnt) : r_new >= th;
  if (mark) {
    part.marked += 1;
    part.marked_deg += cnt;
  }
  c.s.r_u[u] = mark ? -r_new : r_new;
}

// `ring` holds the first units of the warp's U rows, and of its attribute hop's
// for the next round on return.
template <bool COMPACT, bool APPS>
__device__ __forceinline__ void phase2(const Ctx& c, float th, bool per_node, Q1Part& part, Ring& ring,
                                       const uint4* rg, const float* ta_cur, float* ta_next, const SplitAcc& acc,
                                       float* smem) {
  const DevGraph& g = c.g;
  const Q1Layout& Q = g.q1;
  const uint32_t lane = lane_id(), hub_a = Q.hub_a, hub_v = Q.hub_v, na = g.n_a, nsv = Q.v.n_split;
  const float* t_v = c.s.t_v;
  float* s_ta = smem + kQ1RingBytes / 4;
  float* s_tv = s_ta + (hub_a + 3) / 4 * 4;
  const uint32_t v4 = (nsv + 3) / 4;
  for (uint32_t i = v4 + threadIdx.x; i < hub_v / 4; i += kQ1Threads)
    reinterpret_cast<float4*>(s_tv)[i] = reinterpret_cast<const float4*>(t_v)[i];
  for (uint32_t i = threadIdx.x; i < min(4 * v4, hub_v); i += kQ1Threads) s_tv[i] = i < nsv ? acc.v_cur[i] : t_v[i];
  // active attributes and split V rows (Algorithm 4's push counter); the next
  // round's sums start at zero
  if (Q.ta_copies == 1) {
    for (uint32_t i = threadIdx.x; i < hub_a; i += kQ1Threads) s_ta[i] = ta_cur[i];
    for (uint32_t a = c.gt; a < na; a += c.nt) {
      if (ta_cur[a] > 0.f) part.np_flush += Q.deg_a[a];
      ta_next[a] = 0.f;
    }
  } else {                                 // all loads of a sum in flight at once
    const uint32_t n_ta = na * Q.ta_copies;
    auto sum = [&](uint32_t a) {
      float t = 0.f;
#pragma unroll
      for (uint32_t k = 0; k < kTaCopies; ++k) t += a + k * na < n_ta ? ta_cur[a + k * na] : 0.f;
      return t;
    };
    for (uint32_t i = threadIdx.x; i < hub_a; i += kQ1Threads) s_ta[i] = sum(i);
    for (uint32_t a = c.gt; a < na; a += c.nt)
      if (sum(a) > 0.f) part.np_flush += Q.deg_a[a];
    for (uint32_t a = c.gt; a < n_ta; a += c.nt) ta_next[a] = 0.f;
  }
  for (uint32_t v = c.gt; v < nsv; v += c.nt) {
    if (acc.v_cur[v] > 0.f) part.np_flush += Q.deg_v[v];
    acc.v_next[v] = 0.f;
  }
  __syncthreads();
  const uint32_t base_a = smem_addr(s_ta), base_v = smem_addr(s_tv);
  const Q1Rows& L = Q.u;
  const uint4 r = rg[2];
  uint32_t k = r.z, n_chunks = 0;
  uint4 a = r.x < r.y ? L.items[r.x] : make_uint4(0, 0, 0, 0);
  for (uint32_t it = r.x; it < r.y; ++it) {
    const uint4 ca = a;
    if (it + 1 < r.y) a = L.items[it + 1];
    const uint32_t lg = (ca.y >> 8) & 7u, row = lane >> lg, u = ca.x + row, chunk = ca.y >> 31;
    const bool lead = row < (ca.y & 0xffu) && (lane & ((1u << lg) - 1u)) == 0;
    float r_old = 0.f, pv = 0.f, pc = 0.f;
    uint32_t cnt = 0;
    if (lead && !chunk) {
      r_old = c.s.r_u[u];
      pv = c.s.pi[u];
      if (c.p.kahan) pc = c.s.pic[u];
      cnt = Q.deg_u[u];
    }
    float s = 0.f;
#pragma unroll 1
    for (uint32_t j = 0; j < ca.z; ++j) {
      ring.wait<2>();
      const Step st = wide_step(ring, k);
      const float4 x = gather4(st.i, hub_v, base_v, t_v);
      ring.refill<2>();
      s = dot4(st.c, x, s);
    }
#pragma unroll 1
    for (uint32_t i = 0; i < ca.w; ++i) {
      ring.wait<COMPACT ? 1 : 2>();
      const Step st = COMPACT ? compact_step(ring, k) : wide_step(ring, k);
      const float4 x = gather4(st.i, hub_a, base_a, ta_cur);
      ring.refill<COMPACT ? 1 : 2>();
      s = dot4(st.c, x, s);
    }
    s = row_sum(s, lg);
    n_chunks += chunk;
    if (!lead) continue;
    if (chunk) red_add(&acc.u[u], s);
    else finish_row<APPS>(c, u, s, r_old, pv, pc, cnt, th, per_node, part);
  }
  // the warp's chunks, a lane each: the last chunk of a row to be counted
  // finishes it (counted only now, so that no walk waits for the counter)
  for (uint32_t i0 = 0; i0 < n_chunks; i0 += 32) {
    __syncwarp();
    if (i0 + lane >= n_chunks) continue;
    const uint32_t u = L.items[r.x + i0 + lane].x;
    uint32_t seen;
    asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], 1;" : "=r"(seen) : "l"(&c.s.split_cnt[u]) : "memory");
    if (seen != L.chunks_of[u] - 1) continue;
    const float s = __ldcg(&acc.u[u]);
    acc.u[u] = 0.f;
    c.s.split_cnt[u] = 0;
    finish_row<APPS>(c, u, s, c.s.r_u[u], c.s.pi[u], c.p.kahan ? c.s.pic[u] : 0.f, Q.deg_u[u], th, per_node, part);
  }
  ring.start(Q.s.units, rg[0].z, rg[0].w);
}

// --------------------------------------------------------- push (sparse)

template <typename WA>
__device__ void push_u(const Ctx& c, uint32_t n_list) {
  const DevGraph& g = c.g;
  const uint32_t lane = lane_id();
  for (uint32_t i = c.gw; i < n_list; i += c.nw) {
    const uint32_t u = c.s.list_u[i];
    float r = 0.f;
    if (lane == 0) r = c.s.r_u[u];
    r = __shfl_sync(0xffffffffu, r, 0);
    const float p = fmaxf(-r, 0.f);
    if (lane == 0) {
      c.s.r_u[u] = 0.f;
      const float add = c.g.alpha * p;
      if (c.p.kahan) {
        float pv = c.s.pi[u], pc = c.s.pic[u];
        kahan_add(pv, pc, add);
        c.s.pi[u] = pv; c.s.pic[u] = pc;
      } else {
        c.s.pi[u] += add;
      }
    }
    // non-returning reductions: the flush finds the rows it must move by
    // their value, so no first-touch list is kept
    const uint32_t b1 = g.uv_off[u], e1 = g.uv_off[u + 1];
    for (uint32_t k = b1 + lane; k < e1; k += 32) atomicAdd(&c.s.t_v[g.uv_idx[k]], g.uv_c[k] * p);
    const float ka = g.k_attr * g.rnorm_u[u] * p;
    const uint32_t b2 = g.ua_off[u], e2 = g.ua_off[u + 1];
    for (uint32_t k = b2 + lane; k < e2; k += 32) {
      const uint32_t a = g.ua_idx[k];
      atomicAdd(&c.s.t_a[a], wload<WA>(g.ua_w, k) * ka * g.cnorm_a[a]);
    }
  }
}

// One V (or attribute) row's flush over entries [b, e): r_U[j] += w t for its
// U neighbours j (returning atomics: the new residues feed max r_U).
template <typename WA, bool APPS>
__device__ __forceinline__ void flush_row(const Ctx& c, bool is_a, uint32_t b, uint32_t e, float t,
                                          Q1Part& part) {
  const DevGraph& g = c.g;
  const uint32_t* idx = is_a ? g.au_idx : g.vu_idx;
  for (uint32_t k = b + lane_id(); k < e; k += 32) {
    const float w = is_a ? wload<WA>(g.au_w, k) : g.vu_w[k];
    const float add = w * t;
    const uint32_t j = idx[k];
    const float old = atomicAdd(&c.s.r_u[j], add);
    part.max_r = fmaxf(part.max_r, old + add);
    // APP(S): a node's last update sees its new residue (counts of nodes
    // above threshold may repeat a node; only zero is tested)
    if (APPS)
      app_stats(c.p, old + add, (g.uv_off[j + 1] - g.uv_off[j]) + (g.ua_off[j + 1] - g.ua_off[j]), part);
  }
}

// The V and attribute flush of a push round, over the work items of phase 1:
// a short-row item's rows with t > 0 are flushed one after another by the
// warp; a long row's chunk by the warp that owns the chunk.  t_V / t_A are
// only read here (select_frontier clears them after the barrier).
template <typename WA, bool APPS>
__device__ void flush_va(const Ctx& c, Q1Part& part) {
  const DevGraph& g = c.g;
  const uint32_t lane = lane_id();
  const uint32_t nv = g.s1_v.n_items, total = nv + g.s1_a.n_items;
  for (uint32_t it = c.gw; it < total; it += c.nw) {
    const bool is_a = it >= nv;
    const uint4 item = is_a ? g.s1_a.items[it - nv] : g.s1_v.items[it];
    const uint32_t* off = is_a ? g.au_off : g.vu_off;
    const float* t = is_a ? c.s.t_a : c.s.t_v;
    if (item.y & (kItemLong | kItemSplit)) {
      const uint32_t row = item.x;
      const float tv = t[row];
      if (!(tv > 0.f)) continue;
      const uint32_t b = off[row];
      if (item.z == 0 && lane == 0) part.np_flush += off[row + 1] - b;
      flush_row<WA, APPS>(c, is_a, b + item.z, b + item.w, tv, part);
    } else {
      const uint32_t r0 = item.x, nr = item.y;
      const float mine = lane < nr ? t[r0 + lane] : 0.f;
      for (unsigned m = __ballot_sync(0xffffffffu, mine > 0.f); m; m &= m - 1) {
        const uint32_t r = __ffs(m) - 1;
        const float tv = __shfl_sync(0xffffffffu, mine, r);
        const uint32_t b = off[r0 + r], e = off[r0 + r + 1];
        if (lane == 0) part.np_flush += e - b;
        flush_row<WA, APPS>(c, is_a, b, e, tv, part);
      }
    }
  }
}

// Marking of the next frontier in a push round: r_U >= th (per_node: r_U > eps_f cnt(u)),
// and the clearing of t_V / t_A for the next round's U-push.
__device__ void select_frontier(const Ctx& c, float th, bool per_node, RAcc* acc,
                                Q1Part& part) {
  const DevGraph& g = c.g;
  for (uint32_t v = c.gt; v < g.n_v; v += c.nt) c.s.t_v[v] = 0.f;
  for (uint32_t a = c.gt; a < g.n_a; a += c.nt) c.s.t_a[a] = 0.f;
  const uint32_t n = g.n_u;
  // every warp iterates the same number of times so the ballot is warp-uniform
  const uint32_t span = (n + 31) / 32 * 32;
  for (uint32_t u0 = c.gw * 32; u0 < span; u0 += c.nw * 32) {
    const uint32_t u = u0 + lane_id();
    bool m = false;
    uint32_t cnt = 0;
    float r = 0.f;
    if (u < n) {
      r = c.s.r_u[u];
      if (per_node) {
        cnt = (g.uv_off[u + 1] - g.uv_off[u]) + (g.ua_off[u + 1] - g.ua_off[u]);
        m = above_node_threshold(r, c.p.eps_f, c.p.eps_f32, cnt);
      } else {
        m = r >= th;
        if (m) cnt = (g.uv_off[u + 1] - g.uv_off[u]) + (g.ua_off[u + 1] - g.ua_off[u]);
      }
      if (m) {
        c.s.r_u[u] = -r;
        part.marked += 1;
        part.marked_deg += cnt;
      }
    }
    warp_append(m, u, c.s.list_u, &acc->n_list_u);
  }
}

// At the ASRP switch the speculative marks of a pull round used eps_f; the
// first synchronous round pushes every positive residue, so mark the rest.
__device__ void mark_remaining(const Ctx& c, Q1Part& part) {
  const DevGraph& g = c.g;
  for (uint32_t u = c.gt; u < g.n_u; u += c.nt) {
    const float r = c.s.r_u[u];
    if (r > 0.f) {
      c.s.r_u[u] = -r;
      part.marked += 1;
      part.marked_deg += (g.uv_off[u + 1] - g.uv_off[u]) + (g.ua_off[u + 1] - g.ua_off[u]);
    }
  }
}

// Before and after a round, from its accumulators in global memory.
__device__ void begin_round(const Q1State& s, const Q1Params& p, Q1Loop& L) {
  const RAcc* P = &s.racc[(L.rounds + 2) % 3];
  begin_round(p, L, __ldcg(&P->marked), __ldcg(&P->marked_deg));
  if (L.go && blockIdx.x == 0) s.racc[(L.rounds + 1) % 3] = RAcc{};
}
template <bool APPS>
__device__ void end_round(const Q1State& s, const Q1Params& p, Q1Loop& L) {
  const RAcc* A = &s.racc[L.rounds % 3];
  end_round<APPS>(p, L, __uint_as_float(__ldcg(&A->max_r_bits)), __ldcg(&A->np_flush),
                  APPS ? __uint_as_float(__ldcg(&A->max_rel_bits)) : 0.f, APPS ? __ldcg(&A->above) : 0u);
}

}  // namespace

// FORM: how the attribute weights and steps are stored (the graph's bf16 and
// compact_a): 0 FP32, 1 bfloat16 in compact steps, 2 bfloat16, wide U -> A steps.
template <int FORM, bool APPS>
__global__ void __launch_bounds__(kQ1Threads, kQ1Blocks)
k_query1(const __grid_constant__ DevGraph g, const __grid_constant__ Q1State s,
         const __grid_constant__ Q1Params p) {
  using WA = typename std::conditional<FORM == 0, float, __nv_bfloat16>::type;
  extern __shared__ __align__(16) float q1_smem[];
  __shared__ Q1Loop L;
  unsigned int epoch = 0;                  // of the grid barrier
  Ctx c{g, s, p, (blockIdx.x * kQ1Threads + threadIdx.x) >> 5, (gridDim.x * kQ1Threads) >> 5,
        blockIdx.x * kQ1Threads + threadIdx.x, gridDim.x * kQ1Threads};
  const bool leader = blockIdx.x == 0 && threadIdx.x == 0;
  const unsigned int nb = gridDim.x;
  const bool app = p.algo != kAlgoASRP;    // APP's per-node threshold for the source

  // this warp's ranges, and its ring with the first units of the attribute hop
  // (the graph does not change: no barrier needs to come before the copies)
  __shared__ uint4 s_rg[kQ1Warps][3];
  Ring ring;
  ring.base = smem_addr(q1_smem) + (threadIdx.x >> 5) * (kQ1Ring * 512u) + lane_id() * 16u;
  const uint4* rg = s_rg[threadIdx.x >> 5];
  {
    const uint32_t wb = threadIdx.x >> 5, w = blockIdx.x * kQ1Warps + wb, l = lane_id();
    if (l < 3) {
      uint4 r = make_uint4(0, 0, 0, 0);
      if (l == 0 && blockIdx.x < g.q1.s.n_vb) r = g.q1.s.ranges[w];
      if (l == 1) r = g.q1.v.ranges[w];
      if (l == 2) r = g.q1.u.ranges[w];
      s_rg[wb][l] = r;
    }
    __syncwarp();
    ring.start(g.q1.s.units, rg[0].z, rg[0].w);
  }

  // ---- init: zero the state, mark the source (the initial state of Algorithm 3)
  const float r0 = p.lambda_mode ? -1.f : 0.f;
  for (uint32_t u = c.gt; u < g.n_u; u += c.nt) { s.r_u[u] = r0; s.pi[u] = 0.f; s.pic[u] = 0.f; }
  for (uint32_t v = c.gt; v < g.n_v; v += c.nt) s.t_v[v] = 0.f;
  for (uint32_t a = c.gt; a < g.n_a * g.q1.ta_copies; a += c.nt) { s.t_a[a] = 0.f; s.t_a2[a] = 0.f; }
  for (uint32_t i = c.gt; i < p.n_split; i += c.nt) { s.split_acc[i] = 0.f; s.split_cnt[i] = 0; }   // 2 V + U
  if (c.gt < 3) s.racc[c.gt] = RAcc{};
  if (leader) {
    s.ctl->reserve_sum = 0.0;
    s.ctl->resid_sum = 0.0;
    s.final_maxr_bits[0] = 0u;
    s.final_maxr_bits[1] = 0u;
  }
  if (threadIdx.x == 0) {
    L = Q1Loop{};
    L.phase = (p.lambda_mode || p.pi_mode) ? kPhaseSync : kPhaseAsync;
    L.dense = p.lambda_mode ? 1 : 0;
  }
  // a barrier that gives up skips the rounds; the leader still reports the
  // status below, so the host never reads a previous call's control block
  bool ok = grid_sync(s.bar, nb, epoch);
  if (ok && leader) {
    RAcc* a0 = &s.racc[2];
    if (p.lambda_mode) {
      a0->marked = g.n_u;
      a0->marked_deg = p.e_tot;
    } else {
      const uint32_t cnt = (g.uv_off[p.q + 1] - g.uv_off[p.q]) + (g.ua_off[p.q + 1] - g.ua_off[p.q]);
      const double th = app ? p.eps_f * (double)cnt : p.eps_f;
      if (1.0 > th) {
        s.r_u[p.q] = -1.f;
        a0->marked = 1;
        a0->marked_deg = cnt;
        a0->n_list_u = 1;
        s.list_u[0] = p.q;
      } else {
        s.r_u[p.q] = 1.f;
      }
    }
  }
  if (ok) ok = grid_sync(s.bar, nb, epoch, [&] { begin_round(s, p, L); });

  Q1Part part;
  // the sums of a pull round (t_A, split V rows) are added up in one of two
  // buffers, in turn; its phase 2 clears the other for the next round
  int sel = 0;
  while (ok && L.go) {
    RAcc* A = &s.racc[L.rounds % 3];
    if (!L.dense) {
      push_u<WA>(c, L.marked);
      if (!(ok = grid_sync(s.bar, nb, epoch))) break;
      flush_va<WA, APPS>(c, part);
      flush_part<APPS>(part, A);
      if (!(ok = grid_sync(s.bar, nb, epoch, [&] { end_round<APPS>(s, p, L); })) || !L.go) break;
      select_frontier(c, L.theta, L.per_node, A, part);
      flush_part<APPS>(part, A);
      ok = grid_sync(s.bar, nb, epoch, [&] { begin_round(s, p, L); });
    } else {
      float* ta_cur = sel ? s.t_a2 : s.t_a;
      float* ta_next = sel ? s.t_a : s.t_a2;
      const SplitAcc acc = split_acc(s, g.q1, sel);
      phase1<FORM != 0>(c, part, ring, rg, ta_cur, acc, q1_smem);
      if (!(ok = grid_sync(s.bar, nb, epoch))) break;
      phase2<FORM == 1, APPS>(c, L.theta, L.per_node, part, ring, rg, ta_cur, ta_next, acc, q1_smem);
      flush_part<APPS>(part, A);
      ok = grid_sync(s.bar, nb, epoch, [&] {
        ++L.dense_rounds;
        end_round<APPS>(s, p, L);
        if (L.go && !L.switched) begin_round(s, p, L);
      });
      sel ^= 1;
      if (ok && L.go && L.switched) {
        mark_remaining(c, part);
        flush_part<APPS>(part, A);
        ok = grid_sync(s.bar, nb, epoch, [&] { begin_round(s, p, L); });
      }
    }
  }
  __syncthreads();
  const int status = ok ? L.status : (int)kStatusWait;

  // ---- final: reserves pi - compensation, FP64 sums of reserves and residues
  if (status != kStatusWait) {
    double sp = 0.0, sr = 0.0;
    float mr = 0.f, mp = 0.f;
    for (uint32_t u = c.gt; u < g.n_u; u += c.nt) {
      const float v = fmaxf(s.pi[u] - s.pic[u], 0.f);
      const float r = fabsf(s.r_u[u]);
      s.pi[u] = p.pi_mode ? v + r : v;
      s.pic[u] = 0.f;
      sp += v; sr += r; mr = fmaxf(mr, r); mp = fmaxf(mp, v);
    }
    // one atomic per block and sum: FP64 adds to one address take their turns
    __shared__ double s_sum[2][kQ1Warps];
    __shared__ unsigned int s_max[2][kQ1Warps];
    sp = warp_sum_d(sp); sr = warp_sum_d(sr);
    const unsigned int bmr = __reduce_max_sync(0xffffffffu, __float_as_uint(mr));
    const unsigned int bmp = __reduce_max_sync(0xffffffffu, __float_as_uint(mp));
    const uint32_t lane = lane_id(), warp = threadIdx.x >> 5;
    if (lane == 0) { s_sum[0][warp] = sp; s_sum[1][warp] = sr; s_max[0][warp] = bmr; s_max[1][warp] = bmp; }
    __syncthreads();
    if (warp < 2) {
      const double d = warp_sum_d(lane < (uint32_t)kQ1Warps ? s_sum[warp][lane] : 0.0);
      const unsigned int m = __reduce_max_sync(0xffffffffu, lane < (uint32_t)kQ1Warps ? s_max[warp][lane] : 0u);
      if (lane == 0) {
        atomicAdd(warp ? &s.ctl->resid_sum : &s.ctl->reserve_sum, d);
        atomicMax(&s.final_maxr_bits[warp], m);
      }
    }
  }
  if (leader) {
    s.ctl->n_p = L.n_p;
    s.ctl->pushes = L.pushes;
    s.ctl->rounds = L.rounds;
    s.ctl->switch_round = L.switch_round;
    s.ctl->dense_rounds = L.dense_rounds;
    s.ctl->phase = L.phase;
    s.ctl->status = (status == kStatusOk && L.phase != kPhaseDone) ? kStatusCap : status;
  }
}

// Launch helper: persistent cooperative grid (one block per SM).
namespace {
// The instance of a launch: APP(S)'s round statistics are compiled only into
// the APP(S) instances.
template <bool APPS>
const void* q1_form(int form) {
  return form == 0 ? (const void*)k_query1<0, APPS>
                   : form == 1 ? (const void*)k_query1<1, APPS> : (const void*)k_query1<2, APPS>;
}
const void* q1_fn(int form, bool apps) { return apps ? q1_form<true>(form) : q1_form<false>(form); }
}  // namespace

// Carve out of the SM's unified memory just the shared memory the block needs
// (with 1 KB reserved by the system); the rest stays L1, which holds the lines
// of the gathers in flight.  Sets the dynamic shared memory limit of the
// instance too, to that of all graphs: threads that launch for different ones must
// not undo each other's.
int prepare(const void* fn, uint32_t smem_bytes) {
  int dev = 0, per_sm = 0;
  cudaFuncAttributes fa{};
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&per_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev) != cudaSuccess ||
      cudaFuncGetAttributes(&fa, fn) != cudaSuccess || per_sm <= 0)
    return (int)cudaGetLastError();
  cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kQ1SmemMax);
  if (e != cudaSuccess) return (int)e;
  const uint64_t need = (uint64_t)kQ1Blocks * (smem_bytes + fa.sharedSizeBytes + 1024);
  const int pct = (int)std::min<uint64_t>(100, (100 * need + per_sm - 1) / per_sm);
  return (int)cudaFuncSetAttribute(fn, cudaFuncAttributePreferredSharedMemoryCarveout, pct);
}

int launch_query1(const DevGraph& g, const Q1State& s, const Q1Params& p, bool bf16,
                  int grid, cudaStream_t stream) {
  void* args[] = {(void*)&g, (void*)&s, (void*)&p};
  const void* fn = q1_fn(!bf16 ? 0 : g.q1.compact_a ? 1 : 2, p.algo == kAlgoAPPS);
  cudaError_t e = (cudaError_t)prepare(fn, p.smem_bytes);
  if (e == cudaSuccess)
    e = cudaLaunchCooperativeKernel(fn, dim3(grid), dim3(kQ1Threads), args, p.smem_bytes, stream);
  return e == cudaSuccess ? 0 : (int)e;
}

// Co-resident grid of every instance (a graph's layout serves every algorithm).
int query1_max_grid(int sm_count, uint32_t smem_bytes) {
  int best = -1;
  for (int i = 0; i < 6; ++i) {
    const void* fn = q1_fn(i % 3, i >= 3);
    int per_sm = 0;
    cudaError_t e = (cudaError_t)prepare(fn, smem_bytes);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, kQ1Threads, smem_bytes);
    if (e != cudaSuccess || per_sm <= 0) {
      cudaGetLastError();
      return -1;
    }
    best = best < 0 ? per_sm : std::min(best, per_sm);
  }
  return best * sm_count;
}

}  // namespace ahpp
