// Single-query push on one thread-block cluster: every round of APP or ASRP for
// one source, on a graph whose residues, t_V and t_A fit in an SM's shared
// memory.
//
// Why: a round of the grid kernel (ahpp_query1.cu) on such a graph is two grid
// barriers of 2,500 cycles, the atomics of the round's sums and a chain of L2
// latencies, 33,000 cycles for 25,000 edges however little each block has to
// do.  Here every block keeps copies of all residues and of all t values, so
// that lookups never leave its SM; the blocks exchange the rows that each has
// computed through distributed shared memory, and the cluster's hardware
// barrier takes the place of the grid's.  All rounds are pull rounds: rows of V
// and A over U in phase 1, rows of U over both in phase 2 (same linear map; the
// push rounds of the grid kernel are counted as it would have counted them).
// The graph's entries lie in shared memory too.
//
// What bounds it: the chain of a round, about 7,500 cycles (two walks, a row's
// sum, two exchanges of 1,200 cycles that end when the remote writes have
// arrived; tiny graph of 2,000 nodes).  One query there: 1.38 ms on the grid
// kernel, 0.40 here; 4,000 nodes and 160,000 entries: 0.95, 0.58.  Graphs whose
// entries do not fit are left to the grid kernel: read from L2 by 16 SMs (24
// cycles of the SM's data path for a step, and blocks sending each other 17 bytes a
// cycle) they were no faster here (6,000 nodes 0.97 against 1.01 ms, 20,000 nodes
// 1.50 against 1.33).
#include <algorithm>
#include <vector>

#include "ahpp_cluster.cuh"
#include "ahpp_host.h"
#include "ahpp_rounds.cuh"

namespace ahpp {

namespace {

// ------------------------------------------------------------------ device

__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// Address of this block's shared memory address `a` in block `rank`.
__device__ __forceinline__ uint32_t in_block(uint32_t a, uint32_t rank) {
  uint32_t r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
  return r;
}
__device__ __forceinline__ void st_cluster(uint32_t a, float v) {
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory");
}
__device__ __forceinline__ void st_cluster(uint32_t a, uint32_t v) {
  asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ float lds(uint32_t a) {
  float v;
  asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(a) : "memory");
  return v;
}

struct ClStep {
  uint2 i;      // four 16-bit indices
  float4 c;
};

// The step at `at` (of this lane's indices).
__device__ __forceinline__ ClStep load_step(uint32_t at) {
  ClStep s;
  asm volatile("ld.shared.v2.u32 {%0,%1}, [%2];" : "=r"(s.i.x), "=r"(s.i.y) : "r"(at) : "memory");
  asm volatile("ld.shared.v4.f32 {%0,%1,%2,%3}, [%4];"
               : "=f"(s.c.x), "=f"(s.c.y), "=f"(s.c.z), "=f"(s.c.w)
               : "r"(at + 256u + (threadIdx.x & 31) * 8u) : "memory");
  return s;
}

__device__ __forceinline__ float look_up(uint32_t x, uint32_t i) { return lds(x + (i << 2)); }

// The walk of a warp's items, whose steps begin at `st`: each row's (or chunk's)
// sum over its entries of c x_i, to its place.
__device__ __forceinline__ void walk(uint32_t st, uint4 r, const uint2* items, uint32_t x, float* places) {
  const uint32_t lane = threadIdx.x & 31;
  st += lane * 8u;
  uint2 nx = r.x < r.y ? items[r.x] : make_uint2(0, 0);
  for (uint32_t it = r.x; it < r.y; ++it) {
    const uint2 a = nx;
    if (it + 1 < r.y) nx = items[it + 1];
    const uint32_t lg = a.y >> 8, row = lane >> lg, cols = a.x >> 16;
    float s = 0.f;
#pragma unroll 1
    for (uint32_t j = cols >> 2; j > 0; --j, st += kClStepBytes) {
      const ClStep e = load_step(st);
      const float4 v = make_float4(look_up(x, e.i.x & 0xffffu), look_up(x, e.i.x >> 16), look_up(x, e.i.y & 0xffffu),
                                   look_up(x, e.i.y >> 16));
      s = fmaf(e.c.w, v.w, fmaf(e.c.z, v.z, fmaf(e.c.y, v.y, fmaf(e.c.x, v.x, s))));
    }
    if (cols & 3u) {
      const ClStep e = load_step(st);
      st += kClStepBytes;
      const float vx = look_up(x, e.i.x & 0xffffu);
      float vy = 0.f, vz = 0.f;
      if ((cols & 3u) > 1) vy = look_up(x, e.i.x >> 16);
      if ((cols & 3u) > 2) vz = look_up(x, e.i.y & 0xffffu);
      s = fmaf(e.c.z, vz, fmaf(e.c.y, vy, fmaf(e.c.x, vx, s)));
    }
#pragma unroll
    for (uint32_t o = 0; o < 5; ++o)
      if (o < lg) s += __shfl_xor_sync(0xffffffffu, s, 1u << o);
    if (row < (a.y & 0xffu) && (lane & ((1u << lg) - 1u)) == 0) places[(a.x & 0xffffu) + row] = s;
  }
}

// A row's sum: its place and those of its further chunks, in their order.
__device__ __forceinline__ float sum_of(const float* places, uint32_t i, uint32_t more) {
  float s = places[i];
  for (uint32_t k = more & 0xffffu, e = k + (more >> 16); k < e; ++k) s += places[k];
  return s;
}

// How a warp takes part in sending this block's rows to the others: the block it
// sends to, and which of the 16-byte pieces (every step-th from first).
struct Sender {
  uint32_t to, first, step;
  __device__ __forceinline__ Sender(uint32_t rank, uint32_t nb) {
    const uint32_t warp = threadIdx.x >> 5, per = kClWarps / (nb - 1), k = warp / per;   // warps to a block
    to = rank + 1 + k;
    if (to >= nb) to -= nb;
    first = k < nb - 1 ? (warp % per) * 32 + (threadIdx.x & 31) : 0x7fffffffu;           // none
    step = per * 32;
  }
  // the n floats (a multiple of 4) at x
  __device__ __forceinline__ void send(const float* x, uint32_t n) const {
    const uint32_t from = smem_addr(x), at = in_block(from, to);
    for (uint32_t i = first; i < n / 4; i += step)
      asm volatile("{\n\t.reg .f32 a, b, c, d;\n\t"
                   "ld.shared.v4.f32 {a, b, c, d}, [%0];\n\t"
                   "st.shared::cluster.v4.f32 [%1], {a, b, c, d};\n\t}"
                   ::"r"(from + 16 * i), "r"(at + 16 * i) : "memory");
  }
};

constexpr uint32_t kSums = 6;     // marked, marked_deg, np_flush, max_r, max_rel, above

}  // namespace

template <bool APPS>
__global__ void __launch_bounds__(kClThreads, 1)
k_cluster(const __grid_constant__ DevGraph g, const __grid_constant__ ClusterLayout C,
          const __grid_constant__ Q1State s, const __grid_constant__ Q1Params p) {
  extern __shared__ __align__(16) unsigned char cl_smem[];
  __shared__ Q1Loop L;
  __shared__ uint32_t s_part[kSums][kClWarps];
  __shared__ uint32_t s_sums[2][kClBlocks][kSums];   // every block's sums, in turn: a block may share again
                                                   // before another has read the last ones
  __shared__ int s_fine;
  const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t rank = cluster_rank(), nb = C.n_blocks;
  const uint32_t nt = g.n_v + g.n_a;
  const uint4 ct = C.t.cta[rank], cu = C.u.cta[rank];
  const uint2 steps_t = C.t.steps[rank], steps_u = C.u.steps[rank];

  // shared memory (the same places in every block)
  uint32_t at = 0;
  auto take = [&](uint32_t bytes) {
    unsigned char* q = cl_smem + at;
    at += (bytes + 15u) & ~15u;
    return q;
  };
  float* p_u = (float*)take(4 * (g.n_u + 3 & ~3u)); // marked residues of all U nodes, else 0
  float* t = (float*)take(4 * (nt + 3 & ~3u));     // t_V, then t_A
  float* places = (float*)take(4 * max(C.t.places_max, C.u.places_max));
  float* r_u = (float*)take(4 * C.u.rows_max);     // the block's rows: residues (sign = marked),
  float* pi = (float*)take(4 * C.u.rows_max);      // reserves and their compensations
  float* pic = (float*)take(4 * C.u.rows_max);
  uint2* items_t = (uint2*)take(8 * C.t.items_max);
  uint2* items_u = (uint2*)take(8 * C.u.items_max);
  uint2* meta_t = (uint2*)take(8 * C.t.rows_max);
  uint2* meta_u = (uint2*)take(8 * C.u.rows_max);
  uint4* st_t = (uint4*)(cl_smem + at);            // steps
  uint4* st_u = st_t + steps_t.y * (kClStepBytes / 16);

  // ---- init: the graph's part of this block, and the state (Algorithm 3's start)
  for (uint32_t i = tid; i < ct.y; i += kClThreads) meta_t[i] = C.t.meta[ct.x + i];
  for (uint32_t i = tid; i < ct.w; i += kClThreads) items_t[i] = C.t.items[ct.z + i];
  for (uint32_t i = tid; i < cu.w; i += kClThreads) items_u[i] = C.u.items[cu.z + i];
  const float r0 = p.lambda_mode ? -1.f : 0.f;
  for (uint32_t i = tid; i < cu.y; i += kClThreads) {
    meta_u[i] = C.u.meta[cu.x + i];
    r_u[i] = r0;
    pi[i] = 0.f;
    pic[i] = 0.f;
  }
  uint4 rg_t = make_uint4(0, 0, 0, 0), rg_u = rg_t;
  if (warp < kClWalkers) {
    rg_t = C.t.ranges[rank * kClWalkers + warp];
    rg_u = C.u.ranges[rank * kClWalkers + warp];
  }
  for (uint32_t i = tid; i < steps_t.y * (kClStepBytes / 16); i += kClThreads)
    st_t[i] = C.steps[(size_t)steps_t.x * (kClStepBytes / 16) + i];
  for (uint32_t i = tid; i < steps_u.y * (kClStepBytes / 16); i += kClThreads)
    st_u[i] = C.steps[(size_t)steps_u.x * (kClStepBytes / 16) + i];
  const uint32_t a_st_t = smem_addr(st_t) + rg_t.z * kClStepBytes, a_st_u = smem_addr(st_u) + rg_u.z * kClStepBytes;
  for (uint32_t i = tid; i < g.n_u; i += kClThreads) p_u[i] = -r0;
  if (rank == 0 && tid == 0) {
    s.ctl->reserve_sum = 0.0;
    s.ctl->resid_sum = 0.0;
    s.final_maxr_bits[0] = 0u;
    s.final_maxr_bits[1] = 0u;
  }
  if (tid == 0) {
    L = Q1Loop{};
    L.phase = (p.lambda_mode || p.pi_mode) ? kPhaseSync : kPhaseAsync;
    L.dense = p.lambda_mode ? 1 : 0;
  }
  // The grid barrier's one use here: the cluster's own barrier cannot run out,
  // this one reports a wait that does.  What a block saw is settled after the
  // cluster barrier, by the error word that all read.
  unsigned int epoch = 0;
  grid_sync(s.bar, nb, epoch);
  cluster_sync();
  if (tid == 0) {
    s_fine = ld_barrier(s.bar).err == 0;
    if (p.lambda_mode) {
      begin_round(p, L, g.n_u, p.e_tot);
    } else {
      const uint32_t cnt = (g.uv_off[p.q + 1] - g.uv_off[p.q]) + (g.ua_off[p.q + 1] - g.ua_off[p.q]);
      const double th = p.algo != kAlgoASRP ? p.eps_f * (double)cnt : p.eps_f;   // APP's per-node threshold
      const bool mark = 1.0 > th;
      if (mark) p_u[p.q] = 1.f;
      if (p.q - cu.x < cu.y) r_u[p.q - cu.x] = mark ? -1.f : 1.f;
      begin_round(p, L, mark ? 1u : 0u, mark ? cnt : 0u);
    }
  }
  __syncthreads();
  const bool fine = s_fine != 0;

  const Sender sender(rank, nb);
  float *own_t = t + ct.x, *own_p = p_u + cu.x;
  Q1Part part;
  uint32_t turn = 0;
  // A round's end: every block gets this block's residues and its sums.
  auto share = [&] {
    const uint32_t v[kSums] = {__reduce_add_sync(0xffffffffu, part.marked),
                               __reduce_add_sync(0xffffffffu, part.marked_deg),
                               __reduce_add_sync(0xffffffffu, part.np_flush),
                               __reduce_max_sync(0xffffffffu, __float_as_uint(part.max_r)),
                               APPS ? __reduce_max_sync(0xffffffffu, __float_as_uint(part.max_rel)) : 0u,
                               APPS ? __reduce_add_sync(0xffffffffu, part.above) : 0u};
    if (lane == 0) {
#pragma unroll
      for (uint32_t k = 0; k < kSums; ++k) s_part[k][warp] = v[k];
    }
    part = Q1Part();
    turn ^= 1;
    __syncthreads();
    if (warp >= kClWarps - kSums) {                  // a warp per sum
      const uint32_t k = warp - (kClWarps - kSums), x = s_part[k][lane];
      const uint32_t sum = k == 3 || k == 4 ? __reduce_max_sync(0xffffffffu, x) : __reduce_add_sync(0xffffffffu, x);
      if (lane < nb) st_cluster(in_block(smem_addr(&s_sums[turn][rank][k]), lane), sum);
    }
    sender.send(own_p, cu.y + 3 & ~3u);
    cluster_sync();
  };
  // The sums' totals (one warp).
  auto total = [&](uint32_t k) {
    const uint32_t x = lane < nb ? s_sums[turn][lane][k] : 0u;
    return k == 3 || k == 4 ? __reduce_max_sync(0xffffffffu, x) : __reduce_add_sync(0xffffffffu, x);
  };

  const uint32_t a_p = smem_addr(p_u), a_t = smem_addr(t);
  bool counted = true;                     // the last round's control has run
  while (fine) {
    // ---- phase 1: t_V and t_A over the marked nodes' residues; meanwhile the
    // last warp decides from the last round's sums whether there is a round (2,000
    // cycles of one lane, which no other waits for)
    walk(a_st_t, rg_t, items_t, a_p, places);
    if (warp == kClWalkers && !counted) {
      const uint32_t mk = total(0), md = total(1), np = total(2), mr = total(3);
      const uint32_t rel = APPS ? total(4) : 0u, ab = APPS ? total(5) : 0u;
      if (lane == 0) {
        if (L.dense) ++L.dense_rounds;
        end_round<APPS>(p, L, __uint_as_float(mr), np, __uint_as_float(rel), ab);
        if (L.go && !L.switched) begin_round(p, L, mk, md);
        else { L.marked = mk; L.marked_deg = md; }
      }
    }
    if (warp < kClWalkers) {
      uint2 m = tid < ct.y ? meta_t[tid] : make_uint2(0, 0);
      asm volatile("bar.sync 1, %0;" ::"n"(kClWalkers * 32) : "memory");
      for (uint32_t i = tid; i < ct.y; i += kClWalkers * 32) {
        if (i != tid) m = meta_t[i];
        const float v = sum_of(places, i, m.y);
        if (v > 0.f) part.np_flush += m.x;
        own_t[i] = v;
      }
    }
    __syncthreads();
    if (!L.go) break;
    if (L.switched) {
      // at the ASRP switch the marks used eps_f; the first synchronous round
      // pushes every positive residue: mark the rest, and begin the phase again
      part = Q1Part();
      for (uint32_t i = tid; i < cu.y; i += kClThreads) {
        const float r = r_u[i];
        if (r > 0.f) {
          part.marked += 1;
          part.marked_deg += meta_u[i].x;
          r_u[i] = -r;
          own_p[i] = r;
        }
      }
      share();
      if (warp == 0) {
        const uint32_t mk = total(0), md = total(1);
        if (lane == 0) {
          L.switched = 0;
          begin_round(p, L, L.marked + mk, L.marked_deg + md);
        }
      }
      counted = true;
      __syncthreads();
      continue;
    }
    const float th = L.theta;
    const bool per_node = L.per_node != 0;
    sender.send(own_t, ct.y + 3 & ~3u);
    cluster_sync();
    // ---- phase 2: the new residues; reserve update of the nodes pushed, marking
    walk(a_st_u, rg_u, items_u, a_t, places);
    uint2 m = tid < cu.y ? meta_u[tid] : make_uint2(0, 0);
    __syncthreads();
    for (uint32_t i = tid; i < cu.y; i += kClThreads) {
      if (i != tid) m = meta_u[i];
      const uint32_t cnt = m.x;
      const float r_old = r_u[i];
      float kept = r_old;
      if (r_old < 0.f) {
        const float add = g.alpha * (-r_old);
        if (p.kahan) kahan_add(pi[i], pic[i], add);
        else pi[i] += add;
        kept = 0.f;
      }
      const float r_new = kept + sum_of(places, i, m.y);
      part.max_r = fmaxf(part.max_r, r_new);
      if (APPS) app_stats(p, r_new, cnt, part);
      const bool mark = per_node ? above_node_threshold(r_new, p.eps_f, p.eps_f32, cnt) : r_new >= th;
      if (mark) {
        part.marked += 1;
        part.marked_deg += cnt;
      }
      r_u[i] = mark ? -r_new : r_new;
      own_p[i] = mark ? r_new : 0.f;
    }
    share();
    counted = false;
  }
  const int status = fine ? L.status : (int)kStatusWait;

  // ---- final: reserves pi - compensation, FP64 sums of reserves and residues
  if (fine) {
    double sp = 0.0, sr = 0.0;
    float mr = 0.f, mp = 0.f;
    for (uint32_t i = tid; i < cu.y; i += kClThreads) {
      const float v = fmaxf(pi[i] - pic[i], 0.f), r = fabsf(r_u[i]);
      s.pi[cu.x + i] = p.pi_mode ? v + r : v;
      s.r_u[cu.x + i] = r_u[i];
      sp += v; sr += r; mr = fmaxf(mr, r); mp = fmaxf(mp, v);
    }
    __shared__ double s_sum[2][kClWarps];
    __shared__ unsigned int s_max[2][kClWarps];
    sp = warp_sum_d(sp); sr = warp_sum_d(sr);
    const unsigned int bmr = __reduce_max_sync(0xffffffffu, __float_as_uint(mr));
    const unsigned int bmp = __reduce_max_sync(0xffffffffu, __float_as_uint(mp));
    if (lane == 0) { s_sum[0][warp] = sp; s_sum[1][warp] = sr; s_max[0][warp] = bmr; s_max[1][warp] = bmp; }
    __syncthreads();
    if (warp < 2) {
      const double d = warp_sum_d(s_sum[warp][lane]);
      const unsigned int m = __reduce_max_sync(0xffffffffu, s_max[warp][lane]);
      if (lane == 0) {
        atomicAdd(warp ? &s.ctl->resid_sum : &s.ctl->reserve_sum, d);
        atomicMax(&s.final_maxr_bits[warp], m);
      }
    }
  }
  if (rank == 0 && tid == 0) {
    s.ctl->n_p = L.n_p;
    s.ctl->pushes = L.pushes;
    s.ctl->rounds = L.rounds;
    s.ctl->switch_round = L.switch_round;
    s.ctl->dense_rounds = L.dense_rounds;
    s.ctl->phase = L.phase;
    s.ctl->status = (status == kStatusOk && L.phase != kPhaseDone) ? kStatusCap : status;
  }
}

// -------------------------------------------------------------------- host

namespace {

using ClusterFn = void (*)(const DevGraph, const ClusterLayout, const Q1State, const Q1Params);

ClusterFn cluster_fn(bool apps) { return apps ? k_cluster<true> : k_cluster<false>; }

// Dynamic shared memory limit and cluster size of an instance (the limit of all
// graphs, so that threads that launch for different ones do not undo each other's).
cudaError_t allow(ClusterFn fn) {
  cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kClSmemMax);
  return e;
}

cudaLaunchConfig_t config(uint32_t blocks, uint32_t smem_bytes, cudaStream_t stream, cudaLaunchAttribute* attr) {
  attr->id = cudaLaunchAttributeClusterDimension;
  attr->val.clusterDim.x = blocks;
  attr->val.clusterDim.y = attr->val.clusterDim.z = 1;
  cudaLaunchConfig_t c{};
  c.gridDim = dim3(blocks);
  c.blockDim = dim3(kClThreads);
  c.dynamicSmemBytes = smem_bytes;
  c.stream = stream;
  c.attrs = attr;
  c.numAttrs = 1;
  return c;
}

// Whether the device can run a cluster of every instance with that much shared memory.
bool cluster_fits(uint32_t blocks, uint32_t smem_bytes) {
  for (int apps = 0; apps < 2; ++apps) {
    ClusterFn fn = cluster_fn(apps != 0);
    cudaLaunchAttribute attr;
    int n = 0;
    cudaError_t e = allow(fn);
    if (e == cudaSuccess) {
      const cudaLaunchConfig_t c = config(blocks, smem_bytes, nullptr, &attr);
      e = cudaOccupancyMaxActiveClusters(&n, fn, &c);
    }
    if (e != cudaSuccess || n < 1) {
      cudaGetLastError();
      return false;
    }
  }
  return true;
}

constexpr uint32_t kItemCols = 6; // an item's ends cost as much as that many columns

uint32_t cols_of(uint32_t len, uint32_t lg) { return (len + (1u << lg) - 1) >> lg; }

struct HostPhase {
  std::vector<uint4> cta, ranges;
  std::vector<uint2> cta_steps, items, meta;
  std::vector<unsigned char> steps;
  uint32_t rows_max = 0, items_max = 0, places_max = 0;
};

struct HostEntry {
  uint32_t i;
  float c;
};

// Rows [0, n) of len(r) entries, entry(r, k), in `blocks` ranges of about equal
// cost; a slice does not cross row `edge` (rows are sorted by length on either
// side of it).
template <typename Len, typename Entry>
HostPhase cut_phase(uint32_t n, uint32_t edge, uint32_t blocks, Len len, Entry entry) {
  HostPhase h;
  uint64_t entries = 0;
  for (uint32_t r = 0; r < n; ++r) entries += len(r);
  // columns of a warp, half of which a row or chunk may take
  const uint32_t most = (uint32_t)std::min<uint64_t>(32, std::max<uint64_t>(4, entries / 32 / (blocks * kClWalkers) / 2 & ~3ull));
  auto cost = [&](uint32_t r) { return (uint64_t)len(r) + 8; };    // a row: its place in all blocks
  uint64_t left = 0;
  for (uint32_t r = 0; r < n; ++r) left += cost(r);
  uint32_t r0 = 0;
  for (uint32_t b = 0; b < blocks; ++b) {
    uint32_t r1 = r0;
    const uint64_t target = left / (blocks - b);
    uint64_t c = 0;
    while (r1 < n && (b + 1 == blocks || (r1 - r0) % 4 || c + cost(r1) / 2 < target)) c += cost(r1++);
    left -= c;
    const uint32_t rows = r1 - r0, item0 = (uint32_t)h.items.size();
    const uint32_t step0 = (uint32_t)(h.steps.size() / kClStepBytes);
    uint32_t lg_min = 0;                   // a slice for every other warp
    while (lg_min < 5 && ((uint64_t)rows << lg_min) / 32 < kClWalkers / 2) ++lg_min;
    uint32_t places = rows, n_steps = 0;
    uint64_t total = 0, done = 0;
    // rows [row, row + rn), their entries from `first` on, 1 << lg lanes to a row:
    // a lane's places beyond the row's end hold index 0 and coefficient 0
    auto put = [&](uint32_t row, uint32_t rn, uint32_t lg, uint32_t first, uint32_t cols, uint32_t place) {
      h.items.push_back(make_uint2(place | cols << 16, rn | lg << 8));
      h.steps.resize((size_t)(step0 + n_steps + (cols + 3) / 4) * kClStepBytes, 0);
      unsigned char* out = h.steps.data() + (size_t)(step0 + n_steps) * kClStepBytes;
      for (uint32_t l = 0; l < rn << lg; ++l)
        for (uint32_t col = 0; col < cols; ++col) {
          const uint32_t k = first + (col << lg) + (l & ((1u << lg) - 1u));
          if (k >= len(row + (l >> lg))) break;
          const HostEntry e = entry(row + (l >> lg), k);
          unsigned char* step = out + (size_t)(col / 4) * kClStepBytes;
          reinterpret_cast<uint16_t*>(step)[4 * l + col % 4] = (uint16_t)e.i;
          reinterpret_cast<float*>(step + 256)[4 * l + col % 4] = e.c;
        }
      n_steps += (cols + 3) / 4;
      total += kItemCols + cols;
    };
    for (uint32_t r = r0; r < r1;) {
      uint32_t lg = lg_min;
      while (lg < 5 && cols_of(len(r), lg) > most) ++lg;
      const uint32_t need = cols_of(len(r), 5);
      if (lg == 5 && need > 2 * most) {    // chunks
        const uint32_t extra = places;
        for (uint32_t f = 0; f < need; f += most)
          put(r, 1, 5, f * 32, std::min(most, need - f), f ? places++ : r - r0);
        h.meta.push_back(make_uint2(len(r), extra | (places - extra) << 16));
        ++r;
        continue;
      }
      const uint32_t end = r < edge ? std::min(edge, r1) : r1, rn = std::min(32u >> lg, end - r);
      uint32_t cols = 0;
      for (uint32_t i = 0; i < rn; ++i) {
        cols = std::max(cols, cols_of(len(r + i), lg));
        h.meta.push_back(make_uint2(len(r + i), 0));
      }
      put(r, rn, lg, 0, cols, r - r0);
      r += rn;
    }
    const uint32_t items = (uint32_t)h.items.size() - item0;
    uint32_t it = 0, stp = 0;
    for (uint32_t w = 0; w < (uint32_t)kClWalkers; ++w) {
      const uint32_t i0 = it, s0 = stp;
      const uint64_t goal = total * (w + 1) / kClWalkers;
      while (it < items) {
        const uint32_t cols = h.items[item0 + it].x >> 16;
        if (w + 1 < (uint32_t)kClWalkers && done + (kItemCols + cols) / 2 >= goal) break;
        done += kItemCols + cols;
        stp += (cols + 3) / 4;
        ++it;
      }
      h.ranges.push_back(make_uint4(i0, it, s0, stp));
    }
    h.cta.push_back(make_uint4(r0, rows, item0, items));
    h.cta_steps.push_back(make_uint2(step0, n_steps));
    h.rows_max = std::max(h.rows_max, rows);
    h.items_max = std::max(h.items_max, items);
    h.places_max = std::max(h.places_max, places);
    r0 = r1;
  }
  return h;
}

}  // namespace

// The cluster layout of a graph that is small enough for it, else none (g->cl
// stays empty).
int build_cluster_layout(ahpp_graph* g) {
  const DevGraph& G = g->dg;
  g->cl = ClusterLayout();
  const uint32_t nU = G.n_u, nV = G.n_v, nA = G.n_a;
  // without padding: the vectors, and each block's share of both phases' entries
  const uint64_t entries = 2 * ((uint64_t)G.n_e + G.n_ea);
  if (4 * ((uint64_t)nU + nV + nA) + entries / kClBlocks * 6 > kClSmemMax) return AHPP_OK;

  auto down = [&](auto& v, const void* p, size_t n) {
    v.resize(n);
    return n == 0 || cudaMemcpy(v.data(), p, n * sizeof(v[0]), cudaMemcpyDeviceToHost) == cudaSuccess;
  };
  std::vector<uint32_t> uv, uvi, vu, vui, ua, uai, au, aui;
  std::vector<float> uvw, vuc, rn, cn, uaw, auw;
  bool ok = down(uv, G.uv_off, (size_t)nU + 1) && down(uvi, G.uv_idx, G.n_e) && down(uvw, G.uv_w, G.n_e) &&
            down(vu, G.vu_off, (size_t)nV + 1) && down(vui, G.vu_idx, G.n_e) && down(vuc, G.vu_c, G.n_e) &&
            down(ua, G.ua_off, (size_t)nU + 1) && down(uai, G.ua_idx, G.n_ea) &&
            down(au, G.au_off, (size_t)nA + 1) && down(aui, G.au_idx, G.n_ea) &&
            down(rn, G.rnorm_u, nU) && down(cn, G.cnorm_a, nA);
  auto weights = [&](std::vector<float>& w, const void* p) {
    if (!g->bf16) return down(w, p, G.n_ea);
    std::vector<__nv_bfloat16> h;
    if (!down(h, p, G.n_ea)) return false;
    w.resize(h.size());
    for (size_t i = 0; i < h.size(); ++i) w[i] = __bfloat162float(h[i]);
    return true;
  };
  if (!ok || !weights(uaw, G.ua_w) || !weights(auw, G.au_w))
    return cuda_fail(cudaGetLastError(), "cluster layout: adjacency");

  auto len_t = [&](uint32_t r) { return r < nV ? vu[r + 1] - vu[r] : au[r - nV + 1] - au[r - nV]; };
  // t_A[a] = k_attr / W_col(a) sum_u w(u,a) p_u / W_row(u): one coefficient per
  // entry, rounded once
  auto entry_t = [&](uint32_t r, uint32_t k) {
    if (r < nV) return HostEntry{vui[vu[r] + k], vuc[vu[r] + k]};
    const uint32_t e = au[r - nV] + k;
    return HostEntry{aui[e], (float)((double)G.k_attr * cn[r - nV] * auw[e] * rn[aui[e]])};
  };
  auto len_u = [&](uint32_t u) { return (uv[u + 1] - uv[u]) + (ua[u + 1] - ua[u]); };
  auto entry_u = [&](uint32_t u, uint32_t k) {
    const uint32_t d = uv[u + 1] - uv[u];
    if (k < d) return HostEntry{uvi[uv[u] + k], uvw[uv[u] + k]};
    return HostEntry{nV + uai[ua[u] + k - d], uaw[ua[u] + k - d]};
  };
  const uint32_t blocks = kClBlocks;
  const HostPhase t = cut_phase(nV + nA, nV, blocks, len_t, entry_t);
  const HostPhase u = cut_phase(nU, nU, blocks, len_u, entry_u);
  if (std::max(t.places_max, u.places_max) > 0xffff) return AHPP_OK;
  auto up16 = [](uint64_t x) { return (x + 15) / 16 * 16; };
  uint64_t steps = 0;                    // of any block
  for (uint32_t b = 0; b < blocks; ++b) steps = std::max<uint64_t>(steps, (uint64_t)t.cta_steps[b].y + u.cta_steps[b].y);
  const uint64_t smem = up16(4ull * nU) + up16(4ull * (nV + nA)) + up16(4ull * std::max(t.places_max, u.places_max)) +
                        3 * up16(4ull * u.rows_max) + up16(8ull * t.items_max) + up16(8ull * u.items_max) +
                        up16(8ull * t.rows_max) + up16(8ull * u.rows_max) + steps * kClStepBytes;
  if (smem > kClSmemMax || !cluster_fits(blocks, (uint32_t)smem)) return AHPP_OK;

  const uint64_t before = g->layout_bytes;
  auto put = [&](const void* p, size_t bytes) -> void* {
    void* d = g->alloc(std::max<size_t>(bytes, 16));
    if (!d || upload(g, d, p, bytes) != cudaSuccess) ok = false;
    g->layout_bytes += std::max<size_t>(bytes, 16);
    return d;
  };
  auto rows = [&](const HostPhase& h, uint32_t step0, ClusterRows& R) {
    std::vector<uint2> first = h.cta_steps;
    for (auto& x : first) x.x += step0;
    R.cta = (const uint4*)put(h.cta.data(), h.cta.size() * sizeof(uint4));
    R.steps = (const uint2*)put(first.data(), first.size() * sizeof(uint2));
    R.items = (const uint2*)put(h.items.data(), h.items.size() * sizeof(uint2));
    R.meta = (const uint2*)put(h.meta.data(), h.meta.size() * sizeof(uint2));
    R.ranges = (const uint4*)put(h.ranges.data(), h.ranges.size() * sizeof(uint4));
    R.rows_max = h.rows_max;
    R.items_max = h.items_max;
    R.places_max = h.places_max;
  };
  ClusterLayout C;
  rows(t, 0, C.t);
  rows(u, (uint32_t)(t.steps.size() / kClStepBytes), C.u);
  std::vector<unsigned char> all(t.steps);
  all.insert(all.end(), u.steps.begin(), u.steps.end());
  C.steps = (const uint4*)put(all.data(), all.size());
  C.n_blocks = blocks;
  C.smem_bytes = (uint32_t)smem;
  if (!ok) {
    g->layout_bytes = before;
    set_error("cluster layout: device allocation failed");
    return AHPP_ENOMEM;
  }
  g->cl = C;
  return AHPP_OK;
}

int launch_cluster(const DevGraph& g, const ClusterLayout& c, const Q1State& s, const Q1Params& p,
                   cudaStream_t stream) {
  ClusterFn fn = cluster_fn(p.algo == kAlgoAPPS);
  cudaLaunchAttribute attr;
  const cudaLaunchConfig_t cfg = config(c.n_blocks, c.smem_bytes, stream, &attr);
  cudaError_t e = allow(fn);
  if (e == cudaSuccess) e = cudaLaunchKernelEx(&cfg, fn, g, c, s, p);
  return (int)e;
}

}  // namespace ahpp
