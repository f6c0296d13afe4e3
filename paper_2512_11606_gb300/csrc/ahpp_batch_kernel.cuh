// Batched multi-source APP / ASRP: one persistent cooperative launch runs n
// queries packed into tiles of kTile (one query per lane).  Every round of a
// tile is a pull sweep over the whole graph (the synchronous form of
// Algorithm 3's three loops): phase 1 gathers t_V and t_A for all the tile's
// queries from the marked residues, phase 2 gathers the new residues from both,
// applies the reserve update of the pushed nodes and marks the next frontier of
// each query with its own threshold.  Per-query control (termination, the ASRP
// switch test of Algorithm 4) is kept per lane; a query that finishes is
// frozen while the rest of its tile continues, so its result does not depend
// on the other queries of the tile.  Top-k per query is a per-lane radix
// select over (score, caller id) keys.
//
// What bounds a tile's round: 128-byte row gathers, two per edge and two per
// attribute entry, out of L2 (and HBM, where the tables are larger).  A warp
// has 32 rows in flight, 24 warps an SM; the round is short when all warps have
// them in flight all the time, so
//   - a warp's entries lie in the order of its use (TileRows), copied ahead to
//     a ring in shared memory: no index load stands before a gather;
//   - warps share the items by measured cost, the last fifth from a pool;
//   - chunks of long rows go over the table in step (add_chunks), so that each
//     row of a table larger than L2 is fetched once;
//   - the attribute hop is pulled: no reductions (47 G rows/s at best) beside
//     the gathers, and both hops of phase 2 are one list over one table.
// Medium graph, tile of 32, one round: 1,130 us before, 835 now (96 G rows/s;
// 0.69 and 0.98 million cycles in the phases, even to 1 %); 100k nodes: 145 us
// one tile alone, 103 now, 84 with four at once.
// This file is the kernel body of ahpp_batch.cu, which includes it once per
// tile width: AHPP_BT (queries per tile) and AHPP_BT_NS (the namespace of
// that instance) are defined by the includer.  No include guard.
#include "ahpp_batch.cuh"

namespace ahpp {
namespace AHPP_BT_NS {

constexpr int kTile = AHPP_BT;     // queries per tile of this instance


namespace {

constexpr unsigned kFull = 0xffffffffu;

struct BCtx {
  const DevGraph& g;
  const TileBuf& t;
  const BatchParams& p;
  uint32_t gw, nw;     // warp id / count within the group
  uint32_t gt, nt;     // thread id / count within the group
  uint32_t lane;
};

// Shared memory behind the rings: rows copied for a phase, and between phases
// the block reductions, the top-k histograms and the sort buffer.
__device__ __forceinline__ unsigned char* scratch_of(unsigned char* smem) { return smem + kTRingBytes; }

// Per-lane block reduction of a sum and a maximum into acc[lane] (buf: scratch memory).
__device__ __forceinline__ void flush_lane(double sum, float mx, RAcc* acc, unsigned char* buf) {
  double (*s)[32] = reinterpret_cast<double (*)[32]>(buf);
  float (*m)[32] = reinterpret_cast<float (*)[32]>(buf + sizeof(double) * 32 * kBWarps);
  static_assert((sizeof(double) + sizeof(float)) * 32 * kBWarps <= kTHubRows * 128, "fits the scratch memory");
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  __syncthreads();
  s[warp][lane] = sum;
  m[warp][lane] = mx;
  __syncthreads();
  if (warp == 0 && lane < kTile) {
    for (int w = 1; w < kBWarps; ++w) {
      sum += s[w][lane];
      mx = fmaxf(mx, m[w][lane]);
    }
    if (mx > 0.f) atomicMax(&acc[lane].max_r_bits, __float_as_uint(mx));
    if (sum != 0.0) atomicAdd(&acc[lane].sum_r, sum);
  }
  __syncthreads();
}

// ------------------------------------------------------------------------
// Pull phases with row groups: a warp is 4 groups of 8 lanes, each on one row
// (or one chunk of a long row).  A gathered row of the tile is kTile values:
// with 32 queries each lane owns 4 of them (one float4, the group reads a
// 128-byte line); with 16, four lanes own a 64-byte row and the group's halves
// take every other entry.
constexpr int kQL = 4;                 // queries per lane
constexpr int kRL = kTile / kQL;       // lanes per gathered row
constexpr int kEP = 8 / kRL;           // entries a group takes at once
static_assert(kTile == 16 || kTile == 32, "tile of 16 or 32 queries");
static_assert(kAccCopies * kTile <= kBThreads, "one thread per accumulator record");

// Reserves and compensations are read once per round: streamed with the
// evict-first policy so that they do not push the gathered rows out of L2.
template <typename T>
__device__ __forceinline__ T ld_stream(const T* p) {
  return __ldcs(p);
}

// out[0..3] += v as a reduction that returns nothing: an atomicAdd on a
// float4 whose result is unused is still issued as a returning atomic, and
// the returned line then takes L2 -> SM bandwidth that the gathers need.
__device__ __forceinline__ void red_add4(float* out, float4 v) {
  asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(out), "f"(v.x), "f"(v.y), "f"(v.z),
               "f"(v.w)
               : "memory");
}

// The warp's ring: its next kTRing units of the phase's stream (TileRows),
// copied to shared memory ahead of their use and across the barrier.
struct TileRing {
  const uint4* src;            // the lane's place in unit 0
  uint32_t base;               // the warp's ring
  uint32_t next, end;          // next unit to copy, end of the stream

  // no block ends while copies to its shared memory are in flight
  __device__ __forceinline__ ~TileRing() { asm volatile("cp.async.wait_all;" ::: "memory"); }
  __device__ __forceinline__ void refill() {
    if (next < end)
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(base + (next % kTRing) * 512u +
                                                                    (threadIdx.x & 31u) * 16u),
                   "l"(src + (size_t)next * 32) : "memory");
    asm volatile("cp.async.commit_group;" ::: "memory");
    ++next;
  }
  __device__ __forceinline__ void start(const uint4* units, uint32_t b, uint32_t e) {
    src = units + (threadIdx.x & 31u);
    next = b;
    end = e;
    __syncwarp();              // every lane is done with the units of the last stream
#pragma unroll
    for (uint32_t i = 0; i < kTRing; ++i) refill();
  }
  // unit k for every lane of the warp
  __device__ __forceinline__ void wait() const {
    asm volatile("cp.async.wait_group %0;" ::"n"((int)kTRing - 1) : "memory");
    __syncwarp();
  }
};

// Row i of the table (4 of its values for this lane): from the copy of rows
// [first, first + n_hub) in shared memory, else from L2.  s_row: the lane's
// place in the copy's first row.  Half of the rows that a power-law graph's
// long lists name come up again and again; reading those from shared memory
// takes them off the L2 -> SM path, which bounds the gathers.
__device__ __forceinline__ float4 gather_row(uint32_t i, uint32_t first, uint32_t n_hub, uint32_t s_row,
                                             const float* x) {
  float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
  asm volatile("{\n\t.reg .pred p, q, r;\n\t"
               "setp.ne.u32 r, %4, 0xffffffff;\n\t"
               "setp.lt.and.u32 p, %5, %6, r;\n\t"
               "setp.ge.and.u32 q, %5, %6, r;\n\t"
               "@p ld.shared.v4.f32 {%0, %1, %2, %3}, [%7];\n\t"
               "@q ld.global.v4.f32 {%0, %1, %2, %3}, [%8];\n\t}"
               : "+f"(v.x), "+f"(v.y), "+f"(v.z), "+f"(v.w)
               : "r"(i), "r"(i - first), "r"(n_hub), "r"(s_row + (i - first) * (kTile * 4u)),
                 "l"(x + (size_t)i * kTile)
               : "memory");
  return v;
}

// Sum over the `entries` entries (of the warp's longest row) from unit k on of
// coefficient * value(gathered row): waves of eight entries of each row, whose
// gathers are in flight together.  k advances past the item's units.
template <typename Index, typename Value>
__device__ __forceinline__ float4 walk(TileRing& ring, uint32_t& k, uint32_t entries, uint32_t first, uint32_t n_hub,
                                       uint32_t s_row, const float* x, Index index, Value value) {
  const uint32_t lane = threadIdx.x & 31u, r = lane >> 3, sub = (lane & 7u) / kRL;
  float2 a01 = make_float2(0.f, 0.f), a23 = make_float2(0.f, 0.f);
#pragma unroll 1
  for (uint32_t e0 = 0; e0 < entries; e0 += 8) {
    if ((e0 & 8u) == 0) ring.wait();
    const uint32_t row = ring.base + (k % kTRing) * 512u + r * 128u;
    float4 v[8 / kEP];
    float co[8 / kEP];
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      uint32_t i0, i1;
      float c0, c1;
      asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];"
                   : "=r"(i0), "=f"(c0), "=r"(i1), "=f"(c1)
                   : "r"(row + ((((e0 & 8u) >> 1) + t + 2 * r) & 7u) * 16u) : "memory");
      if (kEP == 1) {
        co[2 * t % (8 / kEP)] = c0;
        co[(2 * t + 1) % (8 / kEP)] = c1;
        v[2 * t % (8 / kEP)] = gather_row(index(i0), first, n_hub, s_row, x);
        v[(2 * t + 1) % (8 / kEP)] = gather_row(index(i1), first, n_hub, s_row, x);
      } else {
        co[t % (8 / kEP)] = sub ? c1 : c0;
        v[t % (8 / kEP)] = gather_row(index(sub ? i1 : i0), first, n_hub, s_row, x);
      }
    }
    if ((e0 & 8u) || e0 + 8 >= entries) {          // the unit is used up
      ++k;
      __syncwarp();
      ring.refill();
    }
#pragma unroll
    for (int t = 0; t < 8 / kEP; ++t) {
      const float4 y = value(v[t]);
      const float2 cc = make_float2(co[t], co[t]);
      a01 = __ffma2_rn(cc, make_float2(y.x, y.y), a01);
      a23 = __ffma2_rn(cc, make_float2(y.z, y.w), a23);
    }
  }
  if (kEP == 2) {
    a01.x += __shfl_xor_sync(kFull, a01.x, kRL); a01.y += __shfl_xor_sync(kFull, a01.y, kRL);
    a23.x += __shfl_xor_sync(kFull, a23.x, kRL); a23.y += __shfl_xor_sync(kFull, a23.y, kRL);
  }
  return make_float4(a01.x, a01.y, a23.x, a23.y);
}

// A phase's items of this warp, in segments: its chunks, its slices, then what
// it grabs from the pool while there is any.  rg: its two ranges (tile_ranges);
// first(ring) has been called for the phase already, across the barrier.
struct Segments {
  const TileRows& L;
  const uint4* rg;
  unsigned int* taken;
  uint32_t seg = 0, i0 = 0, i1 = 0, grabbed = 0;

  // the ring's first stream: the chunks', or the slices' where there are none
  static __device__ __forceinline__ void first(TileRing& ring, const TileRows& L, const uint4* rg) {
    const uint4 u = rg[1];
    if (rg[0].x < rg[0].y) ring.start(L.units, u.x, u.y);
    else ring.start(L.units, u.z, u.w);
  }
  __device__ __forceinline__ bool next(TileRing& ring) {
    const uint4 r = rg[0];
    if (seg == 0) {
      seg = 1;
      i0 = r.x;
      i1 = r.y;
      if (i0 < i1) return true;
    }
    if (seg == 1) {
      seg = 2;
      if (r.x < r.y) ring.start(L.units, rg[1].z, rg[1].w);
      i0 = r.z;
      i1 = r.w;
      if (L.pool < L.n_items && (threadIdx.x & 31u) == 0) grabbed = atomicAdd(taken, 1u);   // known by the time it is needed
      if (i0 < i1) return true;
    }
    if (L.pool >= L.n_items) return false;
    i0 = L.pool + __shfl_sync(kFull, grabbed, 0) * L.batch;
    if (i0 >= L.n_items) return false;
    i1 = min(i0 + L.batch, L.n_items);
    if ((threadIdx.x & 31u) == 0) grabbed = atomicAdd(taken, 1u);
    ring.start(L.units, L.items[i0].w, L.items[i1].w);
    return true;
  }
};

// Copies rows [0, n) at x to shared memory (the block).
__device__ __forceinline__ void copy_rows(unsigned char* buf, const float* x, uint32_t n) {
  for (uint32_t i = threadIdx.x; i < n * (kTile / 4); i += kBThreads)
    reinterpret_cast<float4*>(buf)[i] = reinterpret_cast<const float4*>(x)[i];
}

// Per-query partials of one thread (its 4 queries) in phase 2.
template <bool APPS>
struct Q4Partials {
  float max_r[kQL] = {0.f, 0.f, 0.f, 0.f};
  uint32_t marked[kQL] = {0, 0, 0, 0};
  uint32_t mdeg[kQL] = {0, 0, 0, 0};
};
template <>
struct Q4Partials<true> : Q4Partials<false> {
  float max_rel[kQL] = {0.f, 0.f, 0.f, 0.f};   // APP(S) statistics (see RAcc)
  uint32_t above[kQL] = {0, 0, 0, 0};
};

// The block's round partials in shared memory: fields of 32 queries each
// (floats are >= 0, so their bits order them).
enum : int { kAccMax = 0, kAccMarked, kAccDeg, kAccNp, kAccRel, kAccAbove, kAccFields };
using BlockAcc = uint32_t[kAccFields][32];

__device__ __forceinline__ uint32_t bits_of(uint32_t x) { return x; }
__device__ __forceinline__ uint32_t bits_of(float x) { return __float_as_uint(x); }

// v[0..3] (of this lane's queries) into field f, over the warp's lanes first.
template <bool MAX, typename T>
__device__ __forceinline__ void add_field(BlockAcc& acc, int f, const T (&v)[kQL]) {
  const uint32_t lane = threadIdx.x & 31;
#pragma unroll
  for (int j = 0; j < kQL; ++j) {
    uint32_t x = bits_of(v[j]);
#pragma unroll
    for (int o = kRL; o < 32; o <<= 1) {
      const uint32_t y = __shfl_xor_sync(kFull, x, o);
      x = MAX ? max(x, y) : x + y;
    }
    if (lane < kRL && x) {
      if (MAX) atomicMax(&acc[f][lane * kQL + j], x);
      else atomicAdd(&acc[f][lane * kQL + j], x);
    }
  }
}

// The block's partials of the round into one copy of the tile's accumulators,
// cleared for the next round.
template <bool APPS>
__device__ __forceinline__ void flush_round(BlockAcc& acc, TAcc* out) {
  __syncthreads();
  const uint32_t f = threadIdx.x >> 5, q = threadIdx.x & 31;
  if (f >= (APPS ? 5u : 3u)) return;
  TAcc* a = out + q;
  const bool lq = q < (uint32_t)kTile;
  auto take = [&](int field) {
    const uint32_t x = acc[field][q];
    acc[field][q] = 0;
    return x;
  };
  if (f == 0) { const uint32_t x = take(kAccMax); if (lq && x) atomicMax(&a->max_r_bits, x); }
  if (f == 1) { const uint32_t x = take(kAccNp); if (lq && x) atomicAdd(&a->np, x); }
  if (f == 2) {
    const uint32_t m = take(kAccMarked), d = take(kAccDeg);
    if (lq && m) atomicAdd(&a->marked_deg, (unsigned long long)d << 32 | m);
  }
  if (f == 3) { const uint32_t x = take(kAccRel); if (lq && x) atomicMax(&a->max_rel_bits, x); }
  if (f == 4) { const uint32_t x = take(kAccAbove); if (lq && x) atomicAdd(&a->above, x); }
}

// A query's accumulators over their copies.
struct RoundSums {
  uint32_t max_r_bits = 0, np = 0, marked = 0, marked_deg = 0, max_rel_bits = 0, above = 0;
};
template <bool APPS>
__device__ __forceinline__ RoundSums sums_of(const TAcc* a) {
  RoundSums s;
#pragma unroll
  for (uint32_t k = 0; k < kAccCopies; ++k) {
    const TAcc* x = a + k * kTile;
    s.max_r_bits = max(s.max_r_bits, __ldcg(&x->max_r_bits));
    s.np += __ldcg(&x->np);
    const unsigned long long m = __ldcg(&x->marked_deg);
    s.marked += (uint32_t)m;
    s.marked_deg += (uint32_t)(m >> 32);
    if (APPS) {
      s.max_rel_bits = max(s.max_rel_bits, __ldcg(&x->max_rel_bits));
      s.above += __ldcg(&x->above);
    }
  }
  return s;
}

__device__ __forceinline__ void count4(uint32_t (&np)[kQL], float4 t, uint32_t d) {
  np[0] += t.x > 0.f ? d : 0; np[1] += t.y > 0.f ? d : 0;
  np[2] += t.z > 0.f ? d : 0; np[3] += t.w > 0.f ? d : 0;
}

// Phase 1: the table's rows (t_V, t_A) from the marked residues,
//   t_V[v] = sum_u c_uv(u,v) p_u;   t_A[a] = k_attr cnorm_a[a] sum_u w(u,a) rnorm_u[u] p_u.
// The attribute hop is pulled like the V hop: 20M more gathers of 128-byte rows
// take less than the 20M float4 reductions of pushing it from phase 2 (108 G
// rows/s from a 128 MB table against 47 G reductions/s, measured alone).
__device__ __forceinline__ void gphase1(const BCtx& c, BlockAcc& sums, TileRing& ring, const uint4* rg,
                                        GridBarrier* bar, uint32_t set, unsigned char* buf) {
  uint32_t np[kQL] = {0, 0, 0, 0};
  const DevGraph& g = c.g;
  const uint32_t lane = c.lane, ql = kQL * (lane & (kRL - 1)), gi = lane >> 3;
  const bool lead = (lane & 7u) < (uint32_t)kRL;             // this lane writes its queries' sums
  const float* x = c.t.r_u + ql;
  float* acc = c.t.t + (size_t)(g.n_v + set * g.tl.n_acc) * kTile + ql;
  const uint32_t n_hub = min(g.n_u, kTHubRows);
  copy_rows(buf, c.t.r_u, n_hub);
  __syncthreads();
  const uint32_t s_row = smem_addr(buf) + ql * 4u;
  if (c.gt == 0) bar->taken[1] = 0;                          // the other phase's pool is full again
  Segments sg{g.tl.t, rg, &bar->taken[0]};
  while (sg.next(ring)) {
    uint4 a = g.tl.t.items[sg.i0];
    uint32_t k = a.w;
#pragma unroll 1
    for (uint32_t it = sg.i0; it < sg.i1; ++it) {
      const uint4 ca = a;
      if (it + 1 < sg.i1) a = g.tl.t.items[it + 1];
      const bool chunk = ca.y >> 31, ok = gi < (ca.y & 0xffu);
      uint32_t row = ca.x + gi, d = 0;
      if (chunk && ok) row = g.tl.t.chunk_row[ca.x + gi];
      if (!chunk && ok) d = g.q1.deg_v[row];
      const float4 s = walk(ring, k, ca.z, 0u, n_hub, s_row, x, [](uint32_t i) { return i; },
                            [](float4 v) { return make_float4(fmaxf(-v.x, 0.f), fmaxf(-v.y, 0.f), fmaxf(-v.z, 0.f),
                                                              fmaxf(-v.w, 0.f)); });
      if (!ok || !lead) continue;
      if (chunk) {
        red_add4(acc + (size_t)row * kTile, s);
      } else {
        *reinterpret_cast<float4*>(c.t.t + (size_t)row * kTile + ql) = s;
        count4(np, s, d);
      }
    }
  }
  __syncwarp();
  add_field<false>(sums, kAccNp, np);
}

// Residue update of row u for this lane's 4 queries: reserve update of the
// queries that pushed u this round, then the mark for the next round.
// APPLIKE: APP or APP(S) (per-node thresholds possible, r_max read per query);
// APPS: APP(S)'s round statistics too.  ASRP launches compile neither.
template <bool APPLIKE, bool APPS>
__device__ __forceinline__ void gepilogue2(const BCtx& c, uint32_t u, float4 s, const float* th, uint32_t act,
                                           uint32_t pn, const LaneCtl* ctl, Q4Partials<APPS>& part) {
  const uint32_t ql = kQL * (c.lane & (kRL - 1)), cnt = c.g.q1.deg_u[u];
  const size_t i = (size_t)u * kTile + ql;
  float4 r = *reinterpret_cast<const float4*>(c.t.r_u + i);
  float4 pv = ld_stream(reinterpret_cast<const float4*>(c.t.pi + i));
  float4 pc = ld_stream(reinterpret_cast<const float4*>(c.t.pic + i));
  float* rr = &r.x;
  float* pvv = &pv.x;
  float* pcc = &pc.x;
  const float* ss = &s.x;
  bool pushed_any = false;
#pragma unroll
  for (int j = 0; j < kQL; ++j) {
    if (!(act >> j & 1u)) continue;
    float kept = rr[j];
    if (kept < 0.f) {
      const float add = c.g.alpha * (-kept);
      if (c.p.kahan) kahan_add(pvv[j], pcc[j], add);
      else pvv[j] += add;
      kept = 0.f;
      pushed_any = true;
    }
    const float r_new = kept + ss[j];
    part.max_r[j] = fmaxf(part.max_r[j], r_new);
    bool mark;
    if (APPLIKE) {
      const double rmx = ctl[ql + j].eps_f;               // APP's r_max for per-node thresholds
      if constexpr (APPS) {
        if (cnt) part.max_rel[j] = fmaxf(part.max_rel[j], r_new / (float)cnt);
        if (above_node_threshold(r_new, rmx, (float)rmx, cnt)) part.above[j] += 1;
      }
      mark = (pn >> j & 1u) ? above_node_threshold(r_new, rmx, (float)rmx, cnt) : r_new >= th[j];
    } else {
      mark = r_new >= th[j];
    }
    rr[j] = mark ? -r_new : r_new;
    part.marked[j] += mark;
    part.mdeg[j] += mark ? cnt : 0u;
  }
  *reinterpret_cast<float4*>(c.t.r_u + i) = r;
  if (pushed_any) {
    __stcs(reinterpret_cast<float4*>(c.t.pi + i), pv);
    __stcs(reinterpret_cast<float4*>(c.t.pic + i), pc);
  }
}

// Phase 2: new residues of every U node for the tile's queries, over both hops
// at once from the table; the other set of accumulated rows is cleared.
template <bool APPLIKE, bool APPS>
__device__ __forceinline__ void gphase2(const BCtx& c, const LaneCtl* ctl, BlockAcc& sums, TileRing& ring,
                                        const uint4* rg, GridBarrier* bar, uint32_t set, unsigned char* buf) {
  const DevGraph& g = c.g;
  const uint32_t lane = c.lane, ql = kQL * (lane & (kRL - 1)), gi = lane >> 3, n_acc = g.tl.n_acc, n_v = g.n_v;
  const bool lead = (lane & 7u) < (uint32_t)kRL;
  // mark thresholds and activity of this lane's 4 queries: APP's per-node
  // thresholds (pn), or one threshold (eps_f, or 0 once synchronous)
  float th[kQL];
  uint32_t act = 0, pn = 0;
#pragma unroll
  for (int j = 0; j < kQL; ++j) {
    const LaneCtl& q = ctl[ql + j];
    act |= (uint32_t)(q.active != 0) << j;
    if (APPLIKE) pn |= (uint32_t)per_node_threshold(c.p.algo, q.phase) << j;
    th[j] = q.phase == kPhaseSync ? __uint_as_float(1u) : q.th_async;    // smallest float above 0
  }
  const uint32_t shift = set * n_acc, n_hub = min(n_acc, kTHubRows);
  float* cur = c.t.t + (size_t)(n_v + shift) * kTile;
  float* other = c.t.t + (size_t)(n_v + (n_acc - shift)) * kTile;
  copy_rows(buf, cur, n_hub);
  // active accumulated rows (Algorithm 4's push counter); the next round's start at zero
  uint32_t np[kQL] = {0, 0, 0, 0};
  for (uint32_t j = c.gw * 4 + gi; j < n_acc; j += c.nw * 4) {
    const size_t i = (size_t)j * kTile + ql;
    if (!lead) continue;
    count4(np, *reinterpret_cast<const float4*>(cur + i), g.tl.acc_deg[j]);
    *reinterpret_cast<float4*>(other + i) = make_float4(0.f, 0.f, 0.f, 0.f);
  }
  add_field<false>(sums, kAccNp, np);
  Q4Partials<APPS> part;
  __syncthreads();
  const uint32_t s_row = smem_addr(buf) + ql * 4u, first = n_v + shift;
  const float* x = c.t.t + ql;
  if (c.gt == 0) bar->taken[0] = 0;
  Segments sg{g.tl.u, rg, &bar->taken[1]};
  while (sg.next(ring)) {
    uint4 a = g.tl.u.items[sg.i0];
    uint32_t k = a.w;
#pragma unroll 1
    for (uint32_t it = sg.i0; it < sg.i1; ++it) {
      const uint4 ca = a;
      if (it + 1 < sg.i1) a = g.tl.u.items[it + 1];
      const bool chunk = ca.y >> 31, ok = gi < (ca.y & 0xffu);
      const bool mine = ok && lead && !chunk && act;
      uint32_t u = ca.x + gi;
      if (chunk && ok) u = g.tl.u.chunk_row[ca.x + gi];
      const float4 s = walk(ring, k, ca.z, first, n_hub, s_row, x,
                            [&](uint32_t i) { return i >= n_v && i != kNoEntry ? i + shift : i; },
                            [](float4 v) { return v; });
      if (mine) gepilogue2<APPLIKE, APPS>(c, u, s, th, act, pn, ctl, part);
      else if (chunk && ok && lead) red_add4(c.t.split_acc + (size_t)u * kTile + ql, s);
    }
  }
  // the warp's chunks: the last chunk of a row to be counted finishes it
  // (counted only now, so that no walk waits for the counter)
#pragma unroll 1
  for (uint32_t it = rg[0].x; it < rg[0].y; ++it) {
    const uint4 ca = g.tl.u.items[it];
    __syncwarp();
    const bool ok = gi < (ca.y & 0xffu);
    uint32_t u = 0, last = 0;
    if (ok) {
      u = g.tl.u.chunk_row[ca.x + gi];
      if ((lane & 7u) == 0) {
        uint32_t seen;
        asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], 1;" : "=r"(seen) : "l"(&c.t.split_cnt[u]) : "memory");
        last = seen == g.tl.chunks_of[u] - 1;
      }
    }
    last = __shfl_sync(kFull, last, 0, 8);
    if (!last || !lead) continue;
    const size_t i = (size_t)u * kTile + ql;
    float4* sp = reinterpret_cast<float4*>(c.t.split_acc + i);
    const float4 s = __ldcg(sp);
    __stcg(sp, make_float4(0.f, 0.f, 0.f, 0.f));
    if ((lane & 7u) == 0) c.t.split_cnt[u] = 0;
    if (!act) continue;
    gepilogue2<APPLIKE, APPS>(c, u, s, th, act, pn, ctl, part);
  }
  __syncwarp();
  add_field<true>(sums, kAccMax, part.max_r);
  add_field<false>(sums, kAccMarked, part.marked);
  add_field<false>(sums, kAccDeg, part.mdeg);
  if constexpr (APPS) {
    add_field<true>(sums, kAccRel, part.max_rel);
    add_field<false>(sums, kAccAbove, part.above);
  }
}

__device__ __forceinline__ bool switch_now(const BatchParams& p, const LaneCtl& L, float m) {
  return switch_due(p.e_tot, p.switch_rule, L.eps_f, p.lambda, p.log_inv, p.switch_unit,
                    p.switch_rule == 1 ? p.switch_log : L.log_eps, L.n_p, m);
}

// A new lane's thresholds, from its eps_f.
__device__ __forceinline__ void set_eps(LaneCtl& L, double eps_f) {
  L.eps_f = eps_f;
  L.th_async = threshold_up(eps_f);
  const float f = (float)eps_f;
  L.log_eps = f > 1e-30f ? logf(f) : (float)log(eps_f);
}

__device__ __forceinline__ unsigned long long score_key(float score, uint32_t caller_id) {
  return ((unsigned long long)__float_as_uint(fmaxf(score, 0.f)) << 32) |
         (unsigned long long)(0xffffffffu - caller_id);
}

}  // namespace

// One persistent cooperative kernel for both batched queries (SERVE = false:
// n queries packed into tiles, each tile run to completion) and serving steps
// (SERVE = true: every lane of a tile is a slot; NEW slots are admitted into
// tiles already in flight, each live tile advances rounds_per_step rounds,
// slots that finish are finalised and their top-k extracted).
template <int ALGO, bool SERVE>
__global__ void __launch_bounds__(kBThreads, kBMinBlocks)
k_tiles(const __grid_constant__ DevGraph g, const __grid_constant__ BatchParams p,
        const __grid_constant__ ServeParams sv) {
  extern __shared__ __align__(1024) unsigned char smem[];
  // Per-query control of the current tile, one entry per lane / query.  Warp 0
  // of every block makes the decisions (all blocks read the same round
  // accumulators after a barrier, so they agree); the phases read it here.
  __shared__ LaneCtl s_ctl[kTile];
  __shared__ uint32_t s_mdeg[kTile];
  __shared__ int s_switch[kTile];
  __shared__ int s_new[kTile];       // serving: slot admitted at this step
  __shared__ int s_fin[kTile];       // lane finished: finalise and select top-k
  __shared__ uint32_t s_k[kTile];    // top-k size of the lane
  __shared__ int s_pick_d[kTile];    // top-k: digit, keys above it and its count, per lane
  __shared__ uint32_t s_pick_cum[kTile], s_pick_h[kTile];
  __shared__ int s_flag, s_any_switch;
  __shared__ TileBuf s_tb;
  const uint32_t groups = p.groups;
  const uint32_t nbg = gridDim.x / groups;              // blocks per group
  const uint32_t grp = blockIdx.x / nbg;
  if (grp >= groups) return;                            // leftover blocks
  const uint32_t bid = blockIdx.x - grp * nbg;          // block id within the group
  const TileBuf& tb = s_tb;
  BCtx c{g, tb, p, (bid * kBThreads + threadIdx.x) >> 5, (nbg * kBThreads) >> 5,
         bid * kBThreads + threadIdx.x, nbg * kBThreads, threadIdx.x & 31u};
  const uint32_t lane = c.lane;
  const bool lq = lane < (uint32_t)kTile;               // this lane stands for a query
  const bool warp0 = threadIdx.x < 32;
  constexpr bool app = ALGO != kAlgoASRP;  // APP's r_max as eps_f, per-node threshold for the source
  const uint32_t n_work = SERVE ? sv.n_live : (p.n + kTile - 1) / kTile;
  const uint32_t n_split = g.tl.n_split_u, n_acc = g.tl.n_acc;
  const size_t nu32 = (size_t)g.n_u * kTile;
  const uint32_t kmax = p.kmax;
  GridBarrier* bar = p.bars + grp;
  unsigned int epoch = 0;                               // of the group's barrier
  // this warp's items, and its ring with the first units of phase 1 (the graph
  // does not change: no barrier needs to come before the copies)
  __shared__ uint4 s_rg[kBWarps][4];
  __shared__ BlockAcc s_acc;
  const uint4* rg = s_rg[threadIdx.x >> 5];
  if (lane < 4) s_rg[threadIdx.x >> 5][lane] = (lane < 2 ? p.ranges_t : p.ranges_u)[2 * c.gw + (lane & 1u)];
  if (threadIdx.x < kAccFields * 32) s_acc[threadIdx.x >> 5][lane] = 0;
  __syncwarp();
  TileRing ring;
  ring.base = smem_addr(smem) + (threadIdx.x >> 5) * (kTRing * 512u);
  Segments::first(ring, g.tl.t, rg);
  unsigned char* const buf = scratch_of(smem);

  for (uint32_t w = grp; w < n_work; w += groups) {
    const uint32_t tile = SERVE ? sv.live[w] : w;
    const TileBuf* tg = &p.tbufs[SERVE ? tile : grp];
    if (threadIdx.x == 0) s_tb = *tg;
    __syncthreads();
    const uint32_t qi = tile * kTile + lane;            // query (batch) or slot (serve) index
    uint32_t tround = SERVE ? sv.tile_round[tile] : 0u;

    // ---- admission: the initial state of Algorithm 3 (unit residue at the source) for every new lane
    if (!SERVE) {
      for (size_t i = c.gt; i < nu32; i += c.nt) { tb.r_u[i] = 0.f; tb.pi[i] = 0.f; tb.pic[i] = 0.f; }
      for (size_t i = c.gt; i < ((size_t)g.n_v + 2 * n_acc) * kTile; i += c.nt) tb.t[i] = 0.f;
      for (size_t i = c.gt; i < (size_t)n_split * kTile; i += c.nt) tb.split_acc[i] = 0.f;
      for (size_t i = c.gt; i < n_split; i += c.nt) tb.split_cnt[i] = 0;
      for (uint32_t i = c.gt; i < 3 * kAccCopies * kTile; i += c.nt) tb.tacc[i] = TAcc{};
      if (c.gt < 2 * kTile) tb.racc[c.gt] = RAcc{};
    }
    if (warp0) {
      LaneCtl L{0.0, 0, 0, 0, 0, kPhaseAsync, kStatusOk, 0, 0, 0.f, 0.f};
      int is_new = 0;
      uint32_t kk = 0;
      if (!SERVE) {
        const bool in_range = lq && qi < p.n;
        const bool bad = in_range && (p.q[qi] >= g.n_u || !(p.eps[qi] > 0.0));
        if (bad) L.status = kStatusBadArg;
        if (in_range && !bad) {
          set_eps(L, app ? p.eps[qi] / (double)p.e_tot : p.eps[qi] / p.lambda);
          L.active = 1;
          L.valid = 1;
          is_new = 1;
          kk = kmax ? min(min(p.k[qi], kmax), g.n_u) : 0u;
        }
      } else if (lq) {
        const SlotState& S = sv.slots[qi];
        kk = S.k;
        if (S.state == kSlotNew) {
          set_eps(L, S.eps_f);
          L.active = 1;
          L.valid = 1;
          is_new = 1;
        } else if (S.state == kSlotRunning) {
          L = S.ctl;
        }
      }
      if (lq) { s_ctl[lane] = L; s_new[lane] = is_new; s_k[lane] = kk; s_fin[lane] = 0; }
      const int any = __any_sync(kFull, is_new);
      if (lane == 0) s_flag = any;
    }
    __syncthreads();
    if (SERVE && s_flag) {
      // clear the new lanes' columns (the other lanes keep running)
      const bool nw = lq && s_new[lane];
      for (size_t u = c.gw; nw && u < g.n_u; u += c.nw) {
        const size_t i = u * kTile + lane;
        tb.r_u[i] = 0.f; tb.pi[i] = 0.f; tb.pic[i] = 0.f;
      }
      for (size_t j = c.gw; nw && j < 2 * (size_t)n_acc; j += c.nw) tb.t[(g.n_v + j) * kTile + lane] = 0.f;
      if (bid == 0 && nw) {
        for (uint32_t r = 0; r < 3 * kAccCopies; ++r) tb.tacc[r * kTile + lane] = TAcc{};
        for (int r = 0; r < 2; ++r) tb.racc[r * kTile + lane] = RAcc{};
      }
    }
    if (!grid_sync(bar, nbg, epoch)) return;
    if (bid == 0 && warp0 && lq && s_new[lane]) {
      const uint32_t q_new = SERVE ? sv.slots[qi].q_new : p.u_old2new[p.q[qi]];
      const uint32_t cnt = (g.uv_off[q_new + 1] - g.uv_off[q_new]) + (g.ua_off[q_new + 1] - g.ua_off[q_new]);
      const double th = app ? s_ctl[lane].eps_f * (double)cnt : s_ctl[lane].eps_f;
      TAcc* a0 = &tb.tacc[((tround + 2) % 3) * kAccCopies * kTile + lane];
      if (1.0 > th) {
        tb.r_u[(size_t)q_new * kTile + lane] = -1.f;
        a0->marked_deg = (unsigned long long)cnt << 32 | 1u;
      } else {
        tb.r_u[(size_t)q_new * kTile + lane] = 1.f;
      }
    }
    if (!grid_sync(bar, nbg, epoch)) return;

    // ---- rounds (Algorithm 3 / 4) for the active lanes; warp 0 decides, lane by
    // query, in shared memory (registers kept for it would spill in the phases,
    // and after a barrier a spilled register comes back from L2)
    bool wait_fail = false;
    const uint32_t max_r = SERVE ? sv.rounds_per_step : 0xffffffffu;
    uint32_t done_r = 0;
    // before a round: does the tile go on (the marks are in the last round's accumulators)
    auto begin_round = [&](const RoundSums& m) {
      bool act = false;
      if (lq) {
        LaneCtl& L = s_ctl[lane];
        s_mdeg[lane] = m.marked_deg;
        act = L.active;
        if (act && (L.phase == kPhaseDone || m.marked == 0)) { L.phase = kPhaseDone; act = false; s_fin[lane] = 1; }
        if (act && L.rounds >= p.max_rounds) { L.status = kStatusCap; act = false; s_fin[lane] = 1; }
        if (act && done_r < max_r) L.pushes += m.marked;
        L.active = act;
      }
      const int any = __any_sync(kFull, act);
      if (lane == 0) s_flag = any && done_r < max_r;
    };
    auto round_sums = [&](uint32_t r) {
      return lq ? sums_of<ALGO == kAlgoAPPS>(&tb.tacc[(r % 3) * kAccCopies * kTile + lane]) : RoundSums{};
    };
    // after a round: counters, termination and the switch test; whether a lane switches
    auto end_round = [&](const RoundSums& m) {
      bool switched = false;
      if (lq && s_ctl[lane].active) {
        LaneCtl& L = s_ctl[lane];
        const float M = __uint_as_float(m.max_r_bits);
        L.rounds += 1;
        L.n_p += (unsigned long long)s_mdeg[lane] + m.np;
        bool done = false;
        if (ALGO == kAlgoASRP) {
          done = M < L.th_async;                                // M <= eps_f
          switched = !done && L.phase == kPhaseAsync && switch_now(p, L, M);
        } else if (ALGO == kAlgoAPPS) {
          // APP's stopping test; the switch budget in units of APP's thresholds
          const float Mrel = __uint_as_float(m.max_rel_bits);
          done = m.above == 0;
          switched = !done && L.phase == kPhaseAsync && switch_now(p, L, Mrel);
        }
        if (done) {
          L.phase = kPhaseDone;
          L.active = 0;
          s_fin[lane] = 1;
        }
        if (switched) {
          L.phase = kPhaseSync;
          L.switch_round = L.rounds + 1;
        }
      }
      if (lq) s_switch[lane] = switched;
      return __any_sync(kFull, switched);
    };
    if (warp0) begin_round(round_sums(tround + 2));
    __syncthreads();
    while (s_flag) {
      // this block's copy of the round's accumulators; the next round's are cleared
      TAcc* A = &tb.tacc[((tround % 3) * kAccCopies + bid % kAccCopies) * kTile];
      if (bid == 0 && threadIdx.x < kAccCopies * kTile)
        tb.tacc[((tround + 1) % 3) * kAccCopies * kTile + threadIdx.x] = TAcc{};

      const uint32_t set = tround & 1u;                    // accumulated rows of this round
      gphase1(c, s_acc, ring, rg, bar, set, buf);
      Segments::first(ring, g.tl.u, rg + 2);
      if (!grid_sync(bar, nbg, epoch)) { wait_fail = true; break; }
      gphase2<ALGO != kAlgoASRP, ALGO == kAlgoAPPS>(c, s_ctl, s_acc, ring, rg + 2, bar, set, buf);
      flush_round<ALGO == kAlgoAPPS>(s_acc, A);
      Segments::first(ring, g.tl.t, rg);
      if (!grid_sync(bar, nbg, epoch)) { wait_fail = true; break; }
      ++tround;
      ++done_r;
      if (warp0) {
        const RoundSums m = round_sums(tround + 2);
        const bool sw = end_round(m);
        if (lane == 0) s_any_switch = sw;
        if (!sw) begin_round(m);
      }
      __syncthreads();
      if (ALGO != kAlgoAPP && s_any_switch) {
        // first synchronous round pushes every positive residue of that query
        const bool sw = lq && s_switch[lane] != 0;
        uint32_t marked = 0, mdeg = 0;
        for (size_t u = c.gw; sw && u < g.n_u; u += c.nw) {
          const size_t i = u * kTile + lane;
          const float r = tb.r_u[i];
          if (r > 0.f) {
            tb.r_u[i] = -r;
            marked += 1;
            mdeg += g.q1.deg_u[u];
          }
        }
        if (marked) {
          atomicAdd(&s_acc[kAccMarked][lane], marked);
          atomicAdd(&s_acc[kAccDeg][lane], mdeg);
        }
        flush_round<false>(s_acc, A);
        if (!grid_sync(bar, nbg, epoch)) { wait_fail = true; break; }
        if (warp0) begin_round(round_sums(tround + 2));
        __syncthreads();
      }
    }
    if (wait_fail && warp0 && lq && s_ctl[lane].valid) {
      s_ctl[lane].status = kStatusWait;
      s_ctl[lane].active = 0;
      s_fin[lane] = 1;
    }
    __syncthreads();
    const bool fin = lq && s_fin[lane] && s_ctl[lane].valid;
    const uint32_t kq = fin ? s_k[lane] : 0u;
    int any_fin = 0;
    for (int l = 0; l < kTile; ++l) any_fin |= s_fin[l];

    if (any_fin) {
      // ---- reserves = pi - compensation; per-query sums; dense output
      {
        double sum_r = 0.0, sum_p = 0.0;
        float max_r = 0.f;
        for (size_t u = c.gw; fin && u < g.n_u; u += c.nw) {
          const size_t i = u * kTile + lane;
          const float v = fmaxf(tb.pi[i] - tb.pic[i], 0.f);
          tb.pi[i] = v;
          const float r = fabsf(tb.r_u[i]);
          sum_r += (double)r;
          max_r = fmaxf(max_r, r);
          sum_p += (double)v;
          if (!SERVE && p.out_dense) p.out_dense[(size_t)qi * g.n_u + p.u_new2old[u]] = v;
        }
        flush_lane(sum_r, max_r, &tb.racc[0], buf);      // residues
        flush_lane(sum_p, 0.f, &tb.racc[kTile], buf);    // reserves
        for (size_t i = c.gt; i < (size_t)kRadixPasses * kTile * kRadixBins; i += c.nt) tb.hist[i] = 0;
        if (c.gt < kTile) tb.cand_cnt[c.gt] = 0;
      }
      if (!grid_sync(bar, nbg, epoch)) return;

      if (bid == 0 && fin) {
        const LaneCtl L = s_ctl[lane];
        ahpp_stats S;
        S.rounds = L.rounds;
        S.switch_round = L.switch_round;
        S.dense_rounds = L.rounds;
        S.status = (uint32_t)((L.status == kStatusOk && L.phase != kPhaseDone) ? kStatusCap : L.status);
        S.pushes = L.pushes;
        S.n_p = L.n_p;
        S.reserve_sum = __ldcg(&tb.racc[kTile + lane].sum_r);
        S.resid_sum = __ldcg(&tb.racc[lane].sum_r);
        S.mass_err = fabs(S.reserve_sum + S.resid_sum - 1.0);
        S.max_resid = (double)__uint_as_float(__ldcg(&tb.racc[lane].max_r_bits));
        S.lambda = p.lambda;
        S.eps_f = L.eps_f;
        S.served_ms = 0.0;
        if (p.out_stats) p.out_stats[qi] = S;
      }

      // ---- top-k per lane: radix select over 64-bit (score, ~caller id) keys.
      // A lane stops as soon as the bucket holding its k-th key contains
      // exactly the keys it still needs (then every key of that bucket is a
      // winner); with distinct scores that happens once the score bits are
      // resolved, so the caller-id passes are skipped.
      if (kmax) {
        unsigned int* sh = reinterpret_cast<unsigned int*>(buf);    // [kTile][kRadixBins]
        unsigned long long prefix = 0;
        unsigned long long thresh = 0;        // smallest winning key, once known
        uint32_t krem = kq;
        bool known = kq == 0;
        for (int pass = 0; pass < kRadixPasses; ++pass) {
          // every block holds the same per-lane state (read from the same
          // global histograms), so all blocks leave the loop together
          if (!__syncthreads_or(!known)) break;
          const int shift = 64 - kRadixBits * (pass + 1);
          for (int i = threadIdx.x; i < kTile * kRadixBins; i += kBThreads) sh[i] = 0;
          __syncthreads();
          if (!known) {
            for (size_t u = c.gw; u < g.n_u; u += c.nw) {
              const unsigned long long key = score_key(tb.pi[u * kTile + lane], p.u_new2old[u]);
              if (pass == 0 || (key >> (shift + kRadixBits)) == prefix)
                atomicAdd(&sh[lane * kRadixBins + ((key >> shift) & (kRadixBins - 1))], 1u);
            }
          }
          __syncthreads();
          unsigned int* gh = tb.hist + (size_t)pass * kTile * kRadixBins;
          for (int i = threadIdx.x; i < kTile * kRadixBins; i += kBThreads)
            if (sh[i]) atomicAdd(&gh[i], sh[i]);
          if (!grid_sync(bar, nbg, epoch)) return;
          // the merged histograms into shared memory; warp w picks the digit
          // of queries w, w + 8, ... (warp-parallel), lane l reads query l's
          for (int i = threadIdx.x; i < kTile * kRadixBins; i += kBThreads) sh[i] = __ldcg(&gh[i]);
          __syncthreads();
          for (int l = threadIdx.x >> 5; l < kTile; l += kBWarps) {
            const uint32_t kr = __shfl_sync(kFull, krem, l);
            if (__shfl_sync(kFull, (int)known, l)) continue;
            int dd;
            uint32_t cc, hh;
            radix_pick(sh + l * kRadixBins, kRadixBins, kr, &dd, &cc, &hh);
            if ((threadIdx.x & 31) == 0) { s_pick_d[l] = dd; s_pick_cum[l] = cc; s_pick_h[l] = hh; }
          }
          __syncthreads();
          if (!known) {
            const int d = s_pick_d[lane];
            const uint32_t cum = s_pick_cum[lane], h = s_pick_h[lane];
            krem -= cum;
            prefix = (prefix << kRadixBits) | (unsigned long long)d;
            if (h == krem || shift == 0) {
              known = true;
              thresh = prefix << shift;
            }
          }
        }
        // the lane's winners are exactly its keys >= thresh (keys are distinct)
        if (kq) {
          for (size_t u = c.gw; u < g.n_u; u += c.nw) {
            const unsigned long long key = score_key(tb.pi[u * kTile + lane], p.u_new2old[u]);
            if (key >= thresh) {
              const uint32_t pos = atomicAdd(&tb.cand_cnt[lane], 1u);
              if (pos < kmax) tb.cand[(size_t)lane * kmax + pos] = key;
            }
          }
        }
        if (!grid_sync(bar, nbg, epoch)) return;
        // sort each lane's keys descending (bitonic in shared memory), one block per lane
        unsigned long long* sk = reinterpret_cast<unsigned long long*>(buf);
        for (uint32_t l = bid; l < kTile; l += nbg) {
          if (!s_fin[l] || !s_ctl[l].valid) continue;
          const uint32_t ql = tile * kTile + l;
          const uint32_t kl = s_k[l];
          uint32_t m = 1;
          while (m < kl) m <<= 1;
          for (uint32_t i = threadIdx.x; i < m; i += kBThreads)
            sk[i] = i < kl ? tb.cand[(size_t)l * kmax + i] : 0ull;
          __syncthreads();
          for (uint32_t size = 2; size <= m; size <<= 1) {
            for (uint32_t stride = size >> 1; stride > 0; stride >>= 1) {
              for (uint32_t i = threadIdx.x; i < m; i += kBThreads) {
                const uint32_t j = i ^ stride;
                if (j > i) {
                  const bool desc = (i & size) == 0;
                  const unsigned long long a = sk[i], b = sk[j];
                  if (desc ? (a < b) : (a > b)) { sk[i] = b; sk[j] = a; }
                }
              }
              __syncthreads();
            }
          }
          for (uint32_t i = threadIdx.x; i < kl; i += kBThreads) {
            const unsigned long long key = sk[i];
            p.out_nodes[(size_t)ql * kmax + i] = 0xffffffffu - (uint32_t)(key & 0xffffffffu);
            p.out_scores[(size_t)ql * kmax + i] = __uint_as_float((uint32_t)(key >> 32));
          }
          if (threadIdx.x == 0) p.out_n[ql] = kl;
          __syncthreads();
        }
      } else if (bid == 0 && fin && p.out_n) {
        p.out_n[qi] = 0;
      }
    }
    // ---- bad arguments (batch): report and produce no result
    if (!SERVE && bid == 0 && lq && qi < p.n && s_ctl[lane].status == kStatusBadArg) {
      if (p.out_stats) {
        ahpp_stats S{};
        S.status = kStatusBadArg;
        p.out_stats[qi] = S;
      }
      if (p.out_n) p.out_n[qi] = 0;
    }
    // ---- serving: persist the slots' control and the tile's round counter
    if (SERVE && bid == 0 && warp0) {
      if (lq) {
        SlotState& S = sv.slots[qi];
        if (S.state == kSlotNew || S.state == kSlotRunning) {
          S.ctl = s_ctl[lane];
          S.state = s_fin[lane] ? kSlotFinished : kSlotRunning;
        }
      }
      if (lane == 0) sv.tile_round[tile] = tround;
    }
    if (!grid_sync(bar, nbg, epoch)) return;
  }
}

namespace {
template <int ALGO>
const void* tiles_of(bool serve) {
#if AHPP_BT == 32   // serving runs tiles of 32 only
  if (serve) return (const void*)k_tiles<ALGO, true>;
#else
  (void)serve;
#endif
  return (const void*)k_tiles<ALGO, false>;
}
const void* tiles_fn(int algo, bool serve) {
  return algo == kAlgoASRP ? tiles_of<kAlgoASRP>(serve)
                           : algo == kAlgoAPP ? tiles_of<kAlgoAPP>(serve) : tiles_of<kAlgoAPPS>(serve);
}

int launch(bool serve, const DevGraph& g, const BatchParams& p, const ServeParams& sv, int grid, cudaStream_t stream) {
  void* args[] = {(void*)&g, (void*)&p, (void*)&sv};
  const void* fn = tiles_fn(p.algo, serve);
  cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kBatchSmem);
  if (e == cudaSuccess)
    e = cudaLaunchCooperativeKernel(fn, dim3(grid), dim3(kBThreads), args, kBatchSmem, stream);
  return e == cudaSuccess ? 0 : (int)e;
}
}  // namespace

int launch_batch(const DevGraph& g, const BatchParams& p, int grid, cudaStream_t stream) {
  return launch(false, g, p, ServeParams{}, grid, stream);
}

#if AHPP_BT == 32
int launch_serve_step(const DevGraph& g, const BatchParams& p, const ServeParams& sv, int grid, cudaStream_t stream) {
  return launch(true, g, p, sv, grid, stream);
}
#endif

int batch_max_grid(int sm_count) {
  int best = -1;
  for (int i = 0; i < 6; ++i) {
    const void* fn = tiles_fn(i % 3 == 0 ? kAlgoAPP : i % 3 == 1 ? kAlgoASRP : kAlgoAPPS, i >= 3);
    int per_sm = 0;
    if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kBatchSmem) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, kBThreads, kBatchSmem) != cudaSuccess || per_sm <= 0)
      return -1;
    best = best < 0 ? per_sm : std::min(best, per_sm);
  }
  return std::min(best, 1) * sm_count;
}

}  // namespace AHPP_BT_NS
}  // namespace ahpp
