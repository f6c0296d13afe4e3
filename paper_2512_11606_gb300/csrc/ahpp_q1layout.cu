// Sliced layout of the single-query pull phases (Q1Layout), built from a
// loaded graph's adjacency: the host cuts rows into items and balances them
// over the warps of the grid, kernels copy the entries into place.  Built at
// load (both from arrays and from a graph cache, which does not store it) and
// again when the autotuner tries another lane width.
#include <algorithm>
#include <thread>
#include <vector>

#include "ahpp_host.h"

namespace ahpp {

namespace {

constexpr uint32_t kStep = 128;            // entries per step (four per lane)
constexpr uint32_t kLaneStepsMax = 8;      // steps of a slice's rows before vw doubles, at most
constexpr uint32_t kSegMax = 1024;         // entries per attribute segment
constexpr uint32_t kSegWindow = 512;       // segments sorted by length together
constexpr uint32_t kTaEntries = 16000;     // entries of t_A in shared memory
constexpr uint32_t kOwnRows = 16000;       // rows of a block of the attribute hop (64 KB of residues)
constexpr uint32_t kTableFloats = (kQ1SmemMax - kQ1RingBytes) / 4;   // shared memory after the warps' rings

uint32_t steps_of(uint32_t len, uint32_t lg) { return (len + (4u << lg) - 1) >> (2 + lg); }

// Lanes per row (log2) for rows of lv + la entries: at least lg_min, more
// until a lane walks at most lane_steps steps.
uint32_t lanes_of(uint32_t lv, uint32_t la, uint32_t lg_min, uint32_t lane_steps) {
  uint32_t lg = lg_min;
  while (lg < 5 && steps_of(lv, lg) + steps_of(la, lg) > lane_steps) ++lg;
  return lg;
}

// An item before its units have a place (see Q1Rows).
struct Item {
  uint32_t row, rows, lg, split, v_steps, a_steps, slot;
  uint32_t v_first, a_first;               // first V and A entry (local) of a chunk
};

struct HostRows {
  std::vector<Item> items;
  std::vector<uint32_t> chunks_of;         // chunks of each split row
  uint32_t n_chunks = 0;                   // leading items that are chunks
};

// Items of rows [0, n) with lv(r) V entries and la(r) A entries, longest
// first.  Rows of more than 2 chunk_steps steps at 32 lanes are split into
// chunks of chunk_steps (the first max_split of them).
template <typename LV, typename LA>
HostRows make_rows(uint32_t n, LV lv, LA la, uint32_t lg_min, uint32_t lane_steps, uint32_t chunk_steps,
                   uint32_t max_split) {
  HostRows h;
  uint32_t r = 0;
  for (; r < n && r < max_split; ++r) {    // a prefix: rows are sorted by degree
    const uint32_t sv = steps_of(lv(r), 5), sa = steps_of(la(r), 5);
    if (sv + sa <= 2 * chunk_steps) break;
    const uint32_t nch = (sv + sa + chunk_steps - 1) / chunk_steps;
    for (uint32_t c = 0; c < nch; ++c) {
      const uint32_t b = c * chunk_steps, e = std::min(b + chunk_steps, sv + sa);
      const uint32_t v0 = std::min(b, sv), v1 = std::min(e, sv), a0 = std::max(b, sv) - sv, a1 = std::max(e, sv) - sv;
      h.items.push_back(Item{r, 1, 5, 1, v1 - v0, a1 - a0, r, v0 * kStep, a0 * kStep});
    }
    h.chunks_of.push_back(nch);
  }
  h.n_chunks = (uint32_t)h.items.size();
  while (r < n) {
    const uint32_t lg = lanes_of(lv(r), la(r), lg_min, lane_steps), rows = std::min(32u >> lg, n - r);
    Item it{r, rows, lg, 0, 0, 0, 0, 0, 0};
    for (uint32_t i = 0; i < rows; ++i) {
      it.v_steps = std::max(it.v_steps, steps_of(lv(r + i), lg));
      it.a_steps = std::max(it.a_steps, steps_of(la(r + i), lg));
    }
    h.items.push_back(it);
    r += rows;
  }
  return h;
}

// Cycles of an SM that an item takes, fitted to the blocks' measured times: its
// reduction and epilogue, a V step's stream and lookups in shared memory, an
// attribute step's, the L1 lines that lookups outside shared memory touch (two
// cycles each), and a chunk's combination.
uint64_t cost_of(const Item& it, uint32_t lines) {
  return 10 + 25ull * it.v_steps + 20ull * it.a_steps + 2ull * lines + (it.split ? 50 : 0);
}

// What a row space's items become on the device.
struct Cut {
  std::vector<uint4> items;                // in the order of the warps that own them
  std::vector<uint2> place;                // first unit, first V entry; chunks only: first A entry in `a_first`
  std::vector<uint32_t> a_first;
  std::vector<uint4> ranges;
  uint32_t units = 0;
};

// Deals the chunk items evenly to the warps, cuts the slices so that every
// warp's total cost is about the same, and gives the items and their units
// places in the order in which the warps use them.
Cut cut_rows(const HostRows& h, const std::vector<uint32_t>& lines, uint32_t a_units, uint32_t n_warps) {
  Cut c;
  const uint32_t n = (uint32_t)h.items.size();
  std::vector<uint64_t> cost(n);
  uint64_t total = 0, done = 0;            // done: cost handed out to warps <= w
  for (uint32_t i = 0; i < n; ++i) total += cost[i] = cost_of(h.items[i], lines[i]);
  auto put = [&](uint32_t i) {
    const Item& it = h.items[i];
    c.items.push_back(make_uint4(it.row, it.rows | it.lg << 8 | it.split << 31, it.v_steps, it.a_steps));
    c.place.push_back(make_uint2(c.units, it.v_first));
    c.a_first.push_back(it.a_first);
    c.units += 2 * it.v_steps + a_units * it.a_steps;
    done += cost[i];
  };
  uint32_t s = h.n_chunks;
  for (uint32_t w = 0; w < n_warps; ++w) {
    const uint32_t i0 = (uint32_t)c.items.size(), u0 = c.units;
    for (uint64_t k = (uint64_t)h.n_chunks * w / n_warps; k < (uint64_t)h.n_chunks * (w + 1) / n_warps; ++k) put((uint32_t)k);
    const uint64_t target = total * (w + 1) / n_warps;
    while (s < n && (w + 1 == n_warps || done + cost[s] / 2 < target)) put(s++);
    c.ranges.push_back(make_uint4(i0, (uint32_t)c.items.size(), u0, c.units));
  }
  return c;
}

// ---- kernels: one warp per item

// Lane's part of a step: entries k..k+3 of a row (zero past len).
__device__ __forceinline__ void put_step(uint4* units, size_t unit, uint32_t lane, bool compact, const uint32_t* i,
                                         const float* c) {
  uint4* p = units + unit * 32 + lane;
  if (compact) {
    auto bf = [&](int e) { return __float_as_uint(c[e]) >> 16; };       // weights are bfloat16 values
    *p = make_uint4(i[0] | i[1] << 16, i[2] | i[3] << 16, bf(0) | bf(1) << 16, bf(2) | bf(3) << 16);
  } else {
    p[0] = make_uint4(i[0], i[1], i[2], i[3]);
    p[32] = make_uint4(__float_as_uint(c[0]), __float_as_uint(c[1]), __float_as_uint(c[2]), __float_as_uint(c[3]));
  }
}

// L1 lines that the warp's lookups i past the first `hub` entries touch.
__device__ __forceinline__ uint32_t count_lines(uint32_t i, bool valid, uint32_t hub) {
  const bool cold = valid && i >= hub;
  const uint32_t peers = __match_any_sync(0xffffffffu, cold ? i >> 5 : 0xffffffffu);
  return __popc(__ballot_sync(0xffffffffu, cold && __ffs(peers) - 1 == (int)(threadIdx.x & 31)));
}

__global__ void k_count_lines(const Item* items, uint32_t n_items, const uint32_t* off, const uint32_t* idx,
                              uint32_t hub, uint32_t* lines) {
  const uint32_t lane = threadIdx.x & 31, nw = (gridDim.x * blockDim.x) >> 5;
  for (uint32_t it = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; it < n_items; it += nw) {
    const Item a = items[it];
    const uint32_t r = lane >> a.lg, sub = lane & ((1u << a.lg) - 1u);
    const uint32_t base = r < a.rows ? off[a.row + r] : 0u, len = r < a.rows ? off[a.row + r + 1] - base : 0u;
    uint32_t n = 0;
    for (uint32_t j = 0; j < a.v_steps; ++j)
      for (uint32_t e = 0; e < 4; ++e) {
        const uint32_t k = a.v_first + (((j << a.lg) + sub) << 2) + e;
        n += count_lines(k < len ? idx[base + k] : 0u, k < len, hub);
      }
    if (lane == 0) lines[it] = n;
  }
}

template <typename WA>
__global__ void k_fill_rows(const uint4* items, const uint2* place, const uint32_t* a_first, uint32_t n_items,
                            const uint32_t* off, const uint32_t* idx, const float* co, const uint32_t* a_off,
                            const uint32_t* a_idx, const WA* a_w, bool compact, uint4* units) {
  const uint32_t lane = threadIdx.x & 31, nw = (gridDim.x * blockDim.x) >> 5;
  for (uint32_t it = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; it < n_items; it += nw) {
    const uint4 a = items[it];
    const uint2 at = place[it];
    const uint32_t lg = (a.y >> 8) & 7u, r = lane >> lg, sub = lane & ((1u << lg) - 1u);
    const bool ok = r < (a.y & 0xffu);
    size_t unit = at.x;
    uint32_t i4[4];
    float c4[4];
    const uint32_t base = ok ? off[a.x + r] : 0u, len = ok ? off[a.x + r + 1] - base : 0u;
    for (uint32_t j = 0; j < a.z; ++j, unit += 2) {
      for (uint32_t e = 0; e < 4; ++e) {
        const uint32_t k = at.y + (((j << lg) + sub) << 2) + e;
        i4[e] = k < len ? idx[base + k] : 0u;
        c4[e] = k < len ? co[base + k] : 0.f;
      }
      put_step(units, unit, lane, false, i4, c4);
    }
    if (a.w == 0) continue;
    const uint32_t ab = ok ? a_off[a.x + r] : 0u, an = ok ? a_off[a.x + r + 1] - ab : 0u;
    for (uint32_t j = 0; j < a.w; ++j, unit += compact ? 1 : 2) {
      for (uint32_t e = 0; e < 4; ++e) {
        const uint32_t k = a_first[it] + (((j << lg) + sub) << 2) + e;
        i4[e] = k < an ? a_idx[ab + k] : 0u;
        c4[e] = k < an ? (float)a_w[ab + k] : 0.f;
      }
      put_step(units, unit, lane, compact, i4, c4);
    }
  }
}

// segs[s] = {attribute, first entry (in A->U order), entries, first row of the block}
template <typename WA>
__global__ void k_fill_segs(const uint4* items, uint32_t n_items, const uint4* segs, const uint32_t* au_idx,
                            const WA* au_w, bool compact, uint4* units) {
  const uint32_t lane = threadIdx.x & 31, nw = (gridDim.x * blockDim.x) >> 5;
  for (uint32_t it = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; it < n_items; it += nw) {
    const uint4 a = items[it];
    const uint32_t lg = (a.y >> 8) & 7u, r = lane >> lg, sub = lane & ((1u << lg) - 1u);
    const bool ok = r < (a.y & 0xffu);
    const uint4 sg = ok ? segs[a.x + r] : make_uint4(0, 0, 0, 0);
    for (uint32_t j = 0; j < a.w; ++j) {
      uint32_t i4[4];
      float c4[4];
      for (uint32_t e = 0; e < 4; ++e) {
        const uint32_t k = (((j << lg) + sub) << 2) + e;
        i4[e] = k < sg.z ? au_idx[sg.y + k] - sg.w : 0u;
        c4[e] = k < sg.z ? (float)au_w[sg.y + k] : 0.f;
      }
      put_step(units, (size_t)a.z + (size_t)j * (compact ? 1 : 2), lane, compact, i4, c4);
    }
  }
}

// Segment s's place in t_A's copies and the scale of its sum (k_attr / W_col).
__global__ void k_seg_meta(const uint4* segs, uint32_t n, const float* cnorm_a, uint32_t n_a, float k_attr,
                           uint2* meta) {
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
    meta[i] = make_uint2(segs[i].x, __float_as_uint(k_attr * cnorm_a[segs[i].x % n_a]));
}

__global__ void k_diff(const uint32_t* off, uint32_t n, const uint32_t* off2, uint32_t* out) {
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
    out[i] = off[i + 1] - off[i] + (off2 ? off2[i + 1] - off2[i] : 0u);
}

template <typename F>
void over_threads(uint32_t n, F fn) {
  const unsigned hw = std::thread::hardware_concurrency();
  const uint32_t nt = std::max(1u, std::min({hw ? hw : 1u, 32u, n}));
  run_threads(nt, [&](unsigned t) { for (uint32_t i = t; i < n; i += nt) fn(i); });
}

// A block of U rows of the attribute hop.
struct Block {
  std::vector<uint4> segs, items;          // {attribute, first entry, entries, first row}; items
  std::vector<uint4> ranges;               // {item begin, end, unit begin, end} per warp
  uint32_t units = 0;
};

// Segments of rows [r0, r1), sorted by length in windows of consecutive
// attributes: a slice's rows are about equally long, and its sums still go to
// nearby attributes.
Block make_block(uint32_t b, uint32_t r0, uint32_t r1, const std::vector<uint32_t>& au, const std::vector<uint32_t>& au_idx,
                 uint32_t s_units) {
  Block B;
  for (uint32_t a = 0; a + 1 < au.size(); ++a) {
    const uint32_t* s = au_idx.data() + au[a];
    const uint32_t* t = au_idx.data() + au[a + 1];
    const uint32_t* p = std::lower_bound(s, t, r0);
    const uint32_t* q = std::lower_bound(p, t, r1);
    for (; p < q; p += std::min<size_t>(kSegMax, q - p))
      B.segs.push_back(make_uint4(a, (uint32_t)(p - au_idx.data()), (uint32_t)std::min<size_t>(kSegMax, q - p), r0));
  }
  const uint32_t n = (uint32_t)B.segs.size();
  for (uint32_t i = 0; i < n; i += kSegWindow)
    std::stable_sort(B.segs.begin() + i, B.segs.begin() + std::min(n, i + kSegWindow),
                     [](const uint4& x, const uint4& y) { return x.z > y.z; });
  // each block starts with another window: blocks that walked the attributes in
  // step would all reduce into the same lines at the same time (medium graph:
  // 21.15 ms a query against 20.58, mean over six placements in memory)
  const uint32_t windows = (n + kSegWindow - 1) / kSegWindow;
  if (windows) std::rotate(B.segs.begin(), B.segs.begin() + (size_t)(b % windows) * kSegWindow, B.segs.end());
  uint32_t lg_min = 0;                     // enough items for the block's warps
  while (lg_min < 5 && ((uint64_t)n << lg_min) / 32 < kQ1Warps) ++lg_min;
  uint64_t total = 0, done = 0;
  for (uint32_t i = 0; i < n;) {
    const uint32_t lg = lanes_of(0, B.segs[i].z, lg_min, kLaneStepsMax), rows = std::min(32u >> lg, n - i);
    uint32_t k = 0;
    for (uint32_t j = 0; j < rows; ++j) k = std::max(k, steps_of(B.segs[i + j].z, lg));
    B.items.push_back(make_uint4(i, rows | lg << 8, B.units, k));
    B.units += s_units * k;
    total += 2 + k;
    i += rows;
  }
  uint32_t it = 0;
  for (uint32_t w = 0; w < (uint32_t)kQ1Warps; ++w) {
    const uint32_t i0 = it;
    const uint64_t target = total * (w + 1) / kQ1Warps;
    while (it < B.items.size() && (w + 1 == (uint32_t)kQ1Warps || done + (2 + B.items[it].w) / 2 < target))
      done += 2 + B.items[it++].w;
    auto unit = [&](uint32_t i) { return i < B.items.size() ? B.items[i].z : B.units; };
    B.ranges.push_back(make_uint4(i0, it, unit(i0), unit(it)));
  }
  return B;
}

// Blocks of the grid and lanes per short row.
void shape_of(const ahpp_graph* g, uint32_t vec_width, uint32_t* grid, uint32_t* lanes) {
  const DevGraph& G = g->dg;
  // the barrier costs the same from 8 blocks on, so a step of phase 2 is dealt to
  // every fourth warp at least
  const uint64_t steps = ((uint64_t)G.n_e + G.n_ea) / kStep + 1;
  const uint32_t nb = (uint32_t)std::min<uint64_t>(g->q1_max_blocks, std::max<uint64_t>(8, 4 * steps / kQ1Warps));
  // lanes per short row: one (16,000 nodes: 1.77 ms a query with eight lanes, 1.69
  // with one; 44,000: 2.62, 1.70; 100,000: 2.94, 2.64), unless that leaves the
  // warps a long slice of U rows or two each (200,000 nodes of 40 entries: 5.35 with
  // one, 4.89 with two; 277,000 of 36: 10.0, 9.28).  Past either line one lane is
  // faster or as fast (ms with one and two lanes; nodes, entries a node: 140,000 of
  // 34: 3.12, 3.36; 311,000 of 34: 6.59, 6.98; 374,000 of 40: 9.01, 9.10; 176,000 of
  // 22: 3.86, 4.85; 171,000 of 28: 3.26, 3.85; 288,000 of 28: 5.44, 6.12), between
  // them it is one or the other within 3 %, graph by graph (171,000 of 34: 4.17,
  // 4.05; 233,000 of 34: 5.57, 5.68; 288,000 of 34: 6.29, 6.20)
  const uint64_t slices = G.n_u / 32, warps = (uint64_t)nb * kQ1Warps;
  const bool uneven = slices > warps && 10 * slices < 19 * warps;
  *grid = nb;
  *lanes = vec_width ? vec_width : uneven && (uint64_t)G.n_e + G.n_ea >= 30ull * G.n_u ? 2 : 1;
}

int build_q1_layout(ahpp_graph* g, Q1Built* b) {
  const DevGraph& G = g->dg;
  Q1Layout& Q = b->q;
  const uint32_t nU = G.n_u, nV = G.n_v, nA = G.n_a;
  auto down = [&](std::vector<uint32_t>& v, const uint32_t* p, size_t n) {
    v.resize(n);
    return n == 0 || cudaMemcpy(v.data(), p, 4 * n, cudaMemcpyDeviceToHost) == cudaSuccess;
  };
  std::vector<uint32_t> uv, vu, ua, au, au_idx;
  if (!down(uv, G.uv_off, (size_t)nU + 1) || !down(vu, G.vu_off, (size_t)nV + 1) ||
      !down(ua, G.ua_off, (size_t)nU + 1) || !down(au, G.au_off, (size_t)nA + 1) || !down(au_idx, G.au_idx, G.n_ea))
    return cuda_fail(cudaGetLastError(), "single-query layout: adjacency");
  auto lv = [&](uint32_t u) { return uv[u + 1] - uv[u]; };
  auto la = [&](uint32_t u) { return ua[u + 1] - ua[u]; };
  auto lw = [&](uint32_t v) { return vu[v + 1] - vu[v]; };
  auto none = [](uint32_t) { return 0u; };
  g->n_long_u = 0;
  while (g->n_long_u < nU && lv(g->n_long_u) + la(g->n_long_u) > 2048) ++g->n_long_u;
  Q.compact_a = g->bf16 && nA <= 65536;
  Q.compact_s = g->bf16;
  const uint32_t a_units = Q.compact_a ? 1 : 2, s_units = Q.compact_s ? 1 : 2;

  const uint32_t nb = b->grid;
  Q.n_warps = nb * kQ1Warps;
  uint32_t lg_min = 0;
  while ((1u << lg_min) < b->vw) ++lg_min;
  // a lane's walk of a V row: at most half the steps a warp has in the phase, so
  // that the warps' shares can be cut evenly (2M edges: phase 1 from 38,000 to
  // 35,000 cycles); U items and segments, with more to do at their ends, are
  // faster long (12,000 against 10,000 cycles, and 6,000 against 11,000)
  const uint32_t v_steps = (uint32_t)std::min<uint64_t>(
      kLaneStepsMax, std::max<uint64_t>(1, (uint64_t)G.n_e / kStep / Q.n_warps / 2));

  // blocks of U rows of the attribute hop, cut by entries (and rows: each has
  // a residue to load), a multiple of the grid unless rows run out
  std::vector<uint2> vb;
  {
    const uint64_t most = std::max<uint64_t>(1, ((uint64_t)nU + (uint64_t)nb * kOwnRows - 1) / ((uint64_t)nb * kOwnRows));
    const uint64_t want = nb * most;
    uint64_t left = (uint64_t)G.n_ea + nU;
    for (uint32_t r = 0; G.n_ea && r < nU;) {
      const uint64_t blocks = want > vb.size() ? want - vb.size() : 1, target = (left + blocks - 1) / blocks;
      uint64_t c = 0;
      const uint32_t r0 = r;
      while (r < nU && r - r0 < kOwnRows && (c == 0 || c + la(r) + 1 <= target + target / 64)) c += la(r++) + 1;
      left -= c;
      vb.push_back(make_uint2(r0, r - r0));
    }
  }
  const uint32_t n_vb = (uint32_t)vb.size();
  uint32_t own = 0;
  for (const uint2& x : vb) own = std::max(own, x.y);

  // shared memory: t_A first (every U row looks it up), then the leading
  // entries of t_V and p that are looked up often enough by each SM to repay
  // their copy (a copied entry costs 1/16 cycle, a lookup it saves about 3/4)
  const uint32_t least = std::max(1u, nb / 12);
  auto leading = [&](uint32_t n, auto len) {
    uint32_t h = 0;
    for (uint32_t i = 0; i < n; ++i) h += len(i) >= least;
    return h;
  };
  Q.s.own_cap = (own + 3) / 4 * 4;
  Q.hub_u = std::min(leading(nU, lv), kTableFloats - Q.s.own_cap) / 4 * 4;
  Q.hub_a = std::min(nA, kTaEntries);
  Q.hub_v = std::min(leading(nV, lw), kTableFloats - (Q.hub_a + 3) / 4 * 4) / 4 * 4;
  b->smem = kQ1RingBytes + 4 * std::max(Q.s.own_cap + Q.hub_u, (Q.hub_a + 3) / 4 * 4 + Q.hub_v);

  HostRows hv, hu;
  run_threads(2, [&](unsigned t) {
    if (t) hu = make_rows(nU, lv, la, lg_min, kLaneStepsMax, kLaneStepsMax, nU);
    else hv = make_rows(nV, lw, none, lg_min, v_steps, v_steps, Q.hub_v);   // split rows' sums are read from shared memory
  });
  std::vector<Block> blk(n_vb);
  over_threads(n_vb, [&](uint32_t i) {
    blk[i] = make_block(i, vb[i].x, vb[i].x + vb[i].y, au, au_idx, s_units);
  });
  // copies of t_A: at least 16 blocks to a copy (with 39 blocks, eight copies to
  // add up in phase 2 cost 4 % of the query), and few enough attributes that all
  // copies fit in 32 KB and t_A is looked up in shared memory only
  Q.ta_copies = std::max(1u, std::min({kTaCopies, 8192u / std::max(nA, 1u), n_vb / 16}));
  std::vector<uint4> segs, sitems, sranges;
  uint32_t total_s = 0;
  for (uint32_t k = 0; k < n_vb; ++k) {
    const uint32_t s0 = (uint32_t)segs.size(), i0 = (uint32_t)sitems.size();
    for (auto x : blk[k].segs) { x.x += k % Q.ta_copies * nA; segs.push_back(x); }
    for (auto x : blk[k].items) { x.x += s0; x.z += total_s; sitems.push_back(x); }
    for (auto& x : blk[k].ranges) sranges.push_back(make_uint4(x.x + i0, x.y + i0, x.z + total_s, x.w + total_s));
    total_s += blk[k].units;
    blk[k] = Block();
  }

  // ---- device arrays
  bool ok = true;
  auto dev = [&](size_t bytes, const void* src) -> void* {
    void* p = b->put(bytes, src);
    ok = ok && p;
    return p;
  };
  auto put = [&](auto& v) -> void* { return dev(v.size() * sizeof(v[0]), v.data()); };
  ScratchBufs tmp;
  auto scratch = [&](auto& v) -> void* {
    void* p = nullptr;
    const size_t n = v.size() * sizeof(v[0]);
    if (g->dev_malloc(&p, std::max<size_t>(n, 16)) != cudaSuccess) { cudaGetLastError(); ok = false; return nullptr; }
    tmp.bufs.push_back(p);
    if (upload(g, p, v.data(), n) != cudaSuccess) ok = false;
    return p;
  };
  const int grid = std::max(1, 8 * g->sm_count), threads = 256;
  auto rows = [&](HostRows& h, Q1Rows& R, const uint32_t* off, const uint32_t* idx, const float* co, uint32_t hub) {
    const uint32_t n = (uint32_t)h.items.size();
    std::vector<uint32_t> lines(n, 0);
    if (n) {
      const Item* items = (const Item*)scratch(h.items);
      uint32_t* d_lines = (uint32_t*)scratch(lines);
      if (!ok) return;
      k_count_lines<<<grid, threads, 0, g->stream>>>(items, n, off, idx, hub, d_lines);
      ok = cudaStreamSynchronize(g->stream) == cudaSuccess &&
           cudaMemcpy(lines.data(), d_lines, 4ull * n, cudaMemcpyDeviceToHost) == cudaSuccess;
    }
    Cut c = cut_rows(h, lines, a_units, Q.n_warps);
    const uint2* place = (const uint2*)scratch(c.place);
    const uint32_t* a_first = (const uint32_t*)scratch(c.a_first);
    R.items = (const uint4*)put(c.items);
    R.ranges = (const uint4*)put(c.ranges);
    R.chunks_of = (const uint32_t*)put(h.chunks_of);
    R.n_split = (uint32_t)h.chunks_of.size();
    uint4* units = (uint4*)dev((size_t)c.units * 512, nullptr);
    R.units = units;
    if (!ok || n == 0) return;
    if (g->bf16)
      k_fill_rows<<<grid, threads, 0, g->stream>>>(R.items, place, a_first, n, off, idx, co, G.ua_off, G.ua_idx,
                                                   (const __nv_bfloat16*)G.ua_w, Q.compact_a != 0, units);
    else
      k_fill_rows<<<grid, threads, 0, g->stream>>>(R.items, place, a_first, n, off, idx, co, G.ua_off, G.ua_idx,
                                                   (const float*)G.ua_w, Q.compact_a != 0, units);
  };
  rows(hv, Q.v, G.vu_off, G.vu_idx, G.vu_c, Q.hub_u);
  if (ok) rows(hu, Q.u, G.uv_off, G.uv_idx, G.uv_w, Q.hub_v);
  if (ok) {
    const uint32_t n_items = (uint32_t)sitems.size();
    const uint4* sg = (const uint4*)scratch(segs);
    Q.s.items = (const uint4*)put(sitems);
    Q.s.ranges = (const uint4*)put(sranges);
    Q.s.vb = (const uint2*)put(vb);
    uint2* meta = (uint2*)dev(segs.size() * sizeof(uint2), nullptr);
    Q.s.meta = meta;
    Q.s.n_vb = n_vb;
    uint4* units = (uint4*)dev((size_t)total_s * 512, nullptr);
    Q.s.units = units;
    if (ok && n_items) {
      k_seg_meta<<<grid, threads, 0, g->stream>>>(sg, (uint32_t)segs.size(), G.cnorm_a, nA, G.k_attr, meta);
      if (g->bf16)
        k_fill_segs<<<grid, threads, 0, g->stream>>>(Q.s.items, n_items, sg, G.au_idx, (const __nv_bfloat16*)G.au_w,
                                                     true, units);
      else
        k_fill_segs<<<grid, threads, 0, g->stream>>>(Q.s.items, n_items, sg, G.au_idx, (const float*)G.au_w, false,
                                                     units);
    }
  }
  uint32_t* du = (uint32_t*)dev(4ull * nU, nullptr);
  uint32_t* dv = (uint32_t*)dev(4ull * nV, nullptr);
  uint32_t* da = (uint32_t*)dev(4ull * nA, nullptr);
  if (ok) {
    k_diff<<<grid, threads, 0, g->stream>>>(G.uv_off, nU, G.ua_off, du);
    if (nV) k_diff<<<grid, threads, 0, g->stream>>>(G.vu_off, nV, nullptr, dv);
    if (nA) k_diff<<<grid, threads, 0, g->stream>>>(G.au_off, nA, nullptr, da);
  }
  Q.deg_u = du;
  Q.deg_v = dv;
  Q.deg_a = da;
  const cudaError_t e = cudaStreamSynchronize(g->stream);
  const cudaError_t le = cudaGetLastError();
  if (e != cudaSuccess || le != cudaSuccess) return cuda_fail(e != cudaSuccess ? e : le, "single-query layout");
  if (!ok) { set_error("single-query layout: device allocation failed"); return AHPP_ENOMEM; }
  return AHPP_OK;
}

}  // namespace

void use_q1_layout(ahpp_graph* g, Q1Built* b) {
  g->q1_layouts.cur = b;
  g->dg.q1 = b->q;
}

int use_q1_layout(ahpp_graph* g, uint32_t vec_width) {
  Layouts<Q1Built>& L = g->q1_layouts;
  L.drop();
  std::unique_ptr<Q1Built> b(new Q1Built(g));
  shape_of(g, vec_width, &b->grid, &b->vw);
  for (auto& x : L.all)
    if (x->vw == b->vw) { use_q1_layout(g, x.get()); return AHPP_OK; }
  if (int rc = build_q1_layout(g, b.get())) return rc;
  L.all.push_back(std::move(b));
  use_q1_layout(g, L.all.back().get());
  return AHPP_OK;
}

}  // namespace ahpp
