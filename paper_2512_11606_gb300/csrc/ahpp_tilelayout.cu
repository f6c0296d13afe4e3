// Sliced layout of the batched pull phases (TileLayout), built from a loaded
// graph's adjacency: the host cuts rows into items, a kernel copies the entries
// into place.  Built at load (from arrays and from a graph cache, which does
// not store it) and again when the autotuner tries another chunk size.
#include <algorithm>
#include <vector>

#include "ahpp_host.h"

namespace ahpp {

namespace {

constexpr uint32_t kUnit = 16;             // entries of a row per unit

// Where an item's entries come from: rows row .. row + 3 (a slice), or the
// chunks from `row` on (pieces[]).
struct Piece {
  uint32_t row, first, n;                  // entries [first, first + n) of the row
  uint32_t attr;                           // phase 1: an attribute's row
  uint32_t dest;                           // the row that the chunk's sum goes to
  float at;                                // where in the row the chunk begins, 0 to 1
};

struct HostTiles {
  std::vector<uint4> items;
  std::vector<uint32_t> chunk_row;         // row of each chunk
  std::vector<Piece> pieces;
  uint32_t units = 0, n_chunks = 0;
};

void add_item(HostTiles& h, uint32_t first, uint32_t rows, bool chunk, uint32_t entries) {
  h.items.push_back(make_uint4(first, rows | (chunk ? 1u << 31 : 0u), entries, h.units));
  h.units += (entries + kUnit - 1) / kUnit;
}

// The chunks, four to an item.  They are dealt to `warps` warps in the order of
// where they begin in their rows (rows are sorted by column), so that the warps
// pass over the gathered table together: it is larger than L2 on a large graph,
// and each of its rows is then fetched once a phase instead of several times.
void add_chunks(HostTiles& h, uint32_t warps) {
  std::stable_sort(h.pieces.begin(), h.pieces.end(), [](const Piece& a, const Piece& b) { return a.at < b.at; });
  const uint32_t n = (uint32_t)(h.pieces.size() + 3) / 4;
  // warp w has the items [n w / warps, n (w + 1) / warps): one of each pass
  std::vector<uint32_t> order(n);
  uint32_t next = 0;
  for (uint32_t pass = 0; next < n; ++pass)
    for (uint32_t w = 0; w < warps; ++w) {
      const uint32_t b = (uint32_t)((uint64_t)n * w / warps), e = (uint32_t)((uint64_t)n * (w + 1) / warps);
      if (b + pass < e) order[b + pass] = next++;
    }
  std::vector<Piece> dealt;
  dealt.reserve(h.pieces.size());
  for (uint32_t i = 0; i < n; ++i) {
    const size_t p0 = 4 * (size_t)order[i], p1 = std::min(p0 + 4, h.pieces.size());
    uint32_t len = 0;
    for (size_t p = p0; p < p1; ++p) len = std::max(len, h.pieces[p].n);
    add_item(h, (uint32_t)dealt.size(), (uint32_t)(p1 - p0), true, len);
    dealt.insert(dealt.end(), h.pieces.begin() + p0, h.pieces.begin() + p1);
  }
  h.pieces.swap(dealt);
  for (const Piece& p : h.pieces) h.chunk_row.push_back(p.dest);
  h.n_chunks = n;
}

// Relative cost of a slice, fitted to the blocks' measured times on the medium
// graph: tenths of a gathered row (of t_A, a small table: seven), and the
// item's own latencies in kItemT or kItemU.  They only even out the warps' shares
// (on other graphs the pool does the rest).
constexpr uint32_t kRow = 10, kAttr = 7, kItemT = 75, kItemU = 170;
// Share of the slices' cost that is left in the pool, in percent.
constexpr uint32_t kPoolShare = 20;

// An entry of phase 1: row of V or A over its U neighbours.
struct FromU {
  const uint32_t *vu_off, *vu_idx, *au_off, *au_idx;
  const float *vu_c, *au_pc;
  __device__ uint32_t length(uint32_t row) const { return vu_off[row + 1] - vu_off[row]; }
  __device__ uint32_t cost(uint32_t) const { return kRow; }
  __device__ void get(uint32_t row, uint32_t attr, uint32_t k, uint32_t* i, float* c) const {
    const uint32_t e = (attr ? au_off[row] : vu_off[row]) + k;
    *i = attr ? au_idx[e] : vu_idx[e];
    *c = attr ? au_pc[e] : vu_c[e];
  }
};

// An entry of phase 2: row of U over its V neighbours, then its attributes, by
// their places in the table.
template <typename WA>
struct FromTable {
  const uint32_t *uv_off, *uv_idx, *ua_off, *ua_idx;
  const float* uv_w;
  const WA* ua_w;
  uint32_t n_v, n_split_v;
  __device__ uint32_t length(uint32_t row) const {
    return uv_off[row + 1] - uv_off[row] + ua_off[row + 1] - ua_off[row];
  }
  __device__ uint32_t cost(uint32_t i) const {
    return i < n_v + n_split_v ? kRow : kAttr;
  }
  __device__ void get(uint32_t row, uint32_t, uint32_t k, uint32_t* i, float* c) const {
    const uint32_t b = uv_off[row], dv = uv_off[row + 1] - b;
    if (k < dv) {
      const uint32_t v = uv_idx[b + k];
      *i = v < n_split_v ? n_v + v : v;
      *c = uv_w[b + k];
    } else {
      const uint32_t e = ua_off[row] + (k - dv);
      *i = n_v + n_split_v + ua_idx[e];
      *c = (float)ua_w[e];
    }
  }
};

template <typename SRC>
__global__ void k_fill_tiles(const uint4* items, const Piece* pieces, uint32_t n_items, SRC src,
                             uint32_t item_cost, uint4* units, uint32_t* cost) {
  const uint32_t lane = threadIdx.x & 31, r = lane >> 3, j = ((lane & 7u) + 8u - 2u * r) & 7u;
  for (uint32_t it = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; it < n_items; it += (gridDim.x * blockDim.x) >> 5) {
    const uint4 a = items[it];
    const bool ok = r < (a.y & 0xffu);
    Piece p{a.x + r, 0, 0, 0, 0, 0.f};
    if (ok && (a.y >> 31)) p = pieces[a.x + r];
    else if (ok) p.n = src.length(p.row);
    uint32_t sum = 0;
    for (uint32_t u = 0; u * kUnit < a.z; ++u) {
      uint32_t i[2] = {kNoEntry, kNoEntry};
      float c[2] = {0.f, 0.f};
      for (int e = 0; e < 2; ++e) {
        const uint32_t k = u * kUnit + 2 * j + e;
        if (k < p.n) {
          src.get(p.row, p.attr, p.first + k, &i[e], &c[e]);
          sum += src.cost(i[e]);
        }
      }
      units[((size_t)a.w + u) * 32 + lane] =
          make_uint4(i[0], __float_as_uint(c[0]), i[1], __float_as_uint(c[1]));
    }
    sum = __reduce_add_sync(0xffffffffu, sum);
    if (lane == 0) cost[it] = sum / 4 + item_cost;
  }
}

int build_tile_layout(ahpp_graph* g, TileBuilt* b) {
  const DevGraph& G = g->dg;
  TileLayout& T = b->t;
  // a chunk is walked by one warp: on a small graph the configured size would be
  // more than the warps' shares
  uint32_t fine = 64;
  while (fine < 512 && (uint64_t)fine * 16 * g->bt_grid * kBWarps < (uint64_t)G.n_e + G.n_ea) fine *= 2;
  const uint32_t nU = G.n_u, nV = G.n_v, nA = G.n_a, chunk = std::min(kChunkSizes[T.chunk], fine);
  auto down = [&](std::vector<uint32_t>& v, const uint32_t* p, size_t n) {
    v.resize(n);
    return cudaMemcpy(v.data(), p, 4 * n, cudaMemcpyDeviceToHost) == cudaSuccess;
  };
  std::vector<uint32_t> uv, vu, ua, au;
  if (!down(uv, G.uv_off, (size_t)nU + 1) || !down(vu, G.vu_off, (size_t)nV + 1) ||
      !down(ua, G.ua_off, (size_t)nU + 1) || !down(au, G.au_off, (size_t)nA + 1))
    return cuda_fail(cudaGetLastError(), "batched layout: adjacency");
  auto du = [&](uint32_t u) { return uv[u + 1] - uv[u] + ua[u + 1] - ua[u]; };
  auto dv = [&](uint32_t v) { return vu[v + 1] - vu[v]; };
  auto da = [&](uint32_t a) { return au[a + 1] - au[a]; };
  // rows longer than a chunk are a prefix: rows are sorted by degree
  auto longer = [](uint32_t n, auto d, uint32_t c) {
    uint32_t r = 0;
    while (r < n && d(r) > c) ++r;
    return r;
  };
  const uint32_t nsv = longer(nV, dv, chunk);
  T.n_split_u = longer(nU, du, chunk);
  T.n_acc = nsv + nA;
  T.acc_max = longer(nV, dv, std::min(kChunkSizes[0], fine)) + nA;
  T.split_u_max = longer(nU, du, std::min(kChunkSizes[0], fine));

  HostTiles ht, hu;
  std::vector<uint32_t> chunks_of(T.n_split_u), acc_deg(T.n_acc);
  for (uint32_t j = 0; j < T.n_acc; ++j) {
    const bool attr = j >= nsv;
    const uint32_t row = attr ? j - nsv : j, d = attr ? da(row) : dv(row);
    acc_deg[j] = d;
    for (uint32_t z = 0; z < d; z += chunk) {
      ht.pieces.push_back(Piece{row, z, std::min(chunk, d - z), attr ? 1u : 0u, j, (float)z / (float)d});
    }
  }
  const uint32_t warps = (uint32_t)g->bt_grid * kBWarps;
  add_chunks(ht, warps);
  for (uint32_t v = nsv; v < nV && dv(v); v += 4) add_item(ht, v, std::min(4u, nV - v), false, dv(v));
  for (uint32_t u = 0; u < T.n_split_u; ++u) {
    const uint32_t d = du(u);
    chunks_of[u] = (d + chunk - 1) / chunk;
    for (uint32_t z = 0; z < d; z += chunk) {
      hu.pieces.push_back(Piece{u, z, std::min(chunk, d - z), 0, u, (float)z / (float)d});
    }
  }
  add_chunks(hu, warps);
  for (uint32_t u = T.n_split_u; u < nU; u += 4) add_item(hu, u, std::min(4u, nU - u), false, du(u));

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
  auto rows = [&](HostTiles& h, TileRows& R, int which, uint32_t item_cost, auto src) {
    const uint32_t n = (uint32_t)h.items.size();
    h.items.push_back(make_uint4(0, 0, 0, h.units));
    R.items = (const uint4*)put(h.items);
    R.chunk_row = (const uint32_t*)put(h.chunk_row);
    uint4* units = (uint4*)dev((size_t)h.units * 512, nullptr);
    R.units = units;
    const Piece* pieces = (const Piece*)scratch(h.pieces);
    std::vector<uint32_t> cost(n, 0);
    uint32_t* d_cost = (uint32_t*)scratch(cost);
    if (ok && n) {
      k_fill_tiles<<<grid, threads, 0, g->stream>>>(R.items, pieces, n, src, item_cost, units, d_cost);
      ok = cudaStreamSynchronize(g->stream) == cudaSuccess &&
           cudaMemcpy(cost.data(), d_cost, 4ull * n, cudaMemcpyDeviceToHost) == cudaSuccess;
    }
    TileBuilt::Cost& c = b->cost[which];
    c.n_chunks = h.n_chunks;
    c.unit.clear();
    for (const uint4& x : h.items) c.unit.push_back(x.w);
    c.cost.assign(1, 0);
    for (uint64_t x : cost) c.cost.push_back(c.cost.back() + x);
    // the pool: the last slices (the shortest rows), in grabs of about a 40th of
    // a warp's share
    R.n_items = R.pool = n;
    const uint64_t slices = c.cost[n] - c.cost[h.n_chunks];
    if (n - h.n_chunks >= 4 * warps)       // fewer: a grab would cost more than it evens out
      while (R.pool > h.n_chunks && c.cost[n] - c.cost[R.pool] < slices / 100 * kPoolShare) --R.pool;
    R.batch = std::max(1u, (n - R.pool) / (8 * warps));
  };
  rows(ht, T.t, 0, kItemT, FromU{G.vu_off, G.vu_idx, G.au_off, G.au_idx, G.vu_c, G.au_pc});
  if (g->bf16)
    rows(hu, T.u, 1, kItemU, FromTable<__nv_bfloat16>{G.uv_off, G.uv_idx, G.ua_off, G.ua_idx, G.uv_w,
                                              (const __nv_bfloat16*)G.ua_w, nV, nsv});
  else
    rows(hu, T.u, 1, kItemU, FromTable<float>{G.uv_off, G.uv_idx, G.ua_off, G.ua_idx, G.uv_w, (const float*)G.ua_w, nV, nsv});
  T.acc_deg = (const uint32_t*)put(acc_deg);
  T.chunks_of = (const uint32_t*)put(chunks_of);
  const cudaError_t e = cudaStreamSynchronize(g->stream), le = cudaGetLastError();
  if (e != cudaSuccess || le != cudaSuccess) return cuda_fail(e != cudaSuccess ? e : le, "batched layout");
  if (!ok) { set_error("batched layout: device allocation failed"); return AHPP_ENOMEM; }
  return AHPP_OK;
}

int tile_ranges(TileBuilt* b, uint32_t warps, const uint4** t, const uint4** u) {
  for (const auto& c : b->cuts)
    if (c.warps == warps) { *t = c.r[0]; *u = c.r[1]; return AHPP_OK; }
  GrowInCapture grow;
  std::vector<uint4> r;                    // of phase 1, then of phase 2
  for (int k = 0; k < 2; ++k) {
    // chunks evenly, then the slices before the pool so that every warp's cost is
    // about the same: {chunk begin, end, slice begin, end}, and the first units
    // of those four
    const TileBuilt::Cost& c = b->cost[k];
    const uint32_t n = k ? b->t.u.pool : b->t.t.pool;
    uint32_t i = c.n_chunks;
    uint64_t done = 0;
    for (uint32_t w = 0; w < warps; ++w) {
      const uint32_t c0 = (uint32_t)((uint64_t)c.n_chunks * w / warps), c1 = (uint32_t)((uint64_t)c.n_chunks * (w + 1) / warps);
      const uint32_t i0 = i;
      const uint64_t target = c.cost[n] * (w + 1) / warps;
      done += c.cost[c1] - c.cost[c0];
      for (; i < n; ++i) {
        const uint64_t x = c.cost[i + 1] - c.cost[i];
        if (w + 1 < warps && done + x / 2 >= target) break;
        done += x;
      }
      r.push_back(make_uint4(c0, c1, i0, i));
      r.push_back(make_uint4(c.unit[c0], c.unit[c1], c.unit[i0], c.unit[i]));
    }
  }
  const uint4* d = (const uint4*)b->put(r.size() * sizeof(uint4), r.data());
  if (!d) {
    set_error("batched ranges: device allocation failed");
    return AHPP_ENOMEM;
  }
  b->cuts.push_back(TileBuilt::Cut{warps, {d, d + 2 * warps}});
  *t = d;
  *u = d + 2 * warps;
  return AHPP_OK;
}

}  // namespace

void use_tile_layout(ahpp_graph* g, TileBuilt* b) {
  g->tile_layouts.cur = b;
  g->dg.tl = b->t;
}

int use_tile_layout(ahpp_graph* g, uint32_t choice) {
  Layouts<TileBuilt>& L = g->tile_layouts;
  L.drop();
  for (auto& x : L.all)
    if (x->t.chunk == choice) { use_tile_layout(g, x.get()); return AHPP_OK; }
  std::unique_ptr<TileBuilt> b(new TileBuilt(g));
  b->t.chunk = choice;
  if (int rc = build_tile_layout(g, b.get())) return rc;
  const uint4 *t, *u;
  if (int rc = tile_ranges(b.get(), (uint32_t)g->bt_grid * kBWarps, &t, &u)) return rc;
  L.all.push_back(std::move(b));
  use_tile_layout(g, L.all.back().get());
  return AHPP_OK;
}

int tile_ranges(ahpp_graph* g, uint32_t warps, const uint4** t, const uint4** u) {
  return tile_ranges(g->tile_layouts.cur, warps, t, u);
}

int plan_groups(ahpp_graph* g, uint32_t grid, uint32_t* groups, uint32_t* per_group, BatchParams& p) {
  *per_group = grid / *groups;
  int rc = tile_ranges(g, *per_group * kBWarps, &p.ranges_t, &p.ranges_u);
  if (rc == AHPP_ENOMEM && *groups > 1) {
    *groups = 1;
    *per_group = grid;
    rc = tile_ranges(g, grid * kBWarps, &p.ranges_t, &p.ranges_u);
  }
  p.groups = *groups;
  return rc;
}

uint32_t tile_groups(const ahpp_graph* g, uint32_t n_tiles, bool serving) {
  const uint64_t table = 128ull * ((uint64_t)g->n_u + g->n_v + 2ull * g->dg.tl.n_acc);
  return groups_of(g->batch_groups, n_tiles, std::min<uint32_t>(kMaxGroups, (uint32_t)std::max(1, g->bt_grid)), table,
                   serving);
}

}  // namespace ahpp
