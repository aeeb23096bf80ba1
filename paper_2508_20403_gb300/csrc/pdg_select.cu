// Step A4a: select, per graph, a prefix of the global order (score
// descending, id ascending) that is large enough to contain the first k
// recovered edges.
//
// Why a prefix suffices: by Lemma "share LCA" an edge can only be marked by
// an earlier edge of its own subtask, so whether an edge is recovered depends
// only on the edges ranked before it.  Running the greedy on the prefix
// {score >= t} therefore recovers exactly the edges the full pass recovers
// inside that prefix; if at least k of them survive, the first k are the
// answer, otherwise the prefix is enlarged (step A7 reports a retry).
//
// The threshold comes from a two-level radix select on the score bits
// (12 bits: sign + exponent, then the next 12 mantissa bits); every edge of
// the boundary bucket is kept, so the candidate set is always a prefix.
#include <algorithm>

#include "pdg_internal.cuh"

namespace pdg {

namespace {

constexpr int kSelChunkBlocks = 1024;
constexpr int kHistUnroll = 8;  // keys in flight per thread in the histogram passes

__device__ __forceinline__ int64_t sel_chunk(int64_t E, int nb) {
  int64_t c = (E + nb - 1) / nb;
  return (c + kTile - 1) / kTile * kTile;
}

// Level 1: bins of key >> 52 (the lists of a single graph are counted by the
// scoring kernel itself); 0 marks a tree edge.
__global__ void __launch_bounds__(kBlock) k_sel_hist(const uint64_t* __restrict__ key, int64_t E,
                                                     const int64_t* __restrict__ edge_ptr, int32_t G,
                                                     const GraphSel* __restrict__ sel,
                                                     uint32_t* __restrict__ hist) {
  dep_sync();
  __shared__ uint32_t sh[kSelBins];
  const int64_t chunk = sel_chunk(E, gridDim.x);
  const int64_t b0 = (int64_t)blockIdx.x * chunk;
  const int64_t b1 = min(E, b0 + chunk);
  if (b0 >= b1) return;
  const int32_t g0 = (G == 1) ? 0 : part_of(edge_ptr, G, b0);
  const int32_t g1 = (G == 1) ? 0 : part_of(edge_ptr, G, b1 - 1);
  // one graph at a time: a shared-memory histogram for long ranges, direct
  // global atomics for short ones (many small graphs per chunk)
  for (int32_t g = g0; g <= g1; g++) {
    const int64_t r0 = (G == 1) ? b0 : max(b0, edge_ptr[g]);
    const int64_t r1 = (G == 1) ? b1 : min(b1, edge_ptr[g + 1]);
    const GraphSel s = sel[g];
    if (s.take_all || r0 >= r1) continue;
    uint32_t* hg = hist + (int64_t)g * kSelBins;
    if (r1 - r0 < 256) {  // too short to amortise clearing and flushing 4096 shared bins
      for (int64_t i = r0 + threadIdx.x; i < r1; i += blockDim.x)
        if (key[i]) atomicAdd(&hg[key[i] >> 52], 1u);
      continue;
    }
    for (int i = threadIdx.x; i < kSelBins; i += blockDim.x) sh[i] = 0;
    __syncthreads();
    for (int64_t i0 = r0; i0 < r1; i0 += (int64_t)kBlock * kHistUnroll) {
      uint64_t k[kHistUnroll];
#pragma unroll
      for (int u = 0; u < kHistUnroll; u++) {
        const int64_t i = i0 + u * kBlock + threadIdx.x;
        k[u] = i < r1 ? key[i] : 0;
      }
#pragma unroll
      for (int u = 0; u < kHistUnroll; u++)
        if (k[u]) atomicAdd(&sh[k[u] >> 52], 1u);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < kSelBins; i += blockDim.x)
      if (sh[i]) atomicAdd(&hg[i], sh[i]);
    __syncthreads();
  }
}

// One block per graph: walk the bins from the top until `need` edges are
// covered; clears the histogram for the next level.  Thread t owns the 16
// bins just below the 16 t highest ones.
constexpr int kPickPer = kSelBins / kBlock;
static_assert(kPickPer == 16, "pick layout");

__global__ void __launch_bounds__(kBlock) k_sel_pick(uint32_t* __restrict__ hist, GraphSel* __restrict__ sel,
                                                     const int64_t* __restrict__ off_ptr, int32_t G, int lvl,
                                                     int64_t* __restrict__ count_out, int64_t* __restrict__ ptr) {
  dep_sync();
  __shared__ int64_t sm[kBlock / 32 + 1];
  __shared__ int s_owner;
  const int32_t g = blockIdx.x;
  GraphSel s = sel[g];
  uint32_t* hg = hist + (int64_t)g * kSelBins;
  if (s.take_all) {
    if (threadIdx.x == 0) {
      s.count = off_ptr[g + 1] - off_ptr[g];
      s.thresh = 1;  // every off-tree edge (tree edges have key 0)
      sel[g] = s;
      count_out[g] = s.count;
      if (G == 1) {  // a single graph's offsets need no scan
        ptr[0] = 0;
        ptr[1] = s.count;
      }
    }
    return;
  }
  const int64_t need = (lvl == 0) ? s.want : s.want - s.above1;
  const int lo = kSelBins - kPickPer * (threadIdx.x + 1);  // lowest bin of this thread
  uint32_t c[kPickPer];
  const uint4* h4 = reinterpret_cast<const uint4*>(hg + lo);
#pragma unroll
  for (int q = 0; q < kPickPer / 4; q++) {
    const uint4 x = h4[q];
    c[4 * q] = x.x;
    c[4 * q + 1] = x.y;
    c[4 * q + 2] = x.z;
    c[4 * q + 3] = x.w;
  }
  int64_t mine = 0;
#pragma unroll
  for (int i = 0; i < kPickPer; i++) mine += c[i];
  int64_t tot;
  const int64_t excl = block_excl_scan(mine, sm, &tot);  // counts of the higher bins
  // owner: the first thread whose inclusive sum reaches need, else the last
  if (threadIdx.x == 0) s_owner = kBlock - 1;
  __syncthreads();
  if (excl < need && excl + mine >= need) s_owner = threadIdx.x;  // at most one thread
  if (threadIdx.x == 0 && need <= 0) s_owner = 0;
  __syncthreads();
  if (threadIdx.x == s_owner) {
    int64_t run = excl;  // edges in the bins above `bin`
    int bin = lo;        // lowest bin of the thread if need is never reached
    uint32_t bin_count = c[0];
    bool found = false;
#pragma unroll
    for (int i = kPickPer - 1; i >= 0; i--) {
      if (found) continue;
      if (run + c[i] >= need) {
        bin = lo + i;
        bin_count = c[i];
        found = true;
      } else {
        run += c[i];
      }
    }
    if (lvl == 0) {
      s.b1 = bin;
      s.above1 = run;
      s.count = run + bin_count;
      s.thresh = (uint64_t)bin << 52;
    } else {
      s.b2 = bin;
      s.above2 = run;
      s.count = s.above1 + run + bin_count;
      s.thresh = ((uint64_t)s.b1 << 52) | ((uint64_t)bin << 40);
    }
    s.thresh = max(s.thresh, (uint64_t)1);
    count_out[g] = s.count;
    if (G == 1) {
      ptr[0] = 0;
      ptr[1] = s.count;
    }
    sel[g] = s;
  }
  uint4* w4 = reinterpret_cast<uint4*>(hg + lo);
#pragma unroll
  for (int q = 0; q < kPickPer / 4; q++) w4[q] = make_uint4(0u, 0u, 0u, 0u);
}

// The compaction runs in two steps, so that the m keys are read once (for a
// single graph; before, three times: the second histogram, a counting and a
// writing pass, 380 us of 1.47 ms on R-MAT scale 22).
//
// k_sel_list, over all keys with the level-1 threshold, lists the edges of the
// boundary bucket and above.  Every block takes one tile of keys, keeps the
// tile's edges in id order, and places them as one run wherever the list's end
// is at that moment; the tile's place and length go to a table.  (Placing the
// runs themselves in order by a chained look-back passed 20 tiles per us, half
// the rate at which the keys arrive.)  The second histogram and the exact
// compaction then read that short list, tile by tile in id order.
// Tiles of 8192 keys, two blocks per SM: R-MAT scale 22 (64 M keys) 0.15 ms.
constexpr int kListThreads = 1024;
constexpr int kListWarps = kListThreads / 32;
constexpr int kListPairs = 4;  // pairs of keys per thread
constexpr int kListTile = kListThreads * kListPairs * 2;

struct ListArgs {
  const uint64_t* key;      // by id
  int64_t m;
  const int64_t* edge_ptr;  // graphs' ids
  int32_t G;
  const GraphSel* sel;
  int64_t cap;              // of the list
  int32_t* list_id;
  uint64_t* list_key;
  int2* tile;               // per tile: first entry, entries
};

// the graph of position p, found by one warp with 32-way splits
__device__ __forceinline__ int32_t warp_part_of(const int64_t* __restrict__ ptr, int32_t G, int64_t p) {
  const int lane = threadIdx.x & 31;
  int32_t lo = 0, hi = G;  // ptr[lo] <= p < ptr[hi]
  while (hi - lo > 1) {
    const int32_t step = (hi - lo + 31) / 32, q = lo + lane * step;
    const bool ok = q < hi && ptr[q] <= p;
    const int last = 31 - __clz(__ballot_sync(0xffffffffu, ok));  // lane 0 is always ok
    lo += last * step;
    hi = min(hi, lo + step);
  }
  return lo;
}

__global__ void __launch_bounds__(kListThreads, 2) k_sel_list(ListArgs a, DevScalars* dsc) {
  dep_sync();
  __shared__ int sm[kListThreads / 32 + 1];
  __shared__ uint16_t s_pick[kListTile];
  __shared__ int s_count[kListPairs * kListWarps];
  __shared__ int64_t s_base;
  __shared__ int s_graph;
  const int64_t t0 = (int64_t)blockIdx.x * kListTile;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const unsigned below = (1u << lane) - 1;
  // neighbouring threads read neighbouring pairs of keys
  uint64_t k[2 * kListPairs];
#pragma unroll
  for (int i = 0; i < kListPairs; i++) {
    const int64_t p = t0 + 2 * ((int64_t)i * kListThreads + threadIdx.x);
    if (p + 2 <= a.m) {
      const ulonglong2 x = *reinterpret_cast<const ulonglong2*>(a.key + p);
      k[2 * i] = x.x;
      k[2 * i + 1] = x.y;
    } else {
      k[2 * i] = p < a.m ? a.key[p] : 0;
      k[2 * i + 1] = 0;
    }
  }
  if (a.G > 1) {
    if (wid == 0) {
      const int32_t g = warp_part_of(a.edge_ptr, a.G, t0);
      if (lane == 0) s_graph = g;
    }
    __syncthreads();
  }
  // each thread follows its keys' graphs
  int32_t g = a.G > 1 ? s_graph : 0;
  int64_t g_end = a.G > 1 ? a.edge_ptr[g + 1] : INT64_MAX;
  uint64_t th = a.sel[g].thresh;
  uint32_t pick = 0;
#pragma unroll
  for (int i = 0; i < 2 * kListPairs; i++) {
    const int64_t p = t0 + 2 * ((int64_t)(i / 2) * kListThreads + threadIdx.x) + (i & 1);
    if (p < a.m) {
      while (p >= g_end) {
        g++;
        g_end = a.edge_ptr[g + 1];
        th = a.sel[g].thresh;
      }
      if (k[i] >= th) pick |= 1u << i;
    }
  }
  // offsets in key order: rounds, then warps, then lanes
#pragma unroll
  for (int i = 0; i < kListPairs; i++) {
    const unsigned b0 = __ballot_sync(0xffffffffu, pick >> (2 * i) & 1u);
    const unsigned b1 = __ballot_sync(0xffffffffu, pick >> (2 * i + 1) & 1u);
    if (lane == 0) s_count[i * kListWarps + wid] = __popc(b0) + __popc(b1);
  }
  __syncthreads();
  int tot;
  const int before = block_excl_scan_n<kListThreads>(threadIdx.x < kListPairs * kListWarps ? s_count[threadIdx.x] : 0, sm, &tot);
  if (threadIdx.x < kListPairs * kListWarps) s_count[threadIdx.x] = before;
  if (threadIdx.x == 0) {
    int64_t base = tot ? (int64_t)atomicAdd((unsigned long long*)&dsc->n_list, (unsigned long long)tot) : 0;
    const bool fits = base + tot <= a.cap;
    if (!fits) atomicOr(&dsc->err, ERR_CAPACITY);  // the host grows the list (n_list entries) and repeats
    a.tile[blockIdx.x] = make_int2((int)base, fits ? tot : 0);
    s_base = fits ? base : -1;
  }
  __syncthreads();
  if (s_base < 0 || tot == 0) return;  // uniform
#pragma unroll
  for (int i = 0; i < kListPairs; i++) {
    const bool y0 = pick >> (2 * i) & 1u, y1 = pick >> (2 * i + 1) & 1u;
    const unsigned b0 = __ballot_sync(0xffffffffu, y0), b1 = __ballot_sync(0xffffffffu, y1);
    int at = s_count[i * kListWarps + wid] + __popc(b0 & below) + __popc(b1 & below);
    const int j = 2 * (i * kListThreads + threadIdx.x);
    if (y0) s_pick[at++] = (uint16_t)j;
    if (y1) s_pick[at] = (uint16_t)(j + 1);
  }
  __syncthreads();
  for (int j = threadIdx.x; j < tot; j += kListThreads) {
    const int64_t i = t0 + s_pick[j];
    a.list_id[s_base + j] = (int32_t)i;
    a.list_key[s_base + j] = a.key[i];
  }
}

// Blocks of the list's readers: each takes a run of at most kRunTiles tiles,
// whose entries it numbers through in id order.
constexpr int kRunThreads = 512;
constexpr int kRunTiles = 64;

struct ListRun {
  int first[kRunTiles], start[kRunTiles + 1];
  int graph[kRunTiles];     // of the tile's first id
  int64_t ends[kRunTiles];  // where that graph's ids end
  int entries;
  __device__ __forceinline__ void open(const int2* __restrict__ tile, int64_t tiles, const int64_t* __restrict__ edge_ptr,
                                       int32_t G) {
    const int64_t per = (tiles + gridDim.x - 1) / gridDim.x, b = (int64_t)blockIdx.x * per;
    if (threadIdx.x < 32) {
      const int lane = threadIdx.x;
      int run = 0;
      for (int j0 = 0; j0 < kRunTiles; j0 += 32) {
        const int j = j0 + lane;
        const bool mine = j < per && b + j < tiles;
        const int2 t = mine ? tile[b + j] : make_int2(0, 0);
        const int incl = warp_incl_scan(t.y);
        first[j] = t.x;
        start[j] = run + incl - t.y;
        run += __shfl_sync(0xffffffffu, incl, 31);
        const int64_t id0 = (b + j) * kListTile;
        graph[j] = G > 1 && mine ? part_of(edge_ptr, G, id0) : 0;
        ends[j] = G > 1 && mine ? edge_ptr[graph[j] + 1] : INT64_MAX;
      }
      if (lane == 0) start[kRunTiles] = entries = run;
    }
    __syncthreads();
  }
  // place in the list of the run's entry q, and its tile in the run
  __device__ __forceinline__ int64_t at(int q, int& j) const {
    j = 0;
#pragma unroll
    for (int o = kRunTiles / 2; o; o >>= 1)
      if (start[j + o] <= q) j += o;
    return (int64_t)first[j] + (q - start[j]);
  }
  __device__ __forceinline__ int32_t graph_of(int j, int32_t id, const int64_t* __restrict__ edge_ptr) const {
    int32_t g = graph[j];
    if (id >= ends[j])
      while (id >= edge_ptr[g + 1]) g++;
    return g;
  }
};

struct PickArgs {
  const int2* tile;
  int64_t tiles;
  const int32_t* list_id;
  const uint64_t* list_key;
  const int64_t* edge_ptr;
  int32_t G;
  const GraphSel* sel;
  uint32_t* hist;
  int64_t* block_count;     // selected entries per block
  const int64_t* cand_ptr;
  int64_t cap;              // candidates
  int32_t* cand_idx;
  uint64_t* rkey;
  int32_t* rval;
  const int32_t* u;
  const int32_t* v;
  const int32_t* lca;
  int4* rec;                // [2 R]: u, v, LCA, canonical id; score bits
};

// Level 2: bins of (key >> 40) & 0xfff inside the level-1 bucket of the entry's graph.
__global__ void __launch_bounds__(kRunThreads) k_sel_hist2(PickArgs a) {
  dep_sync();
  __shared__ ListRun run;
  __shared__ uint32_t sh[kSelBins];
  run.open(a.tile, a.tiles, a.edge_ptr, a.G);
  if (a.G == 1) {
    if (run.entries == 0) return;  // uniform
    for (int i = threadIdx.x; i < kSelBins; i += kRunThreads) sh[i] = 0;
    __syncthreads();
  }
  for (int q = threadIdx.x; q < run.entries; q += kRunThreads) {
    int j;
    const int64_t at = run.at(q, j);
    const uint64_t k = a.list_key[at];
    const int32_t g = a.G == 1 ? 0 : run.graph_of(j, a.list_id[at], a.edge_ptr);
    const GraphSel& s = a.sel[g];
    if (s.take_all || (int32_t)(k >> 52) != s.b1) continue;
    if (a.G == 1) atomicAdd(&sh[(k >> 40) & 0xfff], 1u);
    else atomicAdd(&a.hist[(int64_t)g * kSelBins + ((k >> 40) & 0xfff)], 1u);
  }
  if (a.G > 1) return;
  __syncthreads();
  for (int i = threadIdx.x; i < kSelBins; i += kRunThreads)
    if (sh[i]) atomicAdd(&a.hist[i], sh[i]);
}

// The candidates: entries at or above their graph's threshold, in id order.
// A count per block, then a write pass whose blocks add up the counts before
// their own.
template <bool WRITE>
__global__ void __launch_bounds__(kRunThreads) k_sel_pick_list(PickArgs a, DevScalars* dsc) {
  dep_sync();
  __shared__ ListRun run;
  __shared__ int64_t sm[kRunThreads / 32 + 1];
  run.open(a.tile, a.tiles, a.edge_ptr, a.G);
  int64_t base = 0;
  if (WRITE) {
    int64_t c = 0, tot;
    for (int i = threadIdx.x; i < (int)blockIdx.x; i += kRunThreads) c += a.block_count[i];
    block_excl_scan_n<kRunThreads>(c, sm, &base);
    if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) {  // the last block's end is the total
      tot = base + a.block_count[blockIdx.x];
      dsc->n_cand_wanted = tot;
      const bool fits = tot <= a.cap && tot == a.cand_ptr[a.G];
      // nothing downstream may touch more than `cap` candidates: run it empty
      if (!fits) atomicOr(&dsc->err, ERR_CAPACITY);
      dsc->n_cand = fits ? tot : 0;
    }
  }
  int64_t count = 0;
  for (int q0 = 0; q0 < run.entries; q0 += kRunThreads) {
    const int q = q0 + threadIdx.x;
    bool in = false;
    int64_t at = 0;
    uint64_t k = 0;
    if (q < run.entries) {
      int j;
      at = run.at(q, j);
      k = a.list_key[at];
      const int32_t g = a.G == 1 ? 0 : run.graph_of(j, a.list_id[at], a.edge_ptr);
      in = k >= a.sel[g].thresh;
    }
    if (!WRITE) {
      count += in ? 1 : 0;
      continue;
    }
    int64_t tot;
    const int64_t pos = base + block_excl_scan_n<kRunThreads>((int64_t)(in ? 1 : 0), sm, &tot);
    base += tot;
    if (!in || pos >= a.cap) continue;
    const int32_t id = a.list_id[at];
    a.cand_idx[pos] = id;
    a.rkey[pos] = ~k;  // ascending ~score = descending score
    a.rval[pos] = (int32_t)pos;
    // what the later steps read of a candidate, in one sector
    a.rec[2 * pos] = make_int4(__ldg(a.u + id), __ldg(a.v + id), __ldg(a.lca + id), id);
    reinterpret_cast<uint64_t*>(a.rec)[4 * pos + 2] = k - 1;
  }
  if (!WRITE) {
    int64_t tot;
    block_excl_scan_n<kRunThreads>(count, sm, &tot);
    if (threadIdx.x == 0) a.block_count[blockIdx.x] = tot;
  }
}

}  // namespace

int64_t select_tiles(int64_t m) { return std::max<int64_t>(1, (m + kListTile - 1) / kListTile); }

int step_select(Handle& h) {
  bool any_select = false;
  for (int32_t g = 0; g < h.G; g++)
    if (h.want_h[g] < h.off_ptr_h[g + 1] - h.off_ptr_h[g]) any_select = true;
  const int64_t tiles = select_tiles(h.m);
  // at most kRunTiles tiles per block, and enough blocks to fill the device when there are many tiles
  const int64_t runs = std::max<int64_t>((tiles + kRunTiles - 1) / kRunTiles, std::min<int64_t>(tiles, (int64_t)h.num_sms * 4));
  if (tiles > 0x7fffffff || runs > kSelRunsMax) return PDG_E_INVALID_ARG;
  auto pick = [&](int lvl, int64_t* ptr) -> int {
    ++h.launches;
    launch_k(h, k_sel_pick, h.G, kBlock, 0, h.hist, h.sel, h.d_off_ptr, h.G, lvl, h.d_graph_tmp, ptr);
    PDG_CUDA(cudaGetLastError());
    return PDG_OK;
  };
  int st;
  if (any_select && !h.fuse_hist) {
    const int nb = (int)std::max<int64_t>(1, std::min<int64_t>(kSelChunkBlocks, (h.m + kTile - 1) / kTile));
    ++h.launches;
    launch_k(h, k_sel_hist, nb, kBlock, 0, h.key, h.m, h.d_edge_ptr, h.G, h.sel, h.hist);
  }
  if ((st = pick(0, h.d_cand_ptr))) return st;
  ListArgs la{h.key, h.m, h.d_edge_ptr, h.G, h.sel, h.list_cap, h.list_id, h.list_key, static_cast<int2*>(h.list_tile)};
  ++h.launches;
  launch_k(h, k_sel_list, (int)tiles, kListThreads, 0, la, h.dsc);
  PickArgs p{};
  p.tile = la.tile;
  p.tiles = tiles;
  p.list_id = h.list_id;
  p.list_key = h.list_key;
  p.edge_ptr = h.d_edge_ptr;
  p.G = h.G;
  p.sel = h.sel;
  p.hist = h.hist;
  p.block_count = h.blk_a;
  p.cand_ptr = h.d_cand_ptr;
  p.cap = h.Rcap;
  p.cand_idx = h.cand_idx;
  p.rkey = h.rk[0];
  p.rval = h.rv[0];
  p.u = h.el_u;
  p.v = h.el_v;
  p.lca = h.lca;
  p.rec = static_cast<int4*>(h.cand_rec);
  if (any_select) {
    ++h.launches;
    launch_k(h, k_sel_hist2, (int)runs, kRunThreads, 0, p);
    if ((st = pick(1, h.d_cand_ptr))) return st;
  }
  if (h.G > 1 && (st = scan_excl_i64(h, h.d_graph_tmp, h.d_cand_ptr, h.G, nullptr, h.G))) return st;
  ++h.launches;
  launch_k(h, k_sel_pick_list<false>, (int)runs, kRunThreads, 0, p, h.dsc);
  ++h.launches;
  launch_k(h, k_sel_pick_list<true>, (int)runs, kRunThreads, 0, p, h.dsc);
  PDG_CUDA(cudaGetLastError());
  return PDG_OK;
}

}  // namespace pdg
