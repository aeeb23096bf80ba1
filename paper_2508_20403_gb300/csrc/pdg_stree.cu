// Spanning-tree generation, the step before recovery (Sec. 2.2: feGRASS
// builds its spanning tree from the effective weight of Eq. weff, then
// recovers off-tree edges against it).
//
// Two trees, both the maximum spanning forest for a strict total order on
// the edges (key descending, canonical edge id ascending), so each is unique:
//   PDG_TREE_MAX_WEIGHT  key = w(e);
//   PDG_TREE_FEGRASS     key = W_eff(e) = fl(fl(w * L) / (d(u) + d(v))) with
//                        L = fl(log(max(deg u, deg v))) and d = unweighted BFS
//                        distance from the maximum-degree vertex (Eq. weff);
//                        the graph must be connected.
// Each tree is rooted at the maximum-degree vertex of its component (ties:
// smaller id) and returned as a parent array.
//
// Forest: Boruvka rounds over the edges that still join two trees.  Every tree
// finds its maximum edge (an atomicMax on the key bits, then an atomicMin on
// the edge id among the edges carrying that key), hooks to the tree across it
// (two trees that chose the same edge: the smaller id stays the root; with a
// strict order no longer cycle exists), and a filter writes the next round's
// list with the new roots.  Rooting: an Euler tour of the forest (arc x->y is
// followed by the arc after y->x in y's tree adjacency, cut at each root),
// ranked; of the two arcs of a tree edge, the earlier one runs from the parent
// to the child.
#include <climits>
#include <cmath>
#include <type_traits>
#include <vector>

#include "pdg_internal.cuh"
#include "pdg_tour.cuh"

namespace pdg {

namespace {

constexpr int32_t kNoEdge = INT_MAX;
constexpr int kStRounds = 40;

__device__ __forceinline__ unsigned long long degree_key(const int64_t* __restrict__ row_ptr, int64_t v) {
  // larger degree first, then smaller id
  return ((unsigned long long)(row_ptr[v + 1] - row_ptr[v]) << 32) | (0xffffffffull - (unsigned long long)v);
}

__global__ void k_st_maxdeg(const int64_t* __restrict__ row_ptr, int64_t n, unsigned long long* best) {
  unsigned long long b = 0;
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x)
    b = max(b, degree_key(row_ptr, v));
  for (int o = 16; o; o >>= 1) b = max(b, __shfl_down_sync(0xffffffffu, b, o));
  if ((threadIdx.x & 31) == 0 && b) atomicMax(best, b);
}

// one BFS level: every vertex at distance `level` labels its unvisited neighbours
__global__ void k_st_bfs(const int64_t* __restrict__ row_ptr, const int32_t* __restrict__ col, int64_t n,
                         int32_t* dist, int32_t level, int32_t* grew) {
  int any = 0;
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x) {
    if (dist[v] != level) continue;
    for (int64_t p = row_ptr[v]; p < row_ptr[v + 1]; p++) {
      const int32_t u = col[p];
      if (dist[u] < 0 && atomicCAS(&dist[u], -1, level + 1) == -1) any = 1;
    }
  }
  if (__any_sync(0xffffffffu, any) && (threadIdx.x & 31) == 0) *grew = 1;
}

// Levels of narrow frontiers in one cluster of 16 blocks, or eight where 16 do
// not fit together.  Every block keeps
// what it discovers in a queue in its shared memory; the next level's vertices
// are the blocks' queues one after another, read across the cluster, eight lanes
// to a vertex.  A cluster barrier ends a level, and the queues' lengths go with
// it.  A level costs the chain of loads from queue, row and neighbours, the
// compare-and-swap and the barrier, 2.0 us on average (with the queue and its length in
// global memory, and the distance looked at before the swap, 3.4 us; a launch
// that looks at every vertex took 6).  It ends where the frontier is empty or
// wider than kBfsNarrow; the distances then say what the frontier is.
constexpr int kBfsThreads = 512, kBfsNarrow = 4096, kBfsLong = 256;

struct BfsState {
  int32_t level, width;
};

__device__ __forceinline__ void cluster_barrier() {
  asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// the address that a block's own shared variable has in block `rank` of the cluster
__device__ __forceinline__ uint32_t cluster_address(const void* own, int rank) {
  uint32_t at;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(at) : "r"((uint32_t)__cvta_generic_to_shared(own)), "r"(rank));
  return at;
}

template <int kBfsCluster>
__global__ void __launch_bounds__(kBfsThreads)
    k_st_bfs_narrow(const int64_t* __restrict__ row_ptr, const int32_t* __restrict__ col, int32_t* dist,
                    const int32_t* __restrict__ first, BfsState* st) {
  __shared__ int32_t s_queue[2][kBfsNarrow];       // of level l: l & 1
  __shared__ int32_t s_count[2][kBfsCluster];      // lengths of all blocks' queues
  __shared__ int32_t s_long[64];
  __shared__ int s_n, s_nlong;
  const int rank = blockIdx.x;  // one cluster
  const int sub = threadIdx.x & 7;
  int level = st->level, width = st->width;
  if (width == 0 || width > kBfsNarrow) return;  // (all blocks)
  {
    const int share = (width + kBfsCluster - 1) / kBfsCluster, p = level & 1;
    if (threadIdx.x < kBfsCluster) s_count[p][threadIdx.x] = max(0, min(share, width - (int)threadIdx.x * share));
    for (int i = threadIdx.x; i < share && rank * share + i < width; i += kBfsThreads)
      s_queue[p][i] = first[rank * share + i];
  }
  __syncthreads();
  cluster_barrier();
  for (;; level++) {
    const int p = level & 1;
    int end[kBfsCluster];  // of the blocks' parts of the frontier
    width = 0;
#pragma unroll
    for (int b = 0; b < kBfsCluster; b++) {
      width += s_count[p][b];
      end[b] = width;
    }
    if (width == 0 || width > kBfsNarrow) break;  // uniform over the cluster
    if (threadIdx.x == 0) s_n = s_nlong = 0;
    __syncthreads();
    auto visit = [&](int32_t u) {
      if (atomicCAS(&dist[u], -1, level + 1) != -1) return;
      const int at = atomicAdd(&s_n, 1);
      if (at < kBfsNarrow) s_queue[p ^ 1][at] = u;  // (a longer queue ends the loop)
    };
    for (int i = (rank * kBfsThreads + (int)threadIdx.x) >> 3; i < width; i += kBfsCluster * kBfsThreads / 8) {
      int b = 0, before = 0;
#pragma unroll
      for (int k = 0; k < kBfsCluster - 1; k++)
        if (i >= end[k]) {
          b = k + 1;
          before = end[k];
        }
      int32_t v;
      asm volatile("ld.shared::cluster.s32 %0, [%1];" : "=r"(v) : "r"(cluster_address(&s_queue[p][i - before], b)) : "memory");
      const int64_t r0 = row_ptr[v], r1 = row_ptr[v + 1];
      if (r1 - r0 > kBfsLong) {  // a long row is shared by the whole block below
        int at = 64;
        if (sub == 0) at = atomicAdd(&s_nlong, 1);
        at = __shfl_sync(0xffu << (threadIdx.x & 24), at, threadIdx.x & 24);  // the eight lanes of this vertex
        if (at < 64) {
          if (sub == 0) s_long[at] = v;
          continue;
        }
      }
      for (int64_t q = r0 + sub; q < r1; q += 8) visit(col[q]);
    }
    __syncthreads();
    for (int k = 0; k < min(s_nlong, 64); k++) {
      const int32_t v = s_long[k];
      for (int64_t q = row_ptr[v] + threadIdx.x; q < row_ptr[v + 1]; q += kBfsThreads) visit(col[q]);
    }
    __syncthreads();
    if (threadIdx.x < kBfsCluster)
      asm volatile("st.shared::cluster.s32 [%0], %1;" ::"r"(cluster_address(&s_count[p ^ 1][rank], threadIdx.x)), "r"(s_n)
                   : "memory");
    cluster_barrier();  // the last access to another block's memory lies before it
  }
  if (rank == 0 && threadIdx.x == 0) {
    st->level = level;
    st->width = width;
  }
}

template <int CLUSTER>
cudaError_t launch_bfs_narrow(const Handle& h, int32_t* dist, const int32_t* first, BfsState* st, cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute at = {};
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = CLUSTER;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cfg.gridDim = dim3(CLUSTER);
  cfg.blockDim = dim3(kBfsThreads);
  cfg.stream = s;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  const int64_t* row_ptr = h.row_ptr;
  const int32_t* col = h.col;
  if (CLUSTER > 8) {  // more than every device takes
    const cudaError_t e =
        cudaFuncSetAttribute(k_st_bfs_narrow<CLUSTER>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
  }
  return cudaLaunchKernelEx(&cfg, k_st_bfs_narrow<CLUSTER>, row_ptr, col, dist, first, st);
}

// the frontier of `level` as a queue, as far as it goes in there (st->width is zero)
__global__ void k_st_bfs_collect(const int32_t* __restrict__ dist, int64_t n, int32_t level, int32_t* __restrict__ queue,
                                 BfsState* st) {
  const int lane = threadIdx.x & 31;
  if (blockIdx.x == 0 && threadIdx.x == 0) st->level = level;
  for (int64_t v0 = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31); v0 < n;
       v0 += (int64_t)gridDim.x * blockDim.x) {  // warp-uniform
    const int64_t v = v0 + lane;
    const bool in = v < n && dist[v] == level;
    const unsigned b = __ballot_sync(0xffffffffu, in);
    if (!b) continue;
    int at = 0;
    if (lane == 0) at = atomicAdd(&st->width, __popc(b));
    at = __shfl_sync(0xffffffffu, at, 0);
    if (in) queue[at + __popc(b & ((1u << lane) - 1))] = (int32_t)v;
  }
}

__global__ void k_st_unreached(const int32_t* __restrict__ dist, int64_t n, int32_t* flag) {
  int any = 0;
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x)
    if (dist[v] < 0) any = 1;
  if (__any_sync(0xffffffffu, any) && (threadIdx.x & 31) == 0) *flag = 1;
}

__global__ void k_st_keys_weight(const double* __restrict__ ew, int64_t m, uint64_t* __restrict__ key) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < m; e += (int64_t)gridDim.x * blockDim.x)
    key[e] = (uint64_t)__double_as_longlong(ew[e]);
}

// W_eff(e) = fl(fl(w * L[max deg]) / (d(u) + d(v))) (Eq. weff); non-negative,
// so its bits order like the value
__global__ void k_st_keys_weff(const int32_t* __restrict__ eu, const int32_t* __restrict__ ev,
                               const double* __restrict__ ew, const int64_t* __restrict__ row_ptr,
                               const int32_t* __restrict__ dist, const double* __restrict__ ltab, int64_t m,
                               uint64_t* __restrict__ key) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < m; e += (int64_t)gridDim.x * blockDim.x) {
    const int32_t u = eu[e], v = ev[e];
    const int64_t du = row_ptr[u + 1] - row_ptr[u], dv = row_ptr[v + 1] - row_ptr[v];
    const double s = (double)((int64_t)dist[u] + (int64_t)dist[v]);  // >= 1: u != v
    const double x = __ddiv_rn(__dmul_rn(ew[e], ltab[max(du, dv)]), s);
    key[e] = (uint64_t)__double_as_longlong(x);
  }
}

// ---- Boruvka over a shrinking list of the edges that still join two trees.
// Every kernel of a round is bound by its random accesses (150 G sectors/s), so
// what counts is how many edges a round touches: on mesh 128^3 (6.2 M edges, 11
// rounds) 1.0 ms; all edges in every round, with the vertices relabelled by
// pointer jumping in between, took 1.4 ms.

// nxt is a union-find forest over the vertices: a tree's root points at itself
__device__ __forceinline__ int32_t st_find(int32_t* nxt, int32_t v) {
  int32_t r = v, p = nxt[r];
  while (p != r) {
    r = p;
    p = nxt[r];
  }
  if (nxt[v] != r) nxt[v] = r;  // a shorter path for the next search; an ancestor either way
  return r;
}

__global__ void k_st_start(int32_t* __restrict__ nxt, unsigned long long* __restrict__ bk, int32_t* __restrict__ bid,
                           int64_t n, int64_t* __restrict__ counts, int64_t m) {
  if (blockIdx.x == 0 && threadIdx.x <= kStRounds) counts[threadIdx.x] = threadIdx.x == 0 ? m : 0;
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x) {
    nxt[v] = (int32_t)v;
    bk[v] = 0;
    bid[v] = kNoEdge;
  }
}

// the edges of a round: the trees at their ends, key, canonical id (null: the place in the list)
struct StEdges {
  const int32_t* u;
  const int32_t* v;
  const uint64_t* key;
  const int32_t* id;
  const int64_t* count;
  __device__ __forceinline__ int32_t id_of(int64_t i) const { return id ? id[i] : (int32_t)i; }
};

__global__ void k_st_best_key(StEdges e, unsigned long long* bk) {
  const int64_t m = *e.count;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < m; i += (int64_t)gridDim.x * blockDim.x) {
    const int32_t u = e.u[i], v = e.v[i];
    const unsigned long long k = e.key[i];
    if (k > bk[u]) atomicMax(&bk[u], k);
    if (k > bk[v]) atomicMax(&bk[v], k);
  }
}

__global__ void k_st_best_id(StEdges e, const unsigned long long* __restrict__ bk, int32_t* bid) {
  const int64_t m = *e.count;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < m; i += (int64_t)gridDim.x * blockDim.x) {
    const int32_t u = e.u[i], v = e.v[i];
    const unsigned long long k = e.key[i];
    if (k == bk[u]) atomicMin(&bid[u], e.id_of(i));
    if (k == bk[v]) atomicMin(&bid[v], e.id_of(i));
  }
}

// Every tree hooks across its chosen edge, which joins the forest; of two trees
// that chose the same edge the smaller id stays a root (a strict order allows
// no longer cycle).  A tree's edge is one entry of the list, so that entry does
// the hooking.
__global__ void k_st_hook(StEdges e, const int32_t* __restrict__ bid, int32_t* __restrict__ nxt,
                          uint8_t* __restrict__ tflag) {
  const int64_t m = *e.count;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < m; i += (int64_t)gridDim.x * blockDim.x) {
    const int32_t u = e.u[i], v = e.v[i], id = e.id_of(i);
    const bool bu = bid[u] == id, bv = bid[v] == id;
    if (!bu && !bv) continue;
    tflag[id] = 1;
    if (bu && !(bv && u < v)) nxt[u] = v;
    if (bv && !(bu && v < u)) nxt[v] = u;
  }
}

// Every vertex points at its root, and the roots' choices are reset (worth a pass while the edges outnumber the
// vertices: each of an edge's two searches is then one load, and it writes nothing at random).
__global__ void k_st_compress(int32_t* nxt, int64_t n, unsigned long long* __restrict__ bk, int32_t* __restrict__ bid) {
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x)
    if (st_find(nxt, (int32_t)v) == (int32_t)v) {
      bk[v] = 0;
      bid[v] = kNoEdge;
    }
}

// The edges that still join two trees, with those trees' roots; without a
// k_st_compress before it, the roots' choices are reset here (roots without
// such an edge take no part any more).  A block's survivors are one run of the
// next list.
__global__ void __launch_bounds__(kBlock) k_st_filter(StEdges e, int32_t* nxt, int32_t* __restrict__ ou,
                                                      int32_t* __restrict__ ov, uint64_t* __restrict__ okey,
                                                      int32_t* __restrict__ oid, int64_t* count,
                                                      bool reset, unsigned long long* __restrict__ bk,
                                                      int32_t* __restrict__ bid) {
  __shared__ int sm[kBlock / 32 + 1];
  __shared__ unsigned long long s_base;
  const int64_t m = *e.count;
  constexpr int kPer = 4;
  for (int64_t i0 = (int64_t)blockIdx.x * kBlock * kPer; i0 < m; i0 += (int64_t)gridDim.x * kBlock * kPer) {
    int32_t u[kPer], v[kPer];
    int mine = 0;
#pragma unroll
    for (int k = 0; k < kPer; k++) {
      const int64_t i = i0 + k * kBlock + threadIdx.x;
      u[k] = v[k] = -1;
      if (i < m) {
        const int32_t a = st_find(nxt, e.u[i]), b = st_find(nxt, e.v[i]);
        if (a != b) {
          u[k] = a;
          v[k] = b;
          mine++;
          if (reset) {
            bk[a] = 0;
            bk[b] = 0;
            bid[a] = kNoEdge;
            bid[b] = kNoEdge;
          }
        }
      }
    }
    int tot;
    int at = block_excl_scan(mine, sm, &tot);
    if (threadIdx.x == 0) s_base = tot ? atomicAdd((unsigned long long*)count, (unsigned long long)tot) : 0;
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kPer; k++) {
      if (u[k] < 0) continue;
      const int64_t i = i0 + k * kBlock + threadIdx.x, o = (int64_t)s_base + at++;
      ou[o] = u[k];
      ov[o] = v[k];
      okey[o] = e.key[i];
      oid[o] = e.id_of(i);
    }
    __syncthreads();
  }
}

// the root of every vertex's tree, and its vertex of maximum degree: a thread keeps the maximum while the tree stays
// the same, and a block whose threads all end in one tree makes one addition to its word (mesh 128^3, one tree: 24 us;
// an addition per vertex, all to that word, took 1340)
__global__ void __launch_bounds__(kBlock) k_st_comp_root(const int64_t* __restrict__ row_ptr, int32_t* nxt,
                                                         int32_t* __restrict__ comp, int64_t n, unsigned long long* rk) {
  __shared__ unsigned long long s_best;
  __shared__ int32_t s_comp;
  __shared__ int s_mixed;
  int32_t cur = -1;
  unsigned long long best = 0;
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x) {
    const int32_t c = st_find(nxt, (int32_t)v);
    comp[v] = c;
    if (c != cur) {
      if (cur >= 0) atomicMax(&rk[cur], best);
      cur = c;
      best = 0;
    }
    best = max(best, degree_key(row_ptr, v));
  }
  if (threadIdx.x == 0) {
    s_best = 0;
    s_comp = cur;
    s_mixed = 0;
  }
  __syncthreads();
  if (cur >= 0 && cur != s_comp) s_mixed = 1;
  __syncthreads();
  if (s_mixed) {
    if (cur >= 0) atomicMax(&rk[cur], best);
    return;
  }
  for (int o = 16; o; o >>= 1) best = max(best, __shfl_down_sync(0xffffffffu, best, o));
  if ((threadIdx.x & 31) == 0) atomicMax(&s_best, best);
  __syncthreads();
  if (threadIdx.x == 0 && s_comp >= 0) atomicMax(&rk[s_comp], s_best);
}

__device__ __forceinline__ bool is_root(const int32_t* __restrict__ comp, const unsigned long long* __restrict__ rk,
                                        int64_t v) {
  return (0xffffffffull - (rk[comp[v]] & 0xffffffffull)) == (unsigned long long)v;
}

// the tour of a component ends with the arc into its root that precedes the
// root's first arc
__global__ void k_st_cut(const int32_t* __restrict__ comp, const unsigned long long* __restrict__ rk,
                         const int64_t* __restrict__ tptr, const int32_t* __restrict__ tdeg,
                         const int32_t* __restrict__ rev, int64_t n, int32_t* __restrict__ succ, RankSpace r) {
  for (int64_t v0 = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31); v0 < n;
       v0 += (int64_t)gridDim.x * blockDim.x) {  // warp-uniform
    const int64_t v = v0 + (threadIdx.x & 31);
    const bool root = v < n && tdeg[v] > 0 && is_root(comp, rk, v);
    if (root) succ[rev[tptr[v] + tdeg[v] - 1]] = -1;
    rank_add_head(root, root ? (int32_t)tptr[v] : 0, r.heads, r.n_heads);
  }
}

// of the two arcs of a tree edge the earlier (farther from the end) leads
// from the parent to the child
__global__ void k_st_parent(const int32_t* __restrict__ eu, const int32_t* __restrict__ ev,
                            const uint8_t* __restrict__ tflag, const int32_t* __restrict__ arc_uv,
                            const int32_t* __restrict__ rev, const uint64_t* __restrict__ own,
                            const uint64_t* __restrict__ walk, int64_t m, int32_t* __restrict__ parent) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < m; e += (int64_t)gridDim.x * blockDim.x) {
    if (!tflag[e]) continue;
    const int32_t a = arc_uv[e];
    if (arc_rank(own, walk, a) > arc_rank(own, walk, rev[a])) parent[ev[e]] = eu[e];
    else parent[eu[e]] = ev[e];
  }
}

}  // namespace

// a failed CUDA call releases the temporaries and reports PDG_E_CUDA
#define ST_CK(x)                                   \
  do {                                             \
    if ((x) != cudaSuccess) return fail(PDG_E_CUDA); \
  } while (0)

int spanning_tree(Handle& h, int tree_kind, int32_t* parent) {
  const int64_t n = h.n, m = h.m;
  const int gn = grid_for(h, n), gm = grid_for(h, std::max<int64_t>(m, 1));
  cudaStream_t s = h.stream;
  std::vector<void*> temps;
  auto cleanup = [&]() {
    for (void* p : temps) cudaFreeAsync(p, s);
    temps.clear();
  };
  auto talloc = [&](auto** p, int64_t count) -> bool {
    void* q = nullptr;
    if (cudaMallocAsync(&q, sizeof(**p) * (size_t)std::max<int64_t>(count, 1), s) != cudaSuccess) return false;
    temps.push_back(q);
    *p = static_cast<std::remove_reference_t<decltype(*p)>>(q);
    return true;
  };
  uint64_t* key = nullptr;
  int32_t *comp = nullptr, *nxt = nullptr, *bid = nullptr, *dist = nullptr, *tdeg = nullptr, *cur = nullptr;
  int32_t *tadj = nullptr, *rev = nullptr, *arc_uv = nullptr, *succ = nullptr, *flags = nullptr;
  int32_t *lu[2] = {nullptr, nullptr}, *lv[2] = {nullptr, nullptr}, *lid[2] = {nullptr, nullptr};
  uint64_t* lkey[2] = {nullptr, nullptr};
  int64_t* counts = nullptr;
  BfsState* bfs = nullptr;
  RankSpace rank;
  unsigned long long *bk = nullptr, *rk = nullptr;
  uint8_t* tflag = nullptr;
  int64_t* tptr = nullptr;
  double* ltab = nullptr;
  const int64_t A = 2 * std::max<int64_t>(n - 1, 0);  // arcs of a spanning forest, at most
  if (!talloc(&key, m) || !talloc(&comp, n) || !talloc(&nxt, n) || !talloc(&bid, n) || !talloc(&bk, n) ||
      !talloc(&rk, n) || !talloc(&tflag, m) || !talloc(&tdeg, n) || !talloc(&cur, n) || !talloc(&tptr, n + 1) ||
      !talloc(&tadj, A) || !talloc(&rev, A) || !talloc(&arc_uv, m) || !talloc(&succ, A) ||
      !rank_space(rank, A, std::max<int64_t>(n / 2, 1), s, talloc) || !talloc(&flags, 64) ||
      !talloc(&counts, kStRounds + 1) || !talloc(&lu[0], m) || !talloc(&lv[0], m) || !talloc(&lid[0], m) ||
      !talloc(&lkey[0], m) || !talloc(&lu[1], m) || !talloc(&lv[1], m) || !talloc(&lid[1], m) || !talloc(&lkey[1], m) ||
      (tree_kind == PDG_TREE_FEGRASS && (!talloc(&dist, n) || !talloc(&bfs, 1)))) {
    cudaGetLastError();
    cleanup();
    return PDG_E_OOM;
  }
  int32_t* hflags = reinterpret_cast<int32_t*>(h.hsc);  // pinned staging of the flags (the scalars are not in use)
  auto read_flags = [&](int count) -> bool {
    return cudaMemcpyAsync(hflags, flags, sizeof(int32_t) * count, cudaMemcpyDeviceToHost, s) == cudaSuccess &&
           cudaStreamSynchronize(s) == cudaSuccess;
  };
  int st = PDG_OK;
  auto fail = [&](int code) {
    cudaGetLastError();
    cleanup();
    return code;
  };
  // 1. edge keys
  if (tree_kind == PDG_TREE_FEGRASS) {
    unsigned long long* best = rk;  // scratch
    ST_CK(cudaMemsetAsync(best, 0, sizeof(unsigned long long), s));
    k_st_maxdeg<<<gn, kBlock, 0, s>>>(h.row_ptr, n, best);
    unsigned long long bh = 0;
    if (cudaMemcpyAsync(&bh, best, sizeof(bh), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
        cudaStreamSynchronize(s) != cudaSuccess)
      return fail(PDG_E_CUDA);
    const int32_t root = (int32_t)(0xffffffffull - (bh & 0xffffffffull));
    const int64_t maxdeg = (int64_t)(bh >> 32);
    // unweighted BFS distances from the root: narrow frontiers in one kernel, wide ones level by level over all
    // vertices, 16 levels per host check
    ST_CK(cudaMemsetAsync(dist, 0xff, sizeof(int32_t) * n, s));
    ST_CK(cudaMemsetAsync(dist + root, 0, sizeof(int32_t), s));
    BfsState* hst = reinterpret_cast<BfsState*>(h.hsc);
    bool done = false;
    int32_t level = 0;
    while (!done) {
      if (level > n) return fail(PDG_E_CUDA);
      ST_CK(cudaMemsetAsync(bfs, 0, sizeof(BfsState), s));
      k_st_bfs_collect<<<gn, kBlock, 0, s>>>(dist, n, level, nxt, bfs);
      if (launch_bfs_narrow<16>(h, dist, nxt, bfs, s) != cudaSuccess) {
        cudaGetLastError();
        ST_CK(launch_bfs_narrow<8>(h, dist, nxt, bfs, s));
      }
      if (cudaMemcpyAsync(hst, bfs, sizeof(BfsState), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
          cudaStreamSynchronize(s) != cudaSuccess)
        return fail(PDG_E_CUDA);
      level = hst->level;
      if (hst->width == 0) break;
      ST_CK(cudaMemsetAsync(flags, 0, sizeof(int32_t) * 16, s));
      for (int i = 0; i < 16; i++) k_st_bfs<<<gn, kBlock, 0, s>>>(h.row_ptr, h.col, n, dist, level + i, flags + i);
      if (!read_flags(16)) return fail(PDG_E_CUDA);
      done = hflags[15] == 0;
      level += 16;
    }
    ST_CK(cudaMemsetAsync(flags, 0, sizeof(int32_t), s));
    k_st_unreached<<<gn, kBlock, 0, s>>>(dist, n, flags);
    if (!read_flags(1)) return fail(PDG_E_CUDA);
    if (hflags[0]) return fail(PDG_E_INVALID_ARG);  // not connected
    // log of the degrees, from the host math library (one table, both sides of every comparison)
    std::vector<double> lh((size_t)maxdeg + 1, 0.0);
    for (int64_t d = 1; d <= maxdeg; d++) lh[d] = std::log((double)d);
    if (!talloc(&ltab, maxdeg + 1)) return fail(PDG_E_OOM);
    ST_CK(cudaMemcpyAsync(ltab, lh.data(), sizeof(double) * lh.size(), cudaMemcpyHostToDevice, s));
    k_st_keys_weff<<<gm, kBlock, 0, s>>>(h.el_u, h.el_v, h.el_w, h.row_ptr, dist, ltab, m, key);
    if (cudaStreamSynchronize(s) != cudaSuccess) return fail(PDG_E_CUDA);  // the host table is released below
  } else {
    k_st_keys_weight<<<gm, kBlock, 0, s>>>(h.el_w, m, key);
  }
  // 2. Boruvka rounds; the host looks at the number of edges left every few rounds
  k_st_start<<<gn, kBlock, 0, s>>>(nxt, bk, bid, n, counts, m);
  ST_CK(cudaMemsetAsync(tflag, 0, (size_t)std::max<int64_t>(m, 1), s));
  int64_t left = m;
  for (int round = 0; left > 0; round++) {
    if (round >= kStRounds) return fail(PDG_E_CUDA);  // every round at least halves the trees
    const int i = round & 1;
    const StEdges e = round == 0 ? StEdges{h.el_u, h.el_v, key, nullptr, counts}
                                 : StEdges{lu[i], lv[i], lkey[i], lid[i], counts + round};
    const int gl = grid_for(h, left);
    k_st_best_key<<<gl, kBlock, 0, s>>>(e, bk);
    k_st_best_id<<<gl, kBlock, 0, s>>>(e, bk, bid);
    k_st_hook<<<gl, kBlock, 0, s>>>(e, bid, nxt, tflag);
    const bool pass = left > n / 2;
    if (pass) k_st_compress<<<gn, kBlock, 0, s>>>(nxt, n, bk, bid);
    k_st_filter<<<gl, kBlock, 0, s>>>(e, nxt, lu[i ^ 1], lv[i ^ 1], lkey[i ^ 1], lid[i ^ 1], counts + round + 1, !pass, bk,
                                      bid);
    if (round < 2 || round % 3 == 1) {
      if (cudaMemcpyAsync(h.hsc, counts + round + 1, sizeof(int64_t), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
          cudaStreamSynchronize(s) != cudaSuccess)
        return fail(PDG_E_CUDA);
      left = *reinterpret_cast<int64_t*>(h.hsc);
    }
  }
  // 3. roots, tree adjacency, Euler tour
  ST_CK(cudaMemsetAsync(rk, 0, sizeof(unsigned long long) * n, s));
  k_st_comp_root<<<std::min(gn, h.num_sms * 4), kBlock, 0, s>>>(h.row_ptr, nxt, comp, n, rk);
  ST_CK(cudaMemsetAsync(tdeg, 0, sizeof(int32_t) * n, s));
  ST_CK(cudaMemsetAsync(cur, 0, sizeof(int32_t) * n, s));
  k_st_tdeg<<<gm, kBlock, 0, s>>>(h.el_u, h.el_v, tflag, m, tdeg);
  if ((st = ensure_scan_status(h, n)) || (st = scan_excl_i32(h, tdeg, tptr, n, nullptr, n))) return fail(st);
  {  // a forest has at most n - 1 edges: the arc arrays are sized for that
    int64_t arcs = 0;
    if (cudaMemcpyAsync(&arcs, tptr + n, sizeof(int64_t), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
        cudaStreamSynchronize(s) != cudaSuccess)
      return fail(PDG_E_CUDA);
    if (arcs < 0 || arcs > A) return fail(PDG_E_CUDA);
  }
  k_st_fill<<<gm, kBlock, 0, s>>>(h.el_u, h.el_v, tflag, m, tptr, cur, tadj, rev, arc_uv);
  const int ga = grid_for(h, std::max<int64_t>(A, 1));
  k_st_succ<<<ga, kBlock, 0, s>>>(tadj, rev, tptr, tdeg, n, succ);
  k_st_cut<<<gn, kBlock, 0, s>>>(comp, rk, tptr, tdeg, rev, n, succ, rank);
  const uint64_t* walk = rank_lists(h, succ, tptr + n, rank, s);
  ST_CK(cudaMemsetAsync(parent, 0xff, sizeof(int32_t) * n, s));
  k_st_parent<<<gm, kBlock, 0, s>>>(h.el_u, h.el_v, tflag, arc_uv, rev, rank.own, walk, m, parent);
  if (cudaGetLastError() != cudaSuccess) return fail(PDG_E_CUDA);
  cleanup();
  return PDG_OK;
}

#undef ST_CK

}  // namespace pdg
