// Euler tours of a forest given by tree-edge flags over the canonical edge
// list: tree adjacency (both arcs of every tree edge, each knowing its
// reverse), the tour successor, and list ranking.  Shared by the tree layout,
// spanning-tree generation (rooting) and the PCG quality measure (tree solves
// as prefix sums over the tour).  After x->y the tour takes the arc following
// y->x in y's adjacency row (cyclically); cutting the tour of a component at
// its root gives a list whose ranks order the arcs.
#pragma once

#include <algorithm>

#include "pdg_internal.cuh"

namespace pdg {

namespace {

__global__ void k_st_tdeg(const int32_t* __restrict__ eu, const int32_t* __restrict__ ev,
                          const uint8_t* __restrict__ tflag, int64_t m, int32_t* tdeg) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < m; e += (int64_t)gridDim.x * blockDim.x) {
    if (!tflag[e]) continue;
    atomicAdd(&tdeg[eu[e]], 1);
    atomicAdd(&tdeg[ev[e]], 1);
  }
}

// tree adjacency: both arcs of every tree edge, each knowing its reverse
__global__ void k_st_fill(const int32_t* __restrict__ eu, const int32_t* __restrict__ ev,
                          const uint8_t* __restrict__ tflag, int64_t m, const int64_t* __restrict__ tptr, int32_t* cur,
                          int32_t* __restrict__ tadj, int32_t* __restrict__ rev, int32_t* __restrict__ arc_uv) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < m; e += (int64_t)gridDim.x * blockDim.x) {
    if (!tflag[e]) continue;
    const int32_t u = eu[e], v = ev[e];
    const int32_t pu = (int32_t)(tptr[u] + atomicAdd(&cur[u], 1));
    const int32_t pv = (int32_t)(tptr[v] + atomicAdd(&cur[v], 1));
    tadj[pu] = v;
    tadj[pv] = u;
    rev[pu] = pv;
    rev[pv] = pu;
    arc_uv[e] = pu;
  }
}

// Euler tour successor: after x->y comes the arc following y->x in y's row
// (cyclically)
__global__ void k_st_succ(const int32_t* __restrict__ tadj, const int32_t* __restrict__ rev,
                          const int64_t* __restrict__ tptr, const int32_t* __restrict__ tdeg, int64_t n,
                          int32_t* __restrict__ succ) {
  const int64_t A = tptr[n];
  for (int64_t a = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; a < A; a += (int64_t)gridDim.x * blockDim.x) {
    const int32_t y = tadj[a];
    const int64_t base = tptr[y];
    const int64_t next = rev[a] - base + 1;
    succ[a] = (int32_t)(base + (next == tdeg[y] ? 0 : next));
  }
}

// List ranking by splitters.  One arc of every eight, chosen by a hash of their
// index so that no order of the arcs makes long gaps likely, starts a walk to
// the next chosen arc (about eight steps; the longest of A / 8 walks about
// eight times its logarithm), noting on every arc on the way the walk and the
// step; pointer jumping then ranks the walks, an eighth of the list, and an
// arc's rank follows from its walk's.  On the 4.2 M arcs of mesh 128^3 this is
// 130 us; pointer jumping over all arcs took 22 rounds, 600 us.
// The first arc of a list need not be chosen: the cuts list those in `heads`.
// A tour that no root cut has no end: its walks never reach one, and arcs that
// no walk visits keep the all-ones word.
struct RankSpace {
  uint64_t* own = nullptr;      // [A] per arc: walk << 32 | step
  uint64_t* walk[2] = {nullptr, nullptr};  // per walk: next walk (-1: the list ends) << 32 | arcs
  int32_t* heads = nullptr;     // first arcs of the lists that no group chose
  int32_t* n_heads = nullptr;
  int64_t groups = 0, max_heads = 0;
};

__device__ __forceinline__ int64_t rank_chosen(int64_t group) { return 8 * group + (int64_t)(mix64((uint64_t)group) & 7); }

// (warp-uniform call) lists the head arcs of the lanes with `pred`
__device__ __forceinline__ void rank_add_head(bool pred, int32_t arc, int32_t* heads, int32_t* n_heads) {
  pred = pred && rank_chosen(arc >> 3) != arc;
  const unsigned b = __ballot_sync(0xffffffffu, pred);
  if (!b) return;
  const int lane = threadIdx.x & 31;
  int at = 0;
  if (lane == 0) at = atomicAdd(n_heads, __popc(b));
  at = __shfl_sync(0xffffffffu, at, 0);
  if (pred) heads[at + __popc(b & ((1u << lane) - 1))] = arc;
}

__global__ void __launch_bounds__(kBlock) k_rank_walk(const int32_t* __restrict__ succ,
                                                      const int64_t* __restrict__ n_arcs, RankSpace r) {
  const int64_t arcs = *n_arcs, walks = r.groups + *r.n_heads;
  for (int64_t id = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; id < walks; id += (int64_t)gridDim.x * blockDim.x) {
    int64_t a = id < r.groups ? rank_chosen(id) : r.heads[id - r.groups];
    uint32_t steps = 0;
    int32_t next = -1;
    while (a < arcs) {  // (a chosen place past the last arc starts no walk)
      r.own[a] = (uint64_t)id << 32 | steps++;
      const int32_t b = succ[a];
      if (b < 0) break;  // the end of the list
      if (rank_chosen(b >> 3) == b) {
        next = b >> 3;
        break;
      }
      a = b;
    }
    r.walk[0][id] = (uint64_t)(uint32_t)next << 32 | steps;
  }
}

// four steps of the walks' list per round
__global__ void __launch_bounds__(kBlock) k_rank_jump(const uint64_t* __restrict__ in, uint64_t* __restrict__ out,
                                                      int64_t groups, const int32_t* __restrict__ n_heads) {
  const int64_t walks = groups + *n_heads;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < walks; i += (int64_t)gridDim.x * blockDim.x) {
    uint64_t w = in[i];
#pragma unroll
    for (int k = 0; k < 3; k++) {
      const int32_t s = (int32_t)(w >> 32);
      if (s < 0) break;
      const uint64_t x = in[s];
      w = (x & 0xffffffff00000000ull) | (uint32_t)((uint32_t)w + (uint32_t)x);
    }
    out[i] = w;
  }
}

// arcs from a to the end of its list (0 for the last one), -1 if it has no end
__device__ __forceinline__ int32_t arc_rank(const uint64_t* __restrict__ own, const uint64_t* __restrict__ walk,
                                            int64_t a) {
  const uint64_t w = own[a];
  if (w == ~0ull) return -1;
  const uint64_t x = walk[w >> 32];
  return (int32_t)(x >> 32) < 0 ? (int32_t)((uint32_t)x - 1 - (uint32_t)w) : -1;
}

// Work space for lists over at most A arcs with at most max_heads heads; alloc(pointer, count) returns success.
template <typename Alloc>
bool rank_space(RankSpace& r, int64_t A, int64_t max_heads, cudaStream_t s, Alloc&& alloc) {
  r.groups = (A + 7) / 8;
  r.max_heads = max_heads;
  return alloc(&r.own, A) && alloc(&r.walk[0], r.groups + max_heads) && alloc(&r.walk[1], r.groups + max_heads) &&
         alloc(&r.heads, max_heads) && alloc(&r.n_heads, 1) &&
         cudaMemsetAsync(r.own, 0xff, sizeof(uint64_t) * (size_t)std::max<int64_t>(A, 1), s) == cudaSuccess &&
         cudaMemsetAsync(r.n_heads, 0, sizeof(int32_t), s) == cudaSuccess;
}

// Ranks the lists of succ (cut, their heads listed in r); the ranked walks are left in the returned array.
inline const uint64_t* rank_lists(const Handle& h, const int32_t* succ, const int64_t* n_arcs, const RankSpace& r,
                                  cudaStream_t s) {
  const int grid = grid_for(h, r.groups + std::min<int64_t>(r.max_heads, r.groups));
  k_rank_walk<<<grid, kBlock, 0, s>>>(succ, n_arcs, r);
  int c = 0;
  for (int64_t reach = 1; reach < r.groups + r.max_heads + 1; reach *= 4) {
    k_rank_jump<<<grid, kBlock, 0, s>>>(r.walk[c], r.walk[c ^ 1], r.groups, r.n_heads);
    c ^= 1;
  }
  return r.walk[c];
}

}  // namespace

}  // namespace pdg

namespace pdg {

namespace {

// Rows of up to kRowShort entries are taken by a thread each, longer ones by the whole block, one after another: a hub
// may have most of the vertices in its row.  row(v, begin, end) and long_row(v, begin, end); every thread of the block
// calls, and runs long_row.
constexpr int kRowShort = 64;

template <typename Row, typename LongRow>
__device__ __forceinline__ void for_rows(const int64_t* __restrict__ ptr, int64_t n, Row&& row, LongRow&& long_row) {
  __shared__ int32_t s_long[kBlock];
  __shared__ int s_n;
  for (int64_t v0 = (int64_t)blockIdx.x * kBlock; v0 < n; v0 += (int64_t)gridDim.x * kBlock) {  // block-uniform
    const int64_t v = v0 + threadIdx.x;
    const int64_t b = v < n ? ptr[v] : 0, e = v < n ? ptr[v + 1] : 0;
    const bool is_long = e - b > kRowShort;
    const bool any = __syncthreads_or(is_long);  // (and the rows listed before are done)
    if (v < n && !is_long) row(v, b, e);
    if (!any) continue;
    if (threadIdx.x == 0) s_n = 0;
    __syncthreads();
    if (is_long) s_long[atomicAdd(&s_n, 1)] = (int32_t)v;
    __syncthreads();
    for (int i = 0; i < s_n; i++) long_row((int64_t)s_long[i], ptr[s_long[i]], ptr[s_long[i] + 1]);
  }
}

__device__ __forceinline__ void sort_few(int32_t* a, int64_t len) {
  for (int64_t p = 1; p < len; p++) {
    const int32_t x = a[p];
    int64_t q = p - 1;
    while (q >= 0 && a[q] > x) {
      a[q + 1] = a[q];
      q--;
    }
    a[q + 1] = x;
  }
}

// The block sorts `len` distinct values: runs of 32 by a thread each, then neighbouring runs are merged, every value
// finding its place by a search in the other run (len log^2 len steps over the block's threads; a thread's insertion
// sort, len^2 / 4, took a hub of 3 x 10^5 neighbours to minutes).  Init of a star of 10^5 leaves and 10^5 more edges 6.6
// ms, of 10^6 and 10^6 78 ms.
__device__ void block_sort_row(int32_t* a, int32_t* tmp, int64_t len) {
  constexpr int kRun = 5;
  for (int64_t r = (int64_t)threadIdx.x << kRun; r < len; r += (int64_t)kBlock << kRun)
    sort_few(a + r, min((int64_t)1 << kRun, len - r));
  __syncthreads();
  int32_t *src = a, *dst = tmp;
  for (int sh = kRun; ((int64_t)1 << sh) < len; sh++) {
    for (int64_t i = threadIdx.x; i < len; i += kBlock) {
      const int32_t x = src[i];
      const int64_t run = i >> sh, other = (run ^ 1) << sh;
      int64_t lo = min(other, len), hi = min(other + ((int64_t)1 << sh), len);
      const int64_t first = lo;
      while (lo < hi) {
        const int64_t mid = (lo + hi) >> 1;
        if (src[mid] < x) lo = mid + 1;
        else hi = mid;
      }
      dst[((run & ~(int64_t)1) << sh) + (i - (run << sh)) + (lo - first)] = x;
    }
    __syncthreads();
    int32_t* const t = src;
    src = dst;
    dst = t;
  }
  if (src != a)
    for (int64_t i = threadIdx.x; i < len; i += kBlock) a[i] = src[i];
  __syncthreads();
}

// Canonical tree adjacency (rows in increasing neighbour order) so that the
// Euler tour, and every sum taken along it, does not depend on the order in
// which the atomic fill placed the arcs.  The values of a row are distinct;
// tmp is as long as they are all together.
__global__ void __launch_bounds__(kBlock) k_tour_sort_rows(const int64_t* __restrict__ ptr, int64_t n, int32_t* vals,
                                                           int32_t* tmp) {
  for_rows(
      ptr, n, [&](int64_t, int64_t b, int64_t e) { sort_few(vals + b, e - b); },
      [&](int64_t, int64_t b, int64_t e) { block_sort_row(vals + b, tmp + b, e - b); });
}

__device__ __forceinline__ int32_t tour_find(const int64_t* __restrict__ tptr, const int32_t* __restrict__ tadj,
                                            int32_t row, int32_t x) {
  int64_t lo = tptr[row], hi = tptr[row + 1];
  while (lo < hi) {
    const int64_t mid = (lo + hi) >> 1;
    if (tadj[mid] < x) lo = mid + 1;
    else hi = mid;
  }
  return (int32_t)lo;
}

// reverse arcs and the u->v arc of every tree edge, after the rows were sorted
__global__ void __launch_bounds__(kBlock) k_tour_fix_rev(const int64_t* __restrict__ tptr,
                                                         const int32_t* __restrict__ tadj, int64_t n,
                                                         int32_t* __restrict__ rev) {
  for_rows(
      tptr, n,
      [&](int64_t x, int64_t b, int64_t e) {
        for (int64_t p = b; p < e; p++) rev[p] = tour_find(tptr, tadj, tadj[p], (int32_t)x);
      },
      [&](int64_t x, int64_t b, int64_t e) {
        for (int64_t p = b + threadIdx.x; p < e; p += kBlock) rev[p] = tour_find(tptr, tadj, tadj[p], (int32_t)x);
      });
}

__global__ void k_tour_fix_arcs(const int32_t* __restrict__ eu, const int32_t* __restrict__ ev,
                                const uint8_t* __restrict__ tflag, int64_t m, const int64_t* __restrict__ tptr,
                                const int32_t* __restrict__ tadj, int32_t* __restrict__ arc_uv) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < m; e += (int64_t)gridDim.x * blockDim.x)
    if (tflag[e]) arc_uv[e] = tour_find(tptr, tadj, eu[e], ev[e]);
}

}  // namespace

}  // namespace pdg
