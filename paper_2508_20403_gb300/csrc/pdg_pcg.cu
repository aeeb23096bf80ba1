// Sparsifier quality: preconditioned conjugate gradients on L_G x = b with
// the sparsifier's Laplacian L_P (spanning tree T plus the recovered edges A)
// as the preconditioner, to a relative residual tol (Sec. 5 measures
// sparsifiers by these iteration counts, tol 1e-3).
//
//   b' = b - mean(b); x = 0, r = b', z = M(r), p = z
//   repeat: a = (r.z) / (p.L_G p); x += a p; r -= a L_G p;
//           stop when ||r|| <= tol ||b'||;
//           z = M(r); beta = (r.z)_new / (r.z)_old; p = z + beta p
//
// M(r) solves L_P z = r grounded at the tree root (z(root) = 0, the root's
// equation dropped), then centres z.  Grounded, L_P = L_T + U W U^T with U
// the incidence columns of the k recovered edges, so (Woodbury)
//   L_P^-1 = L_T^-1 - L_T^-1 U C^-1 U^T L_T^-1,  C = W^-1 + U^T L_T^-1 U (k x k, SPD).
// A grounded tree solve L_T x = y is two prefix sums over the Euler tour:
// the flow on the edge above c is the sum of y over the subtree of c (the
// positions between c's entry and exit arcs), and x(v) sums flow / w over
// the root path of v (+ at each entry, - at each exit, read at v's entry).
// C comes from the root distances of the endpoints' LCAs and is inverted once
// (block sweeps; C is SPD, so no pivoting); every sum runs in a fixed order,
// so the result is deterministic.  Dense C: k <= kPcgMaxEdges.
#include <cmath>
#include <type_traits>
#include <utility>
#include <vector>

#include "pdg_internal.cuh"
#include "pdg_tour.cuh"

namespace pdg {

namespace {

constexpr int kTourThreads = 256;
constexpr int64_t kTourMost = 4096ll * 4096;  // positions

__global__ void k_pc_tflag(const int32_t* __restrict__ eu, const int32_t* __restrict__ ev,
                           const int32_t* __restrict__ parent, int64_t m, uint8_t* __restrict__ tflag) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < m; e += (int64_t)gridDim.x * blockDim.x)
    tflag[e] = (parent[ev[e]] == eu[e] || parent[eu[e]] == ev[e]) ? 1 : 0;
}

// the first vertex without a parent
__global__ void k_pc_root(const int32_t* __restrict__ parent, int64_t n, int32_t* __restrict__ root) {
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x)
    if (parent[v] < 0) atomicMin(root, (int32_t)v);
}

__global__ void k_pc_cut(const int32_t* __restrict__ rev, const int64_t* __restrict__ tptr,
                         const int32_t* __restrict__ tdeg, int32_t root, int32_t* __restrict__ succ, RankSpace r) {
  const bool first = threadIdx.x == 0 && tdeg[root] > 0;  // one warp
  if (first) succ[rev[tptr[root] + tdeg[root] - 1]] = -1;
  rank_add_head(first, (int32_t)tptr[root], r.heads, r.n_heads);
}

// entry / exit positions of every non-root vertex, the weight of the edge above it, and the tour itself (the vertex
// entered, or the complement of the vertex left)
__global__ void k_pc_times(const int32_t* __restrict__ eu, const int32_t* __restrict__ ev,
                           const double* __restrict__ ew, const uint8_t* __restrict__ tflag,
                           const int32_t* __restrict__ arc_uv, const int32_t* __restrict__ rev,
                           const uint64_t* __restrict__ own, const uint64_t* __restrict__ walk,
                           const int64_t* __restrict__ tptr, int64_t n, int64_t m, int32_t* __restrict__ tin,
                           int32_t* __restrict__ tout, double* __restrict__ wup, int32_t* __restrict__ tour,
                           int32_t* __restrict__ bad) {
  const int64_t last = tptr[n] - 1;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < m; e += (int64_t)gridDim.x * blockDim.x) {
    if (!tflag[e]) continue;
    const int32_t a1 = arc_uv[e], a2 = rev[a1];
    const int32_t r1 = arc_rank(own, walk, a1), r2 = arc_rank(own, walk, a2);
    if (r1 < 0 || r2 < 0) {  // on no list that ends: the parent links close a cycle
      *bad = 1;
      continue;
    }
    const bool down1 = r1 > r2;  // u -> v comes first: u is the parent
    const int32_t child = down1 ? ev[e] : eu[e];
    const int32_t in = (int32_t)(last - max(r1, r2)), out = (int32_t)(last - min(r1, r2));
    tin[child] = in;
    tout[child] = out;
    wup[child] = ew[e];
    tour[in] = child;
    tour[out] = ~child;
  }
}

// --- prefix sums over the tour, in a fixed order: tile sums, then every tile adds up the sums before its own and
// scans itself.  What stands at a position is computed from its vertex on the fly, and what the sum is wanted for is
// written at once, so a tree solve is four launches over the tour and no array but E lies between them:
//   flow    y(v) at v's entry; E = exclusive prefix (a subtree's sum is E[exit] - E[entry])
//   drops   +-(flow on the edge above v) / w at v's entry and exit; the inclusive prefix at v's entry is x(v)
//           (kDropsZ: the scan writes z(v) = t(v) - x(v), or x(v) without t, and sums z)
enum { kFlow, kFlowEdges, kDrops, kDropsZ };


__device__ __forceinline__ double warp_incl_scan_d(double v) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const double t = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= o) v += t;
  }
  return v;
}

// sum over the block (a fixed tree), in every thread; sh holds 33 values
__device__ __forceinline__ double block_sum_d(double v, double* sh) {
#pragma unroll
  for (int o = 16; o; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  if (lane == 0) sh[w] = v;
  __syncthreads();
  if (w == 0) {
    double x = lane < nw ? sh[lane] : 0.0;
#pragma unroll
    for (int o = 16; o; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
    if (lane == 0) sh[32] = x;
  }
  __syncthreads();
  const double r = sh[32];
  __syncthreads();
  return r;
}

// Sums over a vector: one number per block, which every block of the kernel that needs the sum adds up for itself, in
// one order (a last block that adds them cost 3 us of fence, counter and second pass in each of four kernels).
constexpr int kDotBlocks = kPcgParts;

struct Parts {
  double* part = nullptr;
  int count = 0;
};

__device__ __forceinline__ void put_part(double s, const Parts& d) {
  __shared__ double sh[33];
  s = block_sum_d(s, sh);
  if (threadIdx.x == 0) d.part[blockIdx.x] = s;
}

__device__ __forceinline__ double sum_of(const Parts& d) {  // in every thread
  __shared__ double sh[33];
  double s = 0.0;
  for (int i = threadIdx.x; i < d.count; i += blockDim.x) s += d.part[i];
  return block_sum_d(s, sh);
}

struct TourArgs {
  const int32_t* tour;
  int64_t A;
  const int32_t* tin;
  const int32_t* tout;
  const double* wup;
  const double* y;        // kFlow
  const int64_t* iptr;    // kFlowEdges: y(v) = sum of +-q over the recovered edges at v, in edge order
  const int32_t* iedge;
  const int32_t* ea;
  const double* q;
  double* E;              // kFlow, kFlowEdges: output; kDrops: input
  double* D;              // values by position
  double* x;              // kDrops: potentials, kDropsZ: z (at the root they are zero)
  const double* t;        // kDropsZ
  Parts z_sum;            // kDropsZ
  int32_t root;
  double* sums;           // per tile
};

template <int MODE>
__device__ __forceinline__ double tour_value(const TourArgs& a, int32_t t) {
  const bool down = t >= 0;
  const int32_t v = down ? t : ~t;
  if (MODE == kFlow) return down ? a.y[v] : 0.0;
  if (MODE == kFlowEdges) {
    double s = 0.0;
    if (down)
      for (int64_t p = a.iptr[v]; p < a.iptr[v + 1]; p++) {
        const int32_t i = a.iedge[p];
        s += a.ea[i] == v ? a.q[i] : -a.q[i];
      }
    return s;
  }
  const double d = (a.E[a.tout[v]] - a.E[a.tin[v]]) / a.wup[v];
  return down ? d : -d;
}

// (kFlowEdges and kDrops leave the values in D for the scan)
template <int MODE, int ITEMS>
__global__ void __launch_bounds__(kTourThreads) k_pc_tour_sums(TourArgs a) {
  __shared__ double sh[kTourThreads / 32];
  const int64_t base = ((int64_t)blockIdx.x * kTourThreads + threadIdx.x) * ITEMS;
  double s = 0.0;
#pragma unroll
  for (int i = 0; i < ITEMS; i++) {
    if (base + i >= a.A) break;
    const double v = tour_value<MODE>(a, a.tour[base + i]);
    if (MODE != kFlow) a.D[base + i] = v;
    s += v;
  }
  // added up as k_pc_tour_scan adds it up, so that a tile's prefixes end where the next tile's begin
  const double incl = warp_incl_scan_d(s);
  if ((threadIdx.x & 31) == 31) sh[threadIdx.x >> 5] = incl;
  __syncthreads();
  if (threadIdx.x == 0) {
    double sum = 0.0;
    for (int i = 0; i < kTourThreads / 32; i++) sum += sh[i];
    a.sums[blockIdx.x] = sum;
  }
}

template <int MODE, int ITEMS>
__global__ void __launch_bounds__(kTourThreads) k_pc_tour_scan(TourArgs a) {
  __shared__ double sh[33], sh2[kTourThreads / 32];
  const int64_t base = ((int64_t)blockIdx.x * kTourThreads + threadIdx.x) * ITEMS;
  int32_t t[ITEMS];
  double v[ITEMS], s = 0.0;
#pragma unroll
  for (int i = 0; i < ITEMS; i++) {
    const bool in = base + i < a.A;
    t[i] = in && MODE != kFlowEdges ? a.tour[base + i] : 0;
    v[i] = !in ? 0.0 : MODE == kFlow ? tour_value<MODE>(a, t[i]) : a.D[base + i];
    s += v[i];
  }
  double pre = 0.0;  // the tiles before this one
  for (int64_t i = threadIdx.x; i < (int64_t)blockIdx.x; i += kTourThreads) pre += a.sums[i];
  pre = block_sum_d(pre, sh);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const double incl = warp_incl_scan_d(s);
  if (lane == 31) sh2[w] = incl;
  __syncthreads();
  // what stands before a position in its tile is added up first, and to the tiles before it last: the sum of the tour so
  // far may be many times larger, and each addition to it rounds at its size
  double run = 0.0;
  for (int i = 0; i < w; i++) run += sh2[i];
  const double left = __shfl_up_sync(0xffffffffu, incl, 1);
  if (lane) run += left;
  double zs = 0.0;
#pragma unroll
  for (int i = 0; i < ITEMS; i++) {
    if (base + i >= a.A) break;
    if (MODE == kFlow || MODE == kFlowEdges) {
      a.E[base + i] = pre + run;
    } else if (t[i] >= 0) {
      double x = pre + (run + v[i]);
      if (MODE == kDropsZ) {
        if (a.t) x = a.t[t[i]] - x;
        zs += x;
      }
      a.x[t[i]] = x;
    }
    run += v[i];
  }
  if (MODE == kDropsZ) {
    if (blockIdx.x == 0 && threadIdx.x == 0) a.x[a.root] = 0.0;
    put_part(zs, a.z_sum);
  }
}

// f(integral constant): the positions of a thread.  FP64 is what the passes are short of (two operations a clock and
// SM), so a short tour is spread over as many tiles as 256 threads make (20,000 positions: 79 tiles, 4 us a pass; five
// tiles of 4096 took 25), a long one over at most 4096, whose sums every tile adds up.
template <typename F>
void with_items(int64_t A, F&& f) {
  if (A <= 1024 * kTourThreads) f(std::integral_constant<int, 1>());
  else if (A <= 1024 * 4 * kTourThreads) f(std::integral_constant<int, 4>());
  else f(std::integral_constant<int, 16>());
}

int64_t tour_tiles(int64_t A) {
  int64_t tiles = 0;
  with_items(A, [&](auto items) { tiles = (A + items() * kTourThreads - 1) / (items() * kTourThreads); });
  return std::max<int64_t>(tiles, 1);
}

// --- the k recovered edges ---
__global__ void k_pc_edges(const int32_t* __restrict__ ids, int64_t k, int64_t m, const int32_t* __restrict__ eu,
                           const int32_t* __restrict__ ev, const double* __restrict__ ew,
                           const uint8_t* __restrict__ tflag, int32_t* __restrict__ ea, int32_t* __restrict__ eb,
                           double* __restrict__ ewk, int32_t* __restrict__ bad) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < k; i += (int64_t)gridDim.x * blockDim.x) {
    const int32_t id = ids[i];
    if (id < 0 || id >= m || tflag[id]) {
      *bad = 1;
      ea[i] = eb[i] = 0;
      ewk[i] = 1.0;
      continue;
    }
    ea[i] = eu[id];
    eb[i] = ev[id];
    ewk[i] = ew[id];
  }
}

__global__ void k_pc_dups(const int32_t* __restrict__ ids, int64_t k, int64_t m, int32_t* __restrict__ seen,
                          int32_t* bad) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < k; i += (int64_t)gridDim.x * blockDim.x) {
    const int32_t id = ids[i];
    if (id >= 0 && id < m && atomicAdd(&seen[id], 1) != 0) *bad = 1;
  }
}

// --- the capacitance matrix.  C[i][j] = u_i^T L_T^-1 u_j (+ 1 / w_i on the diagonal) with u = e_a - e_b, and
// (L_T^-1)(x, y), grounded at the root, is the root distance of LCA(x, y): the vertex of least depth that the tour
// passes between the entries of x and y.  The 2 k endpoints are sorted by entry; gap[r] is the position of least depth
// from endpoint r to endpoint r + 1, both included (depth << 32 | position + 1; zero is the root), and a sparse table
// over the gaps answers every pair.  Depths are whole numbers, so the ancestor is exact; distances are summed along
// the tour in pairs of doubles, since C is made of their differences.  500 edges on the 100 x 100 grid: 0.1 ms; one tree
// solve per column, 14 launches each, took 35 of 44 ms.
struct Dist {
  double hi, lo;
  int32_t depth;
};

__device__ __forceinline__ Dist operator+(const Dist& a, const Dist& b) {
  const double s = a.hi + b.hi, t = s - a.hi;
  const double e = ((a.hi - (s - t)) + (b.hi - t)) + (a.lo + b.lo);
  const double hi = s + e;
  return {hi, e - (hi - s), a.depth + b.depth};
}

__device__ __forceinline__ Dist warp_incl_scan_dist(Dist v) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const Dist t{__shfl_up_sync(0xffffffffu, v.hi, o), __shfl_up_sync(0xffffffffu, v.lo, o),
                 __shfl_up_sync(0xffffffffu, v.depth, o)};
    if (lane >= o) v = t + v;
  }
  return v;
}

__device__ __forceinline__ Dist dist_step(int32_t t, const double* __restrict__ wup) {
  return t >= 0 ? Dist{1.0 / wup[t], 0.0, 1} : Dist{-1.0 / wup[~t], 0.0, -1};
}

// SUM: the tile's sum; else the inclusive prefix of every position, and the largest depth
template <bool SUM, int ITEMS>
__global__ void __launch_bounds__(kTourThreads) k_pc_dist(const int32_t* __restrict__ tour, int64_t A,
                                                          const double* __restrict__ wup, Dist* __restrict__ sums,
                                                          double2* __restrict__ dist, int32_t* __restrict__ depth,
                                                          int32_t* __restrict__ max_depth) {
  constexpr int kWarps = kTourThreads / 32;
  __shared__ Dist sh[kWarps];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int64_t base = ((int64_t)blockIdx.x * kTourThreads + threadIdx.x) * ITEMS;
  Dist v[ITEMS], s{0.0, 0.0, 0};
#pragma unroll
  for (int i = 0; i < ITEMS; i++) {
    v[i] = base + i < A ? dist_step(tour[base + i], wup) : Dist{0.0, 0.0, 0};
    s = s + v[i];
  }
  Dist pre{0.0, 0.0, 0};  // SUM: this tile; else the tiles before it
  if (SUM) pre = s;
  else
    for (int64_t i = threadIdx.x; i < (int64_t)blockIdx.x; i += kTourThreads) pre = pre + sums[i];
  pre = warp_incl_scan_dist(pre);
  if (lane == 31) sh[w] = pre;
  __syncthreads();
  pre = sh[0];
  for (int i = 1; i < kWarps; i++) pre = pre + sh[i];
  if (SUM) {
    if (threadIdx.x == 0) sums[blockIdx.x] = pre;
    return;
  }
  __syncthreads();
  const Dist incl = warp_incl_scan_dist(s);
  if (lane == 31) sh[w] = incl;
  __syncthreads();
  Dist run = pre;
  for (int i = 0; i < w; i++) run = run + sh[i];
  const Dist left{__shfl_up_sync(0xffffffffu, incl.hi, 1), __shfl_up_sync(0xffffffffu, incl.lo, 1),
                  __shfl_up_sync(0xffffffffu, incl.depth, 1)};
  if (lane) run = run + left;
  int deepest = 0;
#pragma unroll
  for (int i = 0; i < ITEMS; i++) {
    if (base + i >= A) break;
    run = run + v[i];
    dist[base + i] = make_double2(run.hi, run.lo);
    depth[base + i] = run.depth;
    deepest = max(deepest, run.depth);
  }
  deepest = __reduce_max_sync(0xffffffffu, deepest);
  if (lane == 0 && deepest > 0) atomicMax(max_depth, deepest);
}

__global__ void k_pc_ends(const int32_t* __restrict__ ea, const int32_t* __restrict__ eb,
                          const int32_t* __restrict__ tin, int32_t root, int64_t k, uint64_t* __restrict__ key) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < 2 * k; i += (int64_t)gridDim.x * blockDim.x) {
    const int32_t v = i < k ? ea[i] : eb[i - k];
    const uint32_t pos = v == root ? 0u : (uint32_t)tin[v] + 1u;  // the root stands before the tour
    key[i] = (uint64_t)pos << 32 | (uint32_t)i;
  }
}

// one block sorts the 2 k <= 16384 keys (bitonic, padded to a power of two) and returns every endpoint's rank
constexpr int kSortMax = 16384;
static_assert(kSortMax >= 2 * kPcgMaxEdges);
__global__ void __launch_bounds__(1024) k_pc_sort_ends(const uint64_t* __restrict__ key, int count, int size,
                                                       int32_t* __restrict__ pos, int32_t* __restrict__ rank) {
  extern __shared__ uint64_t s_key[];
  for (int i = threadIdx.x; i < size; i += 1024) s_key[i] = i < count ? key[i] : ~0ull;
  __syncthreads();
  for (int w = 2; w <= size; w <<= 1)
    for (int o = w >> 1; o; o >>= 1) {
      for (int i = threadIdx.x; i < size / 2; i += 1024) {
        const int a = 2 * o * (i / o) + i % o, b = a + o;
        const uint64_t x = s_key[a], y = s_key[b];
        if ((x > y) == ((a & w) == 0)) {
          s_key[a] = y;
          s_key[b] = x;
        }
      }
      __syncthreads();
    }
  for (int i = threadIdx.x; i < count; i += 1024) {
    pos[i] = (int32_t)(uint32_t)(s_key[i] >> 32) - 1;
    rank[(uint32_t)s_key[i]] = i;
  }
}

// the tour's state at a position (-1: before its first arc, at the root)
__device__ __forceinline__ uint64_t state_at(const int32_t* __restrict__ depth, int64_t pos) {
  return pos < 0 ? 0ull : (uint64_t)(uint32_t)depth[pos] << 32 | (uint32_t)(pos + 1);
}

__global__ void k_pc_gap_ends(const int32_t* __restrict__ pos, const int32_t* __restrict__ depth, int count,
                              uint64_t* __restrict__ gap) {
  for (int r = blockIdx.x * blockDim.x + threadIdx.x; r < count; r += gridDim.x * blockDim.x) {
    const uint64_t a = state_at(depth, pos[r]);
    gap[r] = r + 1 < count ? min(a, state_at(depth, pos[r + 1])) : a;
  }
}

// positions strictly between two neighbouring endpoints
__global__ void k_pc_gap_min(const int32_t* __restrict__ pos, const int32_t* __restrict__ depth, int64_t A, int count,
                             uint64_t* __restrict__ gap) {
  const int lane = threadIdx.x & 31;
  for (int64_t p0 = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31); p0 < A;
       p0 += (int64_t)gridDim.x * blockDim.x) {  // warp-uniform
    const int64_t p = p0 + lane;
    int r = -1;  // the last endpoint at or before p
    unsigned long long v = ~0ull;
    if (p < A) {
      int lo = 0, hi = count;
      while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (pos[mid] <= p) lo = mid + 1;
        else hi = mid;
      }
      r = lo - 1;
      v = state_at(depth, p);
    }
    const bool in = r >= 0 && r + 1 < count;
    const int r0 = __shfl_sync(0xffffffffu, r, 0);
    // a warp's positions are mostly of one gap: its minimum first
    if (__all_sync(0xffffffffu, in && r == r0)) {
#pragma unroll
      for (int o = 16; o; o >>= 1) v = min(v, __shfl_down_sync(0xffffffffu, v, o));
      if (lane == 0) atomicMin(reinterpret_cast<unsigned long long*>(gap + r), v);
    } else if (in) {
      atomicMin(reinterpret_cast<unsigned long long*>(gap + r), v);
    }
  }
}

// the rows of the sparse table after the first, by one block
__global__ void __launch_bounds__(1024) k_pc_gap_rows(uint64_t* table, int rows, int count) {
  for (int t = 1; t < rows; t++) {
    const uint64_t* in = table + (int64_t)(t - 1) * count;
    uint64_t* out = table + (int64_t)t * count;
    const int o = 1 << (t - 1);
    for (int r = threadIdx.x; r < count; r += 1024) out[r] = r + o < count ? min(in[r], in[r + o]) : in[r];
    __syncthreads();
  }
}

__global__ void k_pc_capacitance(const uint64_t* __restrict__ table, const double2* __restrict__ dist,
                                 const int32_t* __restrict__ depth, const int32_t* __restrict__ pos,
                                 const int32_t* __restrict__ rank, const double* __restrict__ ewk, int k,
                                 double* __restrict__ C) {
  const int n = 2 * k;
  // distance of the common ancestor of the endpoints of ranks r and s
  auto common = [&](int r, int s) -> Dist {
    uint64_t st;
    if (r == s) {
      st = state_at(depth, pos[r]);
    } else {
      const int lo = min(r, s), hi = max(r, s), t = 31 - __clz(hi - lo);
      const uint64_t* row = table + (int64_t)t * n;
      st = min(row[lo], row[hi - (1 << t)]);
    }
    if ((st >> 32) == 0) return {0.0, 0.0, 0};  // the root
    const double2 d = dist[(uint32_t)st - 1];
    return {d.x, d.y, 0};
  };
  auto neg = [](const Dist& d) -> Dist { return {-d.hi, -d.lo, 0}; };
  const int64_t kk = (int64_t)k * k;
  for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < kk; q += (int64_t)gridDim.x * blockDim.x) {
    const int i = (int)(q / k), j = (int)(q - (int64_t)i * k);
    if (j > i) continue;  // the lower triangle
    const int ai = rank[i], bi = rank[k + i], aj = rank[j], bj = rank[k + j];
    const Dist d = (common(ai, aj) + neg(common(ai, bj))) + neg(common(bi, aj) + neg(common(bi, bj)));
    C[q] = i == j ? d.hi + 1.0 / ewk[i] : d.hi;
  }
}

// --- inverse of C in place: the symmetric sweep by blocks of kSw pivots, on the lower triangle (C is symmetric
// positive definite: no pivoting).  For the pivot block p, C_pp = M D M^T with M unit lower triangular: Y_i = C_ip M^-T,
// R_i = Y_i D^-1 M^-1 = C_ip inv(C_pp); then C_ij -= (Y_i D^-1) Y_j^T, C_ip = R_i, C_pj = R_j^T, C_pp = -inv(C_pp), and
// after all blocks C is -inv(C).  Two launches per block.
// As accurate as pivot by pivot over the whole matrix.  (With R_i = C_ip inv(C_pp) from the block's explicit inverse and
// C_ij -= C_ip R_j^T, products with inv(C) were 10 to 60 times further off, and the preconditioner's residual, 10^-3
// where off-tree edges outweigh the tree 10^6 times, was of order 1.)
// Bound by FP64 (k^3 / 2 multiply-adds at two a clock and SM) and the chain of k pivots (0.7 us each, mostly the
// reciprocal): k = 500 takes 0.56 ms; pivot by pivot over the whole matrix it was two launches a pivot, 4.4 ms of
// kernels and as much between them.
constexpr int kSw = 32;

// The factors of C_pp (every block for itself: 32 rows in the registers of eight warps, the scaled pivot rows, which are
// the columns of M, through shared memory), then Y, S = Y D^-1 and R of this block's eight rows.  A row of the pivot block takes its
// row of the identity along instead, and its R is its row of inv(C_pp).
__global__ void __launch_bounds__(256) k_pc_sweep_panel(const double* __restrict__ C, int k, int p0,
                                                        double* __restrict__ S, double* __restrict__ R,
                                                        double* __restrict__ Y) {
  __shared__ double b[kSw][kSw + 1];  // b[p][j] = M[j][p], j > p
  __shared__ double s_d[kSw];         // D^-1
  const int nb = min(kSw, k - p0), lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int row = blockIdx.x * 8 + w;  // of Y, S and R
  double x = 0.0;
  if (row >= p0 && row < p0 + nb) x = row - p0 == lane ? 1.0 : 0.0;
  else if (row < k && lane < nb) x = row > p0 ? C[(int64_t)row * k + p0 + lane] : C[(int64_t)(p0 + lane) * k + row];
  double v[4];  // rows w, w + 8, w + 16, w + 24
#pragma unroll
  for (int r = 0; r < 4; r++) {
    const int i = w + 8 * r;
    v[r] = i < nb && lane < nb ? C[(int64_t)(p0 + max(i, lane)) * k + p0 + min(i, lane)] : (i == lane ? 1.0 : 0.0);
  }
  auto pivot_row = [&](double a, int p) {  // row p, up to date: scaled
    const double d = 1.0 / __shfl_sync(0xffffffffu, a, p);
    b[p][lane] = a * d;
    if (lane == p) s_d[p] = d;
  };
  if (w == 0) pivot_row(v[0], 0);
  __syncthreads();
#pragma unroll
  for (int r0 = 0; r0 < 4; r0++)
    for (int q = 0; q < 8; q++) {
      const int p = 8 * r0 + q;  // the pivot: row r0 of warp q
      const double piv = b[p][lane];
      auto update = [&](double a) {
        const double f = __shfl_sync(0xffffffffu, a, p);
        return lane > p ? a - f * piv : a;
      };
      // the next pivot's warp first brings that row up to date and scales it: its division runs beside the others'
      // multiply-adds
      const bool next_here = w == ((q + 1) & 7) && p + 1 < kSw;
      const int rn = q == 7 ? r0 + 1 : r0;
#pragma unroll
      for (int r = 0; r < 4; r++)
        if (next_here && r == rn) pivot_row(update(v[r]), p + 1);
#pragma unroll
      for (int r = 0; r < 4; r++)  // the rows after it
        if (w + 8 * r > p + 1) v[r] = update(v[r]);
      x = update(x);
      __syncthreads();
    }
  if (row >= k) return;  // (warp-uniform)
  Y[(int64_t)row * kSw + lane] = x;
  double t = x * s_d[lane];
  S[(int64_t)row * kSw + lane] = t;
#pragma unroll
  for (int p = kSw - 1; p > 0; p--) {
    const double f = __shfl_sync(0xffffffffu, t, p);
    if (lane < p) t -= f * b[lane][p];
  }
  R[(int64_t)row * kSw + lane] = t;
}

// the t-th tile of the lower triangle, row by row (y: row); the grid holds no others, so that up to 152 of them lie on
// an SM each
__device__ __forceinline__ int2 lower_tile(uint32_t t) {
  int y = (int)((sqrtf(8.0f * (float)t + 1.0f) - 1.0f) * 0.5f);
  while ((uint32_t)(y + 1) * (uint32_t)(y + 2) / 2 <= t) y++;
  while ((uint32_t)y * (uint32_t)(y + 1) / 2 > t) y--;
  return make_int2((int)(t - (uint32_t)y * (uint32_t)(y + 1) / 2), y);
}

__global__ void __launch_bounds__(256) k_pc_sweep_update(double* __restrict__ C, int k, int p0,
                                                         const double* __restrict__ S, const double* __restrict__ R,
                                                         const double* __restrict__ Y) {
  __shared__ double l[kSw][kSw + 1], r[kSw][kSw + 1];  // by row of C
  const int2 tile = lower_tile(blockIdx.x);
  const int i0 = tile.y * kSw, j0 = tile.x * kSw, tid = threadIdx.x;
  const bool pi = i0 == p0, pj = j0 == p0;
  for (int q = tid; q < kSw * kSw; q += 256) {
    const int i = q / kSw, t = q % kSw;
    l[i][t] = i0 + i >= k ? 0.0 : (pj ? R : S)[(int64_t)(i0 + i) * kSw + t];
    r[i][t] = j0 + i >= k ? 0.0 : (pi ? R : Y)[(int64_t)(j0 + i) * kSw + t];
  }
  __syncthreads();
  const int ti = tid / 16, tj = tid % 16;  // rows ti, ti + 16, columns tj, tj + 16
  double acc[2][2] = {};
  if (!pi && !pj) {
#pragma unroll 8
    for (int t = 0; t < kSw; t++) {
      const double x0 = l[ti][t], x1 = l[ti + 16][t], y0 = r[tj][t], y1 = r[tj + 16][t];
      acc[0][0] += x0 * y0;
      acc[0][1] += x0 * y1;
      acc[1][0] += x1 * y0;
      acc[1][1] += x1 * y1;
    }
  }
#pragma unroll
  for (int a = 0; a < 2; a++)
#pragma unroll
    for (int c = 0; c < 2; c++) {
      const int i = ti + 16 * a, j = tj + 16 * c;
      if (i0 + i >= k || j0 + j >= k) continue;
      double* at = C + (int64_t)(i0 + i) * k + j0 + j;
      if (pi && pj) *at = -l[i][j];
      else if (pj) *at = l[i][j];
      else if (pi) *at = r[j][i];
      else *at -= acc[a][c];
    }
}

// C = -C, and its upper triangle
__global__ void __launch_bounds__(256) k_pc_sweep_end(double* __restrict__ C, int k) {
  __shared__ double b[kSw][kSw + 1];
  const int2 tile = lower_tile(blockIdx.x);
  const int i0 = tile.y * kSw, j0 = tile.x * kSw, lane = threadIdx.x & 31;
  for (int i = threadIdx.x >> 5; i < kSw; i += 8)
    if (i0 + i < k && j0 + lane <= i0 + i) b[i][lane] = -C[(int64_t)(i0 + i) * k + j0 + lane];
  __syncthreads();
  for (int i = threadIdx.x >> 5; i < kSw; i += 8) {
    if (i0 + i < k && j0 + lane <= i0 + i) C[(int64_t)(i0 + i) * k + j0 + lane] = b[i][lane];
    if (j0 + i < k && i0 + lane < k && i0 + lane > j0 + i) C[(int64_t)(j0 + i) * k + i0 + lane] = b[lane][i];
  }
}

// q = C^-1 s with s_i = t(a_i) - t(b_i), which every block gathers for itself; one warp per row
constexpr int kGemvThreads = 512;
__global__ void __launch_bounds__(kGemvThreads) k_pc_gemv(const double* __restrict__ Ci, const double* __restrict__ t,
                                                          const int32_t* __restrict__ ea,
                                                          const int32_t* __restrict__ eb, int k,
                                                          double* __restrict__ q) {
  extern __shared__ double s_s[];
  for (int i = threadIdx.x; i < k; i += kGemvThreads) s_s[i] = t[ea[i]] - t[eb[i]];
  __syncthreads();
  const int lane = threadIdx.x & 31, nw = gridDim.x * (kGemvThreads / 32);
  for (int i = blockIdx.x * (kGemvThreads / 32) + (threadIdx.x >> 5); i < k; i += nw) {
    double acc = 0;
#pragma unroll 4
    for (int j = lane; j < k; j += 32) acc += Ci[(int64_t)i * k + j] * s_s[j];
    for (int o = 16; o; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
    if (lane == 0) q[i] = acc;
  }
}

__global__ void k_pc_inc_count(const int32_t* __restrict__ ea, const int32_t* __restrict__ eb, int64_t k,
                               int32_t* __restrict__ cnt) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < k; i += (int64_t)gridDim.x * blockDim.x) {
    atomicAdd(&cnt[ea[i]], 1);
    atomicAdd(&cnt[eb[i]], 1);
  }
}

__global__ void k_pc_inc_fill(const int32_t* __restrict__ ea, const int32_t* __restrict__ eb, int64_t k,
                              const int64_t* __restrict__ iptr, int32_t* __restrict__ cur, int32_t* __restrict__ iedge) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < k; i += (int64_t)gridDim.x * blockDim.x) {
    iedge[iptr[ea[i]] + atomicAdd(&cur[ea[i]], 1)] = (int32_t)i;
    iedge[iptr[eb[i]] + atomicAdd(&cur[eb[i]], 1)] = (int32_t)i;
  }
}

// --- vectors ---
__global__ void k_pc_degw(const int64_t* __restrict__ row_ptr, const double* __restrict__ w, int64_t n,
                          double* __restrict__ dw) {
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x) {
    double s = 0;
    for (int64_t p = row_ptr[v]; p < row_ptr[v + 1]; p++) s += w[p];
    dw[v] = s;
  }
}

// out = L_G p (row order of the CSR), and p . out
__global__ void __launch_bounds__(256) k_pc_spmv(const int64_t* __restrict__ row_ptr, const int32_t* __restrict__ col,
                                                 const double* __restrict__ w, const double* __restrict__ dw,
                                                 const double* __restrict__ p, int64_t n, double* __restrict__ out,
                                                 Parts d) {
  double dot = 0.0;
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x) {
    const double pv = p[v];
    double s = dw[v] * pv;
    for (int64_t q = row_ptr[v]; q < row_ptr[v + 1]; q++) s -= w[q] * p[col[q]];
    out[v] = s;
    dot += pv * s;
  }
  put_part(dot, d);
}

__global__ void __launch_bounds__(256) k_pc_dot(const double* __restrict__ a, const double* __restrict__ b, int64_t n,
                                                Parts d) {
  double s = 0.0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    s += (b ? a[i] * b[i] : a[i]);
  put_part(s, d);
}

// v -= sum / n (centring against the all-ones null space), and v . b (b null: v . v)
__global__ void __launch_bounds__(256) k_pc_center(double* __restrict__ v, int64_t n, Parts sum,
                                                   const double* __restrict__ b, Parts d) {
  const double mu = sum_of(sum) / (double)n;
  double s = 0.0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const double x = v[i] - mu;
    v[i] = x;
    s += x * (b ? b[i] : x);
  }
  put_part(s, d);
}

// x += a p, r -= a Ap with a = rz / pAp, and r . r
__global__ void __launch_bounds__(256) k_pc_step(double* __restrict__ x, double* __restrict__ r,
                                                 const double* __restrict__ p, const double* __restrict__ Ap, int64_t n,
                                                 Parts rz, Parts pAp, Parts d) {
  const double a = sum_of(rz) / sum_of(pAp);
  double s = 0.0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    x[i] += a * p[i];
    const double y = r[i] - a * Ap[i];
    r[i] = y;
    s += y * y;
  }
  put_part(s, d);
}

// p = z + beta p with beta = rz_new / rz
__global__ void k_pc_xpby(double* __restrict__ p, const double* __restrict__ z, Parts rz_new, Parts rz, int64_t n) {
  const double beta = sum_of(rz_new) / sum_of(rz);
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    p[i] = z[i] + beta * p[i];
}

}  // namespace

// a failed CUDA call releases the temporaries and reports PDG_E_CUDA
#define PC_CK(x)                                     \
  do {                                               \
    if ((x) != cudaSuccess) return fail(PDG_E_CUDA); \
  } while (0)

int pcg_quality(Handle& h, const int32_t* ids, int64_t k, const double* b, double tol, int32_t max_iter,
                int32_t* iters, double* relres, double* hist, double* z0) {
  const int64_t n = h.n, m = h.m;
  cudaStream_t s = h.stream;
  const int gn = grid_for(h, n), gm = grid_for(h, std::max<int64_t>(m, 1)), gk = grid_for(h, std::max<int64_t>(k, 1));
  std::vector<void*> temps;
  auto cleanup = [&]() {
    for (void* p : temps) cudaFreeAsync(p, s);
    temps.clear();
  };
  auto fail = [&](int code) {
    cudaGetLastError();
    cleanup();
    return code;
  };
  auto talloc = [&](auto** p, int64_t count) -> bool {
    void* q = nullptr;
    if (cudaMallocAsync(&q, sizeof(**p) * (size_t)std::max<int64_t>(count, 1), s) != cudaSuccess) return false;
    temps.push_back(q);
    *p = static_cast<std::remove_reference_t<decltype(*p)>>(q);
    return true;
  };
  // the arrays lie in one allocation: places are noted first
  std::vector<std::pair<void**, size_t>> places;
  size_t bytes = 0;
  auto place = [&](auto** p, int64_t count) {
    places.emplace_back(reinterpret_cast<void**>(p), bytes);
    bytes += (sizeof(**p) * (size_t)std::max<int64_t>(count, 1) + 255) & ~(size_t)255;
  };
  const int64_t A = 2 * (n - 1);
  if (A >= kTourMost) return fail(PDG_E_INVALID_ARG);  // every tile adds up the sums of those before it
  const int64_t T = tour_tiles(A);
  uint8_t* tflag = nullptr;
  int32_t *tdeg = nullptr, *cur = nullptr, *tadj = nullptr, *rev = nullptr, *arc_uv = nullptr;
  int32_t *succ = nullptr, *tin = nullptr, *tout = nullptr;
  RankSpace rank;
  int32_t *ea = nullptr, *eb = nullptr, *seen = nullptr, *flags = nullptr, *icnt = nullptr, *iedge = nullptr;
  int64_t *tptr = nullptr, *iptr = nullptr;
  double *wup = nullptr, *E = nullptr, *D = nullptr, *sums = nullptr, *ewk = nullptr;
  double *C = nullptr, *swR = nullptr, *swY = nullptr, *swS = nullptr, *dw = nullptr, *bb = nullptr, *x = nullptr;
  double *r = nullptr, *z = nullptr, *p = nullptr, *Ap = nullptr, *t = nullptr;
  double *qv = nullptr, *parts = nullptr;
  double2* dist = nullptr;
  Dist* dsums = nullptr;
  uint64_t *ekey = nullptr, *gaps = nullptr;
  int32_t *epos = nullptr, *erank = nullptr, *tour = nullptr, *depth = nullptr;
  int gap_rows = 1;
  while ((2ll << gap_rows) <= std::max<int64_t>(2 * k, 1)) gap_rows++;
  gap_rows++;
  place(&tflag, m); place(&tdeg, n); place(&cur, n); place(&tptr, n + 1); place(&tadj, A); place(&rev, A);
  place(&arc_uv, m); place(&succ, A); place(&tin, n); place(&tout, n); place(&wup, n); place(&tour, A); place(&E, A);
  place(&sums, T); place(&dist, A); place(&D, A); place(&depth, A); place(&dsums, T); place(&ea, k); place(&eb, k);
  place(&ewk, k); place(&seen, m); place(&flags, 4); place(&icnt, n); place(&iptr, n + 1); place(&iedge, 2 * k);
  place(&C, k * k); place(&swR, kSw * k); place(&swY, kSw * k); place(&swS, kSw * k); place(&ekey, 2 * k);
  place(&epos, 2 * k); place(&erank, 2 * k); place(&gaps, 2 * k * gap_rows); place(&dw, n); place(&bb, n);
  place(&x, n); place(&r, n); place(&z, n); place(&p, n); place(&Ap, n); place(&t, n);
  place(&qv, k); place(&parts, 4 * kDotBlocks + std::max<int64_t>(kDotBlocks, T));
  char* block = nullptr;
  if (!talloc(&block, (int64_t)bytes) || !rank_space(rank, A, 1, s, talloc)) return fail(PDG_E_OOM);
  for (auto& [slot, offset] : places) *slot = block + offset;
  int st = PDG_OK;
  // Euler tour of the tree
  k_pc_tflag<<<gm, kBlock, 0, s>>>(h.el_u, h.el_v, h.parent, m, tflag);
  PC_CK(cudaMemsetAsync(flags, 0x7f, sizeof(int32_t), s));
  k_pc_root<<<gn, kBlock, 0, s>>>(h.parent, n, flags);
  PC_CK(cudaMemsetAsync(tdeg, 0, sizeof(int32_t) * n, s));
  PC_CK(cudaMemsetAsync(cur, 0, sizeof(int32_t) * n, s));
  k_st_tdeg<<<gm, kBlock, 0, s>>>(h.el_u, h.el_v, tflag, m, tdeg);
  if ((st = ensure_scan_status(h, n)) || (st = scan_excl_i32(h, tdeg, tptr, n, nullptr, n))) return fail(st);
  int32_t root = -1;
  {
    int64_t arcs = -1;
    if (cudaMemcpyAsync(&arcs, tptr + n, sizeof(int64_t), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
        cudaMemcpyAsync(&root, flags, sizeof(int32_t), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
        cudaStreamSynchronize(s) != cudaSuccess)
      return fail(PDG_E_CUDA);
    // a root, and the parent links are the n - 1 tree edges
    if (arcs != A || root < 0 || root >= n) return fail(PDG_E_NOT_A_TREE);
  }
  k_st_fill<<<gm, kBlock, 0, s>>>(h.el_u, h.el_v, tflag, m, tptr, cur, tadj, rev, arc_uv);
  // rows in neighbour order: the tour, and so every sum along it, is the same on every run
  k_tour_sort_rows<<<gn, kBlock, 0, s>>>(tptr, n, tadj, succ);  // (succ is written below)
  k_tour_fix_rev<<<gn, kBlock, 0, s>>>(tptr, tadj, n, rev);
  k_tour_fix_arcs<<<gm, kBlock, 0, s>>>(h.el_u, h.el_v, tflag, m, tptr, tadj, arc_uv);
  const int ga = grid_for(h, std::max<int64_t>(A, 1));
  k_st_succ<<<ga, kBlock, 0, s>>>(tadj, rev, tptr, tdeg, n, succ);
  k_pc_cut<<<1, 32, 0, s>>>(rev, tptr, tdeg, root, succ, rank);
  const uint64_t* walk = rank_lists(h, succ, tptr + n, rank, s);
  PC_CK(cudaMemsetAsync(flags, 0, sizeof(int32_t) * 4, s));  // bad ids, repeated ids, a cycle, largest depth
  PC_CK(cudaMemsetAsync(tour, 0, sizeof(int32_t) * (size_t)std::max<int64_t>(A, 1), s));
  k_pc_times<<<gm, kBlock, 0, s>>>(h.el_u, h.el_v, h.el_w, tflag, arc_uv, rev, rank.own, walk, tptr, n, m, tin, tout,
                                   wup, tour, flags + 2);
  // the grounded tree solve x = L_T^-1 y (y: a vector, or null for the recovered edges' +-q)
  const int tiles = (int)T;
  const TourArgs ta{tour, A, tin, tout, wup, nullptr, iptr, iedge, ea, qv, E, D, nullptr, nullptr, {}, root, sums};
  auto tree_solve = [&](const double* yin, double* xout, bool last, const double* t_of_z, const Parts& z_sum) {
    TourArgs a = ta;
    a.y = yin;
    a.x = xout;
    a.t = t_of_z;
    a.z_sum = z_sum;
    with_items(A, [&](auto items) {
      constexpr int I = decltype(items)::value;
      if (yin) {
        k_pc_tour_sums<kFlow, I><<<tiles, kTourThreads, 0, s>>>(a);
        k_pc_tour_scan<kFlow, I><<<tiles, kTourThreads, 0, s>>>(a);
      } else {
        k_pc_tour_sums<kFlowEdges, I><<<tiles, kTourThreads, 0, s>>>(a);
        k_pc_tour_scan<kFlowEdges, I><<<tiles, kTourThreads, 0, s>>>(a);
      }
      k_pc_tour_sums<kDrops, I><<<tiles, kTourThreads, 0, s>>>(a);
      if (last) k_pc_tour_scan<kDropsZ, I><<<tiles, kTourThreads, 0, s>>>(a);
      else k_pc_tour_scan<kDrops, I><<<tiles, kTourThreads, 0, s>>>(a);
    });
  };
  // root distances and depths along the tour
  with_items(A, [&](auto items) {
    constexpr int I = decltype(items)::value;
    k_pc_dist<true, I><<<tiles, kTourThreads, 0, s>>>(tour, A, wup, dsums, dist, depth, flags + 3);
    k_pc_dist<false, I><<<tiles, kTourThreads, 0, s>>>(tour, A, wup, dsums, dist, depth, flags + 3);
  });
  // the recovered edges (distinct off-tree canonical ids)
  PC_CK(cudaMemsetAsync(seen, 0, sizeof(int32_t) * std::max<int64_t>(m, 1), s));
  if (k > 0) {
    k_pc_edges<<<gk, kBlock, 0, s>>>(ids, k, m, h.el_u, h.el_v, h.el_w, tflag, ea, eb, ewk, flags);
    k_pc_dups<<<gk, kBlock, 0, s>>>(ids, k, m, seen, flags + 1);
  }
  {
    int32_t hf[4] = {0, 0, 0, 0};
    if (cudaMemcpyAsync(hf, flags, sizeof(hf), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
        cudaStreamSynchronize(s) != cudaSuccess)
      return fail(PDG_E_CUDA);
    if (hf[2]) return fail(PDG_E_NOT_A_TREE);
    if (!exact_range(*h.hsc, hf[3])) return fail(PDG_E_RANGE);
    if (hf[0] || hf[1]) return fail(PDG_E_INVALID_ARG);
  }
  // capacitance matrix C and its inverse
  if (k > 0) {
    const int ends = (int)(2 * k), g2 = grid_for(h, ends);
    int size = 2;
    while (size < ends) size <<= 1;
    PC_CK(cudaFuncSetAttribute(k_pc_sort_ends, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               kSortMax * (int)sizeof(uint64_t)));
    k_pc_ends<<<g2, kBlock, 0, s>>>(ea, eb, tin, root, k, ekey);
    k_pc_sort_ends<<<1, 1024, sizeof(uint64_t) * (size_t)size, s>>>(ekey, ends, size, epos, erank);
    k_pc_gap_ends<<<g2, kBlock, 0, s>>>(epos, depth, ends, gaps);
    k_pc_gap_min<<<grid_for(h, A), kBlock, 0, s>>>(epos, depth, A, ends, gaps);
    k_pc_gap_rows<<<1, 1024, 0, s>>>(gaps, gap_rows, ends);
    k_pc_capacitance<<<grid_for(h, k * k), kBlock, 0, s>>>(gaps, dist, depth, epos, erank, ewk, (int)k, C);
    const int blocks = (int)((k + kSw - 1) / kSw);
    for (int p0 = 0; p0 < k; p0 += kSw) {
      k_pc_sweep_panel<<<(int)((k + 7) / 8), 256, 0, s>>>(C, (int)k, p0, swS, swR, swY);
      k_pc_sweep_update<<<blocks * (blocks + 1) / 2, 256, 0, s>>>(C, (int)k, p0, swS, swR, swY);
    }
    k_pc_sweep_end<<<blocks * (blocks + 1) / 2, 256, 0, s>>>(C, (int)k);
    // incidence lists of the recovered edges, in edge order
    PC_CK(cudaMemsetAsync(icnt, 0, sizeof(int32_t) * n, s));
    PC_CK(cudaMemsetAsync(cur, 0, sizeof(int32_t) * n, s));
    k_pc_inc_count<<<gk, kBlock, 0, s>>>(ea, eb, k, icnt);
    if ((st = scan_excl_i32(h, icnt, iptr, n, nullptr, n))) return fail(st);
    k_pc_inc_fill<<<gk, kBlock, 0, s>>>(ea, eb, k, iptr, cur, iedge);
    // each list in increasing edge order (a fixed summation order); the sorted endpoints' keys are not needed any more
    k_tour_sort_rows<<<gn, kBlock, 0, s>>>(iptr, n, iedge, reinterpret_cast<int32_t*>(ekey));
  }
  // the root's potential (the solves write every other vertex's)
  PC_CK(cudaMemsetAsync(t + root, 0, sizeof(double), s));
  const int gemv_blocks = std::max(1, std::min(h.num_sms * 2, (int)((k + kGemvThreads / 32 - 1) / (kGemvThreads / 32))));
  PC_CK(cudaFuncSetAttribute(k_pc_gemv, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)(sizeof(double) * kPcgMaxEdges)));
  // sums, by block: rz (two, by turns), p . Ap, r . r, and the one for the mean
  const Parts rz[2] = {{parts, kDotBlocks}, {parts + kDotBlocks, kDotBlocks}};
  const Parts pAp{parts + 2 * kDotBlocks, kDotBlocks}, rr{parts + 3 * kDotBlocks, kDotBlocks};
  const Parts sum_b{parts + 4 * kDotBlocks, kDotBlocks}, sum_z{parts + 4 * kDotBlocks, tiles};
  // the host adds up its copy of r . r, in one order
  double* rr_h = h.pcg_host;
  auto rr_norm = [&]() {
    double v = 0.0;
    for (int i = 0; i < kDotBlocks; i++) v += rr_h[i];
    return std::sqrt(v);
  };
  // the preconditioner M(v) -> zout, and v . zout
  auto precond = [&](const double* vin, double* zout, const Parts& dot) {
    if (k > 0) {
      tree_solve(vin, t, false, nullptr, {});
      k_pc_gemv<<<gemv_blocks, kGemvThreads, sizeof(double) * (size_t)k, s>>>(C, t, ea, eb, (int)k, qv);
      tree_solve(nullptr, zout, true, t, sum_z);
    } else {
      tree_solve(vin, zout, true, nullptr, sum_z);
    }
    k_pc_center<<<kDotBlocks, 256, 0, s>>>(zout, n, sum_z, vin, dot);
  };
  // PCG
  k_pc_degw<<<gn, kBlock, 0, s>>>(h.row_ptr, h.w, n, dw);
  PC_CK(cudaMemcpyAsync(bb, b, sizeof(double) * n, cudaMemcpyDeviceToDevice, s));
  k_pc_dot<<<kDotBlocks, 256, 0, s>>>(bb, nullptr, n, sum_b);
  k_pc_center<<<kDotBlocks, 256, 0, s>>>(bb, n, sum_b, nullptr, rr);
  PC_CK(cudaMemsetAsync(x, 0, sizeof(double) * n, s));
  PC_CK(cudaMemcpyAsync(r, bb, sizeof(double) * n, cudaMemcpyDeviceToDevice, s));
  PC_CK(cudaMemcpyAsync(rr_h, rr.part, sizeof(double) * kDotBlocks, cudaMemcpyDeviceToHost, s));
  PC_CK(cudaStreamSynchronize(s));
  const double nb = rr_norm();
  if (!(nb > 0)) {
    *iters = 0;
    *relres = 0.0;
    cleanup();
    return PDG_OK;
  }
  int c = 0;
  precond(r, z, rz[c]);
  if (z0) {  // the preconditioner applied to b' (host copy for the caller)
    PC_CK(cudaMemcpyAsync(z0, z, sizeof(double) * n, cudaMemcpyDeviceToHost, s));
    PC_CK(cudaStreamSynchronize(s));
  }
  PC_CK(cudaMemcpyAsync(p, z, sizeof(double) * n, cudaMemcpyDeviceToDevice, s));
  double rel = 1.0;
  int32_t it = 0;
  // the host learns of a residual while the device is at the next direction (the last one, past convergence, is not
  // used)
  cudaEvent_t seen_rr = nullptr;
  PC_CK(cudaEventCreateWithFlags(&seen_rr, cudaEventDisableTiming));
  bool ok = true;
  for (it = 1; it <= max_iter; it++) {
    k_pc_spmv<<<kDotBlocks, 256, 0, s>>>(h.row_ptr, h.col, h.w, dw, p, n, Ap, pAp);
    k_pc_step<<<kDotBlocks, 256, 0, s>>>(x, r, p, Ap, n, rz[c], pAp, rr);
    ok = cudaMemcpyAsync(rr_h, rr.part, sizeof(double) * kDotBlocks, cudaMemcpyDeviceToHost, s) == cudaSuccess &&
         cudaEventRecord(seen_rr, s) == cudaSuccess;
    if (!ok) break;
    if (it < max_iter) {
      precond(r, z, rz[c ^ 1]);
      k_pc_xpby<<<gn, kBlock, 0, s>>>(p, z, rz[c ^ 1], rz[c], n);
      c ^= 1;
    }
    if (!(ok = cudaEventSynchronize(seen_rr) == cudaSuccess)) break;
    rel = rr_norm() / nb;
    if (hist) hist[it - 1] = rel;
    if (rel <= tol) break;
  }
  cudaEventDestroy(seen_rr);
  if (!ok) return fail(PDG_E_CUDA);
  *iters = std::min(it, max_iter);
  *relres = rel;
  if (cudaGetLastError() != cudaSuccess) return fail(PDG_E_CUDA);
  cleanup();
  return PDG_OK;
}

#undef PC_CK

}  // namespace pdg
