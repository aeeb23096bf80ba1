// Step A2: tree preprocessing of Algorithm 1 step 1 -- the root distances
// ("dists") and the structure that answers LCA queries (the skip table's
// role), recomputed by every recovery from the tree layout built at init.
//
// Root distances are EXACT: every r(v) = fl(1/w(v, parent v)) is a multiple
// of 2^-S with S = 52 - min_v exponent(r(v)), so D(v) = sum of r on the root
// path is an integer in units of 2^-S, and R_T(u, v) = D(u) + D(v) - 2 D(LCA)
// (Eq. RT) is exact before its single rounding.  Each vertex carries one
// 128-bit word P(v) = D(v) * 2^32 + depth(v); D < 2^96 is checked from the
// exponent range and the maximum depth (PDG_E_RANGE otherwise).
//
// k_tree_sum + k_tree_scan: one prefix sum over the Euler tour.  A down arc
// into v adds word(v) = fixed(r(v)) * 2^32 + 1, an up arc out of v subtracts
// it, so the running sum at v's down arc is P(v).  Integer addition is
// associative: the tiled scan gives the same bits as a sequential walk.
//
// k_rmq_groups + k_rmq_rows: the structure that answers LCA queries.  With
// preorder labels u < v, LCA(u, v) is the SMALLEST parent label among the
// labels (u, v]: all of them lie in the subtree of l = LCA(u, v), whose root
// has its smallest label, and none is l itself, so no parent is below l; and
// the child of l on v's side lies there, so l is among the parents.  So the
// query is a plain range minimum over the 4-byte parent array: inside 32-label
// groups the running minima from both ends (and, for a range inside one group,
// the suffix-minimum mask: bit i of mask[k] set when the parent of entry
// i <= k is below those of all later entries up to k, so the minimum of
// [i, k] stands at the lowest set bit at or above i); over whole groups a
// sparse table, row t the minima of 2^t consecutive groups.
//
// What step A3 gathers of a label is one 32-byte record: P, the two running
// minima, the mask, the parent.  That kernel is bound by the number of
// distinct sectors its lanes touch per edge (one tag lookup each in L1), so
// two records, two table entries and P(l) take the place of nine words.
#include <algorithm>
#include <climits>

#include "pdg_internal.cuh"

namespace pdg {

namespace {

// word(v) of the edge to the parent: fixed(r(v)) * 2^32 + 1, with
// fixed(r) = mant * 2^(e - 52 + S) and S = 52 - e_min
__device__ __forceinline__ u128 edge_word(double r, int e_min, bool range_ok) {
  const uint64_t b = (uint64_t)__double_as_longlong(r);
  const int e = (int)((b >> 52) & 0x7ff) - 1023;
  const uint64_t mant = (b & ((1ull << 52) - 1)) | (1ull << 52);
  const int sh = e - e_min;
  const u128 fixed = (range_ok && sh >= 0 && sh <= 74) ? ((u128)mant << sh) : (u128)0;
  return (fixed << 32) | (u128)1;
}

__device__ __forceinline__ bool range_fits(DevScalars* dsc, int dep_bits) {
  const int e_min = dsc->e_min, e_max = dsc->e_max;
  const bool ok = (e_max == INT_MIN) || (e_max - e_min + 53 + dep_bits <= 96);
  if (blockIdx.x == 0 && threadIdx.x == 0 && !ok) atomicOr(&dsc->err, ERR_RANGE);
  return ok;
}

__device__ __forceinline__ u128 shfl_up_u128(u128 x, int d) {
  const uint64_t lo = __shfl_up_sync(0xffffffffu, (unsigned long long)(uint64_t)x, d);
  const uint64_t hi = __shfl_up_sync(0xffffffffu, (unsigned long long)(uint64_t)(x >> 64), d);
  return ((u128)hi << 64) | lo;
}

__device__ __forceinline__ u128 shfl_xor_u128(u128 x, int d) {
  const uint64_t lo = __shfl_xor_sync(0xffffffffu, (unsigned long long)(uint64_t)x, d);
  const uint64_t hi = __shfl_xor_sync(0xffffffffu, (unsigned long long)(uint64_t)(x >> 64), d);
  return ((u128)hi << 64) | lo;
}

__device__ __forceinline__ u128 warp_incl_scan_u128(u128 x) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const u128 y = shfl_up_u128(x, d);
    if (lane >= d) x += y;
  }
  return x;
}

// The tour is scanned in tiles of 256 threads x 8 arcs, reduce-then-scan:
// k_tree_sum adds each tile's arcs, k_tree_scan adds up the sums of the
// tiles before its own (every block for itself: a few loads per thread,
// no serial pass over the tiles) and rescans its tile from that prefix,
// writing the vertices.  No tile waits on another (a chained scan would
// have to pass the running prefix through every tile in order).
constexpr int kTsThreads = 256;
constexpr int kTsItems = 8;
constexpr int kTsTile = kTsThreads * kTsItems;

struct TreeScanArgs {
  const int32_t* tour;
  int64_t A;
  const double* rtree;
  int dep_bits;
  DevScalars* dsc;
  u128* rec;   // a label's record: P, then the range-minimum words
  u128* tsum;  // [tiles] tile sums
};

// the tile's arcs of this thread (INT_MIN past the end) and the r of their vertices
__device__ __forceinline__ void load_arcs(const TreeScanArgs& a, int64_t base, int32_t (&arc)[kTsItems],
                                          double (&r)[kTsItems]) {
  if (base + kTsItems <= a.A) {
    const int4* p4 = reinterpret_cast<const int4*>(a.tour + base);
    const int4 x = __ldg(p4), y = __ldg(p4 + 1);
    arc[0] = x.x; arc[1] = x.y; arc[2] = x.z; arc[3] = x.w;
    arc[4] = y.x; arc[5] = y.y; arc[6] = y.z; arc[7] = y.w;
  } else {
#pragma unroll
    for (int i = 0; i < kTsItems; i++) arc[i] = (base + i < a.A) ? __ldg(a.tour + base + i) : INT_MIN;
  }
#pragma unroll
  for (int i = 0; i < kTsItems; i++) {
    const int32_t x = arc[i] >= 0 ? arc[i] : ~arc[i];
    r[i] = (arc[i] != INT_MIN) ? __ldg(a.rtree + x) : 0.0;
  }
}

// +word(x) for the down arc into x, -word(x) for the up arc out of x
__device__ __forceinline__ u128 arc_word(int32_t arc, double r, int e_min, bool range_ok) {
  if (arc == INT_MIN) return 0;
  const u128 w = edge_word(r, e_min, range_ok);
  return arc >= 0 ? w : (u128)0 - w;
}

__device__ __forceinline__ u128 block_sum_u128(u128 x, u128* s_warp) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int d = 16; d; d >>= 1) x += shfl_xor_u128(x, d);
  if (lane == 0) s_warp[wid] = x;
  __syncthreads();
  u128 t = 0;
  for (int w = 0; w < (int)(blockDim.x >> 5); w++) t += s_warp[w];
  __syncthreads();
  return t;
}

__global__ void __launch_bounds__(kTsThreads) k_tree_sum(TreeScanArgs a) {
  dep_sync();
  __shared__ u128 s_warp[kTsThreads / 32];
  const bool range_ok = range_fits(a.dsc, a.dep_bits);
  const int e_min = a.dsc->e_min;
  const int64_t t = blockIdx.x;
  int32_t arc[kTsItems];
  double r[kTsItems];
  load_arcs(a, t * kTsTile + (int64_t)threadIdx.x * kTsItems, arc, r);
  u128 s = 0;
#pragma unroll
  for (int i = 0; i < kTsItems; i++) s += arc_word(arc[i], r[i], e_min, range_ok);
  const u128 tot = block_sum_u128(s, s_warp);
  if (threadIdx.x == 0) a.tsum[t] = tot;
}

__global__ void __launch_bounds__(kTsThreads, 4) k_tree_scan(TreeScanArgs a) {
  dep_sync();
  __shared__ u128 s_warp[kTsThreads / 32];
  __shared__ u128 s_pre[kTsThreads / 32];
  const bool range_ok = range_fits(a.dsc, a.dep_bits);
  const int e_min = a.dsc->e_min;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int64_t t = blockIdx.x;
  int32_t arc[kTsItems];
  double r[kTsItems];
  load_arcs(a, t * kTsTile + (int64_t)threadIdx.x * kTsItems, arc, r);
  u128 s = 0;
#pragma unroll
  for (int i = 0; i < kTsItems; i++) s += arc_word(arc[i], r[i], e_min, range_ok);
  const u128 incl = warp_incl_scan_u128(s);
  if (lane == 31) s_warp[wid] = incl;
  __syncthreads();
  // the tile's prefix: the sums of all earlier tiles, added up by this block itself (loads four deep)
  u128 pre[4] = {0, 0, 0, 0};
  for (int64_t i = threadIdx.x; i < t; i += 4 * kTsThreads) {
#pragma unroll
    for (int k = 0; k < 4; k++) {
      const int64_t j = i + (int64_t)k * kTsThreads;
      if (j < t) {
        const ulonglong2 q = __ldg(reinterpret_cast<const ulonglong2*>(a.tsum + j));
        pre[k] += ((u128)q.y << 64) | q.x;
      }
    }
  }
  u128 p = block_sum_u128(pre[0] + pre[1] + pre[2] + pre[3], s_pre);
  for (int w = 0; w < wid; w++) p += s_warp[w];
  p += incl - s;  // prefix of every arc before this thread's first
#pragma unroll
  for (int i = 0; i < kTsItems; i++) {
    if (arc[i] == INT_MIN) continue;
    p += arc_word(arc[i], r[i], e_min, range_ok);
    if (arc[i] >= 0) a.rec[2 * (int64_t)arc[i]] = p;  // the down arc into x: P(x)
  }
}

// One block takes 256 groups of 32 labels: a warp loads 32 of them (coalesced),
// its lanes build one group's masks each from registers (mask[k] =
// (mask[k-1] & {j < k : parent j < parent k}) | bit k, 31 comparisons, no
// data-dependent step), then the warp walks the groups with a lane per label
// for the running minima, so that the records leave as whole runs.  The first
// rows of the sparse table, up to windows of 256 groups, come from the block's
// minima and those of the 256 groups after them, which it recomputes (one
// warp-wide minimum per group) rather than wait for another block.  Padding
// past the last label is larger than any parent.
constexpr int kRmqThreads = 256;
constexpr int kRmqGroups = 256;  // groups per block
constexpr int kRmqRow0 = 8;      // rows 0 .. kRmqRow0 are built with the groups

struct RmqSmem {
  int32_t p[kRmqGroups][33];   // parents, a padded row per group
  uint32_t m[kRmqGroups][33];  // masks
  int32_t row[2][2 * kRmqGroups];
};

__global__ void __launch_bounds__(kRmqThreads) k_rmq_groups(const int32_t* __restrict__ parent, int64_t n, int64_t n1,
                                                            int4* __restrict__ rec, int32_t* __restrict__ table,
                                                            int rows) {
  dep_sync();
  extern __shared__ __align__(16) unsigned char rmq_smem[];
  RmqSmem& sm = *reinterpret_cast<RmqSmem*>(rmq_smem);
  const int lane = threadIdx.x & 31, w0 = threadIdx.x & ~31;  // the warp's first group
  const int64_t g0 = (int64_t)blockIdx.x * kRmqGroups;
  int32_t halo[32];  // the block after this one: this warp's share of its groups
#pragma unroll
  for (int j = 0; j < 32; j++) {
    const int64_t x = (g0 + w0 + j) * 32 + lane;
    sm.p[w0 + j][lane] = x < n ? __ldg(parent + x) : INT_MAX;
  }
  if (rows > 1) {
#pragma unroll
    for (int j = 0; j < 32; j++) {
      const int64_t x = (g0 + kRmqGroups + w0 + j) * 32 + lane;
      halo[j] = x < n ? __ldg(parent + x) : INT_MAX;
    }
#pragma unroll
    for (int j = 0; j < 32; j++) {
      const int32_t m = __reduce_min_sync(0xffffffffu, halo[j]);
      if (lane == j) sm.row[0][kRmqGroups + w0 + j] = m;
    }
  }
  __syncwarp();
  {
    int32_t v[32];
#pragma unroll
    for (int k = 0; k < 32; k++) v[k] = sm.p[w0 + lane][k];
    uint32_t mk = 0;
#pragma unroll
    for (int k = 0; k < 32; k++) {
      uint32_t below = 0;
#pragma unroll
      for (int j = 0; j < k; j++) below |= (v[j] < v[k] ? 1u : 0u) << j;
      mk = (mk & below) | (1u << k);
      sm.m[w0 + lane][k] = mk;
    }
  }
  __syncwarp();
#pragma unroll 4
  for (int j = 0; j < 32; j++) {
    const int64_t x = (g0 + w0 + j) * 32 + lane;
    const int32_t p = sm.p[w0 + j][lane];
    int32_t pre = p, suf = p;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int32_t a = __shfl_up_sync(0xffffffffu, pre, o), b = __shfl_down_sync(0xffffffffu, suf, o);
      if (lane >= o) pre = min(pre, a);
      if (lane + o < 32) suf = min(suf, b);
    }
    const int32_t after = __shfl_down_sync(0xffffffffu, suf, 1);  // the entries after this one
    if (x < n) rec[2 * x + 1] = make_int4(pre, lane < 31 ? after : INT_MAX, (int)sm.m[w0 + j][lane], p);
    if (lane == 31) sm.row[0][w0 + j] = pre;
  }
  __syncthreads();
  int cur = 0;
  for (int t = 0; t < rows && t <= kRmqRow0; t++) {
    if (t > 0) {
      const int o = 1 << (t - 1);
      for (int i = threadIdx.x; i < 2 * kRmqGroups; i += kRmqThreads)
        sm.row[cur ^ 1][i] = min(sm.row[cur][i], i + o < 2 * kRmqGroups ? sm.row[cur][i + o] : INT_MAX);
      cur ^= 1;
      __syncthreads();
    }
    const int64_t g = g0 + threadIdx.x;
    if (g < n1) table[(int64_t)t * n1 + g] = sm.row[cur][threadIdx.x];
  }
}

// Rows t0 + 1 .. t0 + kRmqStep of the sparse table from row t0: row t0 + s at i
// is the minimum of row t0 at i, i + 2^t0, .. (2^s of them), so each further
// row adds coalesced loads of row t0 to the minimum of the row before.
constexpr int kRmqStep = 5;

__global__ void __launch_bounds__(kBlock) k_rmq_rows(int32_t* __restrict__ table, int64_t n1, int t0, int rows) {
  dep_sync();
  const int32_t* base = table + (int64_t)t0 * n1;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n1; i += (int64_t)gridDim.x * blockDim.x) {
    int32_t m = base[i];
#pragma unroll
    for (int s = 1; s <= kRmqStep; s++) {
      if (t0 + s >= rows) break;
#pragma unroll
      for (int j = 1 << (s - 1); j < 1 << s; j++) {
        const int64_t k = i + ((int64_t)j << t0);
        if (k < n1) m = min(m, base[k]);
      }
      table[(int64_t)(t0 + s) * n1 + i] = m;
    }
  }
}

}  // namespace

// the range-minimum build's shared memory, granted once per process (first asked at init, outside any
// stream capture; thread-safe initialisation)
static cudaError_t rmq_smem_attr() {
  static const cudaError_t e =
      cudaFuncSetAttribute(k_rmq_groups, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(RmqSmem));
  return e;
}

int step_tree(Handle& h) {
  int dep_bits = 0;
  while ((1ll << dep_bits) <= h.max_depth) dep_bits++;
  if (h.A > 0) {
    const int64_t tiles = (h.A + kTsTile - 1) / kTsTile;
    TreeScanArgs a{h.tour, h.A, h.rtree, dep_bits, h.dsc, static_cast<u128*>(h.rec), h.ts_sum};
    ++h.launches;
    launch_k(h, k_tree_sum, (int)tiles, kTsThreads, 0, a);
    ++h.launches;
    launch_k(h, k_tree_scan, (int)tiles, kTsThreads, 0, a);
    PDG_CUDA(cudaGetLastError());
  }
  PDG_CUDA(rmq_smem_attr());
  const int64_t n1 = (h.n + 31) / 32;
  ++h.launches;
  launch_k(h, k_rmq_groups, (int)((n1 + kRmqGroups - 1) / kRmqGroups), kRmqThreads, sizeof(RmqSmem), h.parent, h.n, n1,
           static_cast<int4*>(h.rec), h.rmq_table, h.rmq_rows);
  for (int t0 = kRmqRow0; t0 + 1 < h.rmq_rows; t0 += kRmqStep) {
    ++h.launches;
    launch_k(h, k_rmq_rows, grid_for(h, n1), kBlock, 0, h.rmq_table, n1, t0, h.rmq_rows);
  }
  PDG_CUDA(cudaGetLastError());
  return PDG_OK;
}

// the tree scan's work space for a tour of A arcs (tile sums)
int tree_scan_workspace(Handle& h) {
  PDG_CUDA(rmq_smem_attr());
  const int64_t tiles = std::max<int64_t>((h.A + kTsTile - 1) / kTsTile, 1);
  return device_alloc(h, (void**)&h.ts_sum, sizeof(u128) * (size_t)tiles);
}

}  // namespace pdg
