// Step A1: split the edges of G into tree and off-tree edges (Sec. 2.2: every
// edge of G is either a tree edge or an off-tree edge).
//
// Canonical id of {u, v}, u < v: rank of the CSR entry (u, v) among all
// entries with row < col in row-major order.  The handle keeps the graph as
// its canonical edge list (id order; built once from the CSR by
// build_edge_list at init, endpoints then relabelled in the tree's preorder
// as (a, b), a < b): a parent's label is below its child's, so edge (a, b) is a
// tree edge iff parent[b] == a.  Recoveries make that test where the edge is
// scored: the record gathered for b holds its parent, so telling the edges
// apart costs nothing there, and no off-tree list is written and read again
// (compacting one took 0.068 of 0.45 ms on mesh 128^3, 0.63 of 2.05 ms on
// R-MAT scale 22).  What is left of the step is k_resist.
//
// Edge-list layout: each block owns a contiguous chunk of CSR entries, taken in
// tiles of kTile; each thread reads kItems consecutive entries with vector
// loads.  Two passes: a count pass, then a write pass that places each tile's
// output as one contiguous run.
#include <climits>

#include "pdg_fp.cuh"
#include "pdg_internal.cuh"

namespace pdg {

namespace {

__device__ __forceinline__ int64_t cls_chunk(int64_t nnz, int nb) {
  int64_t c = (nnz + nb - 1) / nb;
  return (c + kTile - 1) / kTile * kTile;
}

// Loads kItems column indices starting at base (base is a multiple of kItems).
__device__ __forceinline__ void load_cols(const int32_t* __restrict__ col, int64_t base, int64_t end,
                                          int32_t (&c)[kItems]) {
  if (base + kItems <= end) {
    const int4* c4 = reinterpret_cast<const int4*>(col + base);
    int4 a = __ldg(c4), b = __ldg(c4 + 1);
    c[0] = a.x; c[1] = a.y; c[2] = a.z; c[3] = a.w;
    c[4] = b.x; c[5] = b.y; c[6] = b.z; c[7] = b.w;
  } else {
#pragma unroll
    for (int i = 0; i < kItems; i++) c[i] = (base + i < end) ? __ldg(col + base + i) : 0;
  }
}

__device__ __forceinline__ void load_weights(const double* __restrict__ w, int64_t base, int64_t end,
                                             double (&x)[kItems]) {
  if (base + kItems <= end) {
    const double2* w2 = reinterpret_cast<const double2*>(w + base);
#pragma unroll
    for (int i = 0; i < kItems / 2; i++) {
      double2 t = __ldg(w2 + i);
      x[2 * i] = t.x;
      x[2 * i + 1] = t.y;
    }
  } else {
#pragma unroll
    for (int i = 0; i < kItems; i++) x[i] = (base + i < end) ? __ldg(w + base + i) : 0.0;
  }
}

// Row of CSR entry p (largest u with row_ptr[u] <= p), found by one warp with
// 32-way splits: about log32(n) dependent loads instead of log2(n).
__device__ __forceinline__ int64_t warp_row_of(const int64_t* __restrict__ row_ptr, int64_t n, int64_t p) {
  const int lane = threadIdx.x & 31;
  int64_t lo = 0, hi = n;  // row_ptr[lo] <= p < row_ptr[hi]
  while (hi - lo > 1) {
    const int64_t step = (hi - lo + 31) / 32;
    const int64_t q = lo + lane * step;
    const bool ok = q < hi && __ldg(row_ptr + q) <= p;
    const int last = 31 - __clz(__ballot_sync(0xffffffffu, ok));  // lane 0 is always ok
    lo += last * step;
    hi = min(hi, lo + step);
  }
  return lo;
}

constexpr int kSpanMax = kTile;  // rows staged per tile (enough when no row is empty)

// Edge-list build (init): every CSR entry with row < col, in row-major order.
// The row starts a tile spans are staged in shared memory, so a thread finds
// its row by a short search there and then follows it incrementally; skewed
// rows cost the same as short ones.
template <bool WRITE>
__global__ void __launch_bounds__(kBlock) k_edge_list(const int64_t* __restrict__ row_ptr,
                                                      const int32_t* __restrict__ col,
                                                      const double* __restrict__ w, int64_t n, int64_t nnz,
                                                      int64_t* __restrict__ cnt_up,
                                                      const int64_t* __restrict__ off_up,
                                                      int32_t* __restrict__ eu, int32_t* __restrict__ ev,
                                                      double* __restrict__ ew) {
  dep_sync();
  __shared__ int64_t sm[kBlock / 32 + 1];
  // row starts of the tile, relative to its first entry and clipped to
  // [-1, kTile + 1]: s_rp[j] = row_ptr[r0 + j] - t0
  __shared__ int16_t s_rp[kSpanMax + 1];
  __shared__ int64_t s_r0;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int64_t chunk = cls_chunk(nnz, gridDim.x);
  const int64_t b0 = (int64_t)blockIdx.x * chunk;
  const int64_t b1 = min(nnz, b0 + chunk);
  int64_t run_up = WRITE ? off_up[blockIdx.x] : 0;
  int64_t tot_up = 0;
  if (b0 < b1 && wid == 0) {
    const int64_t r = warp_row_of(row_ptr, n, b0);
    if (lane == 0) s_r0 = r;
  }
  for (int64_t t0 = b0; t0 < b1; t0 += kTile) {
    const int tlen = (int)min((int64_t)kTile, b1 - t0);
    __syncthreads();  // s_r0 is set; the previous tile's shared reads are done
    const int64_t r0 = s_r0;
    // stage row starts kBlock at a time until they cover the tile
    if (threadIdx.x == 0) s_rp[0] = (int16_t)max(__ldg(row_ptr + r0) - t0, (int64_t)-1);
    int span = 0;
    for (;;) {
      const int j = span + 1 + threadIdx.x;
      const int64_t r = r0 + j;
      const int64_t rel = (r <= n) ? __ldg(row_ptr + r) - t0 : (int64_t)kTile + 1;
      s_rp[j] = (int16_t)min(max(rel, (int64_t)-1), (int64_t)kTile + 1);
      __syncthreads();
      span += kBlock;
      if (s_rp[span] >= tlen || span >= kSpanMax) break;  // uniform
    }
    const bool covered = s_rp[span] >= tlen;  // else (many empty rows): global row_ptr
    const int rel0 = threadIdx.x * kItems;
    int32_t c[kItems];
    double x[kItems];
    int32_t rows[kItems];
    uint32_t is_up = 0;
    if (rel0 < tlen) {
      const int64_t base = t0 + rel0;
      load_cols(col, base, t0 + tlen, c);
      if (WRITE) load_weights(w, base, t0 + tlen, x);
      int64_t u, next;
      if (covered) {
        int lo = 0, hi = span;  // s_rp[lo] <= rel0 < s_rp[hi]
        while (hi - lo > 1) {
          const int mid = (lo + hi) >> 1;
          if (s_rp[mid] <= rel0) lo = mid; else hi = mid;
        }
        u = r0 + lo;
        next = t0 + s_rp[lo + 1];
      } else {
        u = row_of(row_ptr, n, base);
        next = __ldg(row_ptr + u + 1);
      }
#pragma unroll
      for (int i = 0; i < kItems; i++) {
        const int64_t p = base + i;
        if (i < tlen - rel0) {
          while (p >= next) {
            u++;
            next = covered ? t0 + s_rp[u - r0 + 1] : __ldg(row_ptr + u + 1);
          }
          rows[i] = (int32_t)u;
          if (u < c[i]) is_up |= 1u << i;
        }
      }
      if (rel0 + kItems >= tlen) s_r0 = u;  // row of the tile's last entry: the next tile starts there
    }
    const int64_t n_up = __popc(is_up);
    if (!WRITE) {
      tot_up += n_up;
      continue;
    }
    int64_t tile_tot;
    int64_t pos = run_up + block_excl_scan(n_up, sm, &tile_tot);
#pragma unroll
    for (int i = 0; i < kItems; i++) {
      if (is_up & (1u << i)) {
        eu[pos] = rows[i];
        ev[pos] = c[i];
        ew[pos] = x[i];
        pos++;
      }
    }
    run_up += tile_tot;
  }
  if (!WRITE) {
    tot_up = block_sum(tot_up, sm);
    if (threadIdx.x == 0) cnt_up[blockIdx.x] = tot_up;
  }
}

// Recovery, tree edges: r(x) = fl(1/w(x, parent x)) of every label from the
// tree's weights in label order, and the exponent range of these r (it fixes
// the fixed-point scale of step A2).  One stream in, one out; the off-tree
// edges are told apart where they are scored.
__global__ void __launch_bounds__(kBlock) k_resist(const double* __restrict__ wup, int64_t n, double* __restrict__ rtree,
                                                   DevScalars* __restrict__ dsc) {
  dep_sync();
  __shared__ int s_lo, s_hi;
  if (threadIdx.x == 0) {
    s_lo = INT_MAX;
    s_hi = INT_MIN;
  }
  __syncthreads();
  int e_lo = INT_MAX, e_hi = INT_MIN;
  // four labels per thread: their loads, then their reciprocals, overlap
  for (int64_t x = ((int64_t)blockIdx.x * kBlock + threadIdx.x) * 4; x < n; x += (int64_t)gridDim.x * kBlock * 4) {
    double w[4], r[4];
    if (x + 4 <= n) {
      const double2 a = __ldg(reinterpret_cast<const double2*>(wup + x)), b = __ldg(reinterpret_cast<const double2*>(wup + x) + 1);
      w[0] = a.x;
      w[1] = a.y;
      w[2] = b.x;
      w[3] = b.y;
    } else {
#pragma unroll
      for (int i = 0; i < 4; i++) w[i] = x + i < n ? __ldg(wup + x + i) : 0.0;
    }
#pragma unroll
    for (int i = 0; i < 4; i++) {
      bool ok;
      const uint64_t rb = rcp_rn_bits((uint64_t)__double_as_longlong(w[i]), &ok);
      r[i] = w[i] == 0.0 ? 0.0 : ok ? __longlong_as_double((long long)rb) : __drcp_rn(w[i]);  // 0: a root
      if (w[i] != 0.0) {
        const int e = (int)(((uint64_t)__double_as_longlong(r[i]) >> 52) & 0x7ff) - 1023;
        e_lo = min(e_lo, e);
        e_hi = max(e_hi, e);
      }
    }
    if (x + 4 <= n) {
      reinterpret_cast<double2*>(rtree + x)[0] = make_double2(r[0], r[1]);
      reinterpret_cast<double2*>(rtree + x)[1] = make_double2(r[2], r[3]);
    } else {
#pragma unroll
      for (int i = 0; i < 4; i++)
        if (x + i < n) rtree[x + i] = r[i];
    }
  }
  e_lo = __reduce_min_sync(0xffffffffu, e_lo);
  e_hi = __reduce_max_sync(0xffffffffu, e_hi);
  if ((threadIdx.x & 31) == 0) {
    atomicMin(&s_lo, e_lo);
    atomicMax(&s_hi, e_hi);
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    if (s_lo != INT_MAX) atomicMin(&dsc->e_min, s_lo);
    if (s_hi != INT_MIN) atomicMax(&dsc->e_max, s_hi);
  }
}

}  // namespace

int build_edge_list(Handle& h) {
  if (h.nnz == 0) return PDG_OK;
  const int nb = (int)std::max<int64_t>(1, std::min<int64_t>(2048, (h.nnz + kTile - 1) / kTile));
  int64_t* cnt = h.blk_a;
  int64_t* off = h.blk_a + 2560;
  ++h.launches;
  launch_k(h, k_edge_list<false>, nb, kBlock, 0, h.row_ptr, h.col, h.w, h.n, h.nnz, cnt, nullptr, nullptr, nullptr,
           nullptr);
  PDG_CUDA(cudaGetLastError());
  int st = scan_excl_i64(h, cnt, off, nb, nullptr, nb);
  if (st) return st;
  ++h.launches;
  launch_k(h, k_edge_list<true>, nb, kBlock, 0, h.row_ptr, h.col, h.w, h.n, h.nnz, nullptr, off, h.el_u, h.el_v, h.el_w);
  PDG_CUDA(cudaGetLastError());
  return PDG_OK;
}

int step_resist(Handle& h) {
  ++h.launches;
  const int grid = (int)std::max<int64_t>(1, std::min<int64_t>((int64_t)h.num_sms * 8, (h.n + 4 * kBlock - 1) / (4 * kBlock)));
  launch_k(h, k_resist, grid, kBlock, 0, h.wup, h.n, h.rtree, h.dsc);
  PDG_CUDA(cudaGetLastError());
  return PDG_OK;
}

}  // namespace pdg
