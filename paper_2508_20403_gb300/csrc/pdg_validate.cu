// Input validation of sparsify_init / sparsify_batch_init (the problem
// statement of Sec. 2.1 and Algorithm 1's input: a weighted undirected graph
// and a spanning tree of it).  Runs once per handle, outside recovery.
//
// Checks: CSR shape (monotone row_ptr, columns in range, no self loops,
// strictly increasing neighbours), symmetric weights (bitwise), weights in
// [2^-900, 2^900], no edge between two graphs of a batch, parent[] with one
// root per graph whose links are edges of G.  That the links are acyclic, and
// the fixed-point range of the exact root distances, which the largest hop
// depth sets, are checked where the Euler tour of the tree is made (the tree
// layout, the PCG measure).
#include <climits>
#include <cmath>

#include "pdg_internal.cuh"

namespace pdg {

namespace {

__device__ __forceinline__ int32_t graph_of_vertex(const int64_t* __restrict__ vtx_ptr, int32_t G, int64_t v) {
  return G == 1 ? 0 : part_of(vtx_ptr, G, v);
}

__global__ void k_val_rowptr(const int64_t* __restrict__ row_ptr, int64_t n, DevScalars* dsc) {
  for (int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; u < n; u += (int64_t)gridDim.x * blockDim.x)
    if (row_ptr[u] > row_ptr[u + 1]) atomicOr(&dsc->err, ERR_NOT_CSR | ERR_NOT_CSR_ROWS);
}

// Every warp takes kValRun * 32 consecutive entries: one search for the row of
// the first, then 32 entries at a time, each lane finding its row among the
// next 32 row ends (one coalesced load, five shuffles).  Only the entries above
// the diagonal look for their mirror image: distinct ones have distinct images
// below it (rows are strictly increasing), so the matrix is symmetric when all
// are found and there are as many entries below as above (dsc->active counts
// the difference).  Bound by the latency of those searches (eight blocks an SM, 32
// registers, against seven: 150 us, 270): 12.5 M entries of mesh 128^3 take 150
// us; a search for every entry, a thread taking eight in a row, took 260.
// The count of the entries above the diagonal in every chunk goes to the
// canonical edge list, which is made of them.
constexpr int kValRun = 16, kValChunk = 32 * kValRun;

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

// Row of entry p = (round's first entry) + lane, for a round whose first entry lies in `row`: its row lies as many rows
// on as of the next 32 row ends are not beyond it.  *u_end: where that row ends (for p < nnz).
__device__ __forceinline__ int64_t warp_entry_row(const int64_t* __restrict__ row_ptr, int64_t n, int64_t nnz,
                                                  int64_t row, int64_t p, int64_t* u_end) {
  const int lane = threadIdx.x & 31;
  const int64_t end = row + 1 + lane <= n ? row_ptr[row + 1 + lane] : nnz;
  int k = 0;
#pragma unroll
  for (int o = 16; o; o >>= 1)
    if (__shfl_sync(0xffffffffu, end, k + o - 1) <= p) k += o;
  int64_t u = row + k;
  *u_end = __shfl_sync(0xffffffffu, end, k);
  if (p < nnz)
    while (*u_end <= p) *u_end = row_ptr[++u + 1];  // past many empty rows (row_ptr is monotone: checked before)
  return u;
}

// WEIGHTS: all checks at once; else (the weights have not come yet) those of the structure, and the places of the mirror
// images are kept, unless row_ptr was found bad.
template <bool WEIGHTS>
__global__ void __launch_bounds__(kBlock, 8) k_val_entries(const int64_t* __restrict__ row_ptr,
                                                        const int32_t* __restrict__ col,
                                                        const double* __restrict__ w, int64_t n, int64_t nnz,
                                                        const int64_t* __restrict__ vtx_ptr, int32_t G,
                                                        int32_t* __restrict__ up_count,
                                                        uint32_t* __restrict__ mirror, DevScalars* dsc) {
  if (!WEIGHTS && (*(volatile int32_t*)&dsc->err & ERR_NOT_CSR_ROWS)) return;
  __shared__ int s_diff;
  if (threadIdx.x == 0) s_diff = 0;
  __syncthreads();
  const double lo = ldexp(1.0, -900), hi = ldexp(1.0, 900);
  const int lane = threadIdx.x & 31;
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t warps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  int err = 0, diff = 0;
  for (int64_t p0 = warp * kValChunk; p0 < nnz; p0 += warps * kValChunk) {
    int64_t row = warp_row_of(row_ptr, n, p0);  // of the round's first entry
    int up = 0;
    for (int64_t b0 = p0; b0 < min(nnz, p0 + kValChunk); b0 += 32) {
      const int64_t p = b0 + lane;
      const bool in = p < nnz;
      int64_t u_end;
      const int64_t u = warp_entry_row(row_ptr, n, nnz, row, p, &u_end);
      const int32_t v = in ? col[p] : 0;
      int32_t next = __shfl_down_sync(0xffffffffu, v, 1);
      if (in) {
        if (lane == 31 && p + 1 < nnz) next = col[p + 1];
        double x = 0.0;
        if (WEIGHTS) {
          x = w[p];
          if (!(x >= lo && x <= hi)) err |= ERR_BAD_WEIGHT;
        }
        if (v < 0 || v >= n || v == u) {
          err |= ERR_NOT_CSR;
        } else {
          if (p + 1 < u_end && !(next > v)) err |= ERR_NOT_CSR;
          if (graph_of_vertex(vtx_ptr, G, u) != graph_of_vertex(vtx_ptr, G, v)) err |= ERR_CROSS_GRAPH;
          diff += u < v ? 1 : -1;
          if (u < v) {
            up++;
            const int64_t b = row_ptr[v], e = row_ptr[v + 1];
            const int64_t q = lower_bound_i32(col, b, e, (int32_t)u);
            if (q >= e || col[q] != (int32_t)u ||
                (WEIGHTS && __double_as_longlong(w[q]) != __double_as_longlong(x)))
              err |= ERR_NOT_SYMMETRIC;
            else if (!WEIGHTS)
              mirror[p] = (uint32_t)q;
          }
        }
      }
      row = __shfl_sync(0xffffffffu, u, 31);  // (not used after a round that ends the entries)
    }
    up = __reduce_add_sync(0xffffffffu, up);
    if (lane == 0) up_count[p0 / kValChunk] = up;
  }
  if (err) atomicOr(&dsc->err, err);
  diff = __reduce_add_sync(0xffffffffu, diff);
  if (lane == 0 && diff) atomicAdd(&s_diff, diff);
  __syncthreads();
  if (threadIdx.x == 0 && s_diff) atomicAdd((unsigned long long*)&dsc->active, (unsigned long long)(long long)s_diff);
}

// The canonical edge list: every entry above the diagonal in row-major order, which is the entries' order, so a warp
// appends the ones of its chunk (columns in range, as many as counted: validated).  Reads the CSR once and writes the
// list, 250 MB for mesh 128^3: 68 us (with a thread's loads eight entries apart and a second pass over the columns to
// count, 133).
// Without WEIGHTS the places of an edge's two entries are kept for k_edge_weights.
template <bool WEIGHTS>
__global__ void __launch_bounds__(kBlock) k_edge_list(const int64_t* __restrict__ row_ptr,
                                                      const int32_t* __restrict__ col, const double* __restrict__ w,
                                                      int64_t n, int64_t nnz, const int64_t* __restrict__ up_off,
                                                      const uint32_t* __restrict__ mirror, int32_t* __restrict__ eu,
                                                      int32_t* __restrict__ ev, double* __restrict__ ew,
                                                      uint2* __restrict__ place) {
  const int lane = threadIdx.x & 31;
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t warps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t p0 = warp * kValChunk; p0 < nnz; p0 += warps * kValChunk) {
    int64_t row = warp_row_of(row_ptr, n, p0), at = up_off[p0 / kValChunk];
    for (int64_t b0 = p0; b0 < min(nnz, p0 + kValChunk); b0 += 32) {
      const int64_t p = b0 + lane;
      const int32_t v = p < nnz ? col[p] : 0;
      const double x = WEIGHTS && p < nnz ? w[p] : 0.0;
      int64_t u_end;
      const int64_t u = warp_entry_row(row_ptr, n, nnz, row, p, &u_end);
      const bool up = p < nnz && u < v;
      const unsigned b = __ballot_sync(0xffffffffu, up);
      if (up) {
        const int64_t o = at + __popc(b & ((1u << lane) - 1));
        eu[o] = (int32_t)u;
        ev[o] = v;
        if (WEIGHTS) ew[o] = x;
        else place[o] = make_uint2((uint32_t)p, mirror[p]);
      }
      at += __popc(b);
      row = __shfl_sync(0xffffffffu, u, 31);
    }
  }
}

// The edges' weights, once they have come, and their checks: an entry below the diagonal has to be its image's equal,
// bit by bit, so every weight is looked at.
__global__ void __launch_bounds__(kBlock) k_edge_weights(const double* __restrict__ w, const uint2* __restrict__ place,
                                                         int64_t m, double* __restrict__ ew, DevScalars* dsc) {
  const double lo = ldexp(1.0, -900), hi = ldexp(1.0, 900);
  int err = 0;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < m; e += (int64_t)gridDim.x * blockDim.x) {
    const uint2 at = place[e];
    const double x = w[at.x], y = w[at.y];
    if (!(x >= lo && x <= hi) || !(y >= lo && y <= hi)) err |= ERR_BAD_WEIGHT;
    if (__double_as_longlong(x) != __double_as_longlong(y)) err |= ERR_NOT_SYMMETRIC;
    ew[e] = x;
  }
  if (err) atomicOr(&dsc->err, err);
}

// WEIGHTS: also the exponent range of the tree edges' resistances
template <bool WEIGHTS>
__global__ void k_val_parent(const int64_t* __restrict__ row_ptr, const int32_t* __restrict__ col,
                             const double* __restrict__ w, const int32_t* __restrict__ parent, int64_t n,
                             const int64_t* __restrict__ vtx_ptr, int32_t G, DevScalars* dsc,
                             int64_t* __restrict__ roots) {
  int err = 0;
  int lmin = INT_MAX, lmax = INT_MIN;
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x) {
    const int32_t p = parent[v];
    if (p == -1) {
      atomicAdd((unsigned long long*)&roots[graph_of_vertex(vtx_ptr, G, v)], 1ull);
      continue;
    }
    if (p < 0 || p >= n || p == v || graph_of_vertex(vtx_ptr, G, p) != graph_of_vertex(vtx_ptr, G, v)) {
      err |= ERR_NOT_A_TREE;
      continue;
    }
    const int64_t b = row_ptr[v], e = row_ptr[v + 1];
    const int64_t q = lower_bound_i32(col, b, e, p);
    if (q >= e || col[q] != p) {
      err |= ERR_NOT_A_TREE;
      continue;
    }
    if (!WEIGHTS) continue;
    const int ex = resist_exponent((unsigned long long)__double_as_longlong(w[q]));
    lmin = min(lmin, ex);
    lmax = max(lmax, ex);
  }
  if (err) atomicOr(&dsc->err, err);
  if (lmin != INT_MAX) {
    atomicMin(&dsc->e_min, lmin);
    atomicMax(&dsc->e_max, lmax);
  }
}

__global__ void k_val_reset(DevScalars* dsc) {
  dsc->err = 0;
  dsc->e_min = INT_MAX;
  dsc->e_max = INT_MIN;
  dsc->active = 0;
  dsc->max_depth = 0;
}

}  // namespace

static int64_t entry_chunks(const Handle& h) { return (h.nnz + kValChunk - 1) / kValChunk; }

static int entry_grid(const Handle& h) { return grid_for(h, 32 * entry_chunks(h)); }

static int alloc_chunks(Handle& h) {
  int st = device_alloc(h, reinterpret_cast<void**>(&h.up_count), sizeof(int32_t) * (size_t)entry_chunks(h));
  if (!st)
    st = device_alloc(h, reinterpret_cast<void**>(&h.up_off), sizeof(int64_t) * (size_t)(entry_chunks(h) + 1));
  return st;
}

int build_edge_list(Handle& h) {
  if (h.nnz == 0) return PDG_OK;
  const int64_t chunks = entry_chunks(h);
  int st = ensure_scan_status(h, chunks);
  if (st || (st = scan_excl_i32(h, h.up_count, h.up_off, chunks, nullptr, chunks))) return st;
  ++h.launches;
  if (h.w_pending)
    k_edge_list<false><<<entry_grid(h), kBlock, 0, h.stream>>>(h.row_ptr, h.col, nullptr, h.n, h.nnz, h.up_off,
                                                               h.w_mirror, h.el_u, h.el_v, nullptr, h.w_place);
  else
    k_edge_list<true><<<entry_grid(h), kBlock, 0, h.stream>>>(h.row_ptr, h.col, h.w, h.n, h.nnz, h.up_off, nullptr,
                                                              h.el_u, h.el_v, h.el_w, nullptr);
  PDG_CUDA(cudaGetLastError());
  device_release(h, h.up_count);
  device_release(h, h.up_off);
  device_release(h, h.w_mirror);
  h.up_count = nullptr;
  h.up_off = nullptr;
  h.w_mirror = nullptr;
  return PDG_OK;
}

int finish_weights(Handle& h) {
  if (!h.w_pending) return PDG_OK;
  h.w_pending = false;
  h.w_late = true;
  PDG_CUDA(cudaStreamWaitEvent(h.stream, h.ev_join, 0));
  ++h.launches;
  k_edge_weights<<<grid_for(h, h.m), kBlock, 0, h.stream>>>(h.w, h.w_place, h.m, h.el_w, h.dsc);
  PDG_CUDA(cudaGetLastError());
  device_release(h, h.w_place);
  device_release(h, h.w);
  h.w_place = nullptr;
  h.w = nullptr;
  return PDG_OK;
}

// (h.hsc holds the scalars as they were after finish_weights)
int late_weight_status(Handle& h) {
  if (h.hsc->err & ERR_BAD_WEIGHT) return PDG_E_BAD_WEIGHT;
  if (h.hsc->err & ERR_NOT_SYMMETRIC) return PDG_E_NOT_SYMMETRIC;
  return PDG_OK;
}

// The CSR checks alone (spanning-tree generation has no parent array yet).
int validate_csr(Handle& h) {
  const int64_t n = h.n;
  const int grid = grid_for(h, std::max<int64_t>(n, h.nnz));
  auto fetch = [&]() -> bool {
    return cudaMemcpyAsync(h.hsc, h.dsc, sizeof(DevScalars), cudaMemcpyDeviceToHost, h.stream) == cudaSuccess &&
           cudaStreamSynchronize(h.stream) == cudaSuccess;
  };
  k_val_reset<<<1, 1, 0, h.stream>>>(h.dsc);
  k_val_rowptr<<<grid, kBlock, 0, h.stream>>>(h.row_ptr, n, h.dsc);
  if (!fetch()) return check_cuda(cudaGetLastError());
  if (h.hsc->err) return PDG_E_NOT_CSR;  // the entry checks below search rows: only on a monotone row_ptr
  if (h.nnz > 0) {
    if (const int st = alloc_chunks(h)) return st;
    k_val_entries<true><<<entry_grid(h), kBlock, 0, h.stream>>>(h.row_ptr, h.col, h.w, n, h.nnz, h.d_vtx_ptr, h.G,
                                                                h.up_count, nullptr, h.dsc);
  }
  if (!fetch()) return check_cuda(cudaGetLastError());
  int err = h.hsc->err;
  if (h.hsc->active != 0) err |= ERR_NOT_SYMMETRIC;
  if (err & ERR_NOT_CSR) return PDG_E_NOT_CSR;
  if (err & ERR_BAD_WEIGHT) return PDG_E_BAD_WEIGHT;
  if (err & ERR_CROSS_GRAPH) return PDG_E_INVALID_ARG;
  if (err & ERR_NOT_SYMMETRIC) return PDG_E_NOT_SYMMETRIC;
  return PDG_OK;
}

constexpr int PDG_RETRY_WITH_WEIGHTS = 1000;

// The checks that need no weights; PDG_RETRY_WITH_WEIGHTS when one of them fails (but row_ptr's).
static int validate_structure(Handle& h, int grid) {
  k_val_reset<<<1, 1, 0, h.stream>>>(h.dsc);
  k_val_rowptr<<<grid, kBlock, 0, h.stream>>>(h.row_ptr, h.n, h.dsc);
  k_val_entries<false><<<entry_grid(h), kBlock, 0, h.stream>>>(h.row_ptr, h.col, nullptr, h.n, h.nnz, h.d_vtx_ptr, h.G,
                                                               h.up_count, h.w_mirror, h.dsc);
  if (cudaMemcpyAsync(h.hsc, h.dsc, sizeof(DevScalars), cudaMemcpyDeviceToHost, h.stream) != cudaSuccess ||
      cudaStreamSynchronize(h.stream) != cudaSuccess)
    return check_cuda(cudaGetLastError());
  if (h.hsc->err & ERR_NOT_CSR) return PDG_E_NOT_CSR;
  if (h.hsc->err || h.hsc->active != 0) return PDG_RETRY_WITH_WEIGHTS;
  int64_t* roots = nullptr;
  if (cudaMallocAsync((void**)&roots, sizeof(int64_t) * h.G, h.stream) != cudaSuccess) {
    cudaGetLastError();
    return PDG_E_OOM;
  }
  cudaMemsetAsync(roots, 0, sizeof(int64_t) * h.G, h.stream);
  k_val_parent<false><<<grid, kBlock, 0, h.stream>>>(h.row_ptr, h.col, nullptr, h.parent, h.n, h.d_vtx_ptr, h.G, h.dsc,
                                                     roots);
  std::vector<int64_t> roots_h(h.G);
  const bool ok =
      cudaMemcpyAsync(roots_h.data(), roots, sizeof(int64_t) * h.G, cudaMemcpyDeviceToHost, h.stream) == cudaSuccess &&
      cudaMemcpyAsync(h.hsc, h.dsc, sizeof(DevScalars), cudaMemcpyDeviceToHost, h.stream) == cudaSuccess &&
      cudaStreamSynchronize(h.stream) == cudaSuccess;
  cudaFreeAsync(roots, h.stream);
  if (!ok) return check_cuda(cudaGetLastError());
  bool tree = h.hsc->err == 0;
  for (int64_t r : roots_h) tree = tree && r == 1;
  return tree ? PDG_OK : PDG_RETRY_WITH_WEIGHTS;
}

int validate_graph(Handle& h) {
  const int64_t n = h.n;
  const int grid = grid_for(h, std::max<int64_t>(n, h.nnz));
  // read the device scalars back on the handle's stream (no legacy-stream sync)
  auto fetch = [&]() -> bool {
    return cudaMemcpyAsync(h.hsc, h.dsc, sizeof(DevScalars), cudaMemcpyDeviceToHost, h.stream) == cudaSuccess &&
           cudaStreamSynchronize(h.stream) == cudaSuccess;
  };
  if (h.nnz > 0)
    if (const int st = alloc_chunks(h)) return st;
  if (h.w_pending) {  // the structure alone; whatever is wrong with it, the weights may be refused for something else
    const int st = validate_structure(h, grid);
    if (st != PDG_RETRY_WITH_WEIGHTS) return st;
    h.w_pending = false;
    if (cudaStreamWaitEvent(h.stream, h.ev_join, 0) != cudaSuccess) return check_cuda(cudaGetLastError());
  }
  k_val_reset<<<1, 1, 0, h.stream>>>(h.dsc);
  k_val_rowptr<<<grid, kBlock, 0, h.stream>>>(h.row_ptr, n, h.dsc);
  if (!fetch()) return check_cuda(cudaGetLastError());
  if (h.hsc->err) return PDG_E_NOT_CSR;
  if (h.nnz > 0) {
    k_val_entries<true><<<entry_grid(h), kBlock, 0, h.stream>>>(h.row_ptr, h.col, h.w, n, h.nnz, h.d_vtx_ptr, h.G,
                                                                h.up_count, nullptr, h.dsc);
  }
  int64_t* roots = nullptr;
  int st = PDG_OK;
  auto cleanup = [&]() { cudaFreeAsync(roots, h.stream); };
  if (cudaMallocAsync((void**)&roots, sizeof(int64_t) * h.G, h.stream) != cudaSuccess) {
    cudaGetLastError();
    return PDG_E_OOM;
  }
  cudaMemsetAsync(roots, 0, sizeof(int64_t) * h.G, h.stream);
  k_val_parent<true><<<grid, kBlock, 0, h.stream>>>(h.row_ptr, h.col, h.w, h.parent, n, h.d_vtx_ptr, h.G, h.dsc, roots);
  std::vector<int64_t> roots_h(h.G);
  if (cudaMemcpyAsync(roots_h.data(), roots, sizeof(int64_t) * h.G, cudaMemcpyDeviceToHost, h.stream) != cudaSuccess ||
      !fetch()) {
    cleanup();
    return check_cuda(cudaGetLastError());
  }
  int err = h.hsc->err;
  if (h.hsc->active != 0) err |= ERR_NOT_SYMMETRIC;
  for (int64_t r : roots_h)
    if (r != 1) err |= ERR_NOT_A_TREE;
  cleanup();
  if (err & ERR_NOT_CSR) st = PDG_E_NOT_CSR;
  else if (err & ERR_BAD_WEIGHT) st = PDG_E_BAD_WEIGHT;
  else if (err & ERR_CROSS_GRAPH) st = PDG_E_INVALID_ARG;
  else if (err & ERR_NOT_SYMMETRIC) st = PDG_E_NOT_SYMMETRIC;
  else if (err & ERR_NOT_A_TREE) st = PDG_E_NOT_A_TREE;
  return st;
}

}  // namespace pdg
