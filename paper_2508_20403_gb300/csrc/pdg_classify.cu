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
#include <climits>

#include "pdg_fp.cuh"
#include "pdg_internal.cuh"

namespace pdg {

namespace {

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

int step_resist(Handle& h) {
  ++h.launches;
  const int grid = (int)std::max<int64_t>(1, std::min<int64_t>((int64_t)h.num_sms * 8, (h.n + 4 * kBlock - 1) / (4 * kBlock)));
  launch_k(h, k_resist, grid, kBlock, 0, h.wup, h.n, h.rtree, h.dsc);
  PDG_CUDA(cudaGetLastError());
  return PDG_OK;
}

}  // namespace pdg
