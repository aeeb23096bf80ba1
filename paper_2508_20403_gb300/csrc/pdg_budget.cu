// Step A7: the recovery budget (Sec. 2.2: recover alpha*|V| edges, one pass).
//
// Recovered flags are indexed by rank, so a prefix count over ranks gives,
// per graph, the order in which the sequential greedy would have recovered
// them.  The first k_g are written out (local canonical ids, recovery order).
// A graph whose prefix held fewer than k_g survivors is marked for a retry
// with a longer prefix unless the prefix already was the whole edge list, in
// which case all survivors are returned (PDG_UNDER_BUDGET).
#include "pdg_internal.cuh"

namespace pdg {

namespace {

// The join's statistics: the shares of its blocks, added up by one block.
struct JoinShares {
  const int4* part;  // subtasks, lone candidates, largest subtask, registrations
  const int32_t* cons;
  int blocks, pair_blocks;  // 0: the tiers have counted
};

__device__ void add_shares(const JoinShares& js, int64_t N, DevScalars* dsc) {
  __shared__ int64_t sm[kBlock / 32 + 1];
  __shared__ int s_max;
  int64_t v[4] = {0, 0, 0, 0};  // subtasks, lone candidates, registrations, constrained
  int mx = 0;
  for (int i = threadIdx.x; i < js.blocks; i += kBlock) {
    const int4 p = js.part[i];
    v[0] += p.x;
    v[1] += p.y;
    mx = max(mx, p.z);
    v[2] += p.w;
  }
  for (int i = threadIdx.x; i < js.pair_blocks; i += kBlock) v[3] += js.cons[i];
  if (threadIdx.x == 0) s_max = 0;
#pragma unroll
  for (int k = 0; k < 4; k++) v[k] = block_sum(v[k], sm);
  atomicMax(&s_max, mx);
  __syncthreads();
  if (threadIdx.x == 0) {
    dsc->n_seg = v[0];
    dsc->n_big = N - v[1];
    dsc->max_seg = s_max;
    dsc->big_regs = v[2];
    dsc->n_constrained = v[3];
    dsc->rounds_used = v[2] > 0 ? 1 : 0;
  }
}

// One pass: each graph's status and count (written by one thread per graph)
// and the output of every recovered candidate within its graph's budget, both
// taken from the prefix count over ranks.
__global__ void __launch_bounds__(kBlock) k_budget_write(
    const uint8_t* __restrict__ acc_flag, const int64_t* __restrict__ scan, const int64_t* __restrict__ cand_ptr,
    int32_t G, const int64_t* __restrict__ kk, const GraphSel* __restrict__ sel, int32_t* __restrict__ gstat,
    int64_t* __restrict__ gcount, const int64_t* __restrict__ out_ptr, const int32_t* __restrict__ rank_cand,
    const int4* __restrict__ cand,
    const int64_t* __restrict__ edge_ptr, DevScalars* __restrict__ dsc, JoinShares js, int32_t* __restrict__ out_ids,
    double* __restrict__ out_scores) {
  dep_sync();
  if (attempt_aborted(dsc)) return;  // the attempt is void
  const int64_t N = dsc->n_cand;
  if (js.blocks && blockIdx.x == gridDim.x - 1) add_shares(js, N, dsc);
  if (N != cand_ptr[G]) return;  // selection overflowed: the host grows and repeats
  const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, nth = (int64_t)gridDim.x * blockDim.x;
  for (int64_t g = tid; g < G; g += nth) {
    const int64_t cnt = scan[cand_ptr[g + 1]] - scan[cand_ptr[g]];
    const int64_t k = kk[g];
    const int64_t c0 = cand_ptr[g], c1 = cand_ptr[g + 1];
    const bool short_does = scan[min(c1, c0 + sel[g].rung)] - scan[c0] >= k;
    gstat[g] = (cnt >= k) ? (short_does ? G_OK_SHORT : G_OK) : (sel[g].take_all ? G_UNDER : G_RETRY);
    gcount[g] = min(cnt, k);
  }
  for (int64_t r = tid; r < N; r += nth) {
    if (!acc_flag[r]) continue;
    const int32_t g = (G == 1) ? 0 : part_of(cand_ptr, G, r);
    const int64_t c0 = scan[cand_ptr[g]], cnt = scan[cand_ptr[g + 1]] - c0, k = kk[g];
    if (cnt < k && !sel[g].take_all) continue;  // the graph is retried with a longer prefix
    const int64_t j = scan[r] - c0;
    if (j >= min(cnt, k)) continue;
    const int4* c = cand + 2 * (int64_t)rank_cand[r];
    const int64_t pos = out_ptr[g] + j;
    out_ids[pos] = (int32_t)(c->w - edge_ptr[g]);
    if (out_scores) out_scores[pos] = __longlong_as_double(*reinterpret_cast<const long long*>(c + 1));
  }
}

}  // namespace

int step_budget(Handle& h, int32_t* out_ids, double* out_scores) {
  const int grid = h.num_sms * 4;
  int st = scan_excl_u8(h, h.acc_flag, h.scan_tmp, &h.dsc->n_cand, h.Rcap);
  if (st) return st;
  ++h.launches;
  const int4* part = static_cast<const int4*>(h.join_part);
  const JoinShares js{part, reinterpret_cast<const int32_t*>(part + h.num_sms * 8), h.tiered ? 0 : h.join_blocks,
                      h.join_pair_blocks};
  launch_k(h, k_budget_write, grid, kBlock, 0, h.acc_flag, h.scan_tmp, h.d_cand_ptr, h.G, h.d_k, h.sel, h.gstat,
           h.gcount, h.d_out_ptr, h.rank_cand, static_cast<const int4*>(h.cand_rec), h.d_edge_ptr, h.dsc, js, out_ids,
           out_scores);
  PDG_CUDA(cudaGetLastError());
  return PDG_OK;
}

}  // namespace pdg
