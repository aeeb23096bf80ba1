// Step A3: score every off-tree edge (Algorithm 1 step 1: LCA_query,
// distance_query, compute_resistance), telling it from the tree edges by the
// parent in the record of its larger label.
//
//   l   = LCA_T(u, v): with preorder labels u < v, the smallest parent among the
//         labels (u, v], one range-minimum query (pdg_tree.cu)
//   R_T = D(u) + D(v) - 2 D(l)                       (Eq. RT), exact integer
//         then ONE round-to-nearest-even conversion to FP64
//   score = fl(w * R_T) (STRETCH) or R_T (RESISTANCE)
//
// Two dependent rounds of gathers per edge: the records of u and v (P, the
// partial groups' minima, the mask) with the two table entries that cover the
// groups between them, all addressed by (u, v) alone; then P(l).  The
// conversion runs on the integer pipes (pdg_fp.cuh); the product is one FP64
// multiply, which the FP64 pipe takes in fewer issue slots than an integer
// version of it.  The edges and the results are streamed past L2 (evict first):
// the records should stay there.
//
// The score is not negative, so its IEEE bit pattern read as an unsigned
// integer orders like the score itself; key[id] stores those bits + 1 for the
// selection and sort steps, and 0 for a tree edge.
#include <algorithm>

#include "pdg_fp.cuh"
#include "pdg_internal.cuh"

namespace pdg {

namespace {


struct ScoreArgs {
  const int32_t* eu;
  const int32_t* ev;
  const double* ew;
  const uint4* rec;       // [2 n]: P; minimum of the group's parents up to the label, after it, mask, parent
  const int32_t* parent;
  const int32_t* table;   // [rows][n1]
  int64_t n1;
  int S;
  int score_mode;
  uint32_t n;
  int* err;
  uint64_t* key;
  int32_t* lca;
  uint32_t* hist;  // nullable: the first-level selection histogram (key >> 52) of a single graph
};

__device__ __forceinline__ void score_edge(const ScoreArgs& A, int64_t i, uint32_t* s_hist) {
  const uint32_t u = (uint32_t)__ldcs(A.eu + i), v = (uint32_t)__ldcs(A.ev + i);  // preorder labels, u < v
  uint4 pu, mu, pv, mv;
  load_sector(A.rec + 2 * (uint64_t)u, pu, mu);
  load_sector(A.rec + 2 * (uint64_t)v, pv, mv);
  if (mv.w == u) {  // a tree edge
    __stcs(A.key + i, (uint64_t)0);
    return;
  }
  int32_t l;
  const uint32_t gu = u >> 5, gv = v >> 5;
  if (gu == gv) {  // (u, v] inside one group: the lowest mask bit after u
    const uint32_t o = (u & 31u) + 1;
    l = __ldg(A.parent + ((v & ~31u) | (o + __ffs(mv.z >> o) - 1)));
  } else {
    l = min((int32_t)mu.y, (int32_t)mv.x);
    if (gv - gu > 1) {  // the groups strictly between
      const int t = 31 - __clz(gv - gu - 1);
      const int32_t* row = A.table + t * A.n1;
      l = min(l, min(__ldg(row + gu + 1), __ldg(row + gv - (1u << t))));
    }
  }
  if ((uint32_t)l >= A.n) {  // cannot happen for a valid layout: report instead of reading out of range
    atomicOr(A.err, ERR_BOUNDS);
    l = (int32_t)u;
  }
  const uint4 pl = __ldg(A.rec + 2 * (uint64_t)(uint32_t)l);
  auto word = [](const uint4& q) { return (u128)((uint64_t)q.w << 32 | q.z) << 64 | ((uint64_t)q.y << 32 | q.x); };
  const u128 r_fixed = (word(pu) >> 32) + (word(pv) >> 32) - ((word(pl) >> 32) << 1);
  const uint64_t rb = fixed_hl_to_bits((uint64_t)(r_fixed >> 64), (uint64_t)r_fixed, A.S);  // below 2^97
  uint64_t sb = rb;
  if (A.score_mode != PDG_SCORE_RESISTANCE)  // one IEEE multiply, rounded to nearest-even
    sb = (uint64_t)__double_as_longlong(__dmul_rn(__ldcs(A.ew + i), __longlong_as_double((long long)rb)));
  sb++;
  __stcs(A.key + i, sb);
  __stcs(A.lca + i, l);
  if (s_hist) atomicAdd(&s_hist[sb >> 52], 1u);
}

// Blocks take tiles of the edge list in order, `tile` edges each: lists that
// one wave of blocks covers are split evenly among them; longer ones are cut
// into tiles of kScoreTile edges, which the hardware hands out in order as
// blocks retire.  The edges in flight then stay a narrow window of the list,
// so the records being gathered (those of a few graphs of a packed batch) stay
// in L2 however long the list is, and no warp draws tickets from one word.
// Tiles of 4096 edges: 192 packed graphs 0.285 ms (8192: 0.36, 16384: 0.51).
// Eight blocks per SM (32 registers): 5 % ahead of six on a mesh.  Measured with
// the tree edges skipped here: mesh 128^3 0.103 ms, R-MAT scale 22 0.815 ms,
// 192 packed graphs 0.331 ms, where a compaction of the off-tree edges and the
// scoring of the list took 0.135, 1.46 and 0.58 ms (queueing the off-tree edges
// of a warp so that every lane scores costs a gather more per edge: slower on
// all of them, 1.27 ms on R-MAT).
constexpr int64_t kScoreTile = 4096;
constexpr int kScoreBlocks = 8;

__global__ void __launch_bounds__(kBlock, kScoreBlocks) k_score(ScoreArgs A, int64_t m, int64_t tile,
                                                                const DevScalars* __restrict__ dsc) {
  dep_sync();
  __shared__ uint32_t s_hist[kSelBins];
  uint32_t* sh = A.hist ? s_hist : nullptr;  // uniform over the grid
  if (sh) {
    for (int i = threadIdx.x; i < kSelBins; i += blockDim.x) sh[i] = 0;
    __syncthreads();
  }
  A.S = 52 - dsc->e_min;
  const int64_t i0 = (int64_t)blockIdx.x * tile, i1 = min(m, i0 + tile);
  for (int64_t i = i0 + threadIdx.x; i < i1; i += kBlock) score_edge(A, i, sh);
  if (sh) {
    __syncthreads();
    for (int i = threadIdx.x; i < kSelBins; i += blockDim.x)
      if (sh[i]) atomicAdd(&A.hist[i], sh[i]);
  }
}

}  // namespace

int step_score(Handle& h, int score_mode) {
  if (h.m == 0) return PDG_OK;
  ++h.launches;
  ScoreArgs A{};
  A.eu = h.el_u;
  A.ev = h.el_v;
  A.ew = h.el_w;
  A.rec = static_cast<const uint4*>(h.rec);
  A.parent = h.parent;
  A.table = h.rmq_table;
  A.n1 = (h.n + 31) / 32;
  A.score_mode = score_mode;
  A.n = (uint32_t)h.n;
  A.err = &h.dsc->err;
  A.key = h.key;
  A.lca = h.lca;
  A.hist = h.fuse_hist ? h.hist : nullptr;
  const int64_t wave = (int64_t)h.num_sms * kScoreBlocks;
  const int64_t even = ((h.m + wave - 1) / wave + kBlock - 1) / kBlock * kBlock;
  const int64_t tile = std::min(even, kScoreTile);
  launch_k(h, k_score, (int)((h.m + tile - 1) / tile), kBlock, 0, A, h.m, tile, h.dsc);
  PDG_CUDA(cudaGetLastError());
  return PDG_OK;
}

}  // namespace pdg
