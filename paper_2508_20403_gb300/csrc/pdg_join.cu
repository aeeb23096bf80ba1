// Steps A5 + A6 as one join: which earlier candidates can mark which later
// ones, found through coarse cells of the tree, and the greedy resolved over
// exactly those pairs.  The tiers of pdg_accept.cu decide the same sets; they
// remain for candidate sets whose cells are too full for a walk (below).
//
// Cells.  Let M = c + 1.  A marker e = (u, v) of the subtask of LCA l, with
// beta = beta*_e >= 1, enters the cell (Q(u), Q(v)): Q(x) is the ancestor of x
// at depth max(M floor((depth x - c) / M), depth l + 1).  If e marks
// e' = (x, y) with x != l, then x and u meet at some vertex a with
// depth a >= depth u - c and a strictly below l, so Q(u) is an ancestor of a
// and hence of x; and |depth x - depth u| <= c leaves at most three depths for
// Q(u), so e' finds e among at most 3 x 3 cells read off its own ancestors
// (5.4 on average).  An edge e' with x = l is reached only by markers with
// beta = hops(u, l) (or v): those also enter (l, Q(v)) (or (Q(u), l)).  Edges
// are oriented by preorder label, so otherwise one orientation suffices.  A
// cell's key determines its subtask (LCA of the two vertices, which are both
// strictly below it or one of them it), so no grouping of the candidates by
// LCA is needed: everything runs in rank order.
//
// k_join_insert   two lanes per rank: the two ancestor chains, the record of
//                 the exact test (one sector), the cells to probe (one sector),
//                 and the insertion of a marker into its cell.  A cell's slot
//                 (16 bytes, two per sector) holds its key, its count and its
//                 first member; the others go to rows of eight ranks, row
//                 g > 0 in a slot of its own keyed (cell, g), so that readers
//                 compute every address from the count.
// k_join_pairs    a warp per 32 ranks: looks the cells up, queues their earlier
//                 members, tests the queue exactly and leaves every candidate
//                 with the list of the earlier ones that mark it if recovered.
//                 Candidates with none (85 % on a mesh) are recovered at once.
// k_join_settle   a thread per rank waits for the candidates on its list:
//                 recovered when all of them are rejected, rejected as soon as
//                 one is recovered.  Blocks take ranks in order from a ticket,
//                 and a candidate waits only for smaller ranks, so whatever it
//                 waits for is running or done; a chain of k dependent
//                 candidates costs k memory round trips, not k launches.
//                 Every wait is bounded (spin_limit -> ERR_TIMEOUT).
//
// What bounds them: the latency of dependent loads (eight and an atomic in the
// first, two per 32 cells and one per 32 pairs in the second), not bandwidth.
// So: one sector per access, read by one 32-byte load (two 16-byte loads took
// 78 us instead of 42 in k_join_pairs on mesh 128^3); lanes filled from queues
// rather than by candidate; every warp the same number of rounds; and no word
// that all warps add to.
// Measured on one GB300, mesh 128^3, alpha .10, c = 2 (314,617 candidates):
// 34 + 42 + 10 us, where the tiers' grouping by LCA, registrations, probes and
// rounds took 340 us (steps A5 + A6 0.298 ms and three sort passes).  A packed
// batch of 192 graphs, 1.43 M candidates: 125 + 325 + 76 us against 1,157; with
// the 784,789 candidates that its first prefixes hold, 65 + 168 + 41.
// When the tiers are the better ones: cells of thousands of members, whose
// pairs grow with the square (kJoinCellMax, kJoinPairsPer).
#include <algorithm>
#include <climits>

#include "pdg_internal.cuh"

namespace pdg {

namespace {

constexpr uint32_t kNoLabel = 0x3fffffffu;  // labels stay below 2^30 - 1
constexpr int kInline = kJoinInline;        // members per slot
constexpr int kMaxProbe = 1024;             // buckets one insertion may visit
constexpr uint32_t kConfInline = 6;
constexpr uint8_t kUndecided = 0xff;

struct __align__(16) JoinSlot {
  unsigned long long key;
  uint32_t count;  // members of the cell
  uint32_t first;  // its first member: nine cells of ten have no other
};
static_assert(sizeof(JoinSlot) == kJoinSlotBytes, "two slots per sector");

struct JoinArgs {
  const int32_t* rank_cand;
  const int4* cand;      // [2 R], candidates in id order: u, v, LCA, canonical id; score bits
  const int4* up;        // per label: parent, grandparent, great-grandparent, depth
  int4* rec;             // [2 R]: u | beta << 30, anc_1..3(u); v, anc_1..3(v)
  int4* probe;           // [2 R]: cells of u (3), u is the LCA; cells of v (3), LCA
  int4* part;            // per block of k_join_insert: subtasks, lone candidates, largest subtask, registrations
  int32_t* part_cons;    // per block of k_join_pairs: candidates with an earlier marker
  JoinSlot* tab;         // cell table: buckets of two slots, one sector
  uint32_t* ranks;       // [slots][kInline]: the members of a slot but its first
  uint32_t buckets;
  int bits;              // of a label
  uint32_t gen_max;      // largest overflow slot number a key can carry
  uint8_t* acc_flag;     // by rank: 1 recovered, 0 rejected, kUndecided
  uint32_t* conf;        // [8 R] by rank: number of earlier markers, the first kConfInline, the others' place in conf_list
  uint32_t* conf_list;
  int64_t conf_cap;
  int32_t* lca_count;    // [n], zero between attempts: candidates per LCA
  int64_t spin_limit;
};

__device__ __forceinline__ int floor_div(int a, int m) { return (a >= 0 ? a : a - m + 1) / m; }

__device__ __forceinline__ uint64_t cell_key(const JoinArgs& a, uint32_t z1, uint32_t z2) {
  return ((uint64_t)z1 << a.bits) | z2;
}

constexpr uint32_t kNoSlot = 0xffffffffu;

__device__ __forceinline__ uint32_t home_bucket(const JoinArgs& a, uint64_t key) {
  return (uint32_t)__umul64hi(mix64(key), a.buckets);
}

__device__ __forceinline__ uint64_t slot_key(const uint4& x) { return (uint64_t)x.y << 32 | x.x; }

// the slot of `key` in a finished table (its words to `found`), or kNoSlot
__device__ __forceinline__ uint32_t find(const JoinArgs& a, uint64_t key, uint4& found) {
  uint32_t b = home_bucket(a, key);
  for (int p = 0; p < kMaxProbe; p++) {
    uint4 x, y;
    load_sector(a.tab + 2 * (uint64_t)b, x, y);
    found = slot_key(x) == key ? x : y;
    if (slot_key(x) == key) return 2 * b;
    if (slot_key(y) == key) return 2 * b + 1;
    if (slot_key(y) == kEmptyKey) break;  // slots fill in order: the key went no further
    if (++b == a.buckets) b = 0;
  }
  return kNoSlot;
}

// the slot of `key`, claimed if it is new; kNoSlot when the table is too full.
// A bucket's slots are taken in order, so two claims of one key meet.
__device__ __forceinline__ uint32_t claim(const JoinArgs& a, uint64_t key) {
  uint32_t b = home_bucket(a, key);
  for (int p = 0; p < kMaxProbe; p++) {
    JoinSlot* t = a.tab + 2 * (uint64_t)b;
    const unsigned long long x = __ldcg(&t[0].key), y = __ldcg(&t[1].key);
    if (x == key) return 2 * b;
    if (x == kEmptyKey) {
      const unsigned long long old = atomicCAS(&t[0].key, (unsigned long long)kEmptyKey, (unsigned long long)key);
      if (old == kEmptyKey || old == key) return 2 * b;
    }
    if (y == key) return 2 * b + 1;
    if (y == kEmptyKey) {
      const unsigned long long old = atomicCAS(&t[1].key, (unsigned long long)kEmptyKey, (unsigned long long)key);
      if (old == kEmptyKey || old == key) return 2 * b + 1;
    }
    if (++b == a.buckets) b = 0;
  }
  return kNoSlot;
}

// Adds rank r to the cell `key`; returns the members before it (kept below
// kJoinCellMax by an error that sends the attempt to the tiers).  Member 0 of
// a cell is kept in its slot, member p > 0 in the row of ranks of slot
// (p - 1) / kInline of the cell: the cell's own, or one claimed for the pair
// (cell, (p - 1) / kInline).
__device__ __forceinline__ uint32_t join_add(const JoinArgs& a, uint64_t key, uint32_t r, int& err) {
  uint32_t pos = 0;
  for (int turn = 0; turn < 2; turn++) {
    const uint32_t g = pos ? (pos - 1) / kInline : 0;
    const uint32_t s = claim(a, key | ((uint64_t)g << (2 * a.bits)));
    if (s == kNoSlot) {
      err |= ERR_TABLE;
      break;
    }
    if (turn == 0) {
      pos = atomicAdd(&a.tab[s].count, 1u);
      if (pos == 0) {
        a.tab[s].first = r;
        break;
      }
      if (pos > kInline) {
        if ((pos - 1) / kInline <= a.gen_max && pos < kJoinCellMax) continue;
        err |= ERR_DENSE;
        break;
      }
    }
    a.ranks[(uint64_t)s * kInline + (pos - 1) % kInline] = r;
    break;
  }
  return pos;
}

// One endpoint's climb from depth `depth`, never above the LCA's depth dl: its
// ancestors 0..C, the cells that the edge probes on this side (their depths
// l0 > l1 > l2, INT_MAX: none), and the cell it enters (lq).  A label's word
// holds three ancestors, so C words cover the 3 C steps it may take.
template <int C>
struct Climb {
  uint32_t anc[C + 1];
  uint32_t cell[3];
  uint32_t q;
  __device__ __forceinline__ void run(uint32_t x, int4 w, int dl, const int4* __restrict__ up) {
    constexpr int M = C + 1;
    const int depth = w.w;
    int l0 = INT_MAX, l1 = INT_MAX, l2 = INT_MAX, lq = INT_MAX, lo = INT_MAX;
    if (depth > dl) {  // an endpoint on the LCA itself has no cells
      const int top = dl + 1, t = depth / M, t0 = floor_div(depth - 2 * C, M);
      lo = l0 = max(M * t, top);
      if (l0 > top && t - 1 >= t0) lo = l1 = max(M * (t - 1), top);
      if (l1 != INT_MAX && l1 > top && t - 2 >= t0) lo = l2 = max(M * (t - 2), top);
      lq = max(M * floor_div(depth - C, M), top);
    }
    // the climb goes as far as an ancestor or a cell needs it
    const int bottom = max(dl, min(lo, depth - C));
    cell[0] = cell[1] = cell[2] = q = kNoLabel;
    uint32_t cur = x;
#pragma unroll
    for (int s = 0; s <= 3 * C; s++) {
      const int d = depth - s;
      if (s <= C) anc[s] = d >= dl ? cur : kNoLabel;
      if (d == l0) cell[0] = cur;
      if (d == l1) cell[1] = cur;
      if (d == l2) cell[2] = cur;
      if (d == lq) q = cur;
      if (s == 3 * C || d <= bottom) continue;
      if (s > 0 && s % 3 == 0) w = __ldg(up + cur);
      cur = (uint32_t)(s % 3 == 0 ? w.x : s % 3 == 1 ? w.y : w.z);
    }
  }
};

// Candidates per LCA (the subtask counts that the statistics report): a block
// keeps the LCAs it met first, the frequent ones among them, in shared memory,
// so that the thousands of candidates of one LCA become one addition per block.
constexpr int kLcaSlots = 512;

// What the additions to the LCAs' counts tell: the first one of an LCA makes a
// subtask, the last one of the largest its size, and a subtask of one
// candidate stays alone until a second addition.
struct SegStats {
  int n_seg = 0, alone = 0, largest = 0;
  __device__ __forceinline__ void add(int32_t* count, int k) {
    const int before = atomicAdd(count, k);
    n_seg += before == 0 ? 1 : 0;
    alone += before == 0 && k == 1 ? 1 : before == 1 ? -1 : 0;
    largest = max(largest, before + k);
  }
};

// Two lanes per candidate, one per endpoint: half the registers of one lane
// doing both, so twice the climbs in flight.
template <int C>
__global__ void __launch_bounds__(kBlock, 6) k_join_insert(JoinArgs a, DevScalars* dsc) {
  dep_sync();
  __shared__ int32_t s_lca[kLcaSlots];
  __shared__ int32_t s_cnt[kLcaSlots];
  __shared__ int s_stat[4];
  __shared__ unsigned long long s_pairs;
  if (attempt_aborted(dsc)) return;  // the attempt is void
  for (int i = threadIdx.x; i < kLcaSlots; i += kBlock) {
    s_lca[i] = -1;
    s_cnt[i] = 0;
  }
  if (threadIdx.x < 4) s_stat[threadIdx.x] = 0;
  if (threadIdx.x == 0) s_pairs = 0;
  __syncthreads();
  const int64_t N = dsc->n_cand;
  const int lane = threadIdx.x & 31, side = lane & 1;
  unsigned long long pairs = 0;
  int err = 0, regs = 0;
  SegStats seg;
  // warp-uniform loop: 16 candidates per warp
  for (int64_t r0 = ((int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31)) / 2; r0 < N;
       r0 += (int64_t)gridDim.x * blockDim.x / 2) {
    const int64_t r = r0 + lane / 2;
    const bool valid = r < N;
    int32_t l = -1;
    int mine = 0, b = 0;
    uint32_t q = kNoLabel;
    const unsigned vm = __ballot_sync(0xffffffffu, valid);  // both lanes of a pair or neither
    if (valid) {
      const int4 e = a.cand[2 * (int64_t)a.rank_cand[r]];  // labels u < v, their LCA
      l = e.z;
      const uint32_t x = (uint32_t)(side ? e.y : e.x);
      const int4 w = __ldg(a.up + x);
      const int dl = __ldg(&a.up[l].w);
      Climb<C> k;
      k.run(x, w, dl, a.up);
      mine = w.w - dl;
      q = k.q;
      const int other = __shfl_xor_sync(vm, mine, 1);
      b = min(min(mine, other), C);
      a.rec[2 * r + side] =
          make_int4((int)(k.anc[0] | (uint32_t)(side ? 0 : b) << 30), C >= 1 ? (int)k.anc[C >= 1 ? 1 : 0] : (int)kNoLabel,
                    C >= 2 ? (int)k.anc[C >= 2 ? 2 : 0] : (int)kNoLabel,
                    C >= 3 ? (int)k.anc[C >= 3 ? 3 : 0] : (int)kNoLabel);
      a.probe[2 * r + side] =
          make_int4((int)k.cell[0], (int)k.cell[1], (int)k.cell[2], side ? l : (mine == 0 ? 1 : 0));
      if (side == 0) a.acc_flag[r] = C == 0 ? 1 : kUndecided;  // c = 0: a neighbourhood is the edge itself
    }
    if (C > 0) {
      const uint32_t q_other = __shfl_xor_sync(0xffffffffu, q, 1);
      // (Q(u), Q(v)) by the first lane; an endpoint within beta hops of the LCA l also marks edges that end on l
#pragma unroll 1
      for (int k = 0; k < 2; k++) {
        if (!valid || b == 0 || (k == 0 ? side != 0 : mine != b)) continue;
        const uint64_t key = k == 0 ? cell_key(a, q, q_other)
                                    : side ? cell_key(a, q_other, (uint32_t)l) : cell_key(a, (uint32_t)l, q_other);
        pairs += join_add(a, key, (uint32_t)r, err);
        regs++;
      }
    }
    if (valid && side == 0) {
      uint32_t s = (uint32_t)l * 2654435761u >> 23;  // 512 slots
      int t = 0;
      for (; t < 8; t++) {
        const int32_t old = atomicCAS(&s_lca[s], -1, l);
        if (old == -1 || old == l) break;
        s = (s + 1) & (kLcaSlots - 1);
      }
      if (t < 8) atomicAdd(&s_cnt[s], 1);
      else seg.add(a.lca_count + l, 1);
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < kLcaSlots; i += kBlock)
    if (s_cnt[i]) seg.add(a.lca_count + s_lca[i], s_cnt[i]);
  // the block's share of the statistics: a word of its own each (additions of every warp to shared words, about
  // 1 ns each, took a third of this kernel on 3 x 10^5 candidates); the last kernel of the recovery adds them up
  seg.n_seg = __reduce_add_sync(0xffffffffu, seg.n_seg);
  seg.alone = __reduce_add_sync(0xffffffffu, seg.alone);
  seg.largest = __reduce_max_sync(0xffffffffu, seg.largest);
  regs = __reduce_add_sync(0xffffffffu, regs);
  for (int o = 16; o; o >>= 1) pairs += __shfl_down_sync(0xffffffffu, pairs, o);
  if (lane == 0) {
    atomicAdd(&s_stat[0], seg.n_seg);
    atomicAdd(&s_stat[1], seg.alone);
    atomicMax(&s_stat[2], seg.largest);
    atomicAdd(&s_stat[3], regs);
    atomicAdd(&s_pairs, pairs);
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    a.part[blockIdx.x] = make_int4(s_stat[0], s_stat[1], s_stat[2], s_stat[3]);
    if (s_pairs > kJoinPairsBase + kJoinPairsPer * (unsigned long long)s_stat[3]) err |= ERR_DENSE;
  }
  if (err) atomicOr(&dsc->err, err);
}

// hops(x, u) <= b from the ancestors of both: anc_i(x) == anc_j(u), i + j <= b
// (every anc_j(u), j <= b, exists; a missing anc_i(x) equals no label)
template <int C>
__device__ __forceinline__ bool within(const uint32_t (&x)[4], const uint32_t (&u)[4], int b) {
  bool hit = false;
#pragma unroll
  for (int j = 0; j <= C; j++)
#pragma unroll
    for (int i = 0; i + j <= C; i++)
      if (i + j <= b && x[i] == u[j]) hit = true;
  return hit;
}

__device__ __forceinline__ uint8_t load_state(const uint8_t* p) { return *(const volatile uint8_t*)p; }

// The walk, a warp at a time over `per` candidates (32, fewer when there are
// not enough candidates to fill the device).  Three steps, each with every
// lane busy whatever the candidates' shapes: the cells of all of them are
// listed; lanes take cells, look them up and queue their earlier members;
// lanes take queued (candidate, member) pairs and test them exactly.  The
// pairs found are counted per candidate and written as runs of conf_list.
constexpr int kJpWarps = 4;
constexpr int kJpBlocks = 6;              // resident per SM
constexpr int kJpQueue = 256;             // pairs queued before they are tested
constexpr int kJpFound = 512;             // pairs found per round of candidates

struct JoinWarp {
  uint4 rec[64];     // records of the candidates
  uint4 probe[64];
  uint32_t q_rank[kJpQueue + 32 * (kInline + 1)];   // queued pairs: the member
  uint32_t f_rank[kJpFound];
  uint16_t item[32 * 9];                          // candidate << 4 | cell
  uint8_t q_cand[kJpQueue + 32 * (kInline + 1)];    // candidate (5 bits) | turned << 5
  uint8_t f_cand[kJpFound];
  uint32_t count[32], base[32];
  uint32_t t_slot[64], t_count[64];               // cells whose further members are still to be queued
  uint16_t t_item[64];
};

template <int C>
__global__ void __launch_bounds__(32 * kJpWarps, kJpBlocks) k_join_pairs(JoinArgs a, DevScalars* dsc) {
  dep_sync();
  __shared__ JoinWarp s_warp[kJpWarps];
  __shared__ int s_cons;
  if (attempt_aborted(dsc)) return;  // the attempt is void
  const int64_t N = dsc->n_cand;
  const int lane = threadIdx.x & 31;
  const unsigned below = (1u << lane) - 1;
  JoinWarp& sm = s_warp[threadIdx.x >> 5];
  bool full = false;
  int cons = 0;
  const int64_t warp = (int64_t)blockIdx.x * kJpWarps + (threadIdx.x >> 5), warps = (int64_t)gridDim.x * kJpWarps;
  // candidates per round: every warp runs the same number of rounds, and all warps have work when there is little
  const int64_t rounds = (N + 32 * warps - 1) / (32 * warps);
  const int per = (int)max((int64_t)4, (N + warps * rounds - 1) / max(warps * rounds, (int64_t)1));
  for (int64_t r0 = warp * per; r0 < N; r0 += warps * per) {
    const int nc = (int)min((int64_t)per, N - r0);
    __syncwarp();
    int ncell = 0;
    if (lane < nc) {
      uint4 pu, pv, x, y;
      load_sector(a.probe + 2 * (r0 + lane), pu, pv);
      load_sector(a.rec + 2 * (r0 + lane), x, y);
      sm.probe[2 * lane] = pu;
      sm.probe[2 * lane + 1] = pv;
      sm.rec[2 * lane] = x;
      sm.rec[2 * lane + 1] = y;
      // the product of the two sides' cells; an edge with an endpoint on the LCA l probes (l, cell) and (cell, l)
      const int na = pu.w ? 2 : 1 + (pu.y != kNoLabel) + (pu.z != kNoLabel);
      const int nb = 1 + (pv.y != kNoLabel) + (pv.z != kNoLabel);
      ncell = na * nb;
    }
    sm.count[lane] = 0;
    const int incl = warp_incl_scan(ncell);
    const int items = __shfl_sync(0xffffffffu, incl, 31);
    for (int t = 0; t < ncell; t++) sm.item[incl - ncell + t] = (uint16_t)(lane << 4 | t);
    __syncwarp();
    int queued = 0, found = 0;
    // tests the queued pairs; the ones found join the round's list
    auto test_queue = [&]() {
      __syncwarp();
      for (int p0 = 0; p0 < queued; p0 += 32) {
        bool hit = false;
        uint32_t j = 0;
        int cd = 0;
        if (p0 + lane < queued) {
          j = sm.q_rank[p0 + lane];
          cd = sm.q_cand[p0 + lane];
          uint4 p, v;
          load_sector(a.rec + 2 * (int64_t)j, p, v);
          // the other way round for markers found through (cell, l)
          const uint4 x = sm.rec[2 * (cd & 31) + (cd >> 5)], y = sm.rec[2 * (cd & 31) + 1 - (cd >> 5)];
          const uint32_t U[4] = {p.x & kNoLabel, p.y, p.z, p.w}, V[4] = {v.x, v.y, v.z, v.w};
          const uint32_t X[4] = {x.x & kNoLabel, x.y, x.z, x.w}, Y[4] = {y.x & kNoLabel, y.y, y.z, y.w};
          const int b = (int)(p.x >> 30);
          hit = within<C>(X, U, b) && within<C>(Y, V, b);
        }
        const unsigned hm = __ballot_sync(0xffffffffu, hit);
        if (hit) {
          const int at = found + __popc(hm & below);
          if (at < kJpFound) {
            sm.f_rank[at] = j;
            sm.f_cand[at] = (uint8_t)(cd & 31);
            atomicAdd(&sm.count[cd & 31], 1u);
          }
        }
        found += __popc(hm);
      }
      queued = 0;
      __syncwarp();
    };
    // a listed cell: its key, and the candidate that asks (| 32: for the other way round)
    auto cell_of = [&](int it, uint64_t& key, int& cd) {
      const int k = it >> 4, t = it & 15;
      const uint4 qu = sm.probe[2 * k], qv = sm.probe[2 * k + 1];
      const int nb = 1 + (qv.y != kNoLabel) + (qv.z != kNoLabel);
      const int i = nb == 1 ? t : nb == 2 ? t >> 1 : (t * 11) >> 5;  // t / nb
      const int j = t - i * nb;
      const uint32_t zu = qu.w ? qv.w : i == 0 ? qu.x : i == 1 ? qu.y : qu.z;
      const uint32_t zv = j == 0 ? qv.x : j == 1 ? qv.y : qv.z;
      const bool turn = qu.w && i == 1;
      key = turn ? cell_key(a, zv, zu) : cell_key(a, zu, zv);
      cd = k | (turn ? 32 : 0);
    };
    int tasks = 0;  // cells with further members than their first
    for (int i0 = 0; i0 < items; i0 += 32) {
      uint4 e = make_uint4(0, 0, 0, 0);
      uint32_t s = kNoSlot, r = 0;
      int cd = 0, it = 0;
      if (i0 + lane < items) {
        it = sm.item[i0 + lane];
        uint64_t key;
        cell_of(it, key, cd);
        r = (uint32_t)r0 + (cd & 31);
        s = find(a, key, e);
      }
      const bool ask = s != kNoSlot && e.w < r, many = s != kNoSlot && e.z > 1;
      const unsigned am = __ballot_sync(0xffffffffu, ask), mm = __ballot_sync(0xffffffffu, many);
      if (ask) {
        const int at = queued + __popc(am & below);
        sm.q_rank[at] = e.w;
        sm.q_cand[at] = (uint8_t)cd;
      }
      if (many) {
        const int at = tasks + __popc(mm & below);
        sm.t_slot[at] = s;
        sm.t_count[at] = e.z - 1;
        sm.t_item[at] = (uint16_t)it;
      }
      queued += __popc(am);
      tasks += __popc(mm);
      const bool last = i0 + 32 >= items;
      __syncwarp();
      // the further members of 32 such cells, a row of kInline per lane
      while (tasks >= 32 || (last && tasks > 0)) {
        const int nt = min(tasks, 32);
        const int tn = lane < nt ? (int)sm.t_count[lane] : 0;
        const int rows = (tn + kInline - 1) / kInline;
        const int upto = warp_incl_scan(rows);
        const int total = __shfl_sync(0xffffffffu, upto, 31);
        for (int q0 = 0; q0 < total; q0 += 32) {
          const int q = q0 + lane;
          int src = 0;  // the cell whose rows hold row q: the cells before it have at most q rows
#pragma unroll
          for (int b = 16; b; b >>= 1)
            if (__shfl_sync(0xffffffffu, upto, src + b - 1) <= q) src += b;
          src = min(src, 31);
          const int g = q - __shfl_sync(0xffffffffu, upto - rows, src);
          uint32_t m[kInline];
          uint32_t want = 0;
          int cc = 0;
          if (q < total) {
            uint64_t key;
            cell_of(sm.t_item[src], key, cc);
            uint32_t gs = sm.t_slot[src];
            uint4 x;
            if (g > 0) gs = find(a, key | ((uint64_t)g << (2 * a.bits)), x);
            if (gs != kNoSlot) {
              const uint32_t left = sm.t_count[src] - (uint32_t)g * kInline, rr = (uint32_t)r0 + (cc & 31);
              uint4 y;
              load_sector(a.ranks + (uint64_t)gs * kInline, x, y);
              m[0] = x.x;
              m[1] = x.y;
              m[2] = x.z;
              m[3] = x.w;
              m[4] = y.x;
              m[5] = y.y;
              m[6] = y.z;
              m[7] = y.w;
#pragma unroll
              for (int z = 0; z < kInline; z++)
                if (z < left && m[z] < rr) want |= 1u << z;
            }
          }
          const int cnt = __popc(want);
          const int incl = warp_incl_scan(cnt);
          int at = queued + incl - cnt;
#pragma unroll
          for (int z = 0; z < kInline; z++)
            if (want >> z & 1u) {
              sm.q_rank[at] = m[z];
              sm.q_cand[at++] = (uint8_t)cc;
            }
          queued += __shfl_sync(0xffffffffu, incl, 31);
          if (queued >= kJpQueue) test_queue();
        }
        __syncwarp();
        if (lane < tasks - nt) {  // fewer than 32 are left
          sm.t_slot[lane] = sm.t_slot[lane + nt];
          sm.t_count[lane] = sm.t_count[lane + nt];
          sm.t_item[lane] = sm.t_item[lane + nt];
        }
        tasks -= nt;
        __syncwarp();
      }
      if (queued >= kJpQueue || last) test_queue();
    }
    __syncwarp();
    // Each candidate's markers: the first kConfInline beside their number, the rest of long lists as a run of
    // conf_list.  (Only those take an addition to the one shared word: an addition per warp to one address,
    // its result awaited, cost 8 to 10 ns each, 90 of this kernel's 100 us on 3 x 10^5 candidates.)
    const uint32_t mine = sm.count[lane];
    const uint32_t more = mine > kConfInline ? mine - kConfInline : 0;
    const uint32_t upto = warp_incl_scan(more);
    const uint32_t spill = __shfl_sync(0xffffffffu, upto, 31);
    full = full || found > kJpFound;
    unsigned long long base = 0;
    if (spill) {
      if (lane == 0) base = atomicAdd(&dsc->join_conf, (unsigned long long)spill);
      base = __shfl_sync(0xffffffffu, base, 0);
      full = full || base + spill > (unsigned long long)a.conf_cap;
    }
    if (!full) {
      sm.base[lane] = (uint32_t)base + upto - more;
      sm.count[lane] = 0;
      __syncwarp();
      for (int f = lane; f < found; f += 32) {
        const int k = sm.f_cand[f];
        const uint32_t at = atomicAdd(&sm.count[k], 1u);
        if (at < kConfInline) a.conf[8 * (r0 + k) + 1 + at] = sm.f_rank[f];
        else a.conf_list[(uint64_t)sm.base[k] + (at - kConfInline)] = sm.f_rank[f];
      }
    }
    if (lane < nc) {
      if (mine == 0) {
        a.acc_flag[r0 + lane] = 1;
      } else {
        a.conf[8 * (r0 + lane)] = mine;
        if (more) a.conf[8 * (r0 + lane) + 7] = (uint32_t)base + upto - more;
        cons++;
      }
    }
  }
  if (full) atomicOr(&dsc->err, ERR_DENSE);
  if (threadIdx.x == 0) s_cons = 0;
  __syncthreads();
  cons = __reduce_add_sync(0xffffffffu, cons);
  if (lane == 0 && cons) atomicAdd(&s_cons, cons);
  __syncthreads();
  if (threadIdx.x == 0) a.part_cons[blockIdx.x] = s_cons;
}

// Candidates in rank order, a block of them per ticket: a candidate waits only
// for smaller ranks, which are in its own block or in blocks that started
// before it.
__global__ void __launch_bounds__(kBlock) k_join_settle(JoinArgs a, DevScalars* dsc) {
  dep_sync();
  if (attempt_aborted(dsc)) return;  // the attempt is void
  __shared__ unsigned long long s_ticket;
  const int64_t N = dsc->n_cand;
  bool timed_out = false;
  for (;;) {
    __syncthreads();
    if (threadIdx.x == 0) s_ticket = atomicAdd(&dsc->block_ticket, 1ull);
    __syncthreads();
    const int64_t r0 = (int64_t)s_ticket * kBlock;
    if (r0 >= N) break;  // uniform
    const int64_t r = r0 + threadIdx.x;
    bool wait = r < N && a.acc_flag[r] == kUndecided;  // written by itself alone
    uint4 x = make_uint4(0, 0, 0, 0), y = x;
    if (wait) {
      load_sector(a.conf + 8 * r, x, y);
    }
    const uint32_t n = x.x;
    uint32_t m[kConfInline] = {x.y, x.z, x.w, y.x, y.y, y.z};
    uint32_t at = 0;  // markers before this one are rejected
    // a warp's lanes wait together: whatever a lane waits for is another lane or another warp
    for (int64_t spins = 0; __any_sync(0xffffffffu, wait); spins++) {
      if (spins >= a.spin_limit) {
        timed_out = true;
        break;
      }
      if (!wait) continue;
      bool rejected = false, waits = false;
      uint8_t st[kConfInline];
#pragma unroll
      for (int q = 0; q < (int)kConfInline; q++) st[q] = at + q < n ? load_state(a.acc_flag + m[q]) : 0;
#pragma unroll
      for (int q = 0; q < (int)kConfInline; q++) {
        rejected = rejected || st[q] == 1;
        waits = waits || st[q] == kUndecided;
      }
      if (!rejected && !waits) {  // these are rejected: on to the next of a long list
        at += kConfInline;
#pragma unroll
        for (int q = 0; q < (int)kConfInline; q++)
          if (at + q < n) m[q] = a.conf_list[(uint64_t)y.w + (at + q - kConfInline)];
      }
      if (rejected || at >= n) {
        *(volatile uint8_t*)(a.acc_flag + r) = rejected ? 0 : 1;
        wait = false;
      }
    }
  }
  if (timed_out) atomicOr(&dsc->err, ERR_TIMEOUT);
}

template <int C>
int run_join(Handle& h, const JoinArgs& a) {
  auto blocks = [&](int64_t threads, int per_block, int per_sm) {
    return (int)std::max<int64_t>(1, std::min<int64_t>((int64_t)h.num_sms * per_sm, (threads + per_block - 1) / per_block));
  };
  h.join_blocks = blocks(2 * h.Rcap, kBlock, 6);
  ++h.launches;
  launch_k(h, k_join_insert<C>, h.join_blocks, kBlock, 0, a, h.dsc);
  h.join_pair_blocks = 0;
  if constexpr (C > 0) {
    h.join_pair_blocks = blocks(h.Rcap, 4 * kJpWarps, kJpBlocks);  // at least four candidates per warp
    ++h.launches;
    launch_k(h, k_join_pairs<C>, h.join_pair_blocks, 32 * kJpWarps, 0, a, h.dsc);
    ++h.launches;
    launch_k(h, k_join_settle, blocks(h.Rcap, kBlock, 8), kBlock, 0, a, h.dsc);
  }
  PDG_CUDA(cudaGetLastError());
  return PDG_OK;
}

}  // namespace

int step_join(Handle& h, int c) {
  JoinArgs a{};
  a.rank_cand = h.rank_cand;
  a.cand = static_cast<const int4*>(h.cand_rec);
  a.up = static_cast<const int4*>(h.up);
  a.rec = static_cast<int4*>(h.join_rec);
  a.probe = static_cast<int4*>(h.join_probe);
  a.tab = static_cast<JoinSlot*>(h.join_tab);
  a.ranks = h.join_ranks;
  a.buckets = (uint32_t)(h.join_slots / 2);
  a.part = static_cast<int4*>(h.join_part);
  a.part_cons = reinterpret_cast<int32_t*>(a.part + h.num_sms * 8);
  a.bits = 1;
  while ((1ll << a.bits) < h.n) a.bits++;
  // keys use 2 bits + generation; all-ones is the empty key
  const int gen_bits = std::min(64 - 2 * a.bits, 16);
  a.gen_max = (1u << gen_bits) - 2;
  a.acc_flag = h.acc_flag;
  a.conf = h.join_conf;
  a.conf_list = h.join_list;
  a.conf_cap = h.join_list_cap;
  a.lca_count = h.lca_count;
  a.spin_limit = h.opt.spin_limit;
  switch (c) {
    case 0: return run_join<0>(h, a);
    case 1: return run_join<1>(h, a);
    case 2: return run_join<2>(h, a);
    default: return run_join<3>(h, a);
  }
}

}  // namespace pdg
