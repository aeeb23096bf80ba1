// The library's host code (handle life cycle, buffers, recovery driver) on the CUDA runtime of fake_cudart.cc: allocations
// fail where a check says so, and what the kernels would report is scripted.  Built and run by tests/test_host_driver.py;
// needs nvcc, no GPU.
#include "pdg_api.cu"

#include <set>

#include "fake_cudart.h"

namespace {

#define CHECK(x)                                                                   \
  do {                                                                             \
    if (!(x)) fake::die("line %d: %s does not hold", __LINE__, #x);                \
  } while (0)

// what the attempts of the following recoveries report
void script(const std::function<void(DevScalars&)>& report) {
  fake::on_copy = [report](void* to, size_t bytes) {
    if (bytes == sizeof(DevScalars)) report(*static_cast<DevScalars*>(to));
  };
}

// what init's kernels would have found in a sound graph
void sound_graph(const std::string& name, void** a) {
  if (fake::named(name, "k_val_parent")) (*static_cast<int64_t**>(a[8]))[0] = 1;  // one root
  if (fake::named(name, "k_gather_rowptr")) {
    const int64_t* row_ptr = *static_cast<const int64_t**>(a[0]);
    const int64_t* vtx_ptr = *static_cast<const int64_t**>(a[1]);
    for (int32_t g = 0; g <= *static_cast<int32_t*>(a[2]); g++) (*static_cast<int64_t**>(a[3]))[g] = row_ptr[vtx_ptr[g]];
  }
}

// a handle over n vertices of `degree` entries each, from host memory
pdg_handle make(int64_t n, int64_t degree, bool use_graph, int* status = nullptr) {
  fake::on_launch = sound_graph;
  fake::on_copy = nullptr;
  std::vector<int64_t> row_ptr(n + 1);
  for (int64_t v = 0; v <= n; v++) row_ptr[v] = v * degree;
  std::vector<int32_t> col(n * degree), parent(n);
  std::vector<double> w(n * degree, 1.0);
  pdg_options o;
  pdg_default_options(&o);
  o.use_graph = use_graph;
  pdg_handle h = nullptr;
  const int st = sparsify_init(&h, n, row_ptr.data(), col.data(), w.data(), parent.data(), PDG_MEM_HOST, &o, nullptr);
  if (status) *status = st;
  else CHECK(st == PDG_OK);
  return h;
}

int recover(pdg_handle h, double alpha, int c = 2) {
  std::vector<int32_t> ids((size_t)h->h.E_off);
  int64_t count = 0;
  return recover_offtree(h, alpha, c, ids.data(), (int64_t)ids.size(), &count, nullptr, PDG_MEM_HOST);
}

// every buffer that the launches of a recovery read or write
void check_buffers(const Handle& h, bool tiers) {
  const size_t R = (size_t)h.Rcap;
  CHECK(R > 0);
  fake::need("cand_idx", h.cand_idx, 4 * R);
  for (int i = 0; i < 2; i++) {
    fake::need("rk", h.rk[i], 8 * R);
    fake::need("rv", h.rv[i], 4 * R);
  }
  fake::need("rank_cand", h.rank_cand, 4 * R);
  fake::need("scan_tmp", h.scan_tmp, 8 * (R + 1));
  fake::need("acc_flag", h.acc_flag, R);
  fake::need("radix_status", h.radix_status, 4);
  for (const void* p : {h.cand_rec, h.join_rec, h.join_probe}) fake::need("records", p, 32 * R);
  fake::need("join_conf", h.join_conf, 32 * R);
  fake::need("join_list", h.join_list, 4 * (size_t)h.join_list_cap);
  CHECK(h.join_slots >= 16 && h.join_list_cap > 0);
  fake::need("join_tab", h.join_tab, (size_t)h.join_slots * kJoinSlotBytes);
  fake::need("join_ranks", h.join_ranks, (size_t)h.join_slots * kJoinInline * 4);
  CHECK(h.list_cap > 0);
  fake::need("list_id", h.list_id, 4 * (size_t)h.list_cap);
  fake::need("list_key", h.list_key, 8 * (size_t)h.list_cap);
  fake::need("scan_status", h.scan_status, 8 * (size_t)h.scan_tiles_cap);
  if (!tiers) return;
  CHECK(h.tier_cap == h.Rcap && h.table_cap > 0 && h.xcap > 0);
  for (const void* p : {(void*)h.lsort_rank, (void*)h.rec_u, (void*)h.rec_v, (void*)h.rec_du, (void*)h.rec_dv,
                        (void*)h.rec_rank, (void*)h.rec_lca, (void*)h.seg_begin, (void*)h.warp_seg, (void*)h.block_seg,
                        (void*)h.big_pos, (void*)h.big_seg, (void*)h.big_chunk, (void*)h.seg_regs, (void*)h.und_list})
    fake::need("tiers", p, 4 * R);
  fake::need("rec_b", h.rec_b, R);
  fake::need("state", h.state, R);
  fake::need("pslot", h.pslot, 32 * R);
  fake::need("reg_slot", h.reg_slot, 16 * R);
  fake::need("ptab", h.ptab, (size_t)h.table_cap);
  fake::need("xtab", h.xtab, 16 * (size_t)h.xcap);
  fake::need("xund1", h.xund1, 16 * (size_t)h.xcap);
}

// Every allocation of a recovery fails in turn; the call says so, and the next one (the same budget, then a smaller
// one) has all its buffers.  `report`: what the recovery's attempts report.
void fail_each(const std::function<void(const Handle&, DevScalars&, int)>& report, bool tiers) {
  for (double next : {0.5, 0.05})
    for (int64_t j = 0;; j++) {
      pdg_handle h = make(2000, 12, false);
      int attempt = 0;
      script([&](DevScalars& d) { report(h->h, d, attempt++); });
      fake::on_launch = [h](const std::string& name, void**) {
        if (fake::named(name, "k_join_insert") || fake::named(name, "k_build_records"))
          check_buffers(h->h, fake::named(name, "k_build_records"));
      };
      fake::fail_from = fake::allocs + j;
      fake::fail_count = 1;
      const int st = recover(h, 0.5);
      const bool failed = fake::allocs > fake::fail_from;
      fake::fail_from = -1;
      CHECK(st == (failed ? PDG_E_OOM : PDG_OK));
      attempt = 0;
      CHECK(recover(h, next) == PDG_OK);
      check_buffers(h->h, tiers);
      sparsifier_free(h);
      CHECK(fake::live.empty());
      if (!failed) break;
    }
}

void oom_join() { fail_each([](const Handle&, DevScalars&, int) {}, false); }

void oom_table() {
  fail_each([](const Handle&, DevScalars& d, int attempt) { d.err = attempt == 0 ? ERR_TABLE : 0; }, false);
}

void oom_tiers() {
  fail_each([](const Handle& h, DevScalars& d, int) { d.err = h.tiered ? 0 : ERR_DENSE; }, true);
}

// a table that could not grow is not asked for at its new size by a call that does without
void oom_table_keeps_size() {
  pdg_handle h = make(2000, 12, false);
  CHECK(recover(h, 0.5) == PDG_OK);
  const int64_t slots = h->h.join_slots;
  int attempt = 0;
  script([&](DevScalars& d) { d.err = attempt++ == 0 ? ERR_TABLE : 0; });
  fake::fail_from = fake::allocs;
  fake::fail_count = 1;
  CHECK(recover(h, 0.5) == PDG_E_OOM);
  fake::fail_from = -1;
  CHECK(recover(h, 0.5) == PDG_OK);
  CHECK(h->h.join_slots == slots);
  sparsifier_free(h);
}

// A captured recovery holds addresses: it is not replayed once its buffers were given back, whatever the sizes of the
// new ones.
void graph_of_old_buffers() {
  pdg_handle h = make(2000, 12, true);
  CHECK(recover(h, 0.1) == PDG_OK && recover(h, 0.1) == PDG_OK);
  CHECK(fake::graphs == 1 && fake::graph_launches == 1);
  const int64_t Rcap = h->h.Rcap;
  fake::fail_from = fake::allocs + 5;  // a larger budget, and memory runs out while its buffers are made
  fake::fail_count = 1;
  CHECK(recover(h, 0.9) == PDG_E_OOM);
  fake::fail_from = -1;
  std::set<void*> taken;  // (the addresses given back are in use elsewhere now)
  for (int i = 0; i < 64; i++) taken.insert(malloc(4096));
  CHECK(recover(h, 0.1) == PDG_OK);
  CHECK(h->h.Rcap == Rcap);
  CHECK(fake::graphs == 2 && fake::graph_launches == 1);
  CHECK(recover(h, 0.1) == PDG_OK);
  CHECK(fake::graphs == 2 && fake::graph_launches == 2);
  sparsifier_free(h);
  for (void* p : taken) free(p);
}

// Memory that is enough for an init whose weights come first is enough for one that may let them come late.
void late_weights_memory() {
  for (int64_t degree : {6, 24, 200}) {
    const int64_t n = (int64_t(1) << 21) / degree;
    fake::no_streams = true;  // no second stream: the weights come first
    fake::peak = 0;
    sparsifier_free(make(n, degree, false));
    const size_t enough = fake::peak;
    fake::no_streams = false;
    for (size_t capacity : {enough, enough + enough / 8, enough + enough / 4, enough + enough / 2, 2 * enough}) {
      fake::capacity = capacity;
      int st = PDG_OK;
      pdg_handle h = make(n, degree, false, &st);
      if (st != PDG_OK) fake::die("degree %d, capacity %zu, enough %zu: status %d", (int)degree, capacity, enough, st);
      sparsifier_free(h);
      CHECK(fake::live.empty());
    }
    fake::capacity = SIZE_MAX;
    const int late = fake::launches("k_edge_weights");
    sparsifier_free(make(n, degree, false));
    CHECK(fake::launches("k_edge_weights") == late + 1);  // with room they do come late
  }
}

// A failed index check ends the recovery; with PDG_DEBUG_BOUNDS set its report reads nothing that is not there: no
// buffers of the tiers after a join, no position the check did not record, no segment that was not made.
void failed_index_check() {
  for (bool tiers : {false, true})
    for (int site : {0, 3})
      for (int64_t pos : {-1ll, 0ll, 64ll * 70, 1ll << 40})
        for (int64_t n : {0, 1, 50}) {
          pdg_handle h = make(2000, 12, false);
          script([&](DevScalars& d) {
            d = DevScalars{};
            d.e_max = INT_MIN;
            if (tiers && !h->h.tiered) {
              d.err = ERR_DENSE;
              return;
            }
            d.err = ERR_BOUNDS;
            d.bounds_site = site;
            d.bounds_pos = pos;
            d.n_cand = d.n_big = n;
            d.n_seg = n / 2;
            d.n_big_seg = n / 3;
          });
          CHECK(recover(h, 0.5) == PDG_E_CUDA);
          CHECK(h->h.stats[11] == site);
          script([](DevScalars&) {});
          sparsifier_free(h);
        }
}

// Budgets from some size on fill the join's cells too much and go to the tiers; the handle remembers that for budgets of
// that size, not for smaller ones, and for the same c.
void tiers_by_budget() {
  pdg_handle h = make(2000, 12, false);
  int joins = 0, tiers = 0;
  fake::on_launch = [&](const std::string& name, void**) {
    joins += fake::named(name, "k_join_insert");
    tiers += fake::named(name, "k_build_records");
  };
  double budget = 0.0;
  script([&](DevScalars& d) { d.err = !h->h.tiered && budget >= 0.4 ? ERR_DENSE : 0; });
  auto run = [&](double b, int c, int want_joins, int want_tiers) {
    budget = b;
    joins = tiers = 0;
    CHECK(recover(h, b, c) == PDG_OK);
    if (joins != want_joins || tiers != want_tiers)
      fake::die("budget %g, c %d: %d joins, %d tiers", b, c, joins, tiers);
  };
  run(0.1, 2, 1, 0);
  run(0.5, 2, 1, 1);  // the join gives up
  run(0.5, 2, 0, 1);  // remembered
  run(0.1, 2, 1, 0);  // a smaller budget never met such cells
  run(0.5, 2, 0, 1);  // still remembered
  run(0.9, 2, 0, 1);  // more candidates, fuller cells
  run(0.4, 2, 1, 1);
  run(0.4, 2, 0, 1);
  run(0.5, 1, 1, 1);  // another c has other cells
  run(0.1, 1, 1, 0);
  sparsifier_free(h);
}

const std::map<std::string, void (*)()> kChecks = {
    {"tiers_by_budget", tiers_by_budget},
    {"failed_index_check", failed_index_check},
    {"late_weights_memory", late_weights_memory},
    {"graph_of_old_buffers", graph_of_old_buffers},
    {"oom_join", oom_join},
    {"oom_table", oom_table},
    {"oom_tiers", oom_tiers},
    {"oom_table_keeps_size", oom_table_keeps_size},
};

}  // namespace

int main(int argc, char** argv) {
  const auto it = argc > 1 ? kChecks.find(argv[1]) : kChecks.end();
  if (it == kChecks.end()) {
    for (const auto& c : kChecks) puts(c.first.c_str());
    return argc > 1 ? 1 : 0;
  }
  it->second();
  return 0;
}
