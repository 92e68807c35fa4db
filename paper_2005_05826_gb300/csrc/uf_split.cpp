// uf_split.cpp -- which branches of a call run through the dense stripe
// kernels and which are scattered pair by pair (uf_sparse.cu), by a cost
// model of the two paths on GB300; plus the count-row lists the split
// needs and a per-tree cache of splits.
#include "uf_runtime.h"

namespace ufg {
namespace rt {

double sparse_regions(const BatchJob &J, double acc_bytes) {
  const double budget = (double)J.region_bytes;
  if (J.tabs.size() != 1 || acc_bytes <= budget) return 1.0;
  return std::ceil(acc_bytes / budget);
}

bool tile_scatter(const BatchJob &J, int acc, bool fixed) {
  if (J.tabs.size() != 1 || !fixed || acc != ACC_MIN || kind_of(J.method) != EMB_SCALED) return false;
  const int64_t n = J.tabs[0].table->n;
  return n >= TILE_MIN_SAMPLES && n <= TILE_MAX_SAMPLES;
}

int64_t tile_least(int64_t n) {
  // a listed row costs a look at its offsets per tile, a direct one an atomic
  // per pair: both over the full stripe range, so that a range call splits
  // the rows as the full run does (FP64 lists have a grid of their own)
  const double full = 0.5 * (double)n * (double)n;
  const double rate = full * 16.0 <= 64e6 ? 1.15e11 : 1.25e10;
  const double row_cost = full / (TILE_I * TILE_J) * 4e-13;
  return std::max<int64_t>(SPARSE_SMALL_ENTRIES + 1,
                           std::min<int64_t>(1024, (int64_t)std::sqrt(2.0 * rate * row_cost)));
}

namespace {

// Per branch v the count entries of table t under v are the CSC run of v's
// tips, ub_t(v) = col_ptr_t[tip_hi] - col_ptr_t[tip_lo] (an upper bound on the
// nonzero samples, exact when no two tips share a sample).  Mode 1 scatters
// v when the modelled time of its pairs is below that of a dense pass over
// its stripe cells; the rates are GB300 measurements of the two kernels and
// of global 64-bit atomics (L2-resident accumulators or not).  Mode 2
// scatters every branch that fits; mode 0 none.  The choice depends on the
// tree and the tables only, not on the stripe range, so that a range run
// gives bitwise the stripes of the full run.
RowSplit split_rows(const uf_tree *tree, const BatchJob &J, const Plan *P, int acc, bool fp32, bool fixed,
                    bool may_list) {
  RowSplit R;
  const bool tiles = may_list && tile_scatter(J, acc, fixed);
  // the variance-adjusted method has no pair-scatter form: every branch dense
  const int mode = acc == ACC_VAW ? 0 : (int)J.sparse;
  bool can_do_without = false;  // the lists other than tiles
  const int64_t nb = tree->n_nodes - 1;
  const size_t nt = J.tabs.size();
  constexpr int NC = 6;
  const int classes[NC] = {SPARSE_SMALL_ENTRIES, 128, 512, 2048, SPARSE_MAX_ENTRIES, SPARSE_LIST_MAX_ENTRIES};
  R.cap.assign(classes, classes + NC);
  R.sparse.resize(NC);
  std::vector<char> is_sparse(std::max<int64_t>(nb, 1), 0);
  if (mode != 0) {
    // accumulator words per cell: FP64 terms are two-word fixed point
    // (uf_device.cuh)
    const int n_acc = (acc == ACC_GEN ? 2 : 1) * (fp32 ? 1 : 2);
    double cells = 0.0, cols = 0.0;  // stripe cells of a full run of every table; samples
    for (size_t t = 0; t < nt; t++) {
      const double n = (double)J.tabs[t].table->n;
      cells += std::floor(n / 2.0) * n;
      cols += n;
    }
    // accumulators beyond L2: one table scatters region by region in L2
    // (sparse_regions), several tables scatter straight into HBM-resident cells
    const bool regions = !tiles && sparse_regions(J, cells * 8.0 * n_acc) > 1;
    // FP32 terms of one table go through lists even when its accumulators fit
    // in L2: a fused list's pair is one atomic (generalized: two) for three
    // branches, and the atomics bound the scatter (2,048 samples weighted 4.73 ->
    // 4.29 ms a call, 1,003 generalized 3.13 -> 2.94)
    const bool listed =
        may_list && nt == 1 && (acc == ACC_MIN || acc == ACC_GEN) && fp32 && J.tabs[0].table->n >= LIST_MIN_SAMPLES;
    R.lists = regions || tiles || listed;
    R.fuse = (int)(acc == ACC_GEN ? std::min<int64_t>(J.fuse, 2) : J.fuse);
    // list mode keeps only sort keys in shared memory: longer runs fit
    const int64_t max_entries = R.lists ? SPARSE_LIST_MAX_ENTRIES : SPARSE_MAX_ENTRIES;
    // the scatter runs table by table (its grid's y is the table), so each
    // table's atomics hit L2 when that table's accumulators fit there
    std::vector<double> pair_cost(nt), entry_cost(nt);
    const double n_regions = regions ? sparse_regions(J, cells * 8.0 * n_acc) : 1.0;
    double dense_rate;  // cell updates per second of the dense kernel
    if (acc == SPLIT_GRAM) dense_rate = fp32 ? 2.5e14 : 2.5e14 * GRAM_SPLITS / GRAM_DIGITS;
    else dense_rate = fp32 ? (acc == ACC_GEN ? 4e12 : 1.3e13) : (acc == ACC_GEN ? 5e10 : fixed ? 3.5e12 : 2e11);
    const double visit_rate = fp32 ? 2e12 : (acc == ACC_GEN ? 3e10 : 1e12);
    const double job_cost = 5e-10;
    // region lists are fused (a listed branch carries its sparse children,
    // and for the min form with option sparse_fuse 6 its grandchildren,
    // region_lists): on the 113k-sample table about 0.57 (0.43) of the pairs
    // and 0.54 (0.39) of the list entries remain, so a scattered branch costs
    // about that share of its own pairs and visits.  The tensor path's
    // scatter runs beside its gram and ends after it already: its split keeps
    // the unfused costs.
    const double fuse = (regions || listed) && acc != SPLIT_GRAM && R.fuse > 0 ? (R.fuse == 6 ? 0.45 : 0.6) : 1.0;
    for (size_t t = 0; t < nt; t++) {
      const double n = (double)J.tabs[t].table->n;
      const double atom_rate = std::floor(n / 2.0) * n * 8.0 * n_acc <= 64e6 || regions ? 2.3e11 : 2.5e10;
      pair_cost[t] = (1.0 / visit_rate + n_acc / atom_rate) * fuse;
      entry_cost[t] = 4.0 / atom_rate;
      if (tiles) {
        pair_cost[t] = 2.4e-12;
        entry_cost[t] = 3e-11;
      }
    }
    // a row's offsets read by every tile
    const double tile_cost = tiles ? cells / (TILE_I * TILE_J) * 4e-13 : 0.0;
    // a dense row also costs its count row and embedding (or planes) in HBM
    const double dense_t = cells / dense_rate + cols * 36.0 / 6e12;
    // node ranges in parallel; each class list is the ranges' lists in order,
    // so the result equals a sequential pass (pair counts are integers < 2^53:
    // their double sums are exact in any order)
    struct Part {
      std::vector<int32_t> cls[NC];
      int64_t n_sparse = 0;
      double pairs = 0.0;
    };
    const int T = (int)std::max<int64_t>(1, std::min<int64_t>(host_threads(), nb / 16384));
    std::vector<Part> part(T);
    parallel_for(T, [&](int c) {
      Part &pt = part[c];
      const int64_t v0 = nb * c / T, v1 = nb * (c + 1) / T;
      for (int64_t v = v0; v < v1; v++) {
        const int32_t lo = tree->tip_lo[v], hi = tree->tip_hi[v];
        if (lo < 0) continue;
        if (tree->length[v] == 0.0) {
          // a zero-length branch adds exactly 0 to every accumulator: skipped
          // (its count row is still built if a dense parent needs it)
          is_sparse[v] = 1;
          pt.n_sparse++;
          continue;
        }
        double cost = 0.0, pairs = 0.0;
        int64_t mx = 0;
        for (size_t t = 0; t < nt; t++) {
          const auto &cp = J.tabs[t].table->col_ptr;
          const int64_t ub = cp[hi] - cp[lo];
          mx = std::max(mx, ub);
          if (ub == 0) continue;
          const double pr = (double)ub * (double)(ub - 1) / 2.0;
          pairs += pr;
          cost += job_cost + pr * pair_cost[t] + (double)ub * entry_cost[t] + tile_cost;
          // one visit per region: a CTA, and each entry's cursors walked to the
          // region (about 7e-12 s per entry and region measured on GB300 with a
          // 113,000-sample table; pairs at 4.3e-12 s)
          if (regions) cost += n_regions * (job_cost + (double)ub * 1e-11 * fuse);
        }
        if (mx > max_entries) continue;
        if (mode == 2 || cost < dense_t) {
          is_sparse[v] = 1;
          // (lists have no kernel of their own for the smallest rows)
          int k = R.lists && !tiles ? 1 : 0;
          while (classes[k] < mx) k++;
          pt.cls[k].push_back((int32_t)v);
          pt.n_sparse++;
          pt.pairs += pairs;
        }
      }
    });
    for (int k = 0; k < NC; k++)
      for (const Part &pt : part) R.sparse[k].insert(R.sparse[k].end(), pt.cls[k].begin(), pt.cls[k].end());
    for (const Part &pt : part) {
      R.n_sparse += pt.n_sparse;
      R.pairs += pt.pairs;
    }
    if (tiles) {
      const auto &cp = J.tabs[0].table->col_ptr;
      const int64_t n = J.tabs[0].table->n, least = tile_least(n);
      int64_t rows = 0, entries = 0;
      for (const auto &c : R.sparse)
        for (int32_t v : c) {
          const int64_t ub = cp[tree->tip_hi[v]] - cp[tree->tip_lo[v]];
          rows += ub >= least;
          entries += ub >= least ? ub : 0;
        }
      R.list_bytes = entries >= (int64_t)UINT32_MAX  // (their places are 32-bit)
                         ? INFINITY
                         : (double)entries * sizeof(TileEnt) + (double)(rows + 31) * (n / TILE_I + 2) * sizeof(uint16_t);
    }
    can_do_without = listed && !regions;
  }
  auto count_rows = [&] {
    const int64_t root = tree->n_nodes - 1;
    auto parent_dense = [&](int64_t v) {
      const int64_t p = tree->parent[v];
      return p != root && !is_sparse[p];
    };
    // per list position: bit 0 = built from CSC columns (tips, and sparse
    // branches under a dense parent), bit 1 = a dense internal node, bit 2 = a
    // dense branch; flagged in parallel, then gathered in list order
    std::vector<uint8_t> flag(P->lists.size(), 0);
    {
      const int64_t np = (int64_t)P->lists.size();
      const int T = (int)std::max<int64_t>(1, std::min<int64_t>(host_threads(), np / 16384));
      parallel_for(T, [&](int c) {
        const int64_t p0 = np * c / T, p1 = np * (c + 1) / T;
        size_t b = 0;
        for (int64_t q = p0; q < p1; q++) {
          // block of position q: blocks cover consecutive ranges of the lists
          while (b + 1 < P->launches.size() && q >= P->launches[b + 1][0].first) b++;
          const auto &l0 = P->launches[b][0];
          const int32_t v = P->lists[q];
          const bool tip = q < l0.first + l0.second;
          flag[q] = (uint8_t)((is_sparse[v] ? parent_dense(v) : tip) | ((!tip && !is_sparse[v]) << 1) |
                              (!is_sparse[v] << 2));
        }
      });
    }
    for (size_t b = 0; b < P->b0.size(); b++) {
      const auto &ls = P->launches[b];
      std::vector<std::pair<int64_t, int>> lb;
      const int64_t q0 = ls[0].first, q1 = ls.back().first + ls.back().second;
      const int64_t at0 = (int64_t)R.cnt_lists.size();
      // (the dense branches among them first: only they get embedding rows)
      std::vector<int32_t> sparse_built;
      for (int64_t q = q0; q < q1; q++)
        if (flag[q] & 1) (flag[q] & 4 ? R.cnt_lists : sparse_built).push_back(P->lists[q]);
      R.cnt_built_dense.push_back((int)((int64_t)R.cnt_lists.size() - at0));
      R.cnt_lists.insert(R.cnt_lists.end(), sparse_built.begin(), sparse_built.end());
      lb.emplace_back(at0, (int)((int64_t)R.cnt_lists.size() - at0));
      for (size_t l = 1; l < ls.size(); l++) {
        const int64_t at = (int64_t)R.cnt_lists.size();
        for (int64_t q = ls[l].first; q < ls[l].first + ls[l].second; q++)
          if (flag[q] & 2) R.cnt_lists.push_back(P->lists[q]);
        if ((int64_t)R.cnt_lists.size() > at) lb.emplace_back(at, (int)((int64_t)R.cnt_lists.size() - at));
      }
      R.cnt_launch.push_back(std::move(lb));
    }
  };
  std::vector<int32_t> row_of(std::max<int64_t>(nb, 1));  // of a dense branch
  auto dense_rows = [&] {
    R.dense_ptr.push_back(0);
    for (size_t b = 0; b < P->b0.size(); b++) {
      for (int64_t v = P->b0[b]; v < P->b1[b]; v++)
        if (!is_sparse[v]) {
          row_of[v] = (int32_t)((int64_t)R.dense.size() - R.dense_ptr[b]);
          R.dense.push_back((int32_t)v);
          R.dense_len.push_back(tree->length[v]);
        }
      R.dense_ptr.push_back((int64_t)R.dense.size());
      R.max_dense = std::max(R.max_dense, R.dense_ptr[b + 1] - R.dense_ptr[b]);
    }
  };
  // the lists of the scattered branches (a table's tiles make their own), of
  // the count rows and of the dense rows side by side: none needs another
  const bool lists = R.lists && R.n_sparse > 0 && !tiles;
  auto part = [&](int c) {
    if (c == 0 && lists) region_lists(tree, J.tabs[0].table, R);
    if (c == 1) count_rows();
    if (c == 2) dense_rows();
  };
  if (nb >= 16384) parallel_for(3, part);
  else
    for (int c = 0; c < 3; c++) part(c);
  if (lists && can_do_without)
    R.list_bytes = (double)R.region->entry_off.back() *
                   (double)(sparse_entry_bytes(fp32, R.fuse, acc, kind_of(J.method) == EMB_PRESENCE) + sizeof(int));
  R.cnt_xrow.resize(R.cnt_lists.size());
  for (size_t q = 0; q < R.cnt_lists.size(); q++) {
    const int32_t v = R.cnt_lists[q];
    R.cnt_xrow[q] = is_sparse[v] ? -1 : row_of[v];
  }
  for (size_t b = 0; b < R.cnt_launch.size(); b++) {
    R.cnt_lev_ptr.push_back((int64_t)R.cnt_levels.size());
    for (const auto &l : R.cnt_launch[b]) {
      R.cnt_levels.push_back((int32_t)l.first);
      R.cnt_levels.push_back((int32_t)(l.first + (&l == &R.cnt_launch[b][0] ? R.cnt_built_dense[b] : l.second)));
    }
  }
  return R;
}

}  // namespace

const RegionLists &region_lists(const uf_tree *tree, const uf_table *table, const RowSplit &sp) {
  RegionLists &L = *sp.region;
  std::call_once(L.once, [&] {
    const int F = sp.fuse, depth = F == 0 ? 0 : F == 6 ? 2 : 1;
    const int64_t nn = tree->n_nodes;
    // A sparse branch whose parent is a listed head rides in the parent's
    // list (its samples are among the parent's and its pairs among the
    // parent's pairs); with six members per head, so does a sparse child of
    // such a member (two levels below the head).  Parents come before
    // children in decreasing node order (parent[v] > v), so every head and
    // member is final when its children are visited.  The pass is sequential
    // and its choices are near coin flips: written without branches.
    std::vector<int8_t> level(nn, -1), used(nn, 0);  // -1: not listed, 0: head, >0: member depth
    std::vector<int32_t> head(nn);                   // a member's head, else the node
    std::vector<int8_t> slot(nn);
    for (const auto &c : sp.sparse)
      for (int32_t v : c) level[v] = 0;
    head[nn - 1] = (int32_t)(nn - 1);
    const int64_t *parent = tree->parent.data();
    for (int64_t v = nn - 2; v >= 0; v--) {
      const int64_t p = parent[v];
      const int32_t h = head[p];
      const int lp = level[p], uh = used[h];
      const int join = (level[v] == 0) & (lp >= 0) & (lp < depth) & (uh < F);
      used[h] = (int8_t)(uh + join);
      slot[v] = (int8_t)uh;
      level[v] = (int8_t)(level[v] + join * (lp + 1));
      head[v] = join ? h : (int32_t)v;
    }
    // the rest in parallel, in pieces of a class that keep its order
    struct Piece {
      size_t k, b, e;
      int64_t heads = 0, entries = 0;
    };
    std::vector<Piece> pc;
    constexpr size_t PIECE = 8192;
    // (the classes with the most entries come first: the region kernel visits
    // the heads in order, and its last wave is then one of small rows: 2,048
    // samples weighted 4.87 -> 4.75 ms, 113,000 samples, 2,048 stripes 921 -> 907 ms)
    for (size_t k = sp.sparse.size(); k-- > 0;)
      for (size_t b = 0; b < sp.sparse[k].size(); b += PIECE)
        pc.push_back(Piece{k, b, std::min(b + PIECE, sp.sparse[k].size())});
    const auto &cp = table->col_ptr;
    const int T = (int)std::max<int64_t>(1, std::min<int64_t>(host_threads(), (int64_t)pc.size()));
    auto pieces = [&](const std::function<void(Piece &)> &body) {
      parallel_for(T, [&](int c) {
        for (size_t i = pc.size() * c / T; i < pc.size() * (c + 1) / T; i++) body(pc[i]);
      });
    };
    pieces([&](Piece &x) {
      const std::vector<int32_t> &rows = sp.sparse[x.k];
      int64_t heads = 0, entries = 0;
      for (size_t i = x.b; i < x.e; i++) {
        const int32_t v = rows[i];
        const int64_t is = level[v] == 0;
        heads += is;
        entries += is * (cp[tree->tip_hi[v]] - cp[tree->tip_lo[v]]);
      }
      x.heads = heads;
      x.entries = entries;
    });
    L.cls_off.assign(sp.sparse.size(), 0);
    L.cls_n.assign(sp.sparse.size(), 0);
    int64_t n_heads = 0, n_entries = 0;
    for (Piece &x : pc) {  // counts -> first positions
      L.cls_n[x.k] += x.heads;
      std::swap(n_heads, x.heads);
      std::swap(n_entries, x.entries);
      n_heads += x.heads;
      n_entries += x.entries;
    }
    for (size_t k = L.cls_n.size(); k-- > 1;) L.cls_off[k - 1] = L.cls_off[k] + L.cls_n[k];
    L.heads.resize(n_heads);
    L.members.resize((size_t)n_heads * F);
    L.entry_off.resize(n_heads + 1);
    L.entry_off[n_heads] = n_entries;
    pieces([&](Piece &x) {
      const std::vector<int32_t> &rows = sp.sparse[x.k];
      int64_t q = x.heads, e = x.entries;
      for (size_t i = x.b; i < x.e; i++) {
        const int32_t v = rows[i];
        if (level[v] != 0) continue;
        L.heads[q] = v;
        L.entry_off[q] = e;
        e += cp[tree->tip_hi[v]] - cp[tree->tip_lo[v]];
        for (int m = used[v]; m < F; m++) L.members[(size_t)q * F + m] = -1;
        head[v] = (int32_t)q++;  // (from here a head's position)
      }
    });
    pieces([&](Piece &x) {
      const std::vector<int32_t> &rows = sp.sparse[x.k];
      for (size_t i = x.b; i < x.e; i++) {
        const int32_t v = rows[i];
        if (level[v] > 0) L.members[(size_t)head[head[v]] * F + slot[v]] = v;
      }
    });
  });
  return L;
}

// The split of a call, cached on the tree by its tables and kind (tables are
// immutable and their ids are never reused).
std::shared_ptr<const RowSplit> get_split(uf_tree *tree, const BatchJob &J, const Plan *P, int acc, bool fp32,
                                          bool fixed, bool may_list) {
  SplitKey key;
  for (const TableJob &t : J.tabs) std::get<0>(key).push_back(t.table->id);
  std::get<1>(key) = acc + (tile_scatter(J, acc, fixed) ? 16 : 0) + (may_list ? 0 : 32);
  std::get<2>(key) = fp32 ? 1 : fixed ? 2 : 0;
  std::get<3>(key) = (int)(J.sparse * 16 + J.fuse);
  std::get<4>(key) = P->block_rows;
  std::get<5>(key) = J.region_bytes;
  std::lock_guard<std::mutex> g(tree->mu);
  auto it = tree->splits.find(key);
  if (it != tree->splits.end()) return it->second;
  if (tree->splits.size() >= 16) tree->splits.clear();
  auto sp = std::make_shared<const RowSplit>(split_rows(tree, J, P, acc, fp32, fixed, may_list));
  tree->splits.emplace(key, sp);
  return sp;
}

}  // namespace rt
}  // namespace ufg
