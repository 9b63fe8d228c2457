// Host generation of the FP64 finish tables (see tables.h for the formulas).
#include "tables.h"

#include <algorithm>
#include <cstring>
#include <map>
#include <tuple>

#include "common.cuh"

namespace mmvm {

namespace {

long double factl(int n) {
  long double r = 1.0L;
  for (int i = 2; i <= n; ++i) r *= (long double)i;
  return r;
}
long double binoml(int n, int k) {
  if (k < 0 || k > n) return 0.0L;
  long double r = 1.0L;
  for (int i = 1; i <= k; ++i) r = r * (long double)(n - k + i) / (long double)i;
  return r;
}
long double pow4l(int e) {
  long double r = 1.0L;
  if (e >= 0)
    for (int i = 0; i < e; ++i) r *= 4.0L;
  else
    for (int i = 0; i < -e; ++i) r *= 0.25L;
  return r;
}

// One row's entries by group l.
struct Group {
  int k, l;
  std::vector<FinEntry> e;
};

// The row blocks and the interleaved entries of t from the groups (by row).
void lay_out(FinishTables& t, const std::vector<std::vector<Group>>& rows) {
  size_t total = 0, groups = 0;
  for (const auto& r : rows)
    for (const Group& g : r) {
      total += g.e.size();
      ++groups;
    }
  // orders above the pair limit serve one particle: a CTA per ~64 groups, four
  // threads each
  const int want = t.M > 8 ? (int)std::min<size_t>(std::max<size_t>(groups / 64, 1), 128) : 1;
  std::vector<int> cut(1, 0);
  size_t run = 0;
  for (int k = 0; k < t.K; ++k) {
    for (const Group& g : rows[k]) run += g.e.size();
    if (run * want >= total * cut.size() && (int)cut.size() < want) cut.push_back(k + 1);
  }
  if (cut.back() != t.K) cut.push_back(t.K);
  t.nrb = (int)cut.size() - 1;
  t.max_groups = 0;
  t.rows_off.assign(1, 0);
  for (int i = 0; i < t.nrb; ++i) {
    RowBlock rb{};
    rb.k0 = cut[i];
    rb.k1 = cut[i + 1];
    rb.len_at = (int)t.glen.size();
    rb.off_at = (int)t.offs.size();
    std::vector<const Group*> gs;
    for (int k = rb.k0; k < rb.k1; ++k)
      for (const Group& g : rows[k]) gs.push_back(&g);
    std::stable_sort(gs.begin(), gs.end(),
                     [](const Group* a, const Group* b) { return a->e.size() > b->e.size(); });
    rb.groups = (int)gs.size();
    t.max_groups = std::max(t.max_groups, rb.groups);
    for (const Group* g : gs) t.glen.push_back((int)g->e.size());
    const size_t longest = gs.empty() ? 0 : gs[0]->e.size();
    for (size_t j = 0; j < longest; ++j) {
      t.offs.push_back((int)t.tab.size());
      for (size_t q = 0; q < gs.size() && gs[q]->e.size() > j; ++q) t.tab.push_back(gs[q]->e[j]);
    }
    std::vector<std::vector<RowGroup>> of_row(rb.k1 - rb.k0);
    for (size_t q = 0; q < gs.size(); ++q) of_row[gs[q]->k - rb.k0].push_back({(int)q, gs[q]->l});
    for (const auto& r : of_row) {
      t.rows.insert(t.rows.end(), r.begin(), r.end());
      t.rows_off.push_back((int)t.rows.size());
    }
    t.blocks.push_back(rb);
  }
}

struct BlobOffsets {
  size_t tab, blocks, glen, offs, rows, rows_off, psi0, bytes;
};
BlobOffsets blob_offsets(const FinishTables& t) {
  BlobOffsets o;
  size_t off = 0;
  auto take = [&](const auto& v) {
    const size_t at = off;
    off = (off + v.size() * sizeof(v[0]) + 255) & ~(size_t)255;
    return at;
  };
  o.tab = take(t.tab);
  o.blocks = take(t.blocks);
  o.glen = take(t.glen);
  o.offs = take(t.offs);
  o.rows = take(t.rows);
  o.rows_off = take(t.rows_off);
  o.psi0 = take(t.psi0);
  o.bytes = off;
  return o;
}

}  // namespace

std::vector<unsigned char> FinishTables::blob() const {
  const BlobOffsets o = blob_offsets(*this);
  std::vector<unsigned char> b(o.bytes, 0);
  auto put = [&](size_t at, const auto& v) {
    if (!v.empty()) std::memcpy(b.data() + at, v.data(), v.size() * sizeof(v[0]));
  };
  put(o.tab, tab);
  put(o.blocks, blocks);
  put(o.glen, glen);
  put(o.offs, offs);
  put(o.rows, rows);
  put(o.rows_off, rows_off);
  put(o.psi0, psi0);
  return b;
}

FinishTab finish_tab(const FinishTables& t, const void* base) {
  const BlobOffsets o = blob_offsets(t);
  const unsigned char* p = static_cast<const unsigned char*>(base);
  FinishTab f;
  f.tab = reinterpret_cast<const FinEntry*>(p + o.tab);
  f.blocks = reinterpret_cast<const RowBlock*>(p + o.blocks);
  f.glen = reinterpret_cast<const int*>(p + o.glen);
  f.offs = reinterpret_cast<const int*>(p + o.offs);
  f.rows = reinterpret_cast<const RowGroup*>(p + o.rows);
  f.rows_off = reinterpret_cast<const int*>(p + o.rows_off);
  f.psi0 = reinterpret_cast<const double*>(p + o.psi0);
  f.nrb = t.nrb;
  f.max_groups = t.max_groups;
  return f;
}

FinishTables build_finish_tables(int M, bool entries) {
  FinishTables t;
  t.M = M;
  t.K = n_moments(M);
  t.NB = n_beta(M);
  t.NJ = jet_order(M);
  std::vector<std::vector<Group>> rows(t.K);  // groups by row
  for (int kn = 0, kcol = 0; entries && kn <= M; ++kn) {
    for (int k2 = 0; k2 <= kn; ++k2, ++kcol) {
      const int k1 = kn - k2;
      std::map<std::pair<int, int>, long double> acc;  // (l col, beta col) -> coef
      for (int ln = 0; ln <= M; ++ln) {
        for (int l2 = 0; l2 <= ln; ++l2) {
          const int l1 = ln - l2;
          const int lcol = mcol(l1, l2);
          const long double sgn = ((kn + ln) & 1) ? -1.0L : 1.0L;
          if (k1 >= 1) {  // Gamma^I, eq:FinalSingleI
            for (int i = 0; i <= (l1 < k1 - 1 ? l1 : k1 - 1); ++i)
              for (int q = 0; q <= (l2 < k2 ? l2 : k2); ++q) {
                const long double v = -sgn * binoml(l1, i) * binoml(l2, q) *
                                      pow4l(i + q + 1 - kn) /
                                      (factl(k1 - i - 1) * factl(k2 - q));
                const int b1 = k1 + l1 - 2 * i - 1, b2 = k2 + l2 - 2 * q + 1;
                acc[{lcol, bcol(b1, b2)}] += v;
              }
          }
          if (k2 >= 1) {  // Gamma^II, eq:FinalSingleII
            for (int i = 0; i <= (l1 < k1 ? l1 : k1); ++i)
              for (int q = 0; q <= (l2 < k2 - 1 ? l2 : k2 - 1); ++q) {
                const long double v = sgn * binoml(l1, i) * binoml(l2, q) *
                                      pow4l(i + q + 1 - kn) /
                                      (factl(k1 - i) * factl(k2 - q - 1));
                const int b1 = k1 + l1 - 2 * i + 1, b2 = k2 + l2 - 2 * q - 1;
                acc[{lcol, bcol(b1, b2)}] += v;
              }
          }
        }
      }
      for (auto& kv : acc) {
        if (kv.second == 0.0L) continue;
        std::vector<Group>& r = rows[kcol];
        if (r.empty() || r.back().l != kv.first.first) r.push_back({kcol, kv.first.first, {}});
        r.back().e.push_back({(double)kv.second, kv.first.second, 0});
      }
    }
  }
  lay_out(t, rows);
  // psi0 (jet of the Gaussian-vortex stream function at the origin, c = 1)
  t.psi0.assign(tri(t.NJ + 1), 0.0);
  const long double inv4pi = 0.0795774715459476678844418816862571810L;
  for (int n = 2; n <= t.NJ; n += 2) {
    for (int a2 = 0; a2 <= n; a2 += 2) {
      const int p = (n - a2) / 2, q = a2 / 2;
      const long double r = factl(2 * p) / factl(p) * (factl(2 * q) / factl(q));
      const long double s = ((p + q) & 1) ? -1.0L : 1.0L;
      t.psi0[tri(n) + a2] = (double)(-inv4pi * s * r / (long double)(p + q));
    }
  }
  return t;
}

SeparableTables build_separable_tables(int M) {
  SeparableTables t;
  t.binom.assign((size_t)(M + 1) * (M + 1), 0.0);
  t.g.assign((size_t)M + 1, 0.0);
  for (int a = 0; a <= M; ++a) {
    for (int b = 0; b <= a; ++b) t.binom[(size_t)a * (M + 1) + b] = (double)binoml(a, b);
    t.g[a] = (double)(pow4l(-a) / factl(a));
  }
  const size_t W = (size_t)M + 1;
  t.cg.assign(W * W * W, 0.0);
  for (int l = 0; l <= M; ++l)
    for (int k = 0; k <= M; ++k)
      for (int q = 0; q <= std::min(l, k); ++q)
        t.cg[((size_t)l * W + k) * W + q] = t.binom[(size_t)l * W + q] * t.g[k - q];
  return t;
}

}  // namespace mmvm
