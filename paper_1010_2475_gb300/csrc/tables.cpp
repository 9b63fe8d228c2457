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

// Pieces, their interleaved layout and the row blocks of t from the rows'
// entries (FinEntry::l holds the group on entry).
void cut_rows(FinishTables& t, const std::vector<std::vector<FinEntry>>& rows) {
  size_t total = 0;
  for (const auto& r : rows) total += r.size();
  // ~128 pieces keep the threads of a CTA busy.  Orders above the pair limit
  // serve one particle: short pieces, since a thread's dependent multiply-adds
  // are what such an evaluation waits for (order 10: 96 entries per thread took
  // 26 us per right-hand side, 16 took 20 us).
  const size_t piece = t.M > 8 ? 8 : std::min<size_t>(std::max<size_t>(total / 128, 8), 96);
  std::vector<std::vector<FinEntry>> ps;
  t.row_off.assign(1, 0);
  for (const auto& r : rows) {
    const size_t cnt = (r.size() + piece - 1) / piece;
    for (size_t i = 0; i < cnt; ++i) {
      const size_t e0 = i * r.size() / cnt, e1 = (i + 1) * r.size() / cnt;
      std::vector<FinEntry> p(r.begin() + e0, r.begin() + e1);
      for (size_t e = 0; e + 1 < p.size(); ++e)
        if (p[e].l == p[e + 1].l) p[e].l = -1;  // only the last entry of a group closes it
      ps.push_back(std::move(p));
    }
    t.row_off.push_back((int)ps.size());
  }
  t.np = (int)ps.size();
  size_t plen = 0;
  for (const auto& p : ps) plen = std::max(plen, p.size());
  t.tab.assign(plen * ps.size(), FinEntry{0.0, 0, -1});
  t.piece_len.clear();
  for (size_t p = 0; p < ps.size(); ++p) {
    t.piece_len.push_back((int)ps[p].size());
    for (size_t j = 0; j < ps[p].size(); ++j) t.tab[j * ps.size() + p] = ps[p][j];
  }
  // row blocks of ~256 pieces, one per thread of a CTA
  const int want = (int)std::min<size_t>(std::max<size_t>(ps.size() / 256, 1), 64);
  t.rb_off.assign(1, 0);
  size_t run = 0;
  for (int k = 0; k < t.K; ++k) {
    run += rows.size() ? rows[k].size() : 0;
    if (run * want >= total * t.rb_off.size() && (int)t.rb_off.size() < want)
      t.rb_off.push_back(k + 1);
  }
  if (t.rb_off.back() != t.K) t.rb_off.push_back(t.K);
  t.nrb = (int)t.rb_off.size() - 1;
  t.rb_pieces = 0;
  for (int i = 0; i < t.nrb; ++i)
    t.rb_pieces = std::max(t.rb_pieces, t.row_off[t.rb_off[i + 1]] - t.row_off[t.rb_off[i]]);
}

struct BlobOffsets {
  size_t tab, piece_len, row_off, rb_off, psi0, bytes;
};
BlobOffsets blob_offsets(const FinishTables& t) {
  BlobOffsets o;
  size_t off = 0;
  auto take = [&](size_t bytes) {
    const size_t at = off;
    off = (off + bytes + 255) & ~(size_t)255;
    return at;
  };
  o.tab = take(t.tab.size() * sizeof(FinEntry));
  o.piece_len = take(t.piece_len.size() * sizeof(int));
  o.row_off = take(t.row_off.size() * sizeof(int));
  o.rb_off = take(t.rb_off.size() * sizeof(int));
  o.psi0 = take(t.psi0.size() * sizeof(double));
  o.bytes = off;
  return o;
}

}  // namespace

std::vector<unsigned char> FinishTables::blob() const {
  const BlobOffsets o = blob_offsets(*this);
  std::vector<unsigned char> b(o.bytes, 0);
  auto put = [&](size_t at, const void* src, size_t bytes) {
    if (bytes) std::memcpy(b.data() + at, src, bytes);
  };
  put(o.tab, tab.data(), tab.size() * sizeof(FinEntry));
  put(o.piece_len, piece_len.data(), piece_len.size() * sizeof(int));
  put(o.row_off, row_off.data(), row_off.size() * sizeof(int));
  put(o.rb_off, rb_off.data(), rb_off.size() * sizeof(int));
  put(o.psi0, psi0.data(), psi0.size() * sizeof(double));
  return b;
}

FinishTab finish_tab(const FinishTables& t, const void* base) {
  const BlobOffsets o = blob_offsets(t);
  const unsigned char* p = static_cast<const unsigned char*>(base);
  FinishTab f;
  f.tab = reinterpret_cast<const FinEntry*>(p + o.tab);
  f.piece_len = reinterpret_cast<const int*>(p + o.piece_len);
  f.row_off = reinterpret_cast<const int*>(p + o.row_off);
  f.rb_off = reinterpret_cast<const int*>(p + o.rb_off);
  f.psi0 = reinterpret_cast<const double*>(p + o.psi0);
  f.np = t.np;
  f.nrb = t.nrb;
  f.rb_pieces = t.rb_pieces;
  return f;
}

FinishTables build_finish_tables(int M, bool entries) {
  FinishTables t;
  t.M = M;
  t.K = n_moments(M);
  t.NB = n_beta(M);
  t.NJ = jet_order(M);
  std::vector<std::vector<FinEntry>> rows(t.K);  // entries by row, grouped by l
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
        rows[kcol].push_back({(double)kv.second, kv.first.second, kv.first.first});
      }
    }
  }
  cut_rows(t, rows);
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
