// FP64 coefficient tables of the MMVM finish step, generated on the host.
//
// In units where c = 2 lambda^2 = 1 (scaled moments a_l = M_l c^{-|l|/2}, and
// the stream-function correlation Psi[beta] of the pair kernel), the moment
// equation of eq:Final_CrossCoef becomes
//   dM_k/dt = c^{|k|/2 - 1} [ sum_l a_l sum_beta coef(k,l,beta) Psi_tot[beta]
//                             + (X_1 a_{k-e1} + X_2 a_{k-e2}) / M_00 ]
// where the (k, l, beta, coef) entries collect the (i, q) double sums of
// eq:FinalSingleI (Gamma^I, velocity component 1, W_1[g] = -Psi[g + e2]) and
// eq:FinalSingleII (Gamma^II, component 2, W_2[g] = Psi[g + e1]) times the
// projection prefactor c_k (eq:coefficient):
//   Gamma^I : coef = -(-1)^{|k|+|l|} C(l1,i) C(l2,q) 4^{i+q+1-|k|} / ((k1-i-1)! (k2-q)!)
//             beta = (k1+l1-2i-1, k2+l2-2q+1)
//   Gamma^II: coef = +(-1)^{|k|+|l|} C(l1,i) C(l2,q) 4^{i+q+1-|k|} / ((k1-i)! (k2-q-1)!)
//             beta = (k1+l1-2i+1, k2+l2-2q-1)
// (the lambda powers of eq:FinalSingleI/II, c_k and the velocity scaling all
// combine into the single factor c^{|k|/2-1}).  Psi_tot adds the self pair,
// Psi_self[beta] = sum_m a_m psi0[m + beta], with psi0 the jet at the origin
// of the stream function of a Gaussian vortex (c = 1):
//   psi0[(2p, 2q)] = -(1/4pi) (-1)^{p+q} [(2p)!/p!] [(2q)!/q!] / (p+q),  p+q >= 1,
// and 0 for any odd index (the closed forms H_1, H_2 of Appendix A.1 are its
// first derivatives: H_1(a) = -psi0[a+e2], H_2(a) = psi0[a+e1]).
#pragma once

#include <vector>

namespace mmvm {

// One (k, l, beta) entry.
struct FinEntry {
  double c;  // coefficient
  int b;     // Psi column beta (bcol)
  int pad;
};

// The moment equation as R_k = sum_l a_l g_kl, g_kl = sum_beta c Psi[beta]: the
// entries form one group per (k, l).  The rows are split into row blocks (one,
// or several CTAs' worth for the single particles of high order); the groups
// of a block are sorted by length, longest first, and entry j of its group q
// sits at tab[off[j] + q], so that threads on neighbouring groups run equally
// long loops over neighbouring entries.
struct RowBlock {
  int k0, k1;    // rows
  int groups;    // groups of the block
  int len_at;    // group lengths: glen[len_at + q]
  int off_at;    // off[j] = offs[off_at + j], j below the longest group's length
  int row_at;    // row k's groups: rows[rows_off[k] .. rows_off[k + 1]) hold (q, l)
};
struct RowGroup {
  int q, l;
};
struct FinishTables {
  int M = 0, K = 0, NB = 0, NJ = 0;
  int nrb = 1;
  int max_groups = 0;              // most groups of a row block
  std::vector<FinEntry> tab;
  std::vector<RowBlock> blocks;    // nrb
  std::vector<int> glen, offs;
  std::vector<RowGroup> rows;
  std::vector<int> rows_off;       // K + 1
  std::vector<double> psi0;        // psi0 for |alpha| <= NJ, column q(|alpha|) + alpha_2
  std::vector<unsigned char> blob() const;  // all of them, 256-byte aligned parts
};

// Device view of a blob() copied to `base`.
struct FinishTab {
  const FinEntry* tab = nullptr;
  const RowBlock* blocks = nullptr;
  const int* glen = nullptr;
  const int* offs = nullptr;
  const RowGroup* rows = nullptr;
  const int* rows_off = nullptr;
  const double* psi0 = nullptr;
  int nrb = 1, max_groups = 0;
};
FinishTab finish_tab(const FinishTables& t, const void* base);

// entries = false leaves out the (k, l, beta) entries (their number grows
// like M^6; the separable single-particle path does not use them).
FinishTables build_finish_tables(int M, bool entries = true);

// Factors of the separable single-particle path (self_high.cu): binom is
// row-major (M+1) x (M+1), binom[l][q] = C(l, q); g[j] = 4^{-j} / j!, j <= M;
// cg[(l (M+1) + k) (M+1) + q] = binom[l][q] * g[k - q] (the FP64 product, 0
// for q > min(l, k)), so that the passes do one multiply-add per term.
struct SeparableTables {
  std::vector<double> binom, g, cg;
};
SeparableTables build_separable_tables(int M);

}  // namespace mmvm
