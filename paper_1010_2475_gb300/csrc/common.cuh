// Shared compile-time index helpers and small device utilities of the MMVM
// kernels.  Index conventions (c = 2 lambda^2, zeta = x / sqrt(c)):
//  * moment column of (k1, k2):  mcol = q(k1+k2) + k2, q(s) = s(s+1)/2;
//  * stream-function correlation Psi[beta] for 1 <= |beta| <= BMAX, column
//    bcol = q(b1+b2) + b2 - 1 (beta = 0 is never needed);
//  * BMAX = 2M covers the velocity jet W[gamma], |gamma| <= 2M-1, that the
//    moment equations need (eq:FinalCrossI/II) and the |m| <= M entries of
//    the centroid equation (eq:xjdot_Final); for M = 0 it is 1.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>
#include <utility>

namespace mmvm {

__host__ __device__ constexpr int tri(int n) { return n * (n + 1) / 2; }
__host__ __device__ constexpr int n_moments(int M) { return tri(M + 1); }
__host__ __device__ constexpr int mcol(int k1, int k2) { return tri(k1 + k2) + k2; }
__host__ __device__ constexpr int bmax_of(int M) { return M == 0 ? 1 : 2 * M; }
__host__ __device__ constexpr int n_beta(int M) { return tri(bmax_of(M) + 1) - 1; }
__host__ __device__ constexpr int bcol(int b1, int b2) { return tri(b1 + b2) + b2 - 1; }
// Highest order of the stream-function jet a pair needs: |m + beta| <= M + BMAX.
__host__ __device__ constexpr int jet_order(int M) { return M + bmax_of(M); }

__host__ __device__ constexpr double binom_d(int n, int k) {
  double r = 1.0;
  for (int i = 1; i <= k; ++i) r = r * (n - k + i) / i;
  return r;
}
__host__ __device__ constexpr double pow2_neg(int n) {
  double r = 1.0;
  for (int i = 0; i < n; ++i) r *= 0.5;
  return r;
}

// Source record: FP32 mode stores zeta split into (hi, lo) floats so that
// differences of nearby centres are exact; FP64 stores zeta directly.
template <typename T> struct Rec;
template <> struct Rec<float> {
  static constexpr int HDR = 4;  // zh1, zh2, zl1, zl2
};
template <> struct Rec<double> {
  static constexpr int HDR = 2;  // z1, z2
};
__host__ __device__ constexpr int round_up(int a, int b) { return (a + b - 1) / b * b; }
// FP32 records also carry the far-field moments A'_n (n = 0..M, complex).
template <typename T>
__host__ __device__ constexpr int rec_far(int M) {
  return sizeof(T) == 4 ? 2 * (M + 1) : 0;
}
template <typename T>
__host__ __device__ constexpr int rec_len(int M) {
  // pad to 16 bytes so a record (and a tile of records) can be bulk-copied
  return round_up(Rec<T>::HDR + n_moments(M) + rec_far<T>(M), 16 / (int)sizeof(T));
}

// Particles per spatial group: the source tile of the pair kernel and the
// unit of the bounding boxes used for the far-field test.
constexpr int kGroup = 32;

// One instance (an independent simulation) of a batch of one order.
//  * state: FP64 blocks y_x (n x 2), y_M (n x K), ys_x, ys_M (RK4 stage
//    state), sum_x, sum_M (RK4 running sum), one after another;
//  * records: n, starting at record slot0 of the batch (slot0 is a multiple
//    of kGroup, so every group of kGroup slots belongs to one instance);
//  * sources split into `chunks` chunks of chunk_len (a multiple of kGroup);
//    partial sums [chunk][beta][target] start part_off doubles into the
//    batch's partials;
//  * core lambda^2 = lam0sq + four_nu t; step size dt; t is advanced on the
//    device after every step.
struct BatchInst {
  double* state;
  int n;
  int slot0;
  int chunk_len;
  int chunks;
  long long part_off;
  double lam0sq;
  double four_nu;
  double t;
  double dt;
};

// Far-field threshold on x = |b|^2 (c = 1 units) per order M: beyond it the
// Gaussian part of every jet entry of order <= 3M is below 2^-25 of the
// largest entry of that order (measured against the FP64 oracle's jet over
// all directions; 6 units of margin added), so a tile pair whose bounding
// boxes are this far apart uses the point-vortex jet.
__host__ __device__ constexpr float x_far(int M) {
  return M <= 0 ? 20.f : M == 1 ? 32.f : M == 2 ? 40.f : M == 3 ? 50.f : M == 4 ? 58.f
       : M == 5 ? 66.f : M == 6 ? 74.f : M == 7 ? 80.f : 88.f;
}

// The same threshold for FP64 pairs: beyond it the Gaussian part of every jet
// entry of order <= 3M is below 2^-54 of the largest entry of that order
// (maximum over all directions; 6 units of margin added), so the point-vortex
// jet equals the full jet to FP64 rounding.
__host__ __device__ constexpr float x_far64(int M) {
  return M <= 0 ? 44.f : M == 1 ? 52.f : M == 2 ? 63.f : M == 3 ? 72.f : M == 4 ? 81.f
       : M == 5 ? 90.f : M == 6 ? 98.f : M == 7 ? 107.f : 115.f;
}

// Far source tiles seen from far enough away are summed through one
// multipole expansion about the tile's centre instead of source by source.
// With u = 1/w, w = target - centre, delta_s = source - centre and
// rho_q(w) = (q-1)! u^q, the shift rho_q(w - delta) = sum_k delta^k/k!
// rho_{q+k}(w) turns the per-source sums sum_n A'_{s,n} rho_{n+nb} into
// sum_j B_j rho_{j+nb}(w), B_j = sum_s sum_{n+k=j} A'_{s,n} delta_s^k / k!.
// Truncating k at m2p_order(M) leaves sum_{k>P} C(q+k-1,k) theta^k below
// 2e-9 for every jet order q <= 3M when the tile radius is at most theta =
// 0.1 of the distance from the target group's box to the tile centre.
__host__ __device__ constexpr int m2p_order(int M) {
  return M <= 0 ? 8 : M == 1 ? 10 : M == 2 ? 12 : M == 3 ? 14 : M == 4 ? 15
       : M == 5 ? 17 : M == 6 ? 18 : M == 7 ? 19 : 21;
}
__host__ __device__ constexpr int m2p_terms(int M) { return M + m2p_order(M) + 1; }
constexpr float kM2PTheta2 = 0.01f;  // theta^2
// Widest tile or node that is taken through its expansion: its terms reach R^j / j!
// of a unit circulation, j < m2p_terms(M), and the shifts of the tree form that power
// too.  The limit keeps them below 1e26, so that circulations up to 1e12 stay inside
// the FP32 range; without it a term overflowed while its derivative underflowed, and
// the far field was NaN (M = 6: groups 1e3 core units wide).  Wider ones are opened, or
// summed source by source.
__host__ __device__ constexpr float m2p_radius(int M) {
  return M <= 0 ? 6700.f : M == 1 ? 1130.f : M == 2 ? 430.f : M == 3 ? 240.f : M == 4 ? 185.f
       : M == 5 ? 135.f : M == 6 ? 118.f : M == 7 ? 104.f : 92.f;
}
// Per group of kGroup records (FP32 far field): (min z1, max z1, min z2,
// max z2) of the hi parts, (centre z1, centre z2, radius, 0), then
// Re/Im B_j for j < m2p_terms(M); padded to whole float4s.
__host__ __device__ constexpr int gdata_len(int M) { return round_up(8 + 2 * m2p_terms(M), 4); }

// Local expansions (pair_local.cuh): extra orders of a group's expansion and of
// a target group's field (2M + extra <= 31: one lane per order), the widest
// group they serve, and the least separation x = |t0 - s0|^2 of two groups, the
// wider of radius r: the further apart, the faster the expansions converge.
// Up to loc_core kLocMinX is enough; beyond, x grows by loc_slope per unit of the
// radius, or (orders 5 and 6) by a second, steeper line.
// What they keep small is the remainder of the Taylor series of the Gaussian
// part, e^{-x} at orders up to 2M + 1 + P.  The double series of two particles at
// the facing ends of two groups at the least separation, in 64 bits against the
// jet itself, over radii, directions and moments (10 % of the circulation per
// order in the weighted norm): the pair's velocity is off by at most 2.4e-7 (M = 3;
// 1.6e-7 at M = 2, 1e-7 or less else), its moment rates by 4e-6 (M = 6) of the sum of
// their terms' magnitudes, below the FP32 jet's rounding at these orders.  (With
// 13 to 15 extra orders and 40 per unit at M <= 3 a velocity was off by up to
// 5e-5; with 40 per unit alone at M = 5 and 6 moment rates by 8e-5 and 1e-3.)
// 17 extra orders at M <= 3 cost 1.4 times the multiply-adds of 14, but 14 would
// have to keep groups further apart: disk of 30011, M = 2, per step 4.07 ms with
// 17, 4.07 with 16, 4.34 with 15, 4.44 with 14 at separations equally safe (3.60
// with the limits that were not).
__host__ __device__ constexpr int loc_extra(int M) { return M == 4 ? 16 : M <= 7 ? 17 : 15; }
__host__ __device__ constexpr float loc_radius(int M) {
  return M == 0 ? 1.75f : M <= 2 ? 2.0f : M <= 4 ? 1.8f : M == 5 ? 1.6f : M == 6 ? 1.7f : M == 7 ? 1.1f : 0.85f;
}
// Widest target group whose far field is taken through its local field.  A box
// may have no width (particles on a line), and then a far source beside it is only
// sqrt(x_far) from the centre: the limits are 0.34 to 0.39 of that, where the Taylor
// series about the centre, to loc_extra orders per axis, ends within FP32 rounding:
// velocities 1e-7 or less, moment rates 1.4e-6 or less of their terms' magnitudes (64 bits,
// over directions and moments; 0.40 to 0.45 at M <= 3 left up to 1.3e-5).
__host__ __device__ constexpr float loc_field_radius(int M) {
  return M <= 0 ? 1.75f : M == 1 ? 2.2f : M == 2 ? 2.45f : M <= 4 ? 2.75f : M == 5 ? 3.2f
       : M == 6 ? 3.3f : M == 7 ? 3.4f : 3.2f;
}
__host__ __device__ constexpr float loc_core(int M) {  // up to this radius kLocMinX is enough
  return M <= 2 ? 0.9f : M == 3 ? 0.8f : M == 4 ? 0.6875f : M <= 7 ? 0.5625f : 0.4375f;
}
__host__ __device__ constexpr float loc_slope(int M) {  // of the least x beyond loc_core
  return M == 0 ? 60.f : M <= 2 ? 54.f : M == 3 ? 56.f : M == 4 ? 55.f : M <= 6 ? 40.f : 60.f;
}
__host__ __device__ constexpr float loc_core2(int M) { return M == 5 ? 0.66f : 0.73f; }
__host__ __device__ constexpr float loc_slope2(int M) { return M == 5 ? 58.f : M == 6 ? 72.f : 0.f; }

// Binary tree over G groups of kGroup sorted records (the far field of the
// list form): level L has ceil(G / 2^L) nodes, node i of level L >= 1 holds
// nodes 2i and 2i+1 of level L-1, the top level one node; the node records
// of levels 1.. are stored one level after another.
__host__ __device__ inline int tree_levels(int G) {
  int L = 0;
  while ((G + (1 << L) - 1) >> L > 1) ++L;
  return L;  // index of the top level (0 if G == 1)
}
__host__ __device__ inline int tree_level_nodes(int G, int L) { return (G + (1 << L) - 1) >> L; }
// Offset (in nodes) of level L >= 1 in the node storage.
__host__ __device__ inline long long tree_level_offset(int G, int L) {
  long long off = 0;
  for (int l = 1; l < L; ++l) off += tree_level_nodes(G, l);
  return off;
}

// Levels of at most this many nodes are built by one CTA in one launch.
constexpr int kTreeTop = 64;  // two nodes per warp
__host__ __device__ inline int tree_build_launches(int G) {
  int L = 1, top = tree_levels(G), k = 0;
  for (; L <= top && tree_level_nodes(G, L) > kTreeTop; ++L) ++k;
  return k + (L <= top ? 1 : 0);
}

// Compile-time loop: f(std::integral_constant<int, i>) for i in [B, E).
template <int B, int E, typename F>
__device__ __forceinline__ void static_for(F&& f) {
  if constexpr (B < E) {
    f(std::integral_constant<int, B>{});
    static_for<B + 1, E>(f);
  }
}
// Descending: i = E-1 down to B.
template <int B, int E, typename F>
__device__ __forceinline__ void static_for_down(F&& f) {
  if constexpr (B < E) {
    f(std::integral_constant<int, E - 1>{});
    static_for_down<B, E - 1>(f);
  }
}

__device__ __forceinline__ float dexp(float v) { return expf(v); }
__device__ __forceinline__ double dexp(double v) { return exp(v); }

}  // namespace mmvm
