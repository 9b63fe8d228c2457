// Single particle at high order: the self term of the moment equation
// (eq:moment_evolutionFinish, the (i,q) double sums of eq:FinalSingleI/II)
// without a table of (k, l, i, q) terms, whose size grows like M^6 (about
// 1e9 terms at M = 60).
//
// In units c = 2 lambda^2 = 1 (a_m = M_m c^{-|m|/2}) the equation reads
//   dM_k/dt = c^{|k|/2-1} R_k,
//   R_k = sum_l a_l sum_{i,q} coef(k,l,i,q) Psi[beta(k,l,i,q)],
//   Psi[beta] = sum_m a_m psi0[m + beta]           (the jet of the self pair),
// and with g(j) = 4^{-j} / j! every coefficient factors into an x part and a
// y part (4^{i+q+1-|k|} / ((k1-1-i)! (k2-q)!) = g(k1-1-i) g(k2-q), and the
// same with the Gamma^II factorials):
//   Gamma^I : -(-1)^{|k|} X1(k1,l1,i) Y1(k2,l2,q),
//             X1 = (-1)^{l1} C(l1,i) g(k1-1-i),  Y1 = (-1)^{l2} C(l2,q) g(k2-q),
//             beta = (k1+l1-2i-1, k2+l2-2q+1)
//   Gamma^II: +(-1)^{|k|} X2(k1,l1,i) Y2(k2,l2,q),
//             X2 = (-1)^{l1} C(l1,i) g(k1-i),    Y2 = (-1)^{l2} C(l2,q) g(k2-1-q),
//             beta = (k1+l1-2i+1, k2+l2-2q-1)
// with beta1 depending only on (k1, l1, i) and beta2 only on (k2, l2, q).
// So the sums are taken one index at a time:
//   pass 1  U[k2, l2, b1] = sum_q  C(l2,q) g(k2(-1)-q) Psi[b1, beta2(k2,l2,q)]
//   pass 2  V[k2, l1, b1] = sum_l2 (-1)^{l2} a_{l1,l2} U[k2, l2, b1]     (l1 + l2 <= M)
//   pass 3  R_k = (-1)^{|k|} sum_l1 (-1)^{l1} sum_i C(l1,i) g(k1(-1)-i)
//                 (-V^I[k2, l1, beta1] + V^II[k2, l1, beta1])
// for about 4.6e7 multiply-adds at M = 60 instead of about 1e9 (the products
// C g come from a host table, so each term is one multiply-add).  Every factor
// g is at most 1, so the intermediate sums stay far inside the FP64 range
// (the jet psi0 reaches ~1e190 at order 3M = 180; binomials ~1e17).  Only
// terms with |beta| <= 2M exist (|k|, |l| <= M); pass 1 skips the rest.
// A lone particle does not move (eq:xjdot_Final has no other particle), so
// dx/dt = 0.  Everything is FP64.
#include <algorithm>

#include "common.cuh"
#include "particle_kernels.h"

namespace mmvm {

namespace {

__device__ __forceinline__ double stage_c_high(const SelfHighArgs& A) {
  const double t = *A.t_dev + A.cs * (A.dt_dev ? *A.dt_dev : 0.0);
  return 2.0 * (A.lam0sq + A.four_nu * t);
}

__device__ __forceinline__ int order_of_col(int col) {  // total order of column col
  int s = 0;
  while (tri(s + 1) <= col) ++s;
  return s;
}

// c^{e/2} by repeated squaring (e may be negative): a few roundings, and a
// fraction of the FP64 operations of pow().
__device__ __forceinline__ double half_power(double c, int e) {
  const double b = e < 0 ? 1.0 / c : c;
  const int h = e < 0 ? -e : e;
  double v = (h & 1) ? sqrt(b) : 1.0, q = b;
  for (int i = h >> 1; i; i >>= 1) {
    if (i & 1) v *= q;
    q *= q;
  }
  return v;
}

// a_m = M_m c^{-|m|/2}
__global__ void self_scale_kernel(SelfHighArgs A) {
  const int m = blockIdx.x * blockDim.x + threadIdx.x;
  if (m >= A.K) return;
  A.at[m] = A.Min[m] * half_power(stage_c_high(A), -order_of_col(m));
}

// Psi[beta] = sum_m a_m psi0[m + beta] for 1 <= |beta| <= 2M (psi0 vanishes at
// odd indices, so only m of the parity of beta contribute).  One warp per
// beta, the lanes take its columns m in turn: one thread per beta ran up to
// 961 dependent multiply-adds on 58 CTAs (92 us at M = 60).
__global__ void self_psi_kernel(SelfHighArgs A) {
  const int b = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (b >= A.NB) return;  // whole warps
  const int bn = order_of_col(b + 1);  // bcol(b1, b2) = tri(|beta|) + b2 - 1
  const int b2 = b + 1 - tri(bn), b1 = bn - b2;
  double acc = 0.0;
#pragma unroll 4
  for (int m1 = b1 & 1; m1 <= A.M; m1 += 2)
    for (int m2 = (b2 & 1) + 2 * lane; m1 + m2 <= A.M; m2 += 64) {
      const int a1 = m1 + b1, a2 = m2 + b2;
      acc = fma(A.at[mcol(m1, m2)], A.psi0[tri(a1 + a2) + a2], acc);
    }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if (lane == 0) A.Psi[b] = acc;
}

// pass 1: U1[k2][l2][b1] (Gamma^I), U2[k2][l2][b1] (Gamma^II).  Pass 3 reads
// V[k2][l1][b1] at b1 <= k1 + l1 + 1 with k1 <= M - k2 only, and pass 2 sums U
// over l1 + l2 <= M, so b1 <= 2M - k2 - l2 + 1 covers all that is used (half
// of the array).
__global__ void self_pass1_kernel(SelfHighArgs A) {
  const int M = A.M, W = 2 * M + 1;
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (M + 1) * (M + 1) * W) return;
  const int b1 = idx % W, l2 = (idx / W) % (M + 1), k2 = idx / (W * (M + 1));
  if (b1 > 2 * M - k2 - l2 + 1) return;
  // C(l2, q) g(k2 - q) and C(l2, q) g(k2 - 1 - q), q = 0, 1, ...
  const double* c1 = A.cg + ((size_t)l2 * (M + 1) + k2) * (M + 1);
  double u1 = 0.0, u2 = 0.0;
#pragma unroll 4
  for (int q = 0; q <= min(l2, k2); ++q) {
    const int bb2 = k2 + l2 - 2 * q + 1;
    if (b1 + bb2 <= 2 * M) u1 = fma(c1[q], A.Psi[bcol(b1, bb2)], u1);
  }
  if (k2 >= 1) {
    const double* c2 = c1 - (M + 1);
#pragma unroll 4
    for (int q = 0; q <= min(l2, k2 - 1); ++q) {
      const int bb2 = k2 + l2 - 2 * q - 1;
      if (b1 + bb2 <= 2 * M && b1 + bb2 >= 1) u2 = fma(c2[q], A.Psi[bcol(b1, bb2)], u2);
    }
  }
  A.U1[idx] = u1;
  A.U2[idx] = u2;
}

// pass 2 (b1 <= M - k2 + l1 + 1, see pass 1): V[k2][l1][b1] = sum_{l2 <= M - l1} (-1)^{l2} a_{l1,l2} U[k2][l2][b1]
__global__ void self_pass2_kernel(SelfHighArgs A) {
  const int M = A.M, W = 2 * M + 1;
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (M + 1) * (M + 1) * W) return;
  const int b1 = idx % W, l1 = (idx / W) % (M + 1), k2 = idx / (W * (M + 1));
  if (b1 > M - k2 + l1 + 1) return;
  const double* u1 = A.U1 + (size_t)k2 * (M + 1) * W + b1;
  const double* u2 = A.U2 + (size_t)k2 * (M + 1) * W + b1;
  double v1 = 0.0, v2 = 0.0;
#pragma unroll 4
  for (int l2 = 0; l1 + l2 <= M; ++l2) {
    const double a = (l2 & 1) ? -A.at[mcol(l1, l2)] : A.at[mcol(l1, l2)];
    v1 = fma(a, u1[(size_t)l2 * W], v1);
    v2 = fma(a, u2[(size_t)l2 * W], v2);
  }
  A.V1[idx] = v1;
  A.V2[idx] = v2;
}

// pass 3 and the finish: one CTA per moment row k, one thread per (l1, Gamma^I or
// Gamma^II), then a sum over the CTA in a fixed order.  R_k, dM_k =
// c^{|k|/2-1} R_k, the RK4 stage.  (A warp per row, the lanes splitting l1, took
// 39 us at M = 60: its longest lane ran 240 dependent multiply-adds.)
constexpr int kPass3Threads = 160;  // >= 2 (M + 1) up to order 64, whole warps
__global__ void __launch_bounds__(kPass3Threads) self_pass3_kernel(SelfHighArgs A) {
  const int M = A.M, W = 2 * M + 1;
  __shared__ double red[kPass3Threads / 32];
  const int lane = threadIdx.x & 31, k = blockIdx.x;
  if (k == 0 && threadIdx.x < 2) {  // the centre does not move
    const int c = threadIdx.x;
    if (A.mode == 0) A.out_dx[c] = 0.0;
    if (A.mode == 1) { A.ys_x[c] = A.y_x[c]; A.sum_x[c] = A.y_x[c]; }
    if (A.mode == 2 || A.mode == 3) A.ys_x[c] = A.y_x[c];
    if (A.mode == 4) A.y_x[c] = A.sum_x[c];
  }
  const int kn = order_of_col(k);
  const int k2 = k - tri(kn), k1 = kn - k2;
  double r = 0.0;
  const int half = threadIdx.x > M, l1 = threadIdx.x - (half ? M + 1 : 0);
  if (l1 <= M) {
    // C(l1, i) g(k1 - i) and C(l1, i) g(k1 - 1 - i), i = 0, 1, ...
    const double* cb = A.cg + ((size_t)l1 * (M + 1) + k1) * (M + 1);
    double s = 0.0;
    if (!half && k1 >= 1) {
      const double* v1 = A.V1 + ((size_t)k2 * (M + 1) + l1) * W;
      const double* ca = cb - (M + 1);
#pragma unroll 4
      for (int i = 0; i <= min(l1, k1 - 1); ++i)
        s = fma(-ca[i], v1[k1 + l1 - 2 * i - 1], s);
    }
    if (half && k2 >= 1) {
      const double* v2 = A.V2 + ((size_t)k2 * (M + 1) + l1) * W;
#pragma unroll 4
      for (int i = 0; i <= min(l1, k1); ++i) {
        const int bb1 = k1 + l1 - 2 * i + 1;
        if (bb1 < W) s = fma(cb[i], v2[bb1], s);
      }
    }
    r = (l1 & 1) ? -s : s;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) r += __shfl_xor_sync(0xffffffffu, r, o);
  if (lane == 0) red[threadIdx.x >> 5] = r;
  __syncthreads();
  if (threadIdx.x != 0) return;
  r = 0.0;
  for (int w = 0; w < kPass3Threads / 32; ++w) r += red[w];
  if (kn & 1) r = -r;  // (-1)^{|k|}
  const double dm = r * half_power(stage_c_high(A), kn - 2);
  if (A.mode == 0) {
    A.out_dM[k] = dm;
    return;
  }
  const double h = *A.dt_dev;
  const double base = A.y_M[k];
  if (A.mode == 1) { A.ys_M[k] = base + 0.5 * h * dm; A.sum_M[k] = base + h / 6.0 * dm; }
  if (A.mode == 2) { A.ys_M[k] = base + 0.5 * h * dm; A.sum_M[k] += h / 3.0 * dm; }
  if (A.mode == 3) { A.ys_M[k] = base + h * dm;       A.sum_M[k] += h / 3.0 * dm; }
  if (A.mode == 4) { A.y_M[k] = A.sum_M[k] + h / 6.0 * dm; }
}

}  // namespace

size_t self_high_scratch_doubles(int M) {
  const size_t P = (size_t)(M + 1) * (M + 1) * (2 * M + 1);
  return (size_t)n_moments(M) + (size_t)n_beta(M) + 4 * P;
}

cudaError_t launch_self_high(SelfHighArgs A, double* scratch, cudaStream_t st) {
  const int M = A.M;
  const size_t P = (size_t)(M + 1) * (M + 1) * (2 * M + 1);
  A.at = scratch;
  A.Psi = A.at + A.K;
  A.U1 = A.Psi + A.NB;
  A.U2 = A.U1 + P;
  A.V1 = A.U2 + P;
  A.V2 = A.V1 + P;
  const int T = 128;
  self_scale_kernel<<<(A.K + T - 1) / T, T, 0, st>>>(A);
  self_psi_kernel<<<(A.NB * 32 + T - 1) / T, T, 0, st>>>(A);
  self_pass1_kernel<<<(int)((P + T - 1) / T), T, 0, st>>>(A);
  self_pass2_kernel<<<(int)((P + T - 1) / T), T, 0, st>>>(A);
  self_pass3_kernel<<<A.K, kPass3Threads, 0, st>>>(A);
  return cudaGetLastError();
}

}  // namespace mmvm
