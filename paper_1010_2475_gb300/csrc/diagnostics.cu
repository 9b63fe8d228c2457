// Diagnostics of a state on the GPU (FP64): the reconstructed vorticity
//   omega(p) = sum_j sum_{|k|<=M} M^j_k D^k phi_00(p - x^j; lambda)
// (eq:vorticity_decomposition; phi_00 = exp(-|x|^2/lambda^2) / (pi lambda^2)),
// with D^k phi_00(x) = (-1/lambda)^{|k|} H_{k1}(t1) H_{k2}(t2) phi_00(x),
// t = x / lambda and H_n the physicists' Hermite polynomials
// (H_{n+1} = 2 t H_n - 2 n H_{n-1}), and the ring sums of the nonaxisymmetric
// enstrophy (eq:nonaxi_enstrophy): per ring of a polar grid, the sum over its
// angles of (omega - ring mean)^2.
//
// One thread per point; the particles pass through shared memory in tiles.
// A particle farther than (sqrt(2M+1) + 6) lambda from the point is skipped:
// every Hermite function of order <= M is below e^-36 of its peak there.
//
// Bound: FP64 arithmetic (2 FMA per cycle and SM).  Orders <= 8 run compiled
// kernels: the Hermite values stay in registers, the moments are scaled by
// (-1/lambda)^|k| once per tile, the double sum is taken one index at a time
// (K + M + 1 multiply-adds instead of 2 K + 2 M), and the cut-off is tested in
// FP32 for a whole tile first, so that each lane walks only its own near
// particles: lanes of a warp then share the FP64 pipe instead of waiting for
// each other's near particles (n = 4096 in a disk of 20 lambda: 20 % of the
// pairs are near per lane, 38 % for some lane of a warp).
#include <algorithm>
#include <cmath>
#include <vector>

#include "common.cuh"
#include "particle_kernels.h"

namespace mmvm {

namespace {

constexpr int kMaxOrderDiag = 64;

__global__ void vorticity_kernel(int n, int M, int K, int tile, const double* __restrict__ x,
                                 const double* __restrict__ mom, const double* t_dev,
                                 double lam0sq, double four_nu, int npts,
                                 const double* __restrict__ pts, double* __restrict__ out) {
  extern __shared__ double sh[];  // tile x (2 + K)
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  const double lam2 = lam0sq + four_nu * (t_dev ? *t_dev : 0.0);
  const double lam = sqrt(lam2), il = 1.0 / lam;
  const double rc = sqrt(2.0 * M + 1.0) + 6.0;
  const double cut2 = rc * rc;
  const double px = p < npts ? pts[2 * p] : 0.0, py = p < npts ? pts[2 * p + 1] : 0.0;
  double hx[kMaxOrderDiag + 1], hy[kMaxOrderDiag + 1];
  double acc = 0.0;
  const int W = 2 + K;
  for (int j0 = 0; j0 < n; j0 += tile) {
    const int cnt = min(tile, n - j0);
    __syncthreads();
    for (int i = threadIdx.x; i < cnt * W; i += blockDim.x) {
      const int jj = i / W, c = i % W;
      sh[i] = c < 2 ? x[2 * (size_t)(j0 + jj) + c] : mom[(size_t)(j0 + jj) * K + (c - 2)];
    }
    __syncthreads();
    if (p >= npts) continue;
    for (int jj = 0; jj < cnt; ++jj) {
      const double* r = sh + jj * W;
      const double t1 = (px - r[0]) * il, t2 = (py - r[1]) * il;
      const double r2 = t1 * t1 + t2 * t2;
      if (r2 > cut2) continue;
      hx[0] = 1.0;
      hy[0] = 1.0;
      if (M >= 1) {
        hx[1] = 2.0 * t1;
        hy[1] = 2.0 * t2;
      }
      for (int q = 1; q < M; ++q) {
        hx[q + 1] = 2.0 * t1 * hx[q] - 2.0 * q * hx[q - 1];
        hy[q + 1] = 2.0 * t2 * hy[q] - 2.0 * q * hy[q - 1];
      }
      const double* mk = r + 2;
      double sum = 0.0, sc = 1.0;  // sc = (-1/lambda)^s
      int col = 0;
      for (int s = 0; s <= M; ++s) {
        double part = 0.0;
        for (int k2 = 0; k2 <= s; ++k2, ++col) part = fma(mk[col], hx[s - k2] * hy[k2], part);
        sum = fma(sc, part, sum);
        sc *= -il;
      }
      acc = fma(sum, exp(-r2), acc);
    }
  }
  if (p < npts) out[p] = acc * (il * il) * 0.31830988618379067154;  // / (pi lambda^2)
}

// Orders <= 8: points [128 blockIdx.x, ...) against particle chunk blockIdx.y;
// writes the sums to out[chunk][point] (divided by pi lambda^2).
constexpr int kVortTile = 128, kVortThreads = 128;

template <int M>
__global__ void __launch_bounds__(kVortThreads)
    vorticity_low_kernel(int n, int chunk, const double* __restrict__ x,
                         const double* __restrict__ mom, const double* t_dev, double lam0sq,
                         double four_nu, int npts, const double* __restrict__ pts,
                         double* __restrict__ out) {
  constexpr int K = n_moments(M), W = 2 + K;
  __shared__ double sh[kVortTile * W];
  __shared__ float2 shf[kVortTile];
  const int p = blockIdx.x * kVortThreads + threadIdx.x;
  const double lam2 = lam0sq + four_nu * (t_dev ? *t_dev : 0.0);
  const double lam = sqrt(lam2), il = 1.0 / lam;
  const double rc = sqrt(2.0 * M + 1.0) + 6.0;
  const double cut2 = rc * rc;
  const double px = p < npts ? pts[2 * p] : 0.0, py = p < npts ? pts[2 * p + 1] : 0.0;
  double scale[M + 1];  // (-1/lambda)^s
  scale[0] = 1.0;
#pragma unroll
  for (int s = 1; s <= M; ++s) scale[s] = scale[s - 1] * -il;
  double acc = 0.0;
  const int j1 = min(n, (int)(blockIdx.y + 1) * chunk);
  for (int j0 = blockIdx.y * chunk; j0 < j1; j0 += kVortTile) {
    const int cnt = min(kVortTile, j1 - j0);
    __syncthreads();
    for (int i = threadIdx.x; i < cnt; i += kVortThreads) {
      const size_t j = (size_t)j0 + i;
      const double x1 = x[2 * j], x2 = x[2 * j + 1];
      sh[i * W] = x1;
      sh[i * W + 1] = x2;
      static_for<0, M + 1>([&](auto sc) {
        constexpr int s = decltype(sc)::value;
#pragma unroll
        for (int k2 = 0; k2 <= s; ++k2) sh[i * W + 2 + tri(s) + k2] = mom[j * K + tri(s) + k2] * scale[s];
      });
    }
    __syncthreads();
    // FP32 offsets from the tile's first particle: exact enough for the test's
    // margin below unless the tile spans 1e5 lambda (then the margin grows)
    const double ox = sh[0], oy = sh[1];
    for (int i = threadIdx.x; i < cnt; i += kVortThreads)
      shf[i] = make_float2((float)((sh[i * W] - ox) * il), (float)((sh[i * W + 1] - oy) * il));
    __syncthreads();
    if (p >= npts) continue;
    const float qx = (float)((px - ox) * il), qy = (float)((py - oy) * il);
#pragma unroll 1
    for (int w0 = 0; w0 < cnt; w0 += 64) {
      unsigned long long near = 0;
      const int wn = min(64, cnt - w0);
      for (int i = 0; i < wn; ++i) {
        const float2 q = shf[w0 + i];
        const float dx = qx - q.x, dy = qy - q.y;
        // rounding of dx is at most 2^-23 (|qx| + |q.x|): widen the radius by that
        const float slack = 2.4e-7f * (fabsf(qx) + fabsf(q.x) + fabsf(qy) + fabsf(q.y)) + 1e-4f;
        const float r = (float)rc + slack;
        if (!(dx * dx + dy * dy > r * r)) near |= 1ull << i;
      }
      while (near) {
        const int i = w0 + __ffsll((long long)near) - 1;
        near &= near - 1;
        const double* r = sh + i * W;
        const double t1 = (px - r[0]) * il, t2 = (py - r[1]) * il;
        const double r2 = t1 * t1 + t2 * t2;
        if (r2 > cut2) continue;
        double hx[M + 1], hy[M + 1];
        hx[0] = 1.0;
        hy[0] = 1.0;
        if constexpr (M >= 1) {
          hx[1] = 2.0 * t1;
          hy[1] = 2.0 * t2;
        }
        static_for<1, M>([&](auto qc) {
          constexpr int q = decltype(qc)::value;
          hx[q + 1] = fma(hx[1], hx[q], -2.0 * q * hx[q - 1]);
          hy[q + 1] = fma(hy[1], hy[q], -2.0 * q * hy[q - 1]);
        });
        double sum = 0.0;
        static_for<0, M + 1>([&](auto kc) {
          constexpr int k2 = decltype(kc)::value;
          double part = r[2 + mcol(0, k2)];
          static_for<1, M - k2 + 1>([&](auto k1c) {
            constexpr int k1 = decltype(k1c)::value;
            part = fma(r[2 + mcol(k1, k2)], hx[k1], part);
          });
          sum = fma(part, hy[k2], sum);
        });
        acc = fma(sum, exp(-r2), acc);
      }
    }
  }
  if (p < npts) out[(size_t)blockIdx.y * npts + p] = acc * (il * il) * 0.31830988618379067154;
}

// out[p] = sum of the chunks' values in order.
__global__ void vorticity_sum_kernel(int npts, int chunks, const double* __restrict__ part,
                                     double* __restrict__ out) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= npts) return;
  double v = 0.0;
  for (int c = 0; c < chunks; ++c) v += part[(size_t)c * npts + p];
  out[p] = v;
}

// One block per ring of ntheta values: sum over the ring of (v - mean)^2.
__global__ void ring_deviation_kernel(int ntheta, const double* __restrict__ v,
                                      double* __restrict__ ring) {
  __shared__ double red[32];
  const double* w = v + (size_t)blockIdx.x * ntheta;
  auto block_sum = [&](double a) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
    __syncthreads();  // red is free
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = a;
    __syncthreads();
    double s = 0.0;
    for (int i = 0; i < (int)(blockDim.x >> 5); ++i) s += red[i];
    return s;
  };
  double a = 0.0;
  for (int i = threadIdx.x; i < ntheta; i += blockDim.x) a += w[i];
  const double mean = block_sum(a) / ntheta;
  double d = 0.0;
  for (int i = threadIdx.x; i < ntheta; i += blockDim.x) d += (w[i] - mean) * (w[i] - mean);
  const double tot = block_sum(d);
  if (threadIdx.x == 0) ring[blockIdx.x] = tot;
}

}  // namespace

int diag_max_order() { return kMaxOrderDiag; }

// Nodes and weights of n-point Gauss-Legendre quadrature on [-1, 1]: Newton's
// method on P_n (three-term recurrence (k+1) P_{k+1} = (2k+1) x P_k - k P_{k-1})
// from the usual cosine start, w = 2 / ((1 - x^2) P_n'(x)^2).
void gauss_legendre(int n, std::vector<double>& xs, std::vector<double>& ws) {
  xs.assign(n, 0.0);
  ws.assign(n, 0.0);
  for (int i = 0; i < (n + 1) / 2; ++i) {
    double z = std::cos(3.14159265358979323846 * (i + 0.75) / (n + 0.5));
    double dp = 1.0;
    for (int it = 0; it < 100; ++it) {
      double p0 = 1.0, p1 = z;
      for (int k = 1; k < n; ++k) {
        const double p2 = ((2.0 * k + 1.0) * z * p1 - k * p0) / (k + 1.0);
        p0 = p1;
        p1 = p2;
      }
      const double pn = n == 0 ? 1.0 : p1, pm = n == 0 ? 0.0 : p0;
      dp = n * (z * pn - pm) / (z * z - 1.0);
      const double dz = pn / dp;
      z -= dz;
      if (std::fabs(dz) < 1e-16) break;
    }
    xs[i] = -z;
    xs[n - 1 - i] = z;
    ws[i] = ws[n - 1 - i] = 2.0 / ((1.0 - z * z) * dp * dp);
  }
}

// Particle chunks of the order <= 8 kernel: ~16 CTAs per SM (points near the
// particles cost far more than points outside), at least 2 tiles per chunk.
int vorticity_chunks(int n, int M, int npts, int sms) {
  if (M > 8) return 1;
  const int blocks = (npts + kVortThreads - 1) / kVortThreads;
  const int want = (16 * sms + blocks - 1) / blocks;
  return std::max(1, std::min(want, n / (2 * kVortTile)));
}

cudaError_t launch_vorticity(int n, int M, const double* x, const double* mom, const double* t_dev,
                             double lam0sq, double four_nu, int npts, const double* pts,
                             double* out, double* work, int chunks, cudaStream_t st) {
  if (M < 0 || M > kMaxOrderDiag) return cudaErrorInvalidValue;
  if (M <= 8) {
    const int chunk = round_up((n + chunks - 1) / chunks, kVortTile);
    const dim3 grid(std::max(1, (npts + kVortThreads - 1) / kVortThreads), chunks);
    double* dst = chunks > 1 ? work : out;
    switch (M) {
#define MMVM_VORT_CASE(m)                                                                  \
  case m:                                                                                  \
    vorticity_low_kernel<m><<<grid, kVortThreads, 0, st>>>(n, chunk, x, mom, t_dev, lam0sq, \
                                                           four_nu, npts, pts, dst);       \
    break;
      MMVM_VORT_CASE(0) MMVM_VORT_CASE(1) MMVM_VORT_CASE(2) MMVM_VORT_CASE(3) MMVM_VORT_CASE(4)
      MMVM_VORT_CASE(5) MMVM_VORT_CASE(6) MMVM_VORT_CASE(7) MMVM_VORT_CASE(8)
#undef MMVM_VORT_CASE
    }
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess || chunks == 1) return e;
    vorticity_sum_kernel<<<(npts + 255) / 256, 256, 0, st>>>(npts, chunks, work, out);
    return cudaGetLastError();
  }
  const int K = n_moments(M);
  const int tile = std::max(1, std::min(64, 6144 / (2 + K)));
  const size_t smem = (size_t)tile * (2 + K) * sizeof(double);
  const int threads = 128;
  vorticity_kernel<<<std::max(1, (npts + threads - 1) / threads), threads, smem, st>>>(
      n, M, K, tile, x, mom, t_dev, lam0sq, four_nu, npts, pts, out);
  return cudaGetLastError();
}

cudaError_t launch_ring_deviation(int nr, int ntheta, const double* v, double* ring,
                                  cudaStream_t st) {
  ring_deviation_kernel<<<std::max(1, nr), 256, 0, st>>>(ntheta, v, ring);
  return cudaGetLastError();
}

}  // namespace mmvm
