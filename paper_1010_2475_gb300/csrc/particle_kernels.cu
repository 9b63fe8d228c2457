// Per-particle kernels of the MMVM right-hand side (FP64):
//  * prep:   core spreading lambda(t)^2 = lambda_0^2 + 4 nu t (eq:phi00) at the
//            stage time, c = 2 lambda^2, and the source records
//            (zeta = x / sqrt(c), a_m = M_m c^{-|m|/2}) for the pair kernel;
//  * finish: sum of the pair partials over source chunks, the Laplacian
//            recursion that turns them into the correlation Psi, the self pair from
//            the jet at the origin, the centroid velocity (eq:xjdot_Final, self
//            pair excluded), the moment equation (eq:Final_CrossCoef with the
//            (i,q) sums of eq:FinalSingleI/II folded into tables) including the
//            transport term C (eq:last_termsimp), and optionally the classic
//            RK4 stage combination;
//  * advance_time: t += dt after the fourth stage.
#include "particle_kernels.h"

#include <algorithm>

#include "common.cuh"

namespace mmvm {

__device__ __forceinline__ double stage_c(const double* t_dev, const double* dt_dev,
                                          double cs, double lam0sq, double four_nu) {
  const double t = *t_dev + cs * (dt_dev ? *dt_dev : 0.0);
  return 2.0 * (lam0sq + four_nu * t);
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

// Powers of the core scale and the step's weights (FinishArgs::scal): c^{-s/2},
// s = 0..M, then c^{s/2-1}, s = 0..M, then h, h/2, h/3, h/6.  One thread per
// value (thread i of at least 2 (M + 1) + 4).
__host__ __device__ constexpr int scal_len(int M) { return 2 * (M + 1) + 4; }
__device__ __forceinline__ void write_scalars(double* o, int i, int M, double c, double h) {
  if (i <= M)
    o[i] = half_power(c, -i);
  else if (i < 2 * (M + 1))
    o[i] = half_power(c, i - (M + 1) - 2);
  else if (i < scal_len(M)) {
    const int w = i - 2 * (M + 1);
    o[i] = w == 0 ? h : w == 1 ? 0.5 * h : w == 2 ? h / 3.0 : h / 6.0;
  }
}

// The source record of one particle (centre xj, moments mj): zeta = x / sqrt(c)
// (FP32: exact (hi, lo) pair), a_m = M_m c^{-|m|/2} and, for FP32 records,
// the far-field multipoles A'_n = sum_{|m|=n} a_m (-i)^{m1+n}.
template <typename T>
__device__ __forceinline__ void make_record(T* __restrict__ r, const double* __restrict__ xj,
                                            const double* __restrict__ mj, int M, int K, int R,
                                            double irc) {
  const double z1 = xj[0] * irc;
  const double z2 = xj[1] * irc;
  int h;
  if constexpr (sizeof(T) == 4) {
    const float h1 = (float)z1, h2 = (float)z2;
    r[0] = h1;
    r[1] = h2;
    r[2] = (float)(z1 - (double)h1);
    r[3] = (float)(z2 - (double)h2);
    h = 4;
  } else {
    r[0] = (T)z1;
    r[1] = (T)z2;
    h = 2;
  }
  double sc = 1.0;
  int col = 0;
  for (int s = 0; s <= M; ++s) {
    double fr = 0.0, fi = 0.0;  // A'_s
    for (int k2 = 0; k2 <= s; ++k2, ++col) {
      const double a = mj[col] * sc;
      r[h + col] = (T)a;
      switch ((s - k2 + s) & 3) {  // (-i)^{m1 + s}, m1 = s - k2
        case 0: fr += a; break;
        case 1: fi -= a; break;
        case 2: fr -= a; break;
        default: fi += a; break;
      }
    }
    if constexpr (sizeof(T) == 4) {
      r[h + K + 2 * s] = (T)fr;
      r[h + K + 2 * s + 1] = (T)fi;
    }
    sc *= irc;
  }
  for (int q = h + K + rec_far<T>(M); q < R; ++q) r[q] = T(0);
}

// The records of kGroup consecutive sorted positions by one CTA (position p
// holds particle perm[p]; perm == null: identity), values as in make_record.
// With gdata, the bounding box of the group's hi-part centres goes to the head
// of its group record (records of GL floats, see gdata_len).  Bound: latency;
// moments and records move as coalesced rows through shared memory (a thread
// per particle waited for K strided loads in turn: 31 us at n = 2011, M = 8).
constexpr int kPrepThreads = 128;
constexpr int kMaxPairM = 8;  // highest order with pair kernels
template <typename T>
__global__ void __launch_bounds__(kPrepThreads)
    prep_kernel(int n, int M, int K, int R, const int* __restrict__ perm,
                const double* __restrict__ x, const double* __restrict__ mom,
                const double* t_dev, const double* dt_dev, double cs, double lam0sq,
                double four_nu, T* __restrict__ rec, float* __restrict__ gdata, int GL,
                double* __restrict__ scal) {
  if (scal != nullptr && blockIdx.x == gridDim.x - 1) {  // the extra CTA: scalars of the finish
    for (int i = threadIdx.x; i < scal_len(M); i += blockDim.x)
      write_scalars(scal, i, M, stage_c(t_dev, dt_dev, cs, lam0sq, four_nu),
                    dt_dev ? *dt_dev : 0.0);
    return;
  }
  constexpr int H = Rec<T>::HDR;
  __shared__ double a_s[kGroup * (n_moments(kMaxPairM) | 1)];  // odd stride
  __shared__ double pw[kMaxPairM + 1];                         // c^{-s/2}
  __shared__ int j_s[kGroup];
  const int p0 = blockIdx.x * kGroup, np = min(kGroup, n - p0), KS = K | 1;
  if (threadIdx.x < kGroup) {
    const int p = p0 + threadIdx.x;
    const bool valid = p < n;
    const int j = valid ? (perm ? perm[p] : p) : 0;
    j_s[threadIdx.x] = j;
    const double irc = 1.0 / sqrt(stage_c(t_dev, dt_dev, cs, lam0sq, four_nu));
    double sc = 1.0;
    for (int s = 0; s <= M; ++s) {
      if (threadIdx.x == 0) pw[s] = sc;
      sc *= irc;
    }
    float lo1 = 3.4e38f, hi1 = -3.4e38f, lo2 = 3.4e38f, hi2 = -3.4e38f;
    if (valid) {
      const double z1 = x[2 * j] * irc, z2 = x[2 * j + 1] * irc;
      T* r = rec + (size_t)p * R;
      r[0] = (T)z1;
      r[1] = (T)z2;
      if constexpr (sizeof(T) == 4) {
        lo1 = hi1 = (float)z1;
        lo2 = hi2 = (float)z2;
        r[2] = (float)(z1 - (double)lo1);
        r[3] = (float)(z2 - (double)lo2);
      }
    }
    if (gdata) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        lo1 = fminf(lo1, __shfl_xor_sync(0xffffffffu, lo1, o));
        hi1 = fmaxf(hi1, __shfl_xor_sync(0xffffffffu, hi1, o));
        lo2 = fminf(lo2, __shfl_xor_sync(0xffffffffu, lo2, o));
        hi2 = fmaxf(hi2, __shfl_xor_sync(0xffffffffu, hi2, o));
      }
      if (threadIdx.x == 0)
        *reinterpret_cast<float4*>(gdata + (size_t)blockIdx.x * GL) =
            make_float4(lo1, hi1, lo2, hi2);
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < np * K; i += kPrepThreads) {
    const int q = i / K, col = i - q * K;
    int s = 0;
    while (tri(s + 1) <= col) ++s;
    const double a = mom[(size_t)j_s[q] * K + col] * pw[s];
    if constexpr (sizeof(T) == 4) a_s[q * KS + col] = a;
    rec[(size_t)(p0 + q) * R + H + col] = (T)a;
  }
  // A'_s = sum_k2 (-i)^{m1 + s} a, m1 = s - k2
  if constexpr (sizeof(T) == 4) {
    __syncthreads();
    const int tail = R - H - K;  // far multipoles and the padding
    for (int i = threadIdx.x; i < np * (M + 1); i += kPrepThreads) {
      const int q = i / (M + 1), s = i - q * (M + 1);
      const double* a = a_s + q * KS + tri(s);
      double fr = 0.0, fi = 0.0;
      for (int k2 = 0; k2 <= s; ++k2) switch ((s - k2 + s) & 3) {
          case 0: fr += a[k2]; break;
          case 1: fi -= a[k2]; break;
          case 2: fr -= a[k2]; break;
          default: fi += a[k2]; break;
        }
      float* r = rec + (size_t)(p0 + q) * R + H + K + 2 * s;
      r[0] = (float)fr;
      r[1] = (float)fi;
    }
    for (int i = threadIdx.x; i < np * (tail - rec_far<T>(M)); i += kPrepThreads) {
      const int w = tail - rec_far<T>(M), q = i / w;
      rec[(size_t)(p0 + q) * R + H + K + rec_far<T>(M) + i - q * w] = T(0);
    }
  } else {
    const int w = R - H - K;
    for (int i = threadIdx.x; i < np * w; i += kPrepThreads) {
      const int q = i / w;
      rec[(size_t)(p0 + q) * R + H + K + i - q * w] = T(0);
    }
  }
}

// Expansion of every group of kGroup FP32 records about its centre (the
// centre of its hi-part box; see m2p_order in common.cuh): one warp per group,
// lane s adds its A'_n delta_s^k / k! into B_{n+k}, then a warp sum; the
// radius is the largest |delta_s|.  Slots past n (or, in a batch, past their
// instance's n) do not count.
template <int M>
__global__ void group_multipole_kernel(int n, const float* __restrict__ rec,
                                       float* __restrict__ gdata,
                                       const BatchInst* __restrict__ inst,
                                       const int* __restrict__ slot_inst,
                                       const int* __restrict__ n_slots) {
  constexpr int K = n_moments(M), R = rec_len<float>(M), P = m2p_order(M);
  constexpr int NA = m2p_terms(M), GL = gdata_len(M), H = Rec<float>::HDR;
  const int total = n_slots ? *n_slots : n;
  const int lane = threadIdx.x & 31;
  const int nwarps = (gridDim.x * blockDim.x) >> 5;
  for (int g = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; g * kGroup < total; g += nwarps) {
    const int p = g * kGroup + lane;
    bool valid = p < total;
    if (valid && inst) {
      const BatchInst& I = inst[slot_inst[g]];
      valid = p - I.slot0 < I.n;
    }
    float* gd = gdata + (size_t)g * GL;
    const float4 box = *reinterpret_cast<const float4*>(gd);
    const float cx = 0.5f * (box.x + box.y), cy = 0.5f * (box.z + box.w);
    float dr = 0.f, di = 0.f, ar[M + 1], ai[M + 1];
#pragma unroll
    for (int q = 0; q <= M; ++q) {
      ar[q] = 0.f;
      ai[q] = 0.f;
    }
    if (valid) {
      const float* r = rec + (size_t)p * R;
      dr = (r[0] - cx) + r[2];
      di = (r[1] - cy) + r[3];
#pragma unroll
      for (int q = 0; q <= M; ++q) {
        ar[q] = r[H + K + 2 * q];
        ai[q] = r[H + K + 2 * q + 1];
      }
    }
    float br[NA], bi[NA];
#pragma unroll
    for (int j = 0; j < NA; ++j) {
      br[j] = 0.f;
      bi[j] = 0.f;
    }
    float er = 1.f, ei = 0.f;  // delta^k / k!
    static_for<0, P + 1>([&](auto kc) {
      constexpr int k = decltype(kc)::value;
      if constexpr (k > 0) {
        const float tr = (er * dr - ei * di) * (1.f / k);
        ei = (er * di + ei * dr) * (1.f / k);
        er = tr;
      }
      static_for<0, M + 1>([&](auto qc) {
        constexpr int q = decltype(qc)::value;
        br[q + k] = fmaf(ar[q], er, fmaf(-ai[q], ei, br[q + k]));
        bi[q + k] = fmaf(ar[q], ei, fmaf(ai[q], er, bi[q + k]));
      });
    });
    float rad2 = dr * dr + di * di;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      rad2 = fmaxf(rad2, __shfl_xor_sync(0xffffffffu, rad2, o));
#pragma unroll
      for (int j = 0; j < NA; ++j) {
        br[j] += __shfl_xor_sync(0xffffffffu, br[j], o);
        bi[j] += __shfl_xor_sync(0xffffffffu, bi[j], o);
      }
    }
    if (lane == 0) {
      *reinterpret_cast<float4*>(gd + 4) = make_float4(cx, cy, sqrtf(rad2), 0.f);
#pragma unroll
      for (int j = 0; j < NA; ++j) {
        gd[8 + 2 * j] = br[j];
        gd[9 + 2 * j] = bi[j];
      }
    }
  }
}

// v[0] + v[stride] + ... (n values) as four interleaved sums: fixed order, a
// quarter of the dependent additions, several loads in flight.
__device__ __forceinline__ double block_sum(const double* __restrict__ v, int n, size_t stride) {
  double s[4] = {0.0, 0.0, 0.0, 0.0};
  int i = 0;
#pragma unroll 2
  for (; i + 4 <= n; i += 4) {
#pragma unroll
    for (int q = 0; q < 4; ++q) s[q] += v[(size_t)(i + q) * stride];
  }
#pragma unroll
  for (int q = 0; q < 3; ++q)
    if (i + q < n) s[q] += v[(size_t)(i + q) * stride];
  return (s[0] + s[1]) + (s[2] + s[3]);
}

// The finish of TG targets (sorted positions j0 .. j0 + TG - 1, those below
// A.n) by one CTA, row blocks [rb0, rb1) of the table.
//
// Bound: FP64 arithmetic.  An FP64 instruction keeps this SM's pipe busy for 16
// cycles however few of its lanes are active, so what counts is lanes in use:
//  * per target NB K / 4 multiply-adds of the self pair, one addition per
//    partial block and column, one multiply-add per table entry and one per
//    (k, l) group (4214 at M = 6);
//  * a thread takes whole groups for one target; groups are sorted by length,
//    so a warp's lanes run loops of (nearly) one length.  (A thread per row, 0
//    to 260 entries, kept 2/3 of the lanes idle; closing groups of mixed
//    lengths inside one loop executed a second multiply-add per entry.)
//  * scalars (powers of c, weights of the step) come from the record kernel;
//    without one (a single particle, batches) two warps form them.
// Before / now: 420 / 327 us at n = 24000, M = 6, 199 / 183 us at n = 2011, M = 8.
// Shared memory holds [column][target] arrays: Psi (NB), a (K), X (2), the
// scalars and the groups' sums.  Every global read of the stage input
// precedes the first write behind a barrier.  All threads of the CTA call this;
// a caller that loops must add a barrier.
template <int TG>
__device__ __forceinline__ void finish_block(const FinishArgs& A, int j0, int rb0, int rb1,
                                             double* sm) {
  const int NB = A.NB, K = A.K, M = A.M, NT = blockDim.x;
  double* psi = sm;                 // NB * TG
  double* at = psi + NB * TG;       // K * TG
  double* X = at + K * TG;          // 2 * TG
  double* cpow = X + 2 * TG;        // the scalars
  double* cinv = cpow + M + 1;
  double* hs = cinv + M + 1;
  double* gsum = hs + 4;            // max_groups * TG
  // 1. the scalars, the stage moments, Psi_excl = sum over the partial blocks
  //    (fixed order)
  if (A.scal) {
    for (int i = threadIdx.x; i < scal_len(M); i += NT) cpow[i] = A.scal[i];
  } else if (threadIdx.x >= NT - 64) {
    write_scalars(cpow, threadIdx.x - (NT - 64), M,
                  stage_c(A.t_dev, A.dt_dev, A.cs, A.lam0sq, A.four_nu),
                  A.dt_dev ? *A.dt_dev : 0.0);
  }
  for (int idx = threadIdx.x; idx < TG * K; idx += NT) {
    const int tt = idx / K, m = idx % K, p = j0 + tt;
    const int j = p < A.n ? (A.perm ? A.perm[p] : p) : 0;
    const double mv = (p < A.n) ? A.Min[(size_t)j * K + m] : 0.0;
    at[m * TG + tt] = p < A.n || m ? mv : 1.0;
  }
  for (int idx = threadIdx.x; idx < TG * NB; idx += NT) {
    const int tt = idx % TG, b = idx / TG, j = j0 + tt;
    double v = 0.0;
    if (j < A.n && A.partial) {
      const double* pb = A.partial + (size_t)b * A.n + j;
      const size_t bs = (size_t)NB * A.n;
      v = block_sum(pb, A.gshares ? A.gshares[j / kGroup] : A.nchunks, bs);
      if (A.local_block >= 0) v += pb[A.local_block * bs];
      // far field of the list form: edge columns only
      if (A.fpart &&
          !(A.rmax > 0.f && A.gdata[(size_t)(j / kGroup) * A.gdata_len + 6] <= A.rmax)) {
        int bn = 1;
        while (tri(bn + 1) - 1 <= b) ++bn;
        const int b1 = bn - (b + 1 - tri(bn));
        if (b1 <= 1)
          v += block_sum(A.fpart + (size_t)(2 * (bn - 1) + b1) * A.n + j, A.nfar,
                         (size_t)A.n_edge * A.n);
      }
    }
    psi[b * TG + tt] = v;
  }
  __syncthreads();
  for (int idx = TG + threadIdx.x; idx < TG * K; idx += NT) {
    int s = 0;
    while (tri(s + 1) <= idx / TG) ++s;  // total order of the column
    at[idx] *= cpow[s];
  }
  if (!A.partial) __syncthreads();
  if (A.partial) {
    // 1b. the pair kernels leave Psi itself only in the edge columns beta1 <= 1;
    //     a column beta1 >= 2 holds R[beta] = sum_m a_m D^{m + beta - 2 e1} Lap psi.
    //     D_1^2 = Lap - D_2^2 gives Psi[beta] = R[beta] - Psi[beta - 2 e1 + 2 e2],
    //     taken per order in increasing beta1.
    const int BM = bmax_of(M);
    for (int idx = threadIdx.x; idx < TG * BM; idx += NT) {
      const int tt = idx % TG, k = idx / TG + 1;
      double* ps = psi + tt;
      for (int b1 = 2; b1 <= k; ++b1)
        ps[bcol(b1, k - b1) * TG] -= ps[bcol(b1 - 2, k - b1 + 2) * TG];
    }
    __syncthreads();  // Psi and the scaled moments
    // 2. centroid sums X_c = sum_m (-1)^{|m|} a_m What_c[m], What_1[m] = -Psi[m+e2],
    //    What_2[m] = Psi[m+e1]  (eq:xjdot_Final in c = 1 units, self pair excluded),
    //    over M_00 (the quotient: 1 / M_00 is infinite below 2^-1024);
    //    the columns m of one (target, component) are split over q lanes
    const int q = min(32, NT / (2 * TG));
    if (threadIdx.x < 2 * TG * q) {  // whole warps: 2 TG q is a multiple of 32 here
      const int part = threadIdx.x % q, tt = (threadIdx.x / q) >> 1, comp = (threadIdx.x / q) & 1;
      double acc = 0.0;
      for (int col = part; col < K; col += q) {
        int s = 0;
        while (tri(s + 1) <= col) ++s;
        const int m2 = col - tri(s), m1 = s - m2;
        const double a = ((s & 1) == comp) ? -at[col * TG + tt] : at[col * TG + tt];
        acc = fma(a, psi[(comp == 0 ? bcol(m1, m2 + 1) : bcol(m1 + 1, m2)) * TG + tt], acc);
      }
      for (int o = q >> 1; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
      if (part == 0) X[2 * tt + comp] = acc / at[tt];
    }
    __syncthreads();
  } else if (threadIdx.x < 2 * TG) {
    X[threadIdx.x] = 0.0;
  }
  // 3. add the self pair: Psi_self[beta] = sum_m a_m psi0[m + beta] (psi0
  //    vanishes at odd indices: only m of the parity of beta contribute).  One
  //    row m1 after another; with few targets the rows of a beta are shared by
  //    SP neighbouring lanes (a lone particle of order 10 waited 6 us for one
  //    thread's 36 terms).
  constexpr int SP = TG == 1 ? 4 : 1;
  for (int i0 = 0; i0 < TG * NB * SP; i0 += NT) {  // whole warps take part in the sums
    const int idx = i0 + threadIdx.x, part = idx % SP, bt = idx / SP;
    const int tt = bt % TG, b = bt / TG;
    double acc = 0.0;
    if (b < NB) {
      int bn = 1;
      while (tri(bn + 1) - 1 <= b) ++bn;
      const int b2 = b + 1 - tri(bn), b1 = bn - b2;
      for (int m1 = (b1 & 1) + 2 * part; m1 <= M; m1 += 2 * SP) {
#pragma unroll 4
        for (int m2 = b2 & 1; m2 <= M - m1; m2 += 2) {
          const int a2 = m2 + b2;
          acc = fma(at[mcol(m1, m2) * TG + tt], __ldg(A.tab.psi0 + tri(m1 + b1 + a2) + a2), acc);
        }
      }
    }
    if constexpr (SP > 1) {
#pragma unroll
      for (int o = SP >> 1; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    }
    if (b < NB && part == 0) psi[b * TG + tt] += acc;
  }
  __syncthreads();
  for (int rb = rb0; rb < rb1; ++rb) {
  const RowBlock B = A.tab.blocks[rb];
  // 4. the groups of the table: g = sum_beta c Psi[beta]; with one target the
  //    entries of a group are shared by GL neighbouring lanes (a lone particle
  //    of order 10 otherwise waits for up to 110 dependent loads and additions)
  {
    constexpr int GL = TG == 1 ? 4 : 1;
    const int tt = threadIdx.x % TG, part = threadIdx.x % GL;
    const double* ps = psi + tt;
    const int* off = A.tab.offs + B.off_at;
    for (int q0 = 0; q0 < B.groups; q0 += NT / (TG * GL)) {  // whole warps stay together
      const int q = q0 + threadIdx.x / (TG * GL);
      const int len = q < B.groups ? __ldg(A.tab.glen + B.len_at + q) : 0;
      const double2* e = reinterpret_cast<const double2*>(A.tab.tab) + q;
      double g = 0.0;
#pragma unroll 4
      for (int j = part; j < len; j += GL) {
        const double2 v = __ldg(e + __ldg(off + j));  // (c, packed b)
        g = fma(v.x, ps[(int)(__double_as_longlong(v.y) & 0xffffffffll) * TG], g);
      }
      if constexpr (GL > 1) {
#pragma unroll
        for (int o = GL >> 1; o > 0; o >>= 1) g += __shfl_xor_sync(0xffffffffu, g, o);
      }
      if (q < B.groups && part == 0) gsum[q * TG + tt] = g;
    }
  }
  __syncthreads();
  // 5. moment equation and stage update per (target, k): R_k = sum_l a_l g_kl,
  //    the l shared by RL neighbouring lanes
  const int k0 = B.k0, nk = B.k1 - B.k0;
  constexpr int RL = TG == 1 ? 16 : 1;
  for (int i0 = 0; i0 < TG * nk * RL; i0 += NT) {  // whole warps take part in the sums
    const int it = i0 + threadIdx.x, part = it % RL, idx = it / RL;
    const bool on = idx < TG * nk;
    const int tt = on ? idx % TG : 0, k = on ? k0 + idx / TG : k0, p = j0 + tt;
    double R = 0.0;
    if (on) {
      const int e1 = A.tab.rows_off[k + 1];
#pragma unroll 4
      for (int e = A.tab.rows_off[k] + part; e < e1; e += RL) {
        const int2 w = __ldg(reinterpret_cast<const int2*>(A.tab.rows) + e);  // (q, l)
        R = fma(at[w.y * TG + tt], gsum[w.x * TG + tt], R);
      }
    }
    if constexpr (RL > 1) {
#pragma unroll
      for (int o = RL >> 1; o > 0; o >>= 1) R += __shfl_xor_sync(0xffffffffu, R, o);
    }
    if (!on || part != 0 || p >= A.n) continue;
    const int j = A.perm ? A.perm[p] : p;
    int kn = 0;
    while (tri(kn + 1) <= k) ++kn;
    const int k2 = k - tri(kn), k1c = kn - k2;
    double ctr = 0.0;
    if (k1c >= 1) ctr += X[2 * tt] * at[mcol(k1c - 1, k2) * TG + tt];
    if (k2 >= 1) ctr += X[2 * tt + 1] * at[mcol(k1c, k2 - 1) * TG + tt];
    const double dm = (R + ctr) * cinv[kn];  // c^{|k|/2 - 1}
    const size_t o = (size_t)j * K + k;
    if (A.mode == 0) {
      A.out_dM[o] = dm;
    } else {
      const double base = A.y_M[o];
      if (A.mode == 1) { A.ys_M[o] = base + hs[1] * dm; A.sum_M[o] = base + hs[3] * dm; }
      if (A.mode == 2) { A.ys_M[o] = base + hs[1] * dm; A.sum_M[o] += hs[2] * dm; }
      if (A.mode == 3) { A.ys_M[o] = base + hs[0] * dm; A.sum_M[o] += hs[2] * dm; }
      if (A.mode == 4) { A.y_M[o] = A.sum_M[o] + hs[3] * dm; }
    }
  }
  if (rb + 1 < rb1) __syncthreads();  // the group sums are reused
  }
  // 6. centroid velocity xdot_c = c^{-1/2} X_c and its stage update
  if (rb0 != 0) return;
  // c^{-1/2} (order 0 has only c^0 in its powers, and c^{-1})
  const double cpow1 = M >= 1 ? cpow[1] : sqrt(cinv[0]);
  for (int idx = threadIdx.x; idx < TG * 2; idx += NT) {
    const int tt = idx >> 1, comp = idx & 1, p = j0 + tt;
    if (p >= A.n) continue;
    const int j = A.perm ? A.perm[p] : p;
    const double dx = X[idx] * cpow1;
    const size_t ox = (size_t)j * 2 + comp;
    if (A.mode == 0) {
      A.out_dx[ox] = dx;
    } else {
      const double base = A.y_x[ox];
      if (A.mode == 1) { A.ys_x[ox] = base + hs[1] * dx; A.sum_x[ox] = base + hs[3] * dx; }
      if (A.mode == 2) { A.ys_x[ox] = base + hs[1] * dx; A.sum_x[ox] += hs[2] * dx; }
      if (A.mode == 3) { A.ys_x[ox] = base + hs[0] * dx; A.sum_x[ox] += hs[2] * dx; }
      if (A.mode == 4) { A.y_x[ox] = A.sum_x[ox] + hs[3] * dx; }
    }
  }
}

constexpr int kFinishThreads = 256;

// Grid: (target blocks, row blocks); row blocks are used for n == 1 only.
template <int TG>
__global__ void __launch_bounds__(kFinishThreads) finish_kernel(FinishArgs A) {
  extern __shared__ double sm[];
  const bool split = gridDim.y > 1;
  finish_block<TG>(A, blockIdx.x * TG, split ? blockIdx.y : 0, split ? blockIdx.y + 1 : A.tab.nrb,
                   sm);
}

__global__ void advance_time_kernel(double* t_dev, const double* dt_dev) {
  if (threadIdx.x == 0 && blockIdx.x == 0) *t_dev += *dt_dev;
}

// Non-finite / zero-circulation scan of a state (flags[0]: non-finite,
// flags[1]: zero circulation); used after set_state and on demand.
__global__ void scan_state_kernel(int n, int K, const double* __restrict__ x,
                                  const double* __restrict__ mom, int* flags) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= n) return;
  bool bad = !isfinite(x[2 * j]) || !isfinite(x[2 * j + 1]);
  for (int m = 0; m < K; ++m) bad |= !isfinite(mom[(size_t)j * K + m]);
  if (bad) atomicOr(flags, 1);
  if (mom[(size_t)j * K] == 0.0) atomicOr(flags + 1, 1);
}

// ------------------------------------------------------------------ batches
// Offsets of the state blocks of one instance (see BatchInst).
__device__ __forceinline__ const double* inst_stage_x(const BatchInst& I, int K, int src) {
  return I.state + (src ? (size_t)I.n * (2 + K) : 0);
}
__device__ __forceinline__ const double* inst_stage_m(const BatchInst& I, int K, int src) {
  return inst_stage_x(I, K, src) + 2 * (size_t)I.n;
}

// Records of every instance of a batch of one order: slot p belongs to
// instance slot_inst[p / kGroup]; padding slots past an instance's n are not
// written (no kernel reads them).  src = 0 reads the step-start state y,
// src = 1 the stage state ys; the core is taken at t + cs dt of each instance.
// With perm_local, sorted slot p holds local particle perm_local[p]; with
// gdata, every warp (one group of kGroup slots: the loop keeps warps aligned
// to groups and n_slots is a multiple of kGroup) writes its group's box at
// the head of the group's record (GL floats).
template <typename T>
__global__ void prep_batch_kernel(int M, int K, int R, const BatchInst* __restrict__ inst,
                                  const int* __restrict__ slot_inst,
                                  const int* __restrict__ n_slots, int src, double cs,
                                  const int* __restrict__ perm_local, T* __restrict__ rec,
                                  float* __restrict__ gdata, int GL) {
  const int total = *n_slots;
  for (int base = blockIdx.x * blockDim.x; base < total; base += gridDim.x * blockDim.x) {
    const int p = base + threadIdx.x;  // whole warps are in or out of range
    if (p >= total) continue;
    const BatchInst& I = inst[slot_inst[p / kGroup]];
    const int j = p - I.slot0;
    float lo1 = 3.4e38f, hi1 = -3.4e38f, lo2 = 3.4e38f, hi2 = -3.4e38f;
    if (j < I.n) {
      const int jj = perm_local ? perm_local[p] : j;
      const double c = 2.0 * (I.lam0sq + I.four_nu * (I.t + cs * I.dt));
      T* r = rec + (size_t)p * R;
      make_record<T>(r, inst_stage_x(I, K, src) + 2 * jj, inst_stage_m(I, K, src) + (size_t)jj * K,
                     M, K, R, 1.0 / sqrt(c));
      if constexpr (sizeof(T) == 4) {
        lo1 = hi1 = r[0];
        lo2 = hi2 = r[1];
      }
    }
    if (gdata) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        lo1 = fminf(lo1, __shfl_xor_sync(0xffffffffu, lo1, o));
        hi1 = fmaxf(hi1, __shfl_xor_sync(0xffffffffu, hi1, o));
        lo2 = fminf(lo2, __shfl_xor_sync(0xffffffffu, lo2, o));
        hi2 = fmaxf(hi2, __shfl_xor_sync(0xffffffffu, hi2, o));
      }
      if ((threadIdx.x & 31) == 0)
        *reinterpret_cast<float4*>(gdata + (size_t)(p / kGroup) * GL) =
            make_float4(lo1, hi1, lo2, hi2);
    }
  }
}

// Finish of every instance of a batch: item (instance, first target) per
// block of TG targets; blocks loop over the items.
template <int TG>
__global__ void __launch_bounds__(kFinishThreads) finish_batch_kernel(BatchFinishArgs B) {
  extern __shared__ double sm[];
  const int total = *B.n_items;
  for (int it = blockIdx.x; it < total; it += gridDim.x) {
    const int2 w = B.items[it];
    const BatchInst& I = B.inst[w.x];
    const size_t blk = (size_t)I.n * (2 + B.K);
    FinishArgs A;
    A.n = I.n;
    A.M = B.M;
    A.K = B.K;
    A.NB = B.NB;
    A.nchunks = I.n > 1 ? I.chunks : 0;
    A.partial = I.n > 1 ? B.partial + I.part_off : nullptr;
    A.perm = B.perm_local ? B.perm_local + I.slot0 : nullptr;
    A.Min = inst_stage_m(I, B.K, B.src);
    A.tab = B.tab;
    A.lam0sq = I.lam0sq;
    A.four_nu = I.four_nu;
    A.t_dev = &I.t;
    A.dt_dev = &I.dt;
    A.cs = B.cs;
    A.mode = B.mode;
    A.y_x = I.state;
    A.y_M = I.state + 2 * (size_t)I.n;
    A.ys_x = I.state + blk;
    A.ys_M = I.state + blk + 2 * (size_t)I.n;
    A.sum_x = I.state + 2 * blk;
    A.sum_M = I.state + 2 * blk + 2 * (size_t)I.n;
    finish_block<TG>(A, w.y, 0, B.tab.nrb, sm);
    __syncthreads();  // shared memory is reused by the next item
  }
}

__global__ void advance_batch_kernel(BatchInst* __restrict__ inst, const int* __restrict__ n_inst) {
  const int total = *n_inst;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < total; i += gridDim.x * blockDim.x)
    inst[i].t += inst[i].dt;
}

// flags[i] = 1 if the step-start state of instance i holds a non-finite value,
// else 0; one block per instance (blocks loop over the instances).
__global__ void scan_batch_kernel(int K, const BatchInst* __restrict__ inst,
                                  const int* __restrict__ n_inst, int* __restrict__ flags) {
  const int total = *n_inst;
  for (int i = blockIdx.x; i < total; i += gridDim.x) {
    const BatchInst& I = inst[i];
    const size_t len = (size_t)I.n * (2 + K);
    bool bad = false;
    for (size_t q = threadIdx.x; q < len; q += blockDim.x) bad |= !isfinite(I.state[q]);
    bad = __syncthreads_or(bad);
    if (threadIdx.x == 0) flags[i] = bad ? 1 : 0;
  }
}

cudaError_t launch_scan_batch(int M, const BatchInst* inst, const int* n_inst, int max_inst,
                              int* flags, cudaStream_t st) {
  scan_batch_kernel<<<std::max(1, std::min(max_inst, 1024)), 256, 0, st>>>(n_moments(M), inst,
                                                                          n_inst, flags);
  return cudaGetLastError();
}

cudaError_t launch_prep_batch(int precision, int M, const BatchInst* inst, const int* slot_inst,
                              const int* n_slots, int max_slots, int src, double cs,
                              const int* perm_local, void* rec, void* gbox, cudaStream_t st) {
  const int K = n_moments(M);
  const int threads = 128, blocks = std::max(1, std::min((max_slots + threads - 1) / threads, 4096));
  if (precision == 1) {
    prep_batch_kernel<float><<<blocks, threads, 0, st>>>(M, K, rec_len<float>(M), inst, slot_inst,
                                                         n_slots, src, cs, perm_local,
                                                         (float*)rec, (float*)gbox,
                                                         gdata_len(M));
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess || !gbox) return e;
    return launch_group_multipole(M, 0, rec, gbox, inst, slot_inst, n_slots, max_slots, st);
  }
  prep_batch_kernel<double><<<blocks, threads, 0, st>>>(M, K, rec_len<double>(M), inst, slot_inst,
                                                        n_slots, src, cs, perm_local,
                                                        (double*)rec, nullptr, 0);
  return cudaGetLastError();
}

// Shared memory of a finish CTA of TG targets.
size_t finish_smem_bytes(int M, int TG, const FinishTab& tab) {
  return sizeof(double) *
         ((size_t)TG * (n_beta(M) + n_moments(M) + 2 + tab.max_groups) + scal_len(M));
}

// Call f(kernel of TG targets) for the run-time TG in {1, 2, 4, 8}.
template <typename F>
cudaError_t with_targets(int TG, F&& f) {
  switch (TG) {
    case 1: return f(std::integral_constant<int, 1>{});
    case 2: return f(std::integral_constant<int, 2>{});
    case 4: return f(std::integral_constant<int, 4>{});
    default: return f(std::integral_constant<int, 8>{});
  }
}

// Targets per batch item: instances of 64 to 8192 particles give 8-target
// items enough CTAs; orders above the pair limit hold one particle.
int finish_batch_targets(int M) { return M > 8 ? 1 : M > 6 ? 4 : 8; }

cudaError_t launch_finish_batch(const BatchFinishArgs& B, int grid, cudaStream_t st) {
  const int TG = finish_batch_targets(B.M);
  const size_t smem = finish_smem_bytes(B.M, TG, B.tab);
  return with_targets(TG, [&](auto tg) {
    constexpr int T = decltype(tg)::value;
    if (smem > 48 * 1024) {
      cudaError_t e = cudaFuncSetAttribute(
          finish_batch_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
      if (e != cudaSuccess) return e;
    }
    finish_batch_kernel<T><<<std::max(1, grid), kFinishThreads, smem, st>>>(B);
    return cudaGetLastError();
  });
}

cudaError_t launch_advance_batch(BatchInst* inst, const int* n_inst, int max_inst,
                                 cudaStream_t st) {
  advance_batch_kernel<<<std::max(1, (max_inst + 127) / 128), 128, 0, st>>>(inst, n_inst);
  return cudaGetLastError();
}

cudaError_t launch_group_multipole(int M, int n, const void* rec, void* gdata,
                                   const BatchInst* inst, const int* slot_inst,
                                   const int* n_slots, int max_slots, cudaStream_t st) {
  const int groups = (max_slots + kGroup - 1) / kGroup;
  const int threads = 128, blocks = std::max(1, std::min((groups * 32 + threads - 1) / threads, 4096));
  const float* r = static_cast<const float*>(rec);
  float* g = static_cast<float*>(gdata);
  switch (M) {
#define MMVM_GM_CASE(m)                                                                  \
  case m:                                                                                \
    group_multipole_kernel<m><<<blocks, threads, 0, st>>>(n, r, g, inst, slot_inst, n_slots); \
    break;
    MMVM_GM_CASE(0) MMVM_GM_CASE(1) MMVM_GM_CASE(2) MMVM_GM_CASE(3) MMVM_GM_CASE(4)
    MMVM_GM_CASE(5) MMVM_GM_CASE(6) MMVM_GM_CASE(7) MMVM_GM_CASE(8)
#undef MMVM_GM_CASE
    default:
      return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

cudaError_t launch_prep(int precision, int n, int M, const int* perm, const double* x,
                        const double* mom, const double* t_dev, const double* dt_dev, double cs,
                        double lam0sq, double four_nu, void* rec, void* gbox, double* scal,
                        cudaStream_t st) {
  const int K = n_moments(M);
  const int threads = kPrepThreads, blocks = (n + kGroup - 1) / kGroup + (scal ? 1 : 0);
  if (precision == 1) {
    prep_kernel<float><<<blocks, threads, 0, st>>>(n, M, K, rec_len<float>(M), perm, x, mom,
                                                   t_dev, dt_dev, cs, lam0sq, four_nu,
                                                   (float*)rec, (float*)gbox, gdata_len(M), scal);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess || !gbox) return e;
    return launch_group_multipole(M, n, rec, gbox, nullptr, nullptr, nullptr, n, st);
  }
  prep_kernel<double><<<blocks, threads, 0, st>>>(n, M, K, rec_len<double>(M), perm, x, mom,
                                                  t_dev, dt_dev, cs, lam0sq, four_nu,
                                                  (double*)rec, nullptr, 0, scal);
  return cudaGetLastError();
}

int finish_scalars(int M) { return scal_len(M); }

// Targets per finish CTA: 8 keep every lane of the FP64 instructions in use (the
// group sums of 8 targets at M = 6 take 48 KB; orders 7 and 8, with up to 127
// KB, take 4), fewer while there are not 3 CTAs per SM.
int finish_targets(int n, int M, int sms) {
  for (int TG : {8, 4, 2})
    if (!(TG == 8 && M > 6) && (n + TG - 1) / TG >= 3 * sms) return TG;
  return 1;
}

cudaError_t launch_finish(const FinishArgs& A, int sms, cudaStream_t st) {
  const int TG = finish_targets(A.n, A.M, sms);
  const int rb = A.n == 1 ? A.tab.nrb : 1;
  const size_t smem = finish_smem_bytes(A.M, TG, A.tab);
  return with_targets(TG, [&](auto tg) {
    constexpr int T = decltype(tg)::value;
    if (smem > 48 * 1024) {
      cudaError_t e = cudaFuncSetAttribute(
          finish_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
      if (e != cudaSuccess) return e;
    }
    finish_kernel<T><<<dim3((A.n + T - 1) / T, rb), kFinishThreads, smem, st>>>(A);
    return cudaGetLastError();
  });
}

cudaError_t launch_advance_time(double* t_dev, const double* dt_dev, cudaStream_t st) {
  advance_time_kernel<<<1, 32, 0, st>>>(t_dev, dt_dev);
  return cudaGetLastError();
}

cudaError_t launch_scan(int n, int K, const double* x, const double* mom, int* flags,
                        cudaStream_t st) {
  scan_state_kernel<<<(n + 127) / 128, 128, 0, st>>>(n, K, x, mom, flags);
  return cudaGetLastError();
}

}  // namespace mmvm
