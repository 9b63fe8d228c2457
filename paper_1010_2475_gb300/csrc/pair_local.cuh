// Local expansions: near pairs of two compact groups through the groups'
// expansions (list form, FP32 records with the far field).
//
// Every term of the pair sums is a derivative of the stream function psi of
// the sqrt(2) lambda Gaussian, an entire function, so the field of a whole
// source group may be expanded about its centre s0 and the field at a target
// group about its centre t0 whatever their distance.  In c = 1 units, with
// P(D) = sum_{|k| <= Q} A_k D^k the expansion of a group,
//     A_k = sum_s sum_{m <= k} a_{s,m} (-delta_s)^{k-m} / (k-m)!,
//     F(t0 + tau) = sum_n F_n tau^n / n!,   F_n = P(D) D^n psi(t0 - s0),
// the correlation at a target is Psi[beta] = D^beta F.  F is carried as its
// Laplacian G = P(D) e^{-x}/pi (|n| <= NL - 2) and its two edge columns per
// order, E0[n] = F_(0,n) and E1[n] = F_(1,n) (order n + 1), from which
// F_n = G_{n - 2 e1} - F_{n - 2 e1 + 2 e2} gives the rest.
//  * G_n = sum_k A_k h_{k1+n1}(b1) h_{k2+n2}(b2) with the Hermite functions of
//    the Gaussian, taken over k2, then over k1.
//  * P = P_e + (D1^2 + D2^2) S with P_e of degree <= 1 in D1, so the edges are
//    P_e on the edge derivatives e_N = D2^N psi, f_N = D1 D2^{N-1} psi plus S on
//    Hermite functions.
//  * r psi_r = (1 - e^{-x}) / 2 pi and the rotation invariance of psi give
//      x1 f_{N+1} + x2 e_{N+1} = -N e_N - h_N,  x1 e_{N+1} - x2 f_{N+1} = N f_N
//    (for 2 pi psi, h_N = D2^N e^{-x}): run upward for N < x, where it is stable, downward
//    from the top order for N > x.  The top order comes from the holomorphic
//    edge and the Gaussian's projection as in pair_kernel.cuh, the binomial
//    sums folded into constants.
// All derivatives of order N carry a factor 4^-N (an exact power of two):
// h_50 would leave the FP32 range.  They are those of 2 pi psi, whose constants
// are exact in FP32; the factor 1 / 2 pi is applied in FP64 at the end (an FP32
// 1 / 2 pi is 4e-8 off, as much as the rounding of a velocity).
//
// Cost at M = 6 (Q = 23, NL = 29): about 1400 multiply-adds per lane for the
// 1024 pairs of two groups, against 32 x 2153 pair by pair.  Groups wider than
// loc_radius(M) and groups close to each other (loc_pair; the target group
// itself among them) stay with the pair kernels.
// Measured (two patches, n = 65536, M = 6, one right-hand side): all-pairs
// kernels 68.6 -> 16.1 ms (near pairs one by one 6.6e8 -> 1.2e8, far field 4.0 ->
// 1.3 ms).
#pragma once

#include "pair_list.cuh"

namespace mmvm {

constexpr float kLocScale = 0.25f;  // factor per derivative order

template <int M>
struct Loc {
  static constexpr int P = loc_extra(M);
  static constexpr int Q = M + P;             // orders of a group's expansion
  static constexpr int NL = bmax_of(M) + P;   // orders of a target group's field
  static constexpr int NG = NL - 2;           // orders of its Laplacian
  static constexpr int NT = Q + NL;           // highest derivative order
  static constexpr int ROWS = 32 + Q + 2;     // table rows (lane + k, k <= Q + 1)
  static_assert(NL <= 31, "one lane per order of the field");
  static_assert(loc_radius(M) <= loc_field_radius(M), "a near field needs its far field's evaluation");
  // Expansion record of a group: rows k1 of A, rows k1 of S (k2 contiguous,
  // rows padded to 4 floats), then the degree 0 and 1 parts of P_e.
  __host__ __device__ static constexpr int row_len(int top, int k1) { return (top - k1 + 1 + 3) / 4 * 4; }
  __host__ __device__ static constexpr int off_a(int k1) {
    int o = 0;
    for (int i = 0; i < k1; ++i) o += row_len(Q, i);
    return o;
  }
  __host__ __device__ static constexpr int off_s(int k1) {
    int o = off_a(Q + 1);
    for (int i = 0; i < k1; ++i) o += row_len(Q - 2, i);
    return o;
  }
  static constexpr int off_p0 = off_s(Q - 1);
  static constexpr int off_p1 = off_p0 + row_len(Q, 0);
  static constexpr int LEN = off_p1 + row_len(Q, 0);
  // Field record of a target group: rows of 32 lanes, G rows n1 = 0..NG (lane
  // n2), then E0 (lane n: beta (0, n)) and E1 (lane n: beta (1, n)).
  static constexpr int FROWS = NG + 3;
};

// ------------------------------------------------------------------ group expansions
// One warp per eligible group: lane k2 sums its column of A over the sources,
// then the division by D1^2 + D2^2, one lane per order.
template <int M>
__global__ void __launch_bounds__(32)
    loc_expand_kernel(const float* __restrict__ rec, int n, int G,
                      const float* __restrict__ gdata, float* __restrict__ gexp) {
  using L = Loc<M>;
  constexpr int R = rec_len<float>(M), K = n_moments(M), GL = gdata_len(M), Q = L::Q;
  constexpr int ST = 33;
  __shared__ float px[(Q + 1) * ST], py[(Q + 1) * ST];
  __shared__ float as[(Q + 1) * (Q + 2)];
  const int lane = threadIdx.x, g = blockIdx.x;  // one warp per CTA: groups spread over the SMs
  const float4 cen = *reinterpret_cast<const float4*>(gdata + (size_t)g * GL + 4);
  if (!(cen.z <= loc_radius(M))) return;
  const int cnt = min(kGroup, n - g * kGroup);
  {  // lane = source: (-delta / scale)^j / j!
    const float* r = rec + (size_t)(g * kGroup + min(lane, cnt - 1)) * R;
    const float tx = -((r[0] - cen.x) + r[2]) * (1.f / kLocScale);
    const float ty = -((r[1] - cen.y) + r[3]) * (1.f / kLocScale);
    float vx = 1.f, vy = 1.f;
#pragma unroll
    for (int j = 0; j <= Q; ++j) {
      if (j > 0) {
        vx *= tx * (1.f / j);
        vy *= ty * (1.f / j);
      }
      px[j * ST + lane] = vx;
      py[j * ST + lane] = vy;
    }
  }
  __syncwarp();
  // rows k1 < 4 hold the largest terms of the low derivatives: their sums over
  // the sources are compensated
  constexpr int KC = 4;
  float A[Q + 1], Al[KC];
#pragma unroll
  for (int k = 0; k <= Q; ++k) A[k] = 0.f;
#pragma unroll
  for (int k = 0; k < KC; ++k) Al[k] = 0.f;
#pragma unroll 1
  for (int s = 0; s < cnt; ++s) {
    const float* a = rec + (size_t)(g * kGroup + s) * R + Rec<float>::HDR;
    float yv[M + 1];
#pragma unroll
    for (int m2 = 0; m2 <= M; ++m2)
      yv[m2] = lane >= m2 && lane <= Q ? py[(lane - m2) * ST + s] : 0.f;
    float W[M + 1];
    float sc1 = 1.f;  // 1 / scale^m1
    static_for<0, M + 1>([&](auto m1c) {
      constexpr int m1 = decltype(m1c)::value;
      float v = 0.f, sc2 = sc1;
      static_for<0, M - m1 + 1>([&](auto m2c) {
        constexpr int m2 = decltype(m2c)::value;
        v = fmaf(__ldg(a + mcol(m1, m2)) * sc2, yv[m2], v);
        sc2 *= 1.f / kLocScale;
      });
      W[m1] = v;
      sc1 *= 1.f / kLocScale;
    });
    static_for<0, Q + 1>([&](auto kc) {
      constexpr int k1 = decltype(kc)::value;
      float v = k1 < KC ? 0.f : A[k1];
      static_for<0, (M < k1 ? M : k1) + 1>([&](auto m1c) {
        constexpr int m1 = decltype(m1c)::value;
        v = fmaf(px[(k1 - m1) * ST + s], W[m1], v);
      });
      if constexpr (k1 < KC)
        two_sum_into(A[k1], Al[k1], v);
      else
        A[k1] = v;
    });
  }
#pragma unroll
  for (int k = 0; k < KC; ++k) A[k] += Al[k];
  float* o = gexp + (size_t)g * L::LEN;
  if (lane <= Q) {
    static_for<0, Q + 1>([&](auto kc) {
      constexpr int k1 = decltype(kc)::value;
      as[k1 * (Q + 2) + lane] = A[k1];
      if (lane < L::row_len(Q, k1)) o[L::off_a(k1) + lane] = lane <= Q - k1 ? A[k1] : 0.f;
    });
  }
  __syncwarp();
  // P = P_e + (D1^2 + D2^2) S: per order N, v[k1] = A[k1] - v[k1 + 2]
  if (lane <= Q) {
    const int N = lane;
    float v0 = 0.f, v1 = 0.f;  // v at the last even / odd k1 (from the top)
    static_for_down<0, Q + 1>([&](auto kc) {
      constexpr int k1 = decltype(kc)::value;
      if (k1 <= N) {
        float& v = (k1 & 1) ? v1 : v0;
        v = as[k1 * (Q + 2) + N - k1] - v;
        if constexpr (k1 >= 2) o[L::off_s(k1 - 2) + N - k1] = v * (kLocScale * kLocScale);
      }
    });
    o[L::off_p0 + N] = v0;
    o[L::off_p1 + N] = v1;
  }
  // the padding of the S rows and of P_e
  static_for<0, Q - 1>([&](auto kc) {
    constexpr int k1 = decltype(kc)::value;
    const int e = Q - 2 - k1 + 1 + lane;
    if (e < L::row_len(Q - 2, k1)) o[L::off_s(k1) + e] = 0.f;
  });
  if (Q + 1 + lane < L::row_len(Q, 0)) {
    o[L::off_p0 + Q + 1 + lane] = 0.f;
    o[L::off_p1 + Q + 1 + lane] = 0.f;
  }
}

// ------------------------------------------------------------------ tables
constexpr int kLocBatch = 16;          // source groups whose tables are formed together
constexpr int kLocST = kLocBatch + 1;  // table row stride (odd: no bank conflicts)

// 2^-N sum_j C(N, a + 2 + 2 j): weight of the Gaussian entry (a, N - 2 - a) in
// the holomorphic derivative of order N.
__host__ __device__ constexpr double loc_weight(int N, int a) {
  double r = 0.0;
  for (int q = a + 2; q <= N; q += 2) r += binom_d(N, q);
  return r * pow2_neg(N);
}

// a - b = d + e exactly.
__device__ __forceinline__ void two_diff(float a, float b, float& d, float& e) {
  d = a - b;
  const float v = d - a;
  e = (a - (d - v)) - (b + v);
}

// (hi, lo) products and sums.
struct Two {
  float h, l;
};
__device__ __forceinline__ Two two_mul(Two a, Two b) {
  const float p = a.h * b.h;
  const float e = fmaf(a.h, b.h, -p) + fmaf(a.h, b.l, a.l * b.h);
  const float s = p + e;
  return {s, e - (s - p)};
}
__device__ __forceinline__ Two two_add(Two a, Two b) {
  const float s = a.h + b.h;
  const float v = s - a.h;
  const float e = (a.h - (s - v)) + (b.h - v) + (a.l + b.l);
  const float r = s + e;
  return {r, e - (r - s)};
}

// Edge derivatives c_N = f_N + i e_N (times scale^N) of orders 1 .. N by the
// upward recursion c_{N+1} = v (i N c_N - g_N), v = 1 / conj(z), from c_1 =
// amp v; g(N) is the Gaussian term.  The first kLocTwo orders are carried as
// (hi, lo) pairs: the low orders are the ones that the velocity and the moment
// rates feel, and an expansion's rounding does not average out over its pairs.
// With xmax > 0 only the orders below min(x, xmax) are written.
constexpr int kLocTwo = 10;
template <int N, typename Gf>
__device__ __forceinline__ void loc_upward(float b1, float b2, float l1, float l2, float x,
                                           float xl, float amp, float s, float* te, float* tf,
                                           Gf&& g, int stride, float xmax) {
  const float rh = 1.f / x;
  // an x beyond the FP32 range leaves zeros (rh = 0), not inf x 0
  const float rl = x <= 3.4e38f ? (fmaf(-x, rh, 1.f) - xl * rh) * rh : 0.f;
  const Two r{rh, rl};
  Two v1 = two_mul({b1, l1}, r), v2 = two_mul({b2, l2}, r);
  v1 = {v1.h * s, v1.l * s};
  v2 = {v2.h * s, v2.l * s};
  Two cf = two_mul(v1, {amp, 0.f}), ce = two_mul(v2, {amp, 0.f});
#pragma unroll 2
  for (int k = 1; k <= kLocTwo; ++k) {
    if (xmax > 0.f && !(x > (float)k)) return;
    te[k * stride] = ce.h;
    tf[k * stride] = cf.h;
    const float fk = (float)k;
    const Two tr = two_add(two_mul({-fk, 0.f}, ce), {-g(k), 0.f}), ti = two_mul({fk, 0.f}, cf);
    const Two a = two_mul(v1, tr), b = two_mul(v2, ti), c = two_mul(v1, ti), d = two_mul(v2, tr);
    cf = two_add(a, {-b.h, -b.l});
    ce = two_add(c, d);
  }
  float pf = cf.h, pe = ce.h;
#pragma unroll 4
  for (int k = kLocTwo + 1; k <= N; ++k) {
    if (xmax > 0.f && !(x > (float)k)) return;
    te[k * stride] = pe;
    tf[k * stride] = pf;
    const float tr = -fmaf((float)k, pe, g(k)), ti = (float)k * pf;
    pf = fmaf(v1.h, tr, fmaf(-v2.h, ti, fmaf(v1.l, tr, -v2.l * ti)));
    pe = fmaf(v1.h, ti, fmaf(v2.h, tr, fmaf(v1.l, ti, v2.l * tr)));
  }
}

// Derivative tables at the separation b = t0 - s0 (one source per lane, its
// column of the tables): hx[n] = 2 h_n(b1), hy[n] = h_n(b2), and e[n], f[n] of
// 2 pi psi, each times 4^-n, rows of kLocST floats.
template <int M>
__device__ __forceinline__ void loc_tables(float2 t0, float2 s0, float* hx, float* hy, float* te,
                                           float* tf) {
  using L = Loc<M>;
  constexpr int N = L::NT;
  constexpr float s = kLocScale, is = 1.f / kLocScale;
  float b1, b2, l1, l2;
  two_diff(t0.x, s0.x, b1, l1);
  two_diff(t0.y, s0.y, b2, l2);
  const float s1 = b1 * b1, s2 = b2 * b2;
  const float q1 = fmaf(b1, b1, -s1), q2 = fmaf(b2, b2, -s2);
  const float x = s1 + s2;
  const float bv = x - s1;
  const float xl = ((s1 - (x - bv)) + (s2 - bv)) + (q1 + 2.f * b1 * l1) + (q2 + 2.f * b2 * l2);
  const float eh1 = expf(-s1) * (1.f - q1), eh2 = expf(-s2) * (1.f - q2);
  const float E = eh1 * (1.f - 2.f * b1 * l1) * (eh2 * (1.f - 2.f * b2 * l2));
  auto hermite = [&](float* h, float b, float l, float h0) {
    const float c = -2.f * s * b, li = l * is;
    float p = h0, q = c * h0;  // orders k, k + 1 at the hi part
#pragma unroll 7
    for (int k = 0; k <= N; ++k) {
      h[k * kLocST] = fmaf(li, q, p);  // first order in the lo part
      const float r = fmaf(c, q, (-2.f * (k + 1) * s * s) * p);
      p = q;
      q = r;
    }
  };
  hermite(hx, b1, l1, 2.f * eh1);
  hermite(hy, b2, l2, eh2);
  // e_N, f_N at the top order (used for N > x)
  float pe, pf;
  {
    const float I = E * kummer_sum<N - 1, float>(fminf(x, (float)(N - 1)));
    float zr = 1.f, zi = 0.f;
    const float u1 = s * (b1 + l1), u2 = s * (b2 + l2);
#pragma unroll 7
    for (int k = 0; k < N; ++k) {
      const float t = fmaf(zr, u1, zi * u2);
      zi = fmaf(zi, u1, -zr * u2);
      zr = t;
    }
    constexpr float sg = ((N - 1) & 1) ? -0.5f : 0.5f;
    float dr = sg * zr * I, di = sg * zi * I;
    static_for<0, N - 1>([&](auto ac) {
      constexpr int a = decltype(ac)::value;
      constexpr int r = (N - 2 - a) & 3;
      constexpr float wgt = (float)(loc_weight(N, a) * s * s);
      const float v = hx[a * kLocST] * hy[(N - 2 - a) * kLocST];
      if constexpr (r == 0) dr = fmaf(-wgt, v, dr);
      if constexpr (r == 1) di = fmaf(wgt, v, di);
      if constexpr (r == 2) dr = fmaf(wgt, v, dr);
      if constexpr (r == 3) di = fmaf(-wgt, v, di);
    });
    if constexpr ((N & 3) == 0) { pe = 2.f * dr;  pf = 2.f * di; }
    if constexpr ((N & 3) == 1) { pe = -2.f * di; pf = 2.f * dr; }
    if constexpr ((N & 3) == 2) { pe = -2.f * dr; pf = -2.f * di; }
    if constexpr ((N & 3) == 3) { pe = 2.f * di;  pf = -2.f * dr; }
  }
  const float gx = hx[0] * 0.5f;  // h_N (scaled) = gx hy_N
  // downward: orders N > x
  if (!(x > (float)N)) {
    te[N * kLocST] = pe;
    tf[N * kLocST] = pf;
  }
#pragma unroll 4
  for (int k = N - 1; k >= 1; --k) {
    const float g = gx * hy[k * kLocST];
    const float ik = 1.f / k;
    const float xe = fmaf(pf, b1, fmaf(pe, b2, fmaf(pf, l1, pe * l2)));
    const float xf = fmaf(pe, b1, fmaf(-pf, b2, fmaf(pe, l1, -pf * l2)));
    pe = -fmaf(xe, is, g) * ik;
    pf = xf * is * ik;
    if (!(x > (float)k)) {
      te[k * kLocST] = pe;
      tf[k * kLocST] = pf;
    }
  }
  // upward: orders N < x.  With c_N = f_N + i e_N and v = 1 / conj(z):
  // c_{N+1} = v (i N c_N - h_N).
  loc_upward<N>(b1, b2, l1, l2, x, xl, 1.f - E, s, te, tf,
                [&](int k) { return gx * hy[k * kLocST]; }, kLocST, (float)N);
}

// ------------------------------------------------------------------ near groups
constexpr int kLocWarps = 4;  // warps (target groups) per CTA
constexpr int kLocSlots = 2;  // expansion records in flight per warp

template <int M>
struct LocSmem {
  using L = Loc<M>;
  static constexpr size_t tab = (size_t)4 * L::ROWS * kLocST * 4;
  static constexpr size_t slots = (size_t)kLocSlots * L::LEN * 4;
  static constexpr size_t acc = (size_t)2 * L::FROWS * 32 * 4;
  static constexpr size_t warp = (slots + acc + tab + 15) / 16 * 16;
  static constexpr size_t bytes = kLocWarps * warp + kLocWarps * kLocSlots * 8;
};

// One warp: the field of target group tg from segment blockIdx.y of its list of
// compact near groups (entries counted from the end of its list row).
// fld: [segment][group][FROWS][32] (hi, lo) pairs.  err as in near_pair_kernel.
template <int M>
__global__ void __launch_bounds__(kLocWarps * 32, 2)
    loc_near_kernel(int n, int G, const float* __restrict__ gdata,
                    const float* __restrict__ gexp, const int2* __restrict__ ent,
                    const int* __restrict__ mcnt, int C, float2* __restrict__ fld,
                    unsigned long long* __restrict__ counts, int* __restrict__ err) {
  using L = Loc<M>;
  using SM = LocSmem<M>;
  constexpr int GL = gdata_len(M), Q = L::Q, NG = L::NG, ST = kLocST;
  extern __shared__ __align__(16) unsigned char smem_loc[];
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  unsigned char* base = smem_loc + (size_t)w * SM::warp;
  float* slots = reinterpret_cast<float*>(base);
  float* ahi = reinterpret_cast<float*>(base + SM::slots);
  float* alo = ahi + L::FROWS * 32;
  float* hx = alo + L::FROWS * 32;
  float* hy = hx + L::ROWS * ST;
  float* te = hy + L::ROWS * ST;
  float* tf = te + L::ROWS * ST;
  unsigned long long* bar =
      reinterpret_cast<unsigned long long*>(smem_loc + (size_t)kLocWarps * SM::warp) +
      w * kLocSlots;
  const int tg = blockIdx.x * kLocWarps + w;
  if (tg >= G) return;  // whole warps, no CTA barrier
  const int cnt = mcnt[tg];
  const int i0 = (int)((long long)blockIdx.y * cnt / C);
  const int i1 = (int)((long long)(blockIdx.y + 1) * cnt / C);
  float2* out = fld + ((size_t)blockIdx.y * G + tg) * L::FROWS * 32 + lane;
  if (i0 >= i1) {
#pragma unroll
    for (int r = 0; r < L::FROWS; ++r) out[r * 32] = make_float2(0.f, 0.f);
    return;
  }
  for (int i = lane; i < 2 * L::FROWS * 32; i += 32) ahi[i] = 0.f;
  // rows past the highest order are read by lanes whose sums nothing uses
  for (int i = lane; i < 4 * L::ROWS * ST; i += 32) hx[i] = 0.f;
  if (lane == 0) {
    for (int s = 0; s < kLocSlots; ++s) mbar_init(bar + s, 1);
    fence_mbar_init();
  }
  __syncwarp();
  const float4 tc = *reinterpret_cast<const float4*>(gdata + (size_t)tg * GL + 4);
  const int2* lst = ent + (size_t)tg * G + (G - 1);
  float acc[L::FROWS];
#pragma unroll
  for (int r = 0; r < L::FROWS; ++r) acc[r] = 0.f;
  constexpr int KC = 4;  // rows of G summed as (hi, lo) pairs source by source, as are the edges
  float accl[KC + 2];
#pragma unroll
  for (int r = 0; r < KC + 2; ++r) accl[r] = 0.f;
  bool timeout = false;
  unsigned nsrc = 0;
  auto issue = [&](int t, int g) {  // lane 0: record of group g into slot t % kLocSlots
    unsigned long long* b = bar + t % kLocSlots;
    mbar_arrive_expect_tx(b, (unsigned)(L::LEN * 4));
    bulk_copy_g2s(slots + (size_t)(t % kLocSlots) * L::LEN, gexp + (size_t)g * L::LEN,
                  (unsigned)(L::LEN * 4), b);
  };
  int t = 0;  // sources taken so far (slot t % kLocSlots, phase t / kLocSlots)
#pragma unroll 1
  for (int b0 = i0; b0 < i1; b0 += kLocBatch) {
    const int nb = min(kLocBatch, i1 - b0);
    int g = tg;
    if (lane < nb) g = lst[-(b0 + lane)].x;
    // the slots are free: the previous batch waited for all its copies
    {
      const int g0 = __shfl_sync(0xffffffffu, g, 0), g1 = __shfl_sync(0xffffffffu, g, 1);
      if (lane == 0) {
        fence_proxy_async_smem();
        issue(t, g0);
        if (nb > 1) issue(t + 1, g1);
      }
    }
    if (lane < nb) {
      const float4 sc = *reinterpret_cast<const float4*>(gdata + (size_t)g * GL + 4);
      loc_tables<M>(make_float2(tc.x, tc.y), make_float2(sc.x, sc.y), hx + lane, hy + lane,
                    te + lane, tf + lane);
      nsrc += min(kGroup, n - g * kGroup);
    }
    __syncwarp();
#pragma unroll 1
    for (int s = 0; s < nb; ++s, ++t) {
      if (!mbar_wait_bounded(bar + t % kLocSlots, (unsigned)((t / kLocSlots) & 1))) timeout = true;
      const float* xr = slots + (size_t)(t % kLocSlots) * L::LEN;
      float hyr[Q + 1], hxr[Q + NG + 1];
#pragma unroll
      for (int k = 0; k <= Q; ++k) hyr[k] = hy[(lane + k) * ST + s];
#pragma unroll
      for (int k = 0; k <= Q + NG; ++k) hxr[k] = hx[k * ST + s];
      {  // edges: P_e on e, f (E1: D1^2 = Lap - D2^2 once), S on Hermite functions
        float v0 = 0.f, v1 = 0.f, vl = 0.f;
        static_for<0, Q + 1>([&](auto kc) {
          constexpr int k = decltype(kc)::value;
          const float p0 = xr[L::off_p0 + k], p1 = xr[L::off_p1 + k];
          const float e0 = te[(lane + k) * ST + s], f0 = tf[(lane + k) * ST + s];
          const float e1 = te[(lane + k + 1) * ST + s], f1 = tf[(lane + k + 1) * ST + s];
          v0 = fmaf(p0, e0, v0);
          v1 = fmaf(p0, f1, v1);
          if constexpr (k > 0) {
            v0 = fmaf(p1, f0, v0);
            v1 = fmaf(-p1, e1, v1);
            vl = fmaf(p1, hyr[k - 1], vl);
          }
        });
        v1 = fmaf(vl, hxr[0] * (kLocScale * kLocScale), v1);
        float u0 = 0.f, u1 = 0.f;
        static_for<0, Q - 1>([&](auto kc) {
          constexpr int k1 = decltype(kc)::value;
          float u = 0.f;
          static_for<0, L::row_len(Q - 2, k1) / 4>([&](auto jc) {
            constexpr int j = 4 * decltype(jc)::value;
            const float4 a = *reinterpret_cast<const float4*>(xr + L::off_s(k1) + j);
            u = fmaf(a.x, hyr[j], u);
            if constexpr (j + 1 <= Q) u = fmaf(a.y, hyr[j + 1], u);
            if constexpr (j + 2 <= Q) u = fmaf(a.z, hyr[j + 2], u);
            if constexpr (j + 3 <= Q) u = fmaf(a.w, hyr[j + 3], u);
          });
          u0 = fmaf(hxr[k1], u, u0);
          u1 = fmaf(hxr[k1 + 1], u, u1);
        });
        two_sum_into(acc[NG + 1], accl[KC], v0 + u0);
        two_sum_into(acc[NG + 2], accl[KC + 1], v1 + u1);
      }
      float U[Q + 1];
      static_for<0, Q + 1>([&](auto kc) {
        constexpr int k1 = decltype(kc)::value;
        float u = 0.f;
        static_for<0, L::row_len(Q, k1) / 4>([&](auto jc) {
          constexpr int j = 4 * decltype(jc)::value;
          const float4 a = *reinterpret_cast<const float4*>(xr + L::off_a(k1) + j);
          u = fmaf(a.x, hyr[j], u);
          if constexpr (j + 1 <= Q - k1) u = fmaf(a.y, hyr[j + 1], u);
          if constexpr (j + 2 <= Q - k1) u = fmaf(a.z, hyr[j + 2], u);
          if constexpr (j + 3 <= Q - k1) u = fmaf(a.w, hyr[j + 3], u);
        });
        U[k1] = u;
      });
      static_for<0, NG + 1>([&](auto nc) {
        constexpr int n1 = decltype(nc)::value;
        float v = 0.f;
        static_for<0, Q + 1>([&](auto kc) {
          constexpr int k1 = decltype(kc)::value;
          v = fmaf(hxr[k1 + n1], U[k1], v);
        });
        if constexpr (n1 < KC)
          two_sum_into(acc[n1], accl[n1], v);
        else
          acc[n1] += v;
      });
      __syncwarp();  // every lane has read this slot before it is refilled
      if (s + kLocSlots < nb) {
        const int gn = __shfl_sync(0xffffffffu, g, (s + kLocSlots) & 31);
        if (lane == 0) {
          fence_proxy_async_smem();
          issue(t + kLocSlots, gn);
        }
      }
    }
#pragma unroll
    for (int r = 0; r < L::FROWS; ++r) flush_one(acc[r], ahi, alo, r * 32 + lane);
#pragma unroll
    for (int r = 0; r < KC + 2; ++r) {
      alo[(r < KC ? r : NG + 1 + r - KC) * 32 + lane] += accl[r];
      accl[r] = 0.f;
    }
  }
#pragma unroll
  for (int r = 0; r < L::FROWS; ++r)
    out[r * 32] = make_float2(ahi[r * 32 + lane], alo[r * 32 + lane]);
  if (timeout && lane == 0) {
    // a copy may still be in flight: wait (bounded) before the CTA ends
    for (int q = max(0, t - kLocSlots); q < t; ++q)
      mbar_wait_bounded(bar + q % kLocSlots, (unsigned)((q / kLocSlots) & 1));
    atomicExch(err, 1);
  }
  if (counts != nullptr) {  // near pairs covered
    const unsigned tot = __reduce_add_sync(0xffffffffu, nsrc);
    const unsigned long long p = (unsigned long long)tot * (unsigned)min(kGroup, n - tg * kGroup);
    if (lane == 0 && p) {
      atomicAdd(counts, p);
      atomicAdd(counts + 4, p);
    }
  }
}

// ------------------------------------------------------------------ far field
// The far field of the target groups that take local expansions, as in
// far_tree_kernel and far_pair_kernel (the same walk, the same criteria) but summed into the edge
// rows of the group's field instead of target by target: a node costs 4 (NA)
// multiply-adds per lane instead of 2902 flops per target, a far source 4 (M +
// 1) instead of 838 flops per target.  The lanes first form the point-vortex
// edge derivatives of up to 32 nodes or sources (one each), then run through
// them with one order of the field per lane.  For a target group of radius
// loc_field_radius or less the field's Taylor series loses less than FP32
// rounding (common.cuh).
//
// A node is taken at a radius of up to 0.2 of the distance (0.15 at order 0, which
// has the fewest terms), twice that of the target-by-target kernels, which hold
// every order q <= 3M of the jet to 2e-9 of the node's own term of that order.
// Here a velocity is off by at most 4e-8 (M = 0; 0.2 would leave 5e-7), 2.4e-8 (M =
// 1), 1e-9 (M = 2) and less (M >= 3) of a source's at the near edge of its node, and
// the moment rates by 2e-9 (M = 2) of their terms' magnitudes: the high orders, off by up
// to 1e-5 of their own term, count that little at a distance of sqrt(x_far).
template <int M>
__device__ __forceinline__ bool loc_takes(const float4 tb, const float4 c) {
  constexpr float theta2 = M == 0 ? 0.0225f : 0.04f;
  const float dx = fmaxf(0.f, fmaxf(tb.x - c.x, c.x - tb.y));
  const float dy = fmaxf(0.f, fmaxf(tb.z - c.y, c.y - tb.w));
  return c.z <= m2p_radius(M) && c.z * c.z <= theta2 * (dx * dx + dy * dy);
}

template <int M>
struct LocFarSmem {
  using L = Loc<M>;
  static constexpr int NA = m2p_terms(M);
  static constexpr int ROWS = 32 + NA + 1;  // rows lane + n + 1, n < NA
  static constexpr int ST = 33;
  static constexpr size_t tab = (size_t)2 * ROWS * ST * 4;
  static constexpr size_t warp = tab + 32 * 4 + kTreeStack * 4;
  static constexpr size_t bytes = kLocWarps * warp;
};

template <int M>
__global__ void __launch_bounds__(kLocWarps * 32)
    loc_far_kernel(const float* __restrict__ rec, int n, int G, const float* __restrict__ gdata,
                   const float* __restrict__ tree, int Lc, int S, float2* __restrict__ ffld,
                   unsigned long long* __restrict__ counts) {
  using L = Loc<M>;
  using SM = LocFarSmem<M>;
  constexpr int R = rec_len<float>(M), K = n_moments(M), HDR = Rec<float>::HDR;
  constexpr int GL = gdata_len(M), NA = SM::NA, ST = SM::ST, NL = L::NL;
  constexpr float rmax = loc_radius(M);  // near groups (loc_pair)
  extern __shared__ __align__(16) unsigned char smem_lf[];
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  unsigned char* base = smem_lf + (size_t)w * SM::warp;
  float* te = reinterpret_cast<float*>(base);
  float* tf = te + SM::ROWS * ST;
  int* node_s = reinterpret_cast<int*>(base + SM::tab);  // nodes waiting for a batch
  int* stack = node_s + 32;
  const int tg = blockIdx.x * kLocWarps + w;
  if (tg >= G) return;  // whole warps, no CTA barrier
  const float4 tb = *reinterpret_cast<const float4*>(gdata + (size_t)tg * GL);
  const float4 tc = *reinterpret_cast<const float4*>(gdata + (size_t)tg * GL + 4);
  if (!(tc.z <= loc_field_radius(M))) return;  // the target-by-target far kernels'
  for (int i = lane; i < 2 * SM::ROWS * ST; i += 32) te[i] = 0.f;
  __syncwarp();
  float h0 = 0.f, q0 = 0.f, h1 = 0.f, q1 = 0.f;  // edge rows E0, E1 of this lane's order
  auto node_rec = [&](int L_, int i) -> const float* {
    return L_ == 0 ? gdata + (size_t)i * GL
                   : tree + (size_t)(tree_level_offset(G, L_) + i) * GL;
  };
  // point-vortex tables of this lane's centre (cx, cy) + (lx, ly), orders <= TOP
  auto tables = [&](float cx, float cy, float lx, float ly, auto topc) {
    constexpr int TOP = decltype(topc)::value;
    float b1, b2, l1, l2;
    two_diff(tc.x, cx, b1, l1);
    two_diff(tc.y, cy, b2, l2);
    l1 -= lx;
    l2 -= ly;
    const float s1 = b1 * b1, s2 = b2 * b2;
    const float e1 = fmaf(b1, b1, -s1), e2 = fmaf(b2, b2, -s2);
    const float x = s1 + s2;
    const float bv = x - s1;
    const float xl = ((s1 - (x - bv)) + (s2 - bv)) + (e1 + 2.f * b1 * l1) + (e2 + 2.f * b2 * l2);
    loc_upward<TOP>(b1, b2, l1, l2, x, xl, 1.f, 1.f, te + lane, tf + lane,
                    [](int) { return 0.f; }, ST, 0.f);
  };
  // add the source in table column s with NT multipole terms B_n = (br, bi)(n):
  // i^n B_n = p0_n - i p1_n acts as p0 D2^n + p1 D1 D2^{n-1} on a harmonic field
  auto add = [&](int s, auto ntc, auto&& term) {
    constexpr int NTm = decltype(ntc)::value;
    float v0 = 0.f, v1 = 0.f;
    float e0 = te[lane * ST + s], f0 = tf[lane * ST + s];
    static_for<0, NTm>([&](auto kc) {
      constexpr int k = decltype(kc)::value;
      const float2 t = term(kc);
      const float br = t.x, bi = t.y;
      float p0, p1;
      if constexpr ((k & 3) == 0) { p0 = br;  p1 = -bi; }
      if constexpr ((k & 3) == 1) { p0 = -bi; p1 = -br; }
      if constexpr ((k & 3) == 2) { p0 = -br; p1 = bi; }
      if constexpr ((k & 3) == 3) { p0 = bi;  p1 = br; }
      const float en = te[(lane + k + 1) * ST + s], fn = tf[(lane + k + 1) * ST + s];
      v0 = fmaf(p0, e0, v0);
      v1 = fmaf(p0, fn, v1);
      if constexpr (k > 0) {
        v0 = fmaf(p1, f0, v0);
        v1 = fmaf(-p1, en, v1);
      }
      e0 = en;
      f0 = fn;
    });
    two_sum_into(h0, q0, v0);
    two_sum_into(h1, q1, v1);
  };
  int nq = 0;  // nodes waiting
  auto run_nodes = [&]() {
    __syncwarp();
    const float* nd = nullptr;
    int id = 0;
    if (lane < nq) {
      id = node_s[lane];
      nd = node_rec(id >> kTreeShift, id & ((1 << kTreeShift) - 1));
      const float4 c = *reinterpret_cast<const float4*>(nd + 4);
      tables(c.x, c.y, 0.f, 0.f, std::integral_constant<int, NL + NA>{});
    }
    __syncwarp();
#pragma unroll 1
    for (int s = 0; s < nq; ++s) {
      const float* b =
          reinterpret_cast<const float*>(__shfl_sync(0xffffffffu, (unsigned long long)nd, s)) + 8;
      add(s, std::integral_constant<int, NA>{}, [&](auto kc) {
        constexpr int k = decltype(kc)::value;
        return __ldg(reinterpret_cast<const float2*>(b) + k);
      });
    }
    nq = 0;
    __syncwarp();
  };
  unsigned n_far = 0, n_m2p = 0, n_m2p_pairs = 0;
  // the walk from node blockIdx.y of level Lc, or (no tree) the groups of
  // source range blockIdx.y one after another
  int sp = 0, gnext = 0, gend = 0;
  if (tree != nullptr) {
    if (lane == 0) stack[0] = (Lc << kTreeShift) | blockIdx.y;
    sp = 1;
  } else {
    gnext = (int)((long long)blockIdx.y * G / S);
    gend = (int)((long long)(blockIdx.y + 1) * G / S);
  }
  __syncwarp();
  while (sp > 0 || gnext < gend) {
    const int top = sp > 0 ? stack[--sp] : gnext++;
    __syncwarp();
    const int Lv = top >> kTreeShift, i = top & ((1 << kTreeShift) - 1);
    const float* nd = node_rec(Lv, i);
    const float4 box = *reinterpret_cast<const float4*>(nd);
    const float4 cen = *reinterpret_cast<const float4*>(nd + 4);
    const bool far_box = box_dist2(tb, box) >= x_far(M);
    if (far_box && loc_takes<M>(tb, cen)) {
      if (lane == 0) node_s[nq] = top;
      n_m2p += 1;
      n_m2p_pairs += Lv == 0 ? min(kGroup, n - kGroup * i) : (unsigned)cen.w;
      if (++nq == 32) run_nodes();
      continue;
    }
    if (Lv > 0) {  // open the node: children 2i (taken first) and 2i+1 (if any)
      const bool two = 2 * i + 1 < tree_level_nodes(G, Lv - 1);
      if (lane == 0) {
        if (two) stack[sp] = ((Lv - 1) << kTreeShift) | (2 * i + 1);
        stack[sp + (two ? 1 : 0)] = ((Lv - 1) << kTreeShift) | (2 * i);
      }
      sp += two ? 2 : 1;
      __syncwarp();
      continue;
    }
    if (!far_box && loc_pair<M>(rmax, tc, cen)) continue;  // a near group of loc_near_kernel
    // source by source, as in far_tree_kernel
    const int nsrc = min(kGroup, n - i * kGroup);
    const float* r = rec + (size_t)(i * kGroup + min(lane, nsrc - 1)) * R;
    const float4 z = *reinterpret_cast<const float4*>(r);
    const bool mine = lane < nsrc && (far_box || point_is_far<M>(tb, z.x, z.y));
    unsigned fm = __ballot_sync(0xffffffffu, mine);
    if (!fm) continue;
    n_far += __popc(fm);
    if (mine) tables(z.x, z.y, z.z, z.w, std::integral_constant<int, NL + M + 1>{});
    __syncwarp();
    while (fm) {
      const int s = __ffs(fm) - 1;
      fm &= fm - 1;
      const float* a = rec + (size_t)(i * kGroup + s) * R + HDR + K;
      add(s, std::integral_constant<int, M + 1>{}, [&](auto kc) {
        constexpr int k = decltype(kc)::value;
        return make_float2(__ldg(a + 2 * k), __ldg(a + 2 * k + 1));
      });
    }
    __syncwarp();
  }
  if (nq) run_nodes();
  // the field's rows carry scale^order; the tables here do not: at large
  // distances scaled multipoles would leave the FP32 range
  float2* out = ffld + ((size_t)blockIdx.y * G + tg) * 64 + lane;
  const float s0 = __int_as_float((127 - 2 * lane) << 23);  // 4^-lane
  out[0] = make_float2(h0 * s0, q0 * s0);
  out[32] = make_float2(h1 * (s0 * kLocScale), q1 * (s0 * kLocScale));
  if (counts != nullptr && lane == 0) {
    const unsigned long long nt = (unsigned)min(kGroup, n - tg * kGroup);
    if (n_far) atomicAdd(counts + 1, nt * n_far);
    if (n_m2p) atomicAdd(counts + 2, nt * n_m2p);
    if (n_m2p_pairs) atomicAdd(counts + 3, nt * n_m2p_pairs);
  }
}

// ------------------------------------------------------------------ targets
// One CTA per target group: the sum of the C segments' fields, then Psi (edge
// columns) and R (columns beta1 >= 2) at its 32 targets into partial block
// `out` ([NB][n] FP64).  The value at the centre is added in FP64, the rest of
// the Taylor sum in FP32.  Groups without a local field get zeros.  A warp
// takes every kEvalWarps-th row of the field and of the results: with one warp per
// group the chain of dependent shared loads and multiply-adds took 77 us at n =
// 2011, M = 8 (now 33 us) and 97 us at n = 24000, M = 6, with 5 warps on an SM.
constexpr int kEvalWarps = 4;
template <int M>
__global__ void __launch_bounds__(kEvalWarps * 32)
    loc_eval_kernel(const float* __restrict__ rec, int n, int G, const float* __restrict__ gdata,
                    int C, const float2* __restrict__ fld, int nfar,
                    const float2* __restrict__ ffld, double* __restrict__ out) {
  using L = Loc<M>;
  constexpr int R = rec_len<float>(M), GL = gdata_len(M), NL = L::NL, NG = L::NG, P = L::P;
  constexpr int BM = bmax_of(M), NB = n_beta(M);
  constexpr int GS = (NG + 1 + 3) / 4 * 4;  // row strides, whole float4s
  constexpr int FS = 36;
  __shared__ __align__(16) float gs[(NG + 1) * GS];
  __shared__ __align__(16) float fs[(P + 2) * FS];  // F rows n1 = 0 .. P + 1
  __shared__ double gd[n_moments(BM >= 2 ? BM - 2 : 0)];
  __shared__ double fd[2 * 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, tg = blockIdx.x;
  const int j = tg * kGroup + lane;
  const float4 cen = *reinterpret_cast<const float4*>(gdata + (size_t)tg * GL + 4);
  if (!(cen.z <= loc_field_radius(M))) {  // the whole CTA
    if (j < n)
      for (int b = warp; b < NB; b += kEvalWarps) out[(size_t)b * n + j] = 0.0;
    return;
  }
  // sum of the segments; G rows as FP32, the low orders and the edges in FP64
  for (int r = L::FROWS - 1 - warp; r >= 0; r -= kEvalWarps) {  // the long edge rows first
    float h = 0.f, l = 0.f;
#pragma unroll 4
    for (int c = 0; c < C; ++c) {
      const float2 v = fld[(((size_t)c * G + tg) * L::FROWS + r) * 32 + lane];
      two_sum_into(h, l, v.x);
      l += v.y;
    }
    if (r > NG)
#pragma unroll 8
      for (int c = 0; c < nfar; ++c) {
        const float2 v = ffld[(((size_t)c * G + tg) * 2 + r - NG - 1) * 32 + lane];
        two_sum_into(h, l, v.x);
        l += v.y;
      }
    if (r <= NG) {  // zeros beyond order NG: the sums below run over whole rows
      if (lane < GS) gs[r * GS + lane] = r + lane <= NG ? h + l : 0.f;
      if constexpr (BM >= 2)
        if (r + lane <= BM - 2) gd[tri(r + lane) + lane] = (double)h + (double)l;
    } else {
      fd[(r - NG - 1) * 32 + lane] = (double)h + (double)l;
      fs[(r - NG - 1) * FS + lane] = r - NG - 1 + lane <= NL ? h + l : 0.f;
    }
  }
  __syncthreads();
  // F_(n1, n2) = scale^2 G_(n1-2, n2) - F_(n1-2, n2+2), rows n1 >= 2: the even
  // rows by warp 0, the odd ones by warp 1 (orders n1 + n2 > NL are zero, so the
  // top lanes need no neighbour)
  if (warp < 2) {
    float v = fs[warp * FS + lane];
    for (int n1 = 2 + warp; n1 <= P + 1; n1 += 2) {
      const float up = __shfl_down_sync(0xffffffffu, v, 2);
      v = n1 + lane <= NL ? kLocScale * kLocScale * gs[(n1 - 2) * GS + lane] - up : 0.f;
      fs[n1 * FS + lane] = v;
    }
  }
  __syncthreads();
  if (j >= n) return;  // no further CTA-wide step
  const float* r = rec + (size_t)j * R;
  const float t1 = ((r[0] - cen.x) + r[2]) * (1.f / kLocScale);
  const float t2 = ((r[1] - cen.y) + r[3]) * (1.f / kLocScale);
  float px[P + 1], py[P + 1];
  px[0] = py[0] = 1.f;
#pragma unroll
  for (int k = 1; k <= P; ++k) {
    px[k] = px[k - 1] * (t1 * (1.f / k));
    py[k] = py[k - 1] * (t2 * (1.f / k));
  }
  // D^(q1, q2), q2 <= Q2, of a table with rows T[n1][n2] (NX columns), without
  // the value at the centre: X over n1, then over n2
  auto row = [&](int q1, auto nxc, auto stridec, const float* T, auto q2maxc, auto&& emit) {
    constexpr int NX = decltype(nxc)::value, SD = decltype(stridec)::value;
    constexpr int Q2 = decltype(q2maxc)::value, V = (NX + 3) / 4;
    float X[4 * V], X0[Q2 + 1];
#pragma unroll
    for (int i = 0; i < 4 * V; ++i) X[i] = 0.f;
#pragma unroll
    for (int jj = P; jj >= 1; --jj) {
      const float* t = T + (q1 + jj) * SD;
#pragma unroll
      for (int v = 0; v < V; ++v) {
        const float4 a = *reinterpret_cast<const float4*>(t + 4 * v);
        X[4 * v] = fmaf(a.x, px[jj], X[4 * v]);
        X[4 * v + 1] = fmaf(a.y, px[jj], X[4 * v + 1]);
        X[4 * v + 2] = fmaf(a.z, px[jj], X[4 * v + 2]);
        X[4 * v + 3] = fmaf(a.w, px[jj], X[4 * v + 3]);
      }
    }
#pragma unroll
    for (int i = 0; i <= Q2; ++i) X0[i] = X[i];
#pragma unroll
    for (int i = 0; i < NX; ++i) X[i] += T[q1 * SD + i];
    static_for<0, Q2 + 1>([&](auto qc) {
      constexpr int q2 = decltype(qc)::value;
      float v = 0.f;
      static_for_down<1, P + 1>([&](auto jc) {
        constexpr int jj = decltype(jc)::value;
        if constexpr (q2 + jj < NX) v = fmaf(X[q2 + jj], py[jj], v);
      });
      emit(q2, v + X0[q2]);
    });
  };
  auto inv_scale = [](int q) {  // scale^-q / 2 pi, the power 4^q exact
    return __longlong_as_double((long long)(1023 + 2 * q) << 52) * 0.15915494309189533577;
  };
  static_assert(kLocScale == 0.25f, "inv_scale");
  if constexpr (BM >= 2) {
#pragma unroll 1
    for (int q1 = warp; q1 <= BM - 2; q1 += kEvalWarps)
      row(q1, std::integral_constant<int, NG + 1>{}, std::integral_constant<int, GS>{}, gs,
          std::integral_constant<int, BM - 2>{}, [&](int q2, float v) {
            if (q1 + q2 <= BM - 2)
              out[(size_t)bcol(q1 + 2, q2) * n + j] =
                  (gd[tri(q1 + q2) + q2] + (double)v) * inv_scale(q1 + q2);
          });
  }
  // the edge rows to the warps with the fewest rows so far
  const int q1 = ((BM >= 2 ? BM - 1 : 0) + kEvalWarps - 1 - warp) % kEvalWarps;
  if (q1 < 2)
    row(q1, std::integral_constant<int, NL + 1>{}, std::integral_constant<int, FS>{}, fs,
        std::integral_constant<int, BM>{}, [&](int q2, float v) {
          if (q1 + q2 >= 1 && q1 + q2 <= BM)
            out[(size_t)bcol(q1, q2) * n + j] =
                (fd[q1 * 32 + q2] + (double)v) * inv_scale(q1 + q2);
        });
}

}  // namespace mmvm
