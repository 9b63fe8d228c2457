// Dispatch from (order, precision, variant) to the compiled slice kernels.
#include <algorithm>

#include "pair_registry.h"
#include "common.cuh"

namespace mmvm {

// the slice entry points of every compiled variant, and fill_slices()
#include "pair_registry_table.inc"
// the near-kernel and far-kernel entry points of the list form, and fill_list()
#include "pair_list_table.inc"

int pair_variant_count(int M, int precision) {
  if (M < 0 || M > 8 || (precision != 0 && precision != 1)) return 0;
  return n_variants(M, precision);
}

PairEntry pair_entry(int M, int precision, int v) {
  PairEntry e;
  if (v < 0 || v >= pair_variant_count(M, precision)) return e;
  const VariantSpec sp = variant_spec(M, precision, v);
  if (!fill_slices((M * 2 + precision) * kMaxVariants + v, e)) return e;
  e.M = M;
  e.precision = precision;
  e.variant = v;
  e.tpc = sp.TPC;
  e.minb = sp.MINB;
  e.sync = sp.SYNC;
  e.nslices = sp.nslices;
  for (int k = 0; k < e.nslices; ++k)
    if (e.slices[k].tpc != e.tpc) e.uniform_tpc = false;
  e.rec_len = precision == 1 ? rec_len<float>(M) : rec_len<double>(M);
  e.elem_bytes = precision == 1 ? 4 : 8;
  return e;
}

cudaError_t pair_prepare(const PairEntry& e, int S) {
  for (int s = 0; s < e.nslices; ++s) {
    cudaError_t r = e.slices[s].prepare(S);
    if (r != cudaSuccess) return r;
  }
  return cudaSuccess;
}

int pair_occupancy(const PairEntry& e, int S) {
  int best = 1 << 30;
  for (int s = 0; s < e.nslices; ++s) {
    int b = 0;
    if (e.slices[s].occupancy(S, &b) != cudaSuccess) {
      cudaGetLastError();
      return 0;
    }
    best = std::min(best, b);
  }
  return e.nslices ? best : 0;
}

cudaError_t pair_launch(const PairEntry& e, const void* rec, int n, int chunks, int S,
                        const void* gbox, double* partial, int grid_y_limit, cudaStream_t st,
                        unsigned long long* counts) {
  // FP32 chunks start on group boundaries so every source tile is one group
  // (its record decides near or far); FP64 reads no group records
  const int len = (n + chunks - 1) / chunks;
  const int chunk_len = e.precision == 1 ? round_up(len, S) : len;
  const int gy = (grid_y_limit > 0 && chunks > grid_y_limit) ? grid_y_limit : chunks;
  for (int s = 0; s < e.nslices; ++s) {
    cudaError_t r = e.slices[s].launch(rec, n, chunk_len, gy, S, gbox, partial, counts, st);
    if (r != cudaSuccess) return r;
  }
  return cudaSuccess;
}

int pair_batch_occupancy(const PairEntry& e, int S) {
  int best = 1 << 30;
  for (int s = 0; s < e.nslices; ++s) {
    int b = 0;
    if (e.slices[s].occupancy_batch(S, &b) != cudaSuccess) {
      cudaGetLastError();
      return 0;
    }
    best = std::min(best, b);
  }
  return e.nslices ? best : 0;
}

cudaError_t pair_launch_batch(const PairEntry& e, const void* rec, const BatchInst* inst,
                              const int4* items, const int* n_items, int* counters, int grid,
                              int S, const void* gbox, double* partial, cudaStream_t st) {
  for (int s = 0; s < e.nslices; ++s) {
    cudaError_t r = e.slices[s].launch_batch(rec, inst, items, n_items, counters + s, grid, S,
                                             gbox, partial, st);
    if (r != cudaSuccess) return r;
  }
  return cudaSuccess;
}

int list_variant_count(int M) {
  if (M < 0 || M > 8) return 0;
  return n_list_variants(M);
}

ListEntry list_entry(int M, int v) {
  ListEntry e;
  if (v < 0 || v >= list_variant_count(M)) return e;
  if (!fill_list(M * kMaxListVariants + v, e)) return e;
  e.M = M;
  e.variant = v;
  e.nslices = list_variant_spec(M, v).nslices;
  return e;
}

cudaError_t list_prepare(const ListEntry& e) {
  for (int s = 0; s < e.nslices; ++s) {
    cudaError_t r = e.slices[s].prepare();
    if (r != cudaSuccess) return r;
  }
  return cudaSuccess;
}

int list_occupancy(const ListEntry& e) {
  int best = 1 << 30;
  for (int s = 0; s < e.nslices; ++s) {
    int b = 0;
    if (e.slices[s].occupancy(&b) != cudaSuccess) {
      cudaGetLastError();
      return 0;
    }
    best = std::min(best, b);
  }
  return e.nslices ? best : 0;
}

long long tree_nodes(int G) { return tree_level_offset(G, tree_levels(G) + 1); }

int tree_chunk_level(int G, int blocks, int* nodes) {
  int L = 0;
  while (tree_level_nodes(G, L) > std::max(blocks, 1)) ++L;
  *nodes = tree_level_nodes(G, L);
  return L;
}

namespace {

constexpr int kCutThreads = 1024;
constexpr int kMinShare = 32;  // sources: about 3 rounds of a CTA's warps

// One CTA: the near sources nsrc[g] of the G target groups, put one group after
// another, in at most T equal shares, so that no group falls into more than C
// of them: pre[g] = sources before group g, pre[G] = all, pre[G + 1] = sources
// per share, gshares[g] = shares that group g falls into, start[t] = group in
// which share t starts (only set for shares that exist).
__global__ void __launch_bounds__(kCutThreads)
    near_cut_kernel(int G, int T, int C, const int* nsrc, unsigned long long* pre, int* gshares,
                    int* start) {
  __shared__ unsigned long long wsum[32], total;
  __shared__ int wmax[32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  unsigned long long run = 0;
  int most = 0;
  for (int g0 = 0; g0 < G; g0 += kCutThreads) {
    const int g = g0 + threadIdx.x;
    const int w = g < G ? nsrc[g] : 0;
    most = max(most, w);
    unsigned long long incl = w;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned long long v = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += v;
    }
    if (lane == 31) wsum[warp] = incl;
    __syncthreads();
    if (warp == 0) {
      unsigned long long s = wsum[lane];
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long v = __shfl_up_sync(0xffffffffu, s, o);
        if (lane >= o) s += v;
      }
      wsum[lane] = s;
      if (lane == 31) total = s;
    }
    __syncthreads();
    if (g < G) pre[g] = run + (warp ? wsum[warp - 1] : 0) + incl - w;
    run += total;
    __syncthreads();  // wsum and total are rewritten
  }
  most = __reduce_max_sync(0xffffffffu, most);
  if (lane == 0) wmax[warp] = most;
  __syncthreads();
  most = __reduce_max_sync(0xffffffffu, wmax[lane]);
  // a group of w sources falls into at most ceil(w / share) + 1 shares
  unsigned long long share = (run + T - 1) / T;
  share = max(share, (unsigned long long)((most + C - 2) / (C - 1)));
  share = max(share, (unsigned long long)kMinShare);
  if (threadIdx.x == 0) {
    pre[G] = run;
    pre[G + 1] = share;
  }
  __syncthreads();
  for (int g = threadIdx.x; g < G; g += kCutThreads) {
    const unsigned long long a = pre[g], b = pre[g + 1];
    gshares[g] = b > a ? (int)((b - 1) / share - a / share) + 1 : 0;
  }
  for (int t = threadIdx.x; t < T; t += kCutThreads) {
    const unsigned long long at = t * share;
    if (at >= run) break;
    int l = 0, h = G - 1;  // the last group with pre <= at: it has sources
    while (l < h) {
      const int m = (l + h + 1) >> 1;
      if (pre[m] <= at) l = m;
      else h = m - 1;
    }
    start[t] = l;
  }
}

}  // namespace

cudaError_t list_launch(const ListEntry& e, const ListArgs& A, cudaStream_t st,
                        cudaEvent_t* marks) {
  const int n = A.n, G = (n + kGroup - 1) / kGroup;
  const float rmax = A.local ? e.far.loc_radius : 0.f;
  const float frad = A.local ? e.far.loc_field_radius : 0.f;
  cudaError_t r = e.far.build(A.rec, n, G, A.gdata, rmax, A.ent, A.cnt, A.cnt + G, A.cut, st);
  if (r == cudaSuccess) {
    near_cut_kernel<<<1, kCutThreads, 0, st>>>(G, A.shares, A.segments, A.cut, A.pre, A.cut + G,
                                               A.cut + 2 * (size_t)G);
    r = cudaGetLastError();
  }
  if (A.tree && r == cudaSuccess) r = e.far.tree_build(A.gdata, n, G, A.tree, st);
  if (marks && r == cudaSuccess) r = cudaEventRecord(marks[0], st);
  if (r == cudaSuccess)
    r = A.tree ? e.far.far_tree(A.rec, n, G, A.gdata, A.tree, A.Lc, frad, A.fpart, A.counts, st)
               : e.far.far(A.rec, n, G, A.gdata, A.far_ranges, frad, A.fpart, A.counts, st);
  if (A.local && r == cudaSuccess)
    r = e.far.loc_far(A.rec, n, G, A.gdata, A.tree, A.Lc, A.far_ranges, A.ffld, A.counts, st);
  if (marks && r == cudaSuccess) r = cudaEventRecord(marks[1], st);
  if (A.local && r == cudaSuccess)
    r = e.far.loc_near(A.rec, n, G, A.gdata, A.gexp, A.ent, A.cnt + G, A.loc_segments, A.fld,
                       A.tree ? tree_level_nodes(G, A.Lc) : A.far_ranges, A.ffld,
                       A.partial + (size_t)A.segments * n_beta(e.M) * n, A.counts, A.err, st);
  for (int s = 0; s < e.nslices && r == cudaSuccess; ++s) {
    r = e.slices[s].launch(A.rec, n, G, A.ent, A.cnt, A.shares, A.pre, A.cut + 2 * (size_t)G, A.partial,
                           A.counts, A.err, st);
    if (marks && r == cudaSuccess) r = cudaEventRecord(marks[2 + s], st);
  }
  return r;
}

}  // namespace mmvm
