// Spatial ordering of the particles for the all-pairs kernel: consecutive
// positions are close in space, so the 32-particle groups (source tiles and
// target warps) have small bounding boxes and the far-field test of the pair
// kernel can take the point-vortex jet for whole tiles.  Keys: the position
// along a Hilbert curve of the centres quantised to 16 bits per axis over the
// bounding square, sorted with a stable radix sort (ties keep the index
// order), so the order is deterministic.  Neighbours on a Hilbert curve are
// always neighbours in the plane; a Z-order curve jumps across the plane, and
// the groups that straddle a jump have boxes many times larger (two patches,
// n = 65536: median group radius 0.60 core units against 1.06, mean box area
// 0.88 against 1.96).
#include <cub/device/device_radix_sort.cuh>

#include <algorithm>

#include "common.cuh"
#include "particle_kernels.h"

namespace mmvm {

namespace {

// Distance along the order-16 Hilbert curve of the cell (x, y), both below
// 2^16: per level the quadrant's rank along the curve, then the rotation or
// reflection that maps the quadrant's curve onto the parent's.
__device__ __forceinline__ unsigned hilbert16(unsigned x, unsigned y) {
  unsigned d = 0;
#pragma unroll
  for (int b = 15; b >= 0; --b) {
    const unsigned rx = (x >> b) & 1u, ry = (y >> b) & 1u;
    d = (d << 2) | ((3u * rx) ^ ry);
    if (!ry) {
      if (rx) {
        x = 65535u - x;
        y = 65535u - y;
      }
      const unsigned t = x;
      x = y;
      y = t;
    }
  }
  return d;
}

// Morton (Z-order) code of a centre, each axis scaled to its own extent: the
// server's order.  Its batched kernel (direct form, no expansions) gains 2 % from
// the Hilbert order, within the spread of its runs.
__device__ __forceinline__ unsigned spread16(unsigned v) {
  v &= 0xffffu;
  v = (v | (v << 8)) & 0x00ff00ffu;
  v = (v | (v << 4)) & 0x0f0f0f0fu;
  v = (v | (v << 2)) & 0x33333333u;
  v = (v | (v << 1)) & 0x55555555u;
  return v;
}
__device__ __forceinline__ unsigned morton_key(double x1, double x2, const double4 b) {
  const double s1 = fmax(b.z - b.x, 1e-300), s2 = fmax(b.w - b.y, 1e-300);
  const double q1 = fmin(fmax((x1 - b.x) / s1, 0.0), 1.0) * 65535.0;
  const double q2 = fmin(fmax((x2 - b.y) / s2, 0.0), 1.0) * 65535.0;
  return spread16((unsigned)q1) | (spread16((unsigned)q2) << 1);
}

// Hilbert key of the centre (x1, x2) in the box (min1, min2, max1, max2).
__device__ __forceinline__ unsigned order_key(double x1, double x2, double lo1, double lo2,
                                              double hi1, double hi2) {
  const double s = fmax(fmax(hi1 - lo1, hi2 - lo2), 1e-300);
  const double q1 = fmin(fmax((x1 - lo1) / s, 0.0), 1.0) * 65535.0;
  const double q2 = fmin(fmax((x2 - lo2) / s, 0.0), 1.0) * 65535.0;
  return hilbert16((unsigned)q1, (unsigned)q2);
}

// Bounding box of the centres of one CTA's share -> box[4 blockIdx.x ...] = (min1,
// min2, max1, max2); keys_kernel joins the shares' boxes.  (One CTA for all
// took 85 us at n = 65536.)
__device__ __forceinline__ void warp_box(double& lo1, double& lo2, double& hi1, double& hi2) {
  for (int o = 16; o > 0; o >>= 1) {
    lo1 = fmin(lo1, __shfl_xor_sync(0xffffffffu, lo1, o));
    hi1 = fmax(hi1, __shfl_xor_sync(0xffffffffu, hi1, o));
    lo2 = fmin(lo2, __shfl_xor_sync(0xffffffffu, lo2, o));
    hi2 = fmax(hi2, __shfl_xor_sync(0xffffffffu, hi2, o));
  }
}
__global__ void bbox_kernel(int n, const double* __restrict__ x, double* __restrict__ box) {
  __shared__ double red[4][32];
  double lo1 = 1e300, lo2 = 1e300, hi1 = -1e300, hi2 = -1e300;
#pragma unroll 4
  for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < n; j += gridDim.x * blockDim.x) {
    const double a = x[2 * j], b = x[2 * j + 1];
    lo1 = fmin(lo1, a);
    hi1 = fmax(hi1, a);
    lo2 = fmin(lo2, b);
    hi2 = fmax(hi2, b);
  }
  warp_box(lo1, lo2, hi1, hi2);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  if (l == 0) {
    red[0][w] = lo1;
    red[1][w] = lo2;
    red[2][w] = hi1;
    red[3][w] = hi2;
  }
  __syncthreads();
  if (w == 0) {
    const int nw = blockDim.x >> 5;
    lo1 = l < nw ? red[0][l] : 1e300;
    lo2 = l < nw ? red[1][l] : 1e300;
    hi1 = l < nw ? red[2][l] : -1e300;
    hi2 = l < nw ? red[3][l] : -1e300;
    warp_box(lo1, lo2, hi1, hi2);
    if (l == 0) {
      double* o = box + 4 * blockIdx.x;
      o[0] = lo1;
      o[1] = lo2;
      o[2] = hi1;
      o[3] = hi2;
    }
  }
}

__global__ void keys_kernel(int n, int boxes, const double* __restrict__ x,
                            const double* __restrict__ box, unsigned* __restrict__ keys,
                            int* __restrict__ idx) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x, l = threadIdx.x & 31;
  double lo1 = l < boxes ? box[4 * l] : 1e300, lo2 = l < boxes ? box[4 * l + 1] : 1e300;
  double hi1 = l < boxes ? box[4 * l + 2] : -1e300, hi2 = l < boxes ? box[4 * l + 3] : -1e300;
  warp_box(lo1, lo2, hi1, hi2);
  if (j >= n) return;
  keys[j] = order_key(x[2 * j], x[2 * j + 1], lo1, lo2, hi1, hi2);
  idx[j] = j;
}

// scratch layout: [boxes of the CTAs, 4 doubles each][keys_in n][keys_out n][idx_in n][cub temp]
size_t cub_bytes(int n) {
  size_t b = 0;
  cub::DeviceRadixSort::SortPairs(nullptr, b, (const unsigned*)nullptr, (unsigned*)nullptr,
                                  (const int*)nullptr, (int*)nullptr, n);
  return b;
}

// Batches: one block per instance -> bounding box of its step-start centres,
// ibox[i] = (min1, min2, max1, max2).
__global__ void bbox_batch_kernel(const BatchInst* __restrict__ inst, const int* __restrict__ n_inst,
                                  double4* __restrict__ ibox) {
  __shared__ double red[4][32];
  const int total = *n_inst;
  for (int i = blockIdx.x; i < total; i += gridDim.x) {
    const BatchInst& I = inst[i];
    double lo1 = 1e300, lo2 = 1e300, hi1 = -1e300, hi2 = -1e300;
    for (int j = threadIdx.x; j < I.n; j += blockDim.x) {
      const double a = I.state[2 * j], b = I.state[2 * j + 1];
      lo1 = fmin(lo1, a);
      hi1 = fmax(hi1, a);
      lo2 = fmin(lo2, b);
      hi2 = fmax(hi2, b);
    }
    for (int o = 16; o > 0; o >>= 1) {
      lo1 = fmin(lo1, __shfl_xor_sync(0xffffffffu, lo1, o));
      hi1 = fmax(hi1, __shfl_xor_sync(0xffffffffu, hi1, o));
      lo2 = fmin(lo2, __shfl_xor_sync(0xffffffffu, lo2, o));
      hi2 = fmax(hi2, __shfl_xor_sync(0xffffffffu, hi2, o));
    }
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    if (l == 0) {
      red[0][w] = lo1;
      red[1][w] = lo2;
      red[2][w] = hi1;
      red[3][w] = hi2;
    }
    __syncthreads();
    if (w == 0) {
      const int nw = blockDim.x >> 5;
      lo1 = l < nw ? red[0][l] : 1e300;
      lo2 = l < nw ? red[1][l] : 1e300;
      hi1 = l < nw ? red[2][l] : -1e300;
      hi2 = l < nw ? red[3][l] : -1e300;
      for (int o = 16; o > 0; o >>= 1) {
        lo1 = fmin(lo1, __shfl_xor_sync(0xffffffffu, lo1, o));
        hi1 = fmax(hi1, __shfl_xor_sync(0xffffffffu, hi1, o));
        lo2 = fmin(lo2, __shfl_xor_sync(0xffffffffu, lo2, o));
        hi2 = fmax(hi2, __shfl_xor_sync(0xffffffffu, hi2, o));
      }
      if (l == 0) ibox[i] = make_double4(lo1, lo2, hi1, hi2);
    }
    __syncthreads();  // red is reused by the next instance
  }
}

// Key of slot p: (instance << 32) | Morton code in the instance's own box;
// padding slots of an instance sort after its particles, slots past the
// batch after everything.
__global__ void keys_batch_kernel(int slot_cap, const int* __restrict__ n_slots,
                                    const BatchInst* __restrict__ inst,
                                    const int* __restrict__ slot_inst,
                                    const double4* __restrict__ ibox,
                                    unsigned long long* __restrict__ keys, int* __restrict__ idx) {
  const int total = *n_slots;
  for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < slot_cap; p += gridDim.x * blockDim.x) {
    unsigned long long key = ~0ull;
    if (p < total) {
      const int i = slot_inst[p / kGroup];
      const BatchInst& I = inst[i];
      const int j = p - I.slot0;
      unsigned code = 0xffffffffu;
      if (j < I.n) {
        code = morton_key(I.state[2 * j], I.state[2 * j + 1], ibox[i]);
      }
      key = ((unsigned long long)i << 32) | code;
    }
    keys[p] = key;
    idx[p] = p;
  }
}

// Sorted slot p of instance i holds its particle perm_local[p] (local index).
__global__ void perm_batch_kernel(const int* __restrict__ n_slots, const BatchInst* __restrict__ inst,
                                  const int* __restrict__ slot_inst, const int* __restrict__ sorted,
                                  int* __restrict__ perm_local) {
  const int total = *n_slots;
  for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < total; p += gridDim.x * blockDim.x) {
    const BatchInst& I = inst[slot_inst[p / kGroup]];
    perm_local[p] = (p - I.slot0 < I.n) ? sorted[p] - I.slot0 : 0;
  }
}

size_t cub_bytes64(int n) {
  size_t b = 0;
  cub::DeviceRadixSort::SortPairs(nullptr, b, (const unsigned long long*)nullptr,
                                  (unsigned long long*)nullptr, (const int*)nullptr, (int*)nullptr,
                                  n);
  return b;
}

}  // namespace

size_t batch_order_temp_bytes(int slot_cap) { return cub_bytes64(slot_cap) + 256; }

cudaError_t launch_batch_order(int slot_cap, const int* n_slots, const BatchInst* inst,
                               const int* n_inst, int inst_cap, const int* slot_inst, void* ibox,
                               unsigned long long* kin, unsigned long long* kout, int* iin,
                               int* iout, void* temp, size_t temp_bytes, int* perm_local,
                               cudaStream_t st) {
  size_t cb = cub_bytes64(slot_cap);
  if (cb > temp_bytes) return cudaErrorInvalidValue;
  bbox_batch_kernel<<<std::max(1, std::min(inst_cap, 1024)), 256, 0, st>>>(
      inst, n_inst, static_cast<double4*>(ibox));
  const int blocks = std::max(1, std::min((slot_cap + 255) / 256, 4096));
  keys_batch_kernel<<<blocks, 256, 0, st>>>(slot_cap, n_slots, inst, slot_inst,
                                              static_cast<const double4*>(ibox), kin, iin);
  cudaError_t e = cub::DeviceRadixSort::SortPairs(temp, cb, kin, kout, iin, iout, slot_cap, 0, 64,
                                                  st);
  if (e != cudaSuccess) return e;
  perm_batch_kernel<<<blocks, 256, 0, st>>>(n_slots, inst, slot_inst, iout, perm_local);
  return cudaGetLastError();
}

size_t spatial_order_temp_bytes(int n) {
  return 32 * kBoxBlocks + (size_t)3 * ((size_t)n * 4 + 256) + cub_bytes(n) + 256;
}

cudaError_t launch_boxes(int n, const double* x, double* boxes, int* count, cudaStream_t st) {
  *count = std::max(1, std::min(kBoxBlocks, (n + 255) / 256));
  bbox_kernel<<<*count, 256, 0, st>>>(n, x, boxes);
  return cudaGetLastError();
}

cudaError_t launch_spatial_order(int n, const double* x, void* temp, size_t temp_bytes,
                                 int* perm, cudaStream_t st) {
  auto align = [](size_t v) { return (v + 255) & ~(size_t)255; };
  char* base = static_cast<char*>(temp);
  double* box = reinterpret_cast<double*>(base);
  size_t off = 32 * kBoxBlocks;
  unsigned* kin = reinterpret_cast<unsigned*>(base + off);
  off = align(off + (size_t)n * 4);
  unsigned* kout = reinterpret_cast<unsigned*>(base + off);
  off = align(off + (size_t)n * 4);
  int* iin = reinterpret_cast<int*>(base + off);
  off = align(off + (size_t)n * 4);
  size_t cb = cub_bytes(n);
  if (off + cb > temp_bytes) return cudaErrorInvalidValue;
  int boxes = 0;
  cudaError_t e = launch_boxes(n, x, box, &boxes, st);
  if (e != cudaSuccess) return e;
  keys_kernel<<<(n + 255) / 256, 256, 0, st>>>(n, boxes, x, box, kin, iin);
  return cub::DeviceRadixSort::SortPairs(base + off, cb, kin, kout, iin, perm, n, 0, 32, st);
}

}  // namespace mmvm
