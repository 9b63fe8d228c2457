// One near-pair kernel of one interaction-list variant (pair_list.cuh,
// pair_list_variants.h), built with -DMMVM_INST_M, -DMMVM_INST_V and
// -DMMVM_INST_S so the kernels compile in parallel; with -DMMVM_INST_FAR
// instead of -DMMVM_INST_V / -DMMVM_INST_S, the list build and the far
// kernel of order MMVM_INST_M.
#include <algorithm>

#include "pair_local.cuh"
#include "pair_registry.h"

#if !defined(MMVM_INST_M)
#error "MMVM_INST_M must be defined"
#endif

namespace mmvm {

#if defined(MMVM_INST_FAR)

namespace {
constexpr int kM = MMVM_INST_M;
cudaError_t build_fn(const float* rec, int n, int G, const float* gdata, float rmax, int2* ent,
                     int* cnt, int* mcnt, int* nsrc, cudaStream_t st) {
  // a warp per target group; one warp per CTA while that spreads them over the SMs
  const int wpc = G <= 1024 ? 1 : 8;
  near_list_kernel<kM><<<(G + wpc - 1) / wpc, 32 * wpc, 0, st>>>(rec, n, G, gdata, rmax, ent,
                                                                    cnt, mcnt, nsrc);
  return cudaGetLastError();
}
cudaError_t far_fn(const float* rec, int n, int G, const float* gdata, int S, float frad,
                   double* fpart, unsigned long long* counts, cudaStream_t st) {
  dim3 grid((G + kFarWarps - 1) / kFarWarps, S);
  far_pair_kernel<kM><<<grid, kFarWarps * 32, 0, st>>>(rec, n, G, gdata, S, frad, fpart, counts);
  return cudaGetLastError();
}
cudaError_t far_occ_fn(int* blocks) {
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks, far_pair_kernel<kM>,
                                                       kFarWarps * 32, 0);
}
cudaError_t tree_build_fn(const float* gdata, int n, int G, float* tree, cudaStream_t st) {
  const int top = tree_levels(G);
  int L = 1;
  for (; L <= top && tree_level_nodes(G, L) > kTreeTop; ++L)
    tree_level_kernel<kM><<<(tree_level_nodes(G, L) + 3) / 4, 128, 0, st>>>(gdata, n, G, L, L, tree);
  if (L <= top) {
    const int warps = std::min(tree_level_nodes(G, L), 32);
    tree_level_kernel<kM><<<1, 32 * warps, 0, st>>>(gdata, n, G, L, top, tree);
  }
  return cudaGetLastError();
}
cudaError_t far_tree_fn(const float* rec, int n, int G, const float* gdata, const float* tree,
                        int Lc, float frad, double* fpart, unsigned long long* counts,
                        cudaStream_t st) {
  dim3 grid((G + kFarWarps - 1) / kFarWarps, tree_level_nodes(G, Lc));
  far_tree_kernel<kM><<<grid, kFarWarps * 32, 0, st>>>(rec, n, G, gdata, tree, Lc, frad, fpart,
                                                    counts);
  return cudaGetLastError();
}
cudaError_t loc_prepare_fn() {
  cudaError_t e = cudaFuncSetAttribute(
      loc_near_kernel<kM>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)LocSmem<kM>::bytes);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(loc_far_kernel<kM>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)LocFarSmem<kM>::bytes);
}
cudaError_t loc_far_fn(const float* rec, int n, int G, const float* gdata, const float* tree,
                       int Lc, int S, float2* ffld, unsigned long long* counts,
                       cudaStream_t st) {
  const dim3 grid((G + kLocWarps - 1) / kLocWarps, tree ? tree_level_nodes(G, Lc) : S);
  loc_far_kernel<kM><<<grid, kLocWarps * 32, LocFarSmem<kM>::bytes, st>>>(
      rec, n, G, gdata, tree, Lc, S, ffld, counts);
  return cudaGetLastError();
}
cudaError_t loc_near_fn(const float* rec, int n, int G, const float* gdata, float* gexp,
                        const int2* ent, const int* mcnt, int C, float2* fld, int nfar,
                        const float2* ffld, double* out, unsigned long long* counts, int* err,
                        cudaStream_t st) {
  const int blocks = (G + kLocWarps - 1) / kLocWarps;
  loc_expand_kernel<kM><<<G, 32, 0, st>>>(rec, n, G, gdata, gexp);
  loc_near_kernel<kM><<<dim3(blocks, C), kLocWarps * 32, LocSmem<kM>::bytes, st>>>(
      n, G, gdata, gexp, ent, mcnt, C, fld, counts, err);
  loc_eval_kernel<kM><<<G, kEvalWarps * 32, 0, st>>>(rec, n, G, gdata, C, fld, nfar, ffld, out);
  return cudaGetLastError();
}
}  // namespace

#define MMVM_CAT2(a, b) a##b
#define MMVM_FAR_NAME(m) MMVM_CAT2(list_far_m, m)
#define MMVM_FAR(m) MMVM_FAR_NAME(m)

ListFarEntry MMVM_FAR(MMVM_INST_M)() {
  ListFarEntry e;
  e.build = build_fn;
  e.far = far_fn;
  e.far_occupancy = far_occ_fn;
  e.tree_build = tree_build_fn;
  e.far_tree = far_tree_fn;
  e.n_edge = n_edge(kM);
  e.loc_prepare = loc_prepare_fn;
  e.loc_far = loc_far_fn;
  e.loc_near = loc_near_fn;
  e.loc_len = Loc<kM>::LEN;
  e.loc_rows = Loc<kM>::FROWS;
  e.loc_radius = loc_radius(kM);
  e.loc_field_radius = loc_field_radius(kM);
  return e;
}

#else

#if !defined(MMVM_INST_V) || !defined(MMVM_INST_S)
#error "MMVM_INST_V and MMVM_INST_S must be defined"
#endif

namespace {
constexpr int kM = MMVM_INST_M;
constexpr ListVariantSpec kSpec = list_variant_spec(kM, MMVM_INST_V);
static_assert(MMVM_INST_S < kSpec.nslices, "slice index out of range");
constexpr ListSliceSpec kS = kSpec.s[MMVM_INST_S];
constexpr size_t kSmem = near_list_smem_bytes<kM, kS.lo, kS.hi, kS.part, kS.w, kS.nst>();
static_assert(kSmem <= 232448, "near-pair kernel needs more shared memory than a CTA has");
#define MMVM_NEAR_KERNEL near_pair_kernel<kM, kS.lo, kS.hi, kS.part, kS.w, kS.minb, kS.nst, kS.sync>

cudaError_t prepare_fn() {
  return cudaFuncSetAttribute(MMVM_NEAR_KERNEL, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)kSmem);
}
cudaError_t launch_fn(const float* rec, int n, int G, const int2* ent, const int* cnt, int T,
                      const unsigned long long* pre, const int* start, double* partial, unsigned long long* counts, int* err, cudaStream_t st) {
  MMVM_NEAR_KERNEL<<<T, kS.w * 32, kSmem, st>>>(rec, n, G, ent, cnt, pre, start, partial, counts,
                                                err);
  return cudaGetLastError();
}
cudaError_t occ_fn(int* blocks) {
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks, MMVM_NEAR_KERNEL, kS.w * 32,
                                                       kSmem);
}
}  // namespace

#define MMVM_CAT4(a, b, c, d) a##b##c##d
#define MMVM_LSLICE_NAME(m, v, s) MMVM_CAT4(list_slice_m, m, _v##v, _s##s)
#define MMVM_LSLICE(m, v, s) MMVM_LSLICE_NAME(m, v, s)

ListSliceEntry MMVM_LSLICE(MMVM_INST_M, MMVM_INST_V, MMVM_INST_S)() {
  ListSliceEntry e;
  e.lo = kS.lo;
  e.hi = kS.hi;
  e.part = kS.part;
  e.warps = kS.w;
  e.prepare = prepare_fn;
  e.launch = launch_fn;
  e.occupancy = occ_fn;
  return e;
}

#endif

}  // namespace mmvm
