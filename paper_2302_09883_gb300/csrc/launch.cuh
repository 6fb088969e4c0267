// Launch glue for one instantiation of the fused patch kernel.
#pragma once
#include "patch2d.cuh"
#include "registry.h"

namespace wcs {

// A step behind the step before it in its stream (see after_last_step): the
// next step's launch latency, 3 to 4 us, hides behind the last wave.
inline cudaError_t launch_step(void (*kernel)(PatchArgs), const PatchArgs& a, int blocks, int threads, size_t smem,
                               cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(unsigned(blocks));
  cfg.blockDim = dim3(unsigned(threads));
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, a);
}

// hi + lo coarse storage: INIT and STEP kernels of their own (HL = 1)
template <int SCH, int WV, typename T, int ST, int P, int L>
cudaError_t prepare_hilo() {
  typedef Cfg<SCH, WV, T, ST, P, L> C;
  if constexpr (C::HILO) {
    cudaError_t e;
    if ((e = cudaFuncSetAttribute(patch_kernel<SCH, WV, T, ST, P, L, MODE_INIT, 0, 1>,
                                  cudaFuncAttributeMaxDynamicSharedMemorySize, int(C::SMEM))) != cudaSuccess)
      return e;
    return cudaFuncSetAttribute(patch_kernel<SCH, WV, T, ST, P, L, MODE_STEP, 0, 1>,
                                cudaFuncAttributeMaxDynamicSharedMemorySize, int(C::SMEM));
  }
  return cudaSuccess;
}

// Clusters for the steps of small grids: D2Q9 with a ghost ring in FP64, five
// CTAs (two of the nine fields each at most) or three (three each) per patch.
// More would not shorten the transforms until there are nine, and GB300's
// GPCs hold 28 clusters of five but only 15 of eight (one short of the 16
// patches of the 128^2 grid: 65 us a step in two rounds, five: 40 us).
template <int SCH, int WV, typename T, int ST, int P, int L> constexpr bool has_cluster() {
  return SCH == SCH_D2Q9 && !Cfg<SCH, WV, T, ST, P, L>::RINGFREE && sizeof(T) == 8;
}
template <int SCH, int WV, typename T, int ST, int P, int L, int CL> bool cluster_fits(int npatch) {
  typedef Cfg<SCH, WV, T, ST, P, L> C;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(unsigned(npatch) * CL);
  cfg.blockDim = dim3(C::NT);
  cfg.dynamicSmemBytes = C::SMEM;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = CL;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, patch_kernel_cluster<SCH, WV, T, ST, P, L, CL>, &cfg) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return npatch <= n;
}
// Steps with two CTAs per SM: 33^2-node patches have at most 297 lines per
// pass, so a CTA of a whole SM leaves most threads at the barriers, but it
// finishes a patch sooner.  Shallow water 992 x 512 (496 patches, 30 steps) 1.91
// -> 1.60 ms, 512^2 (256) 1.32 -> 1.10, FP64 512^2 18.7 -> 15.8.  D2Q9 1632 x
// 1024 (1632 patches, 30 steps) 3.36 -> 2.39, FP32 details 992^2 (961) 7.13 ->
// 6.29; where a few patches hold most of the survivors the step waits for
// them: a bump, 53 steps, 1024 patches 4.23 -> 4.00, 640 equal, 480 3.02 ->
// 3.15, 304 2.55 -> 2.69.  So nine fields take it from four patches per SM on,
// three from one and a half (on 16 patches 5.5 -> 6.0).  Nine FP64 fields need
// more warps and registers than half an SM has.
constexpr int HALF_SM = -1;
template <int SCH, int P, typename T> constexpr bool has_half() {
  return P <= 32 && scheme_fields(SCH) > 1 && (sizeof(T) == 4 || scheme_fields(SCH) <= 3);
}
// Shape of a step of npatch patches: the largest cluster of which all run at
// once (beyond that an SM steps a whole patch in less time than its share of
// several), HALF_SM: CTAs of half an SM, 0: one CTA per patch and SM.
template <int SCH, int WV, typename T, int ST, int P, int L> int pick_shape(int npatch) {
  if constexpr (has_cluster<SCH, WV, T, ST, P, L>()) {
    if (cluster_fits<SCH, WV, T, ST, P, L, 5>(npatch)) return 5;
    if (cluster_fits<SCH, WV, T, ST, P, L, 3>(npatch)) return 3;
  } else if constexpr (has_half<SCH, P, T>()) {
    int dev = 0, nsm = 0;
    if (cudaGetDevice(&dev) == cudaSuccess &&
        cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess &&
        2 * (long long)npatch >= (scheme_fields(SCH) > 4 ? 8 : 3) * (long long)nsm)
      return HALF_SM;
    cudaGetLastError();
  }
  return 0;
}
template <int SCH, int WV, typename T, int ST, int P, int L>
cudaError_t launch_shape(const PatchArgs& a, int npatch, int shape, cudaStream_t s) {
  typedef Cfg<SCH, WV, T, ST, P, L> C;
  if (npatch <= 0) return cudaSuccess;
  if constexpr (has_cluster<SCH, WV, T, ST, P, L>()) {
    if (shape == 5) return launch_step(patch_kernel_cluster<SCH, WV, T, ST, P, L, 5>, a, npatch * 5, C::NT, C::SMEM, s);
    if (shape == 3) return launch_step(patch_kernel_cluster<SCH, WV, T, ST, P, L, 3>, a, npatch * 3, C::NT, C::SMEM, s);
  } else if constexpr (has_half<SCH, P, T>()) {
    typedef Cfg<SCH, WV, T, ST, P, L, 1> H;
    if (shape == HALF_SM)
      return launch_step(patch_kernel<SCH, WV, T, ST, P, L, MODE_STEP, 0, 0, 1>, a, npatch, H::NT, H::SMEM, s);
  }
  return cudaErrorInvalidValue;
}
template <int SCH, int WV, typename T, int ST, int P, int L>
cudaError_t prepare_half() {
  if constexpr (has_half<SCH, P, T>() && !has_cluster<SCH, WV, T, ST, P, L>())
    return cudaFuncSetAttribute(patch_kernel<SCH, WV, T, ST, P, L, MODE_STEP, 0, 0, 1>,
                                cudaFuncAttributeMaxDynamicSharedMemorySize, int(Cfg<SCH, WV, T, ST, P, L, 1>::SMEM));
  return cudaSuccess;
}

template <int SCH, int WV, typename T, int ST, int P, int L>
cudaError_t prepare_patch() {
  typedef Cfg<SCH, WV, T, ST, P, L> C;
  cudaError_t e;
  if constexpr (has_cluster<SCH, WV, T, ST, P, L>()) {
    if ((e = cudaFuncSetAttribute(patch_kernel_cluster<SCH, WV, T, ST, P, L, 5>,
                                  cudaFuncAttributeMaxDynamicSharedMemorySize, int(C::SMEM))) != cudaSuccess)
      return e;
    if ((e = cudaFuncSetAttribute(patch_kernel_cluster<SCH, WV, T, ST, P, L, 3>,
                                  cudaFuncAttributeMaxDynamicSharedMemorySize, int(C::SMEM))) != cudaSuccess)
      return e;
  }
  if ((e = cudaFuncSetAttribute(patch_kernel<SCH, WV, T, ST, P, L, MODE_INIT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                int(C::SMEM))) != cudaSuccess)
    return e;
  if ((e = cudaFuncSetAttribute(patch_kernel<SCH, WV, T, ST, P, L, MODE_STEP>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                int(C::SMEM))) != cudaSuccess)
    return e;
  if ((e = cudaFuncSetAttribute(patch_kernel<SCH, WV, T, ST, P, L, MODE_EXPORT>,
                                cudaFuncAttributeMaxDynamicSharedMemorySize, int(C::SMEM))) != cudaSuccess)
    return e;
  if ((e = cudaFuncSetAttribute(patch_kernel<SCH, WV, T, ST, P, L, MODE_STEP, 1>,
                                cudaFuncAttributeMaxDynamicSharedMemorySize, int(C::SMEM))) != cudaSuccess)
    return e;
  if ((e = prepare_hilo<SCH, WV, T, ST, P, L>()) != cudaSuccess) return e;
  if ((e = prepare_half<SCH, WV, T, ST, P, L>()) != cudaSuccess) return e;
  return cudaFuncSetAttribute(patch_kernel_batch<SCH, WV, T, ST, P, L>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              int(C::SMEM));
}

// step that also writes the per-patch features of the new state
template <int SCH, int WV, typename T, int ST, int P, int L>
cudaError_t launch_feat(const PatchArgs& a, int npatch, cudaStream_t s) {
  typedef Cfg<SCH, WV, T, ST, P, L> C;
  if (npatch <= 0) return cudaSuccess;
  if (a.coarse_lo) return cudaErrorInvalidValue;  // no learned-threshold kernel keeps hi + lo
  return launch_step(patch_kernel<SCH, WV, T, ST, P, L, MODE_STEP, 1>, a, npatch, C::NT, C::SMEM, s);
}

template <int SCH, int WV, typename T, int ST, int P, int L, int MODE>
cudaError_t launch_mode(const PatchArgs& a, int npatch, cudaStream_t s) {
  typedef Cfg<SCH, WV, T, ST, P, L> C;
  if (a.coarse_lo && MODE != MODE_EXPORT) {  // hi + lo coarse storage
    if constexpr (C::HILO && MODE == MODE_STEP) return launch_step(patch_kernel<SCH, WV, T, ST, P, L, MODE, 0, 1>, a, npatch, C::NT, C::SMEM, s);
    else if constexpr (C::HILO && MODE != MODE_EXPORT) patch_kernel<SCH, WV, T, ST, P, L, MODE, 0, 1><<<npatch, C::NT, C::SMEM, s>>>(a);
    else return cudaErrorInvalidValue;
  } else if constexpr (MODE == MODE_STEP) {
    return launch_step(patch_kernel<SCH, WV, T, ST, P, L, MODE>, a, npatch, C::NT, C::SMEM, s);
  } else {
    patch_kernel<SCH, WV, T, ST, P, L, MODE><<<npatch, C::NT, C::SMEM, s>>>(a);
  }
  return cudaGetLastError();
}

// (batches take no simulation with hi + lo coarse storage: wcs_batch_create)
template <int SCH, int WV, typename T, int ST, int P, int L>
cudaError_t launch_batch(const PatchArgs* args, const unsigned int* work, int nblocks, cudaStream_t s) {
  typedef Cfg<SCH, WV, T, ST, P, L> C;
  if (nblocks <= 0) return cudaSuccess;
  patch_kernel_batch<SCH, WV, T, ST, P, L><<<nblocks, C::NT, C::SMEM, s>>>(args, work);
  return cudaGetLastError();
}

template <int SCH, int WV, typename T, int ST, int P, int L>
cudaError_t launch_patch(int mode, const PatchArgs& a, int npatch, cudaStream_t s) {
  if (npatch <= 0) return cudaSuccess;
  if (mode == MODE_INIT) return launch_mode<SCH, WV, T, ST, P, L, MODE_INIT>(a, npatch, s);
  if (mode == MODE_STEP) return launch_mode<SCH, WV, T, ST, P, L, MODE_STEP>(a, npatch, s);
  return launch_mode<SCH, WV, T, ST, P, L, MODE_EXPORT>(a, npatch, s);
}

// Init / step / export only (no batch and no learned-threshold variants).
template <int SCH, int WV, typename T, int ST, int P, int L>
cudaError_t prepare_patch_lite() {
  typedef Cfg<SCH, WV, T, ST, P, L> C;
  cudaError_t e;
  if ((e = cudaFuncSetAttribute(patch_kernel<SCH, WV, T, ST, P, L, MODE_INIT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                int(C::SMEM))) != cudaSuccess)
    return e;
  if ((e = cudaFuncSetAttribute(patch_kernel<SCH, WV, T, ST, P, L, MODE_STEP>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                int(C::SMEM))) != cudaSuccess)
    return e;
  if ((e = prepare_hilo<SCH, WV, T, ST, P, L>()) != cudaSuccess) return e;
  if ((e = prepare_half<SCH, WV, T, ST, P, L>()) != cudaSuccess) return e;
  return cudaFuncSetAttribute(patch_kernel<SCH, WV, T, ST, P, L, MODE_EXPORT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              int(C::SMEM));
}

template <int SCH, int WV, typename T, int ST, int P, int L>
KernelEntry make_entry_lite() {
  typedef Cfg<SCH, WV, T, ST, P, L> C;
  KernelEntry k;
  k.scheme = SCH;
  k.wavelet = WV;
  k.prec = sizeof(T) == 8 ? 0 : 1;
  k.store = ST;
  k.P = P;
  k.L = L;
  k.ring = C::RING;
  k.pitch = C::PW;
  k.hilo = C::HILO ? 1 : 0;
  k.smem = C::SMEM;
  k.threads = C::NT;
  k.launch = &launch_patch<SCH, WV, T, ST, P, L>;
  k.launch_batch = nullptr;
  k.launch_feat = nullptr;
  k.pick_shape = &pick_shape<SCH, WV, T, ST, P, L>;
  k.launch_shape = &launch_shape<SCH, WV, T, ST, P, L>;
  k.prepare = &prepare_patch_lite<SCH, WV, T, ST, P, L>;
  return k;
}

template <int SCH, int WV, typename T, int ST, int P, int L>
KernelEntry make_entry() {
  typedef Cfg<SCH, WV, T, ST, P, L> C;
  KernelEntry k;
  k.scheme = SCH;
  k.wavelet = WV;
  k.prec = sizeof(T) == 8 ? 0 : 1;
  k.store = ST;
  k.P = P;
  k.L = L;
  k.ring = C::RING;
  k.pitch = C::PW;
  k.hilo = C::HILO ? 1 : 0;
  k.smem = C::SMEM;
  k.threads = C::NT;
  k.launch = &launch_patch<SCH, WV, T, ST, P, L>;
  k.launch_batch = &launch_batch<SCH, WV, T, ST, P, L>;
  k.launch_feat = &launch_feat<SCH, WV, T, ST, P, L>;
  k.pick_shape = &pick_shape<SCH, WV, T, ST, P, L>;
  k.launch_shape = &launch_shape<SCH, WV, T, ST, P, L>;
  k.prepare = &prepare_patch<SCH, WV, T, ST, P, L>;
  return k;
}

}  // namespace wcs

#define WCS_INSTANTIATE(NAME, SCH, WV, T, ST, P, L)                                        \
  namespace wcs {                                                                           \
  void NAME(std::vector<KernelEntry>& v) { v.push_back(make_entry<SCH, WV, T, ST, P, L>()); } \
  }

#define WCS_INSTANTIATE_LITE(NAME, SCH, WV, T, ST, P, L)                                        \
  namespace wcs {                                                                                \
  void NAME(std::vector<KernelEntry>& v) { v.push_back(make_entry_lite<SCH, WV, T, ST, P, L>()); } \
  }

namespace wcs {
template <int SCH, int WV, typename T, int ST, int P0, int L0, int P1, int L1>
cudaError_t launch_mixed(const PatchArgs* args0, const PatchArgs* args1, const unsigned int* work, int nitems, int grid,
                         cudaStream_t s) {
  typedef Cfg<SCH, WV, T, ST, P0, L0> C0;
  typedef Cfg<SCH, WV, T, ST, P1, L1> C1;
  if (nitems <= 0) return cudaSuccess;
  const size_t smem = C0::SMEM > C1::SMEM ? C0::SMEM : C1::SMEM;
  patch_kernel_batch_mixed<SCH, WV, T, ST, P0, L0, P1, L1><<<grid, C0::NT, smem, s>>>(args0, args1, work, nitems);
  return cudaGetLastError();
}

template <int SCH, int WV, typename T, int ST, int P0, int L0, int P1, int L1>
cudaError_t prepare_mixed() {
  typedef Cfg<SCH, WV, T, ST, P0, L0> C0;
  typedef Cfg<SCH, WV, T, ST, P1, L1> C1;
  const size_t smem = C0::SMEM > C1::SMEM ? C0::SMEM : C1::SMEM;
  return cudaFuncSetAttribute(patch_kernel_batch_mixed<SCH, WV, T, ST, P0, L0, P1, L1>,
                              cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
}

template <int SCH, int WV, typename T, int ST, int P0, int L0, int P1, int L1>
MixedBatchEntry make_mixed() {
  typedef Cfg<SCH, WV, T, ST, P0, L0> C0;
  typedef Cfg<SCH, WV, T, ST, P1, L1> C1;
  MixedBatchEntry m;
  m.scheme = SCH;
  m.wavelet = WV;
  m.prec = sizeof(T) == 8 ? 0 : 1;
  m.store = ST;
  m.P0 = P0;
  m.L0 = L0;
  m.P1 = P1;
  m.L1 = L1;
  m.smem = C0::SMEM > C1::SMEM ? C0::SMEM : C1::SMEM;
  m.threads = C0::NT;
  m.launch = &launch_mixed<SCH, WV, T, ST, P0, L0, P1, L1>;
  m.prepare = &prepare_mixed<SCH, WV, T, ST, P0, L0, P1, L1>;
  return m;
}
}  // namespace wcs
