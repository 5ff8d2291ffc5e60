// k_batch.cuh — dispatch of the batched kernels over their instances.
#pragma once
#include "launch.h"

namespace cfr {

#define CFR_BATCH_LANES(X, MA, TH) X(MA, 2, TH) X(MA, 4, TH) X(MA, 8, TH) X(MA, 32, TH)
#define CFR_BATCH_ALL(X) \
  CFR_BATCH_LANES(X, 4, 256) CFR_BATCH_LANES(X, 4, 1024) CFR_BATCH_LANES(X, 8, 256) CFR_BATCH_LANES(X, 8, 1024)

template <typename K, typename... More>
static cudaError_t launch_batch_any(K kern, int threads, const BatchLaunch &l, cudaStream_t s, const InstDesc *table,
                                    const InstDesc &one, More... more) {
  if (l.cluster > 8) {
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
  }
  // The limit belongs to the kernel, not to a launch: every caller sets the
  // same one, so that a launch from another thread cannot find a lower one.
  if (l.smem > 0) {
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kResidentBytes);
    if (e != cudaSuccess) return e;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(l.count * l.cluster));
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = l.smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  cfg.attrs = attr;
  if (l.cluster > 1) {
    attr[cfg.numAttrs].id = cudaLaunchAttributeClusterDimension;
    attr[cfg.numAttrs].val.clusterDim.x = (unsigned)l.cluster;
    attr[cfg.numAttrs].val.clusterDim.y = 1;
    attr[cfg.numAttrs].val.clusterDim.z = 1;
    ++cfg.numAttrs;
  }
  if (l.chained) {
    attr[cfg.numAttrs].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[cfg.numAttrs].val.programmaticStreamSerializationAllowed = 1;
    ++cfg.numAttrs;
  }
  return cudaLaunchKernelEx(&cfg, kern, table, one, l.count, more...);
}

template <typename T, int MA, int L, int TH>
static cudaError_t launch_batch_one(const BatchLaunch &l, cudaStream_t s, const InstDesc *table, const InstDesc &one) {
  constexpr int NT = kBatchThreads<T, MA, TH>;
  if (l.mode == kResident) return launch_batch_any(batch_iterate_kernel<T, MA, L, NT, kResident>, NT, l, s, table, one);
  if (l.mode == kCluster) return launch_batch_any(batch_iterate_kernel<T, MA, L, NT, kCluster>, NT, l, s, table, one);
  return launch_batch_any(batch_iterate_kernel<T, MA, L, NT, kSolo>, NT, l, s, table, one);
}

// FP64 sums do not depend on the lane count: chains of four or eight lanes.
template <typename T, int L> constexpr int kBatchLanes = sizeof(T) == 4 ? L : (L <= 4 ? 4 : 8);

template <typename T>
cudaError_t launch_batch_iterate(int maxa, int lanes, int threads, const BatchLaunch &l, cudaStream_t s,
                                 const InstDesc *table, const InstDesc &one) {
  if (l.push) return launch_batch_push<T>(maxa, lanes, threads, l, s, table, one);
#define IT_CASE(MA, L, TH)                       \
  if (maxa == MA && lanes == L && threads == TH) \
    return launch_batch_one<T, MA, kBatchLanes<T, L>, TH>(l, s, table, one);
  CFR_BATCH_ALL(IT_CASE)
#undef IT_CASE
  return cudaErrorInvalidValue;
}

}  // namespace cfr
