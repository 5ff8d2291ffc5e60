// k_batch.cuh — dispatch of the batched kernels over their instances.
#pragma once
#include "launch.h"

namespace cfr {

#define CFR_BATCH_LANES(X, MA, TH) X(MA, 2, TH) X(MA, 4, TH) X(MA, 8, TH) X(MA, 32, TH)
#define CFR_BATCH_ALL(X) \
  CFR_BATCH_LANES(X, 4, 256) CFR_BATCH_LANES(X, 4, 1024) CFR_BATCH_LANES(X, 8, 256) CFR_BATCH_LANES(X, 8, 1024)

// `cluster` CTAs per instance; chained: the launch before in the stream is the
// same call's and need not be complete (chain_enter).
template <typename K>
static cudaError_t launch_batch_any(K kern, int threads, int cluster, bool chained, int n, cudaStream_t s,
                                    const InstDesc *table, const InstDesc &one) {
  if (cluster > 8) {
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(n * cluster));
  cfg.blockDim = dim3((unsigned)threads);
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  cfg.attrs = attr;
  if (cluster > 1) {
    attr[cfg.numAttrs].id = cudaLaunchAttributeClusterDimension;
    attr[cfg.numAttrs].val.clusterDim.x = (unsigned)cluster;
    attr[cfg.numAttrs].val.clusterDim.y = 1;
    attr[cfg.numAttrs].val.clusterDim.z = 1;
    ++cfg.numAttrs;
  }
  if (chained) {
    attr[cfg.numAttrs].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[cfg.numAttrs].val.programmaticStreamSerializationAllowed = 1;
    ++cfg.numAttrs;
  }
  return cudaLaunchKernelEx(&cfg, kern, table, one, n);
}

template <typename T, int MA, int L, int TH>
static cudaError_t launch_batch_one(int cluster, bool chained, int n, cudaStream_t s, const InstDesc *table,
                                    const InstDesc &one) {
  constexpr int NT = kBatchThreads<T, MA, TH>;
  if (cluster == 1) return launch_batch_any(batch_iterate_kernel<T, MA, L, NT, false>, NT, 1, chained, n, s, table, one);
  return launch_batch_any(batch_iterate_kernel<T, MA, L, NT, true>, NT, cluster, chained, n, s, table, one);
}

// FP64 sums do not depend on the lane count: chains of four or eight lanes.
template <typename T>
cudaError_t launch_batch_iterate(int maxa, int lanes, int threads, int cluster, bool chained, int n, cudaStream_t s,
                                 const InstDesc *table, const InstDesc &one) {
#define IT_CASE(MA, L, TH)                          \
  if (maxa == MA && lanes == L && threads == TH)    \
    return launch_batch_one<T, MA, sizeof(T) == 4 ? L : (L <= 4 ? 4 : 8), TH>(cluster, chained, n, s, table, one);
  CFR_BATCH_ALL(IT_CASE)
#undef IT_CASE
  return cudaErrorInvalidValue;
}

}  // namespace cfr
