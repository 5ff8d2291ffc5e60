// k_top.cuh — dispatch of the near-root kernel over its instances.
#pragma once
#include "launch.h"

namespace cfr {

#define CFR_TOP_ALL(X) X(4, 4) X(4, 8) X(8, 4) X(8, 8)

template <typename T> cudaError_t prepare_top(int maxa, int lanes) {
#define TOP_CASE(MA, L)          \
  if (maxa == MA && lanes == L)  \
    return cudaFuncSetAttribute(top_kernel<T, MA, L>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kResidentBytes);
  CFR_TOP_ALL(TOP_CASE)
#undef TOP_CASE
  return cudaErrorInvalidValue;
}

template <typename T>
cudaError_t launch_top(int maxa, int lanes, uint32_t smem, cudaStream_t s, const InstDesc &in, int K, int v_new, int phase,
                       int upd, bool pdl) {
#define TOP_CASE(MA, L)         \
  if (maxa == MA && lanes == L) \
    return launch_k(top_kernel<T, MA, L>, 1, kTopThreads<T, MA>, smem, s, pdl, in, K, v_new, phase, upd);
  CFR_TOP_ALL(TOP_CASE)
#undef TOP_CASE
  return cudaErrorInvalidValue;
}

}  // namespace cfr
