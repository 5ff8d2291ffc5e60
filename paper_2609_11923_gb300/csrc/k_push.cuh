// k_push.cuh — dispatch of the batched kernels of the pushing reach orders (in
// files of their own: compiled beside k_batch.cuh's, and loaded when used).
#pragma once
#include "k_batch.cuh"

namespace cfr {

// (FP64 sums do not depend on the lane count, and a thread holds fewer of their
// terms with four: 200 endgames of 10,400 nodes 20 iterations 4.9 ms, by eight
// lanes 7.1.)
template <typename T, int MA, int L, int TH>
static cudaError_t push_one(const BatchLaunch &l, cudaStream_t s, const InstDesc *table, const InstDesc &one) {
  constexpr int NT = kBatchThreads<T, MA, TH>;
  if (l.mode == kCluster) return launch_batch_any(batch_iterate_push_kernel<T, MA, L, NT, kCluster>, NT, l, s, table, one);
  return launch_batch_any(batch_iterate_push_kernel<T, MA, L, NT, kSolo>, NT, l, s, table, one);
}

template <typename T>
cudaError_t launch_batch_push(int maxa, int lanes, int threads, const BatchLaunch &l, cudaStream_t s,
                              const InstDesc *table, const InstDesc &one) {
#define PUSH_CASE(MA, L, TH)                     \
  if (maxa == MA && lanes == L && threads == TH) return push_one<T, MA, sizeof(T) == 8 ? 4 : L, TH>(l, s, table, one);
  CFR_BATCH_ALL(PUSH_CASE)
#undef PUSH_CASE
  return cudaErrorInvalidValue;
}

}  // namespace cfr
