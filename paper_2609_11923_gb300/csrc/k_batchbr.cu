// Batched best-response kernel instances (see batch.cuh).
#include "k_batch.cuh"
namespace cfr {
template <int MA, int L, int TH>
static cudaError_t br_one(const BatchLaunch &l, cudaStream_t s, const InstDesc *table, const InstDesc &one) {
  constexpr int NT = kBatchThreads<double, MA, TH>, PARTS = TH <= 256 ? 256 : 512;
  static_assert(PARTS == NT || PARTS == 2 * NT, "one or two partial sums a thread");
  if (l.mode == kCluster) return launch_batch_any(batch_br_kernel<MA, L, NT, true>, NT, l, s, table, one, PARTS);
  return launch_batch_any(batch_br_kernel<MA, L, NT, false>, NT, l, s, table, one, PARTS);
}

cudaError_t launch_batch_br(int maxa, int lanes, int threads, const BatchLaunch &l, cudaStream_t s,
                            const InstDesc *table, const InstDesc &one) {
#define BR_CASE(MA, L, TH) \
  if (maxa == MA && lanes == L && threads == TH) return br_one<MA, L, TH>(l, s, table, one);
  CFR_BATCH_ALL(BR_CASE)
#undef BR_CASE
  return cudaErrorInvalidValue;
}
}  // namespace cfr
