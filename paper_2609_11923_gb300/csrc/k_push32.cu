// Pushing batched-iteration kernel instances, FP32 (see batch.cuh).
#include "k_push.cuh"
namespace cfr {
template cudaError_t launch_batch_push<float>(int, int, int, const BatchLaunch &, cudaStream_t, const InstDesc *, const InstDesc &);
}
