// Near-root kernel instances, FP32 (see top.cuh).
#include "k_top.cuh"
namespace cfr {
template cudaError_t prepare_top<float>(int, int);
template cudaError_t launch_top<float>(int, int, uint32_t, cudaStream_t, const InstDesc &, int, int, int, int, bool);
}
