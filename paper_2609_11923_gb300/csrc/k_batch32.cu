// Batched-iteration kernel instances, FP32 (see batch.cuh).
#include "k_batch.cuh"
namespace cfr {
template cudaError_t launch_batch_iterate<float>(int, int, int, const BatchLaunch &, cudaStream_t, const InstDesc *, const InstDesc &);

cudaError_t batch_cluster_room(int cluster, int *clusters) {
  auto kern = batch_iterate_kernel<float, 8, 8, 512, kCluster>;
  const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)cluster);
  cfg.blockDim = dim3(512);
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)cluster;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaOccupancyMaxActiveClusters(clusters, kern, &cfg);
}
}  // namespace cfr
