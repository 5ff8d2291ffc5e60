// launch.h — host wrappers that pick the kernel instance (actions tier x
// lanes per information set). Each wrapper is defined in its own translation
// unit so the instances compile in parallel.
#pragma once
#include <cuda_runtime.h>

#include "kernels.cuh"
#include "bwd_stream.cuh"

namespace cfr {

// Launch of a per-level kernel; with pdl set, as a programmatic dependent
// launch (the kernel waits for its predecessor itself: pdl_enter).
template <typename... KArgs, typename... Args>
inline cudaError_t launch_k(void (*kern)(KArgs...), int grid, int block, size_t smem, cudaStream_t s, bool pdl,
                            Args... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3((unsigned)block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = pdl ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kern, args...);
}

// The streaming FP32 backward of one depth (bwd_stream_kernel); grid = the
// streaming CTAs over the depth's chunks [c0, c1) (set and chance chunks).
// early (with pdl only, and only when the launch before is the backward
// launch of the next depth): copy every input but the children's values
// before waiting for that launch.
cudaError_t launch_bwd_stream(int maxa, int grid, cudaStream_t s, GameView g, StateView<float> st,
                              const SetInfo *info, const StreamChunk *chunks, int c0, int c1, int rule, int upd,
                              int *err, bool pdl, bool early, StreamShape shape);
// Allows the streaming kernel its dynamic shared memory (call before the
// first launch, outside any stream capture; idempotent).
cudaError_t prepare_bwd_stream();

template <typename T>
cudaError_t launch_bwd_level(int maxa, int lanes, int grid, cudaStream_t s, GameView g, StateView<T> st,
                             LevelWork w, int nb_chance, int rule, int upd, int bump, bool pdl = false,
                             int flags = 0);

// query_occupancy != nullptr: only report resident blocks per SM of the
// chosen instance (nothing is launched).
template <typename T>
cudaError_t launch_persistent(int maxa, int lanes, int grid, cudaStream_t s, PersistArgs<T> a,
                              int *query_occupancy);

cudaError_t launch_br_level(int maxa, int lanes, int grid, cudaStream_t s, GameView g, const double2 *reach2,
                            const double *sbs, double2 *vb, double *vavg, LevelWork w, int nb_chance, bool pdl);

}  // namespace cfr

#include "batch.cuh"
#include "top.cuh"

namespace cfr {
// One launch of a batched call: `count` instances from `first` of the table,
// `cluster` CTAs each, their arrays where `mode` says (kSolo, kCluster,
// kResident with `smem` bytes of them). push: the pushing forward (reach
// orders other than member order). chained: the launch before in the stream
// is the same call's and need not be complete (chain_enter).
struct BatchLaunch {
  int first = 0, count = 0, cluster = 1, mode = kSolo;
  uint32_t smem = 0;
  bool push = false, chained = false;
};

// Clusters of `cluster` CTAs of the batched kernel (one CTA an SM) that run at
// the same time.
cudaError_t batch_cluster_room(int cluster, int *clusters);

template <typename T>
cudaError_t launch_batch_iterate(int maxa, int lanes, int threads, const BatchLaunch &l, cudaStream_t s,
                                 const InstDesc *table, const InstDesc &one);
// launch_batch_iterate's launches with l.push.
template <typename T>
cudaError_t launch_batch_push(int maxa, int lanes, int threads, const BatchLaunch &l, cudaStream_t s,
                              const InstDesc *table, const InstDesc &one);
cudaError_t launch_batch_br(int maxa, int lanes, int threads, const BatchLaunch &l, cudaStream_t s,
                            const InstDesc *table, const InstDesc &one);

// The depths near the root as one launch (top_kernel). smem: the bytes of its
// arrays (prepare_top first, outside any capture).
template <typename T> cudaError_t prepare_top(int maxa, int lanes);
template <typename T>
cudaError_t launch_top(int maxa, int lanes, uint32_t smem, cudaStream_t s, const InstDesc &in, int K, int v_new, int phase,
                       int upd, bool pdl);
}  // namespace cfr
