// top.cuh — the depths near the root as one launch of one CTA.
//
// A game's first depths are small (a tree of branching 3 has a thousand nodes
// in its first seven), but in the per-level form each costs a forward and a
// backward launch, about 2.7 us apiece whatever its size. This kernel takes
// depths 0 .. K at once: it copies their part of the game and the state into
// shared memory (sets, members, slots, internal ranks and value slots are all
// numbered by depth, so each array's part is a prefix), passes the values of
// depth K + 1 up to the root, updates the slots, and runs the forward pass of
// the next iteration (or half-iteration) down to depth K with the new
// strategy. A call to cfr_iterate starts with the forward part alone. The
// device functions are those of the resident batched solves. It is a chain of
// short steps in one CTA: what bounds it is their latency. An iteration of the
// random tree of depth 14 (depths 0-6 of 13 here): 107.8 -> 84.5 us.
#pragma once
#include "batch.cuh"

namespace cfr {

// FP64 with up to 8 actions: 256 threads (rows of its sums in shared memory).
template <typename T, int MAXA> constexpr int kTopThreads = sizeof(T) == 8 && MAXA > 4 ? 256 : 512;
constexpr int kTopBackward = 1, kTopForward = 2;  // phases of a launch

// in: the prefix counts (n_sets, n_slots, n_int, n_dec, n_chance of depths
// 0 .. K; n_nodes = value slots of the children of these depths), arrays and
// options of the game. v_new: the first value slot of depth K's children, the
// only input that the launch before (the backward launch of depth K + 1)
// writes: everything else is copied before waiting for it.
template <typename T, int MAXA, int LANES>
__global__ void __launch_bounds__(kTopThreads<T, MAXA>, 1) top_kernel(const __grid_constant__ InstDesc in, int K, int v_new,
                                                             int phase, int upd) {
  constexpr int NT = kTopThreads<T, MAXA>;
  extern __shared__ __align__(128) unsigned char s_solve[];
  __shared__ double s_rows[NT / 32][kChainDoubles<T, MAXA, LANES>];
  __shared__ LevelWork s_lw[kBatchLevels];
  const int tid = threadIdx.x;
  const ResidentLayout L = resident_layout(in, sizeof(T));
  const uint32_t I = (uint32_t)in.n_sets, A = (uint32_t)in.n_slots;
  // elements [e0, e1) of a global array into its place, in 16-byte pieces
  // (arena arrays are 256-byte aligned and padded to 256 bytes)
  auto stage = [&](uint32_t off, const void *src, uint32_t b0, uint32_t b1) {
    const uint32_t dst = (uint32_t)__cvta_generic_to_shared(s_solve + off);
    for (uint32_t i = (b0 & ~15u) + tid * 16u; i < b1; i += NT * 16u)
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + i), "l"((const char *)src + i) : "memory");
  };
  for (int i = tid; i < (K + 1) * (int)(sizeof(LevelWork) / 4); i += NT)
    reinterpret_cast<int *>(s_lw)[i] = reinterpret_cast<const int *>(in.lw)[i];
  stage(L.int_edge, in.g.int_edge, 0, 8 * (uint32_t)in.n_int);
  stage(L.sigma, in.sigma, 0, (uint32_t)sizeof(T) * A);
  if (phase & kTopBackward) {
    stage(L.iset_slot, in.g.iset_slot, 0, 4 * (I + 1));
    stage(L.iset_mem, in.g.iset_mem, 0, 4 * (I + 1));
    stage(L.iset_vb, in.g.iset_vb, 0, 4 * I);
    stage(L.iset_rank, in.g.iset_rank, 0, 8 * I);
    stage(L.mem_vs, in.g.mem_vs, 0, 4 * (uint32_t)in.n_dec);
    stage(L.ch_vb, in.g.ch_vb, 0, 4 * (uint32_t)in.n_chance);
    stage(L.ch_nch, in.g.ch_nch, 0, 4 * (uint32_t)in.n_chance);
    stage(L.ch_vs, in.g.ch_vs, 0, 4 * (uint32_t)in.n_chance);
    stage(L.R, in.R, 0, 8 * A);
    stage(L.avg, in.avg, 0, 8 * A);
    stage(L.reach, in.reach, 0, 2 * (uint32_t)sizeof(T) * (uint32_t)in.n_int);
    stage(L.v, in.v, 0, (uint32_t)sizeof(T) * (uint32_t)v_new & ~15u);  // terminals of these depths
  } else {
    stage(L.reach, in.reach, 0, 2 * (uint32_t)sizeof(T));  // the root's
  }
  pdl_enter();
  if (phase & kTopBackward) stage(L.v, in.v, (uint32_t)sizeof(T) * (uint32_t)v_new, (uint32_t)sizeof(T) * (uint32_t)in.n_nodes);
  const double wt = avg_weight(*in.t + 1, in.rule);
  asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 0;" ::: "memory");
  GroupView<T> g;
  g.iset_slot = (const int32_t *)(s_solve + L.iset_slot);
  g.iset_mem = (const int32_t *)(s_solve + L.iset_mem);
  g.iset_vb = (const int32_t *)(s_solve + L.iset_vb);
  g.iset_rank = (const int2 *)(s_solve + L.iset_rank);
  g.mem_vs = (const int32_t *)(s_solve + L.mem_vs);
  g.int_edge = (const int2 *)(s_solve + L.int_edge);
  g.ch_vb = (const int32_t *)(s_solve + L.ch_vb);
  g.ch_nch = (const int32_t *)(s_solve + L.ch_nch);
  g.ch_vs = (const int32_t *)(s_solve + L.ch_vs);
  g.reach = (vec2_t<T> *)(s_solve + L.reach);
  g.v = (T *)(s_solve + L.v);
  g.sigma = (T *)(s_solve + L.sigma);
  g.R = (double *)(s_solve + L.R);
  g.avg = (double *)(s_solve + L.avg);
  g.def_r = (T *)(s_solve + L.def_r);
  g.def_m = (T *)(s_solve + L.def_m);
  __syncthreads();
  if (phase & kTopBackward) {
    // the root's own value has no reader and no place here
    if (tid == 0 && s_lw[0].is1 > s_lw[0].is0) reinterpret_cast<int32_t *>(s_solve + L.mem_vs)[0] = -1;
    __syncthreads();
    double *rows = s_rows[tid / 32];
    for (int d = K; d >= 0; --d) {
      const LevelWork &w = s_lw[d];
      const int is0 = w.is0, is2 = w.is2, is1 = w.is1;
      if (d == 0 && is0 == is1) break;  // a chance root's value has no reader in an iteration
      if (d > 0) {
        for (int32_t i = w.ch0 + tid; i < w.ch1; i += NT) {  // left to right
          const int32_t cb = g.ch_vb[i], n = g.ch_nch[i];
          T s = T(0);
          for (int32_t c = 0; c < n; ++c) s = s + g.v[cb + c];
          g.v[g.ch_vs[i]] = s;
        }
      }
      group_sets<T, MAXA, LANES, kResident>(g, is0, is2, is1, tid, NT, upd, rows);
      __syncthreads();
    }
    if (upd == 3) {
      group_updates<T, MAXA, kResident>(g, 0, (int32_t)I, tid, NT, wt, in.rule);
    } else {
      for (int d = 0; d <= K; ++d)
        group_updates<T, MAXA, kResident>(g, upd & 1 ? s_lw[d].is0 : s_lw[d].is2, upd & 1 ? s_lw[d].is2 : s_lw[d].is1, tid,
                                          NT, wt, in.rule);
    }
    __syncthreads();
    for (uint32_t q = tid; q < A; q += NT) {
      ((T *)in.sigma)[q] = g.sigma[q];
      in.R[q] = g.R[q];
      in.avg[q] = g.avg[q];
    }
    if (tid == 0 && (upd & 2)) *in.t += 1;
  }
  if (phase & kTopForward) {
    for (int d = 1; d <= K; ++d) {
      group_pull<T, kResident>(g, s_lw[d].ib + tid, NT, s_lw[d].ie);
      __syncthreads();
    }
    for (int q = tid; q < in.n_int; q += NT) ((vec2_t<T> *)in.reach)[q] = g.reach[q];
  }
}

}  // namespace cfr
