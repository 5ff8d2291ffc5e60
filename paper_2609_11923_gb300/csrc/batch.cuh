// batch.cuh — many independent solves in one launch (batched serving).
//
// One CTA, or one thread-block cluster of up to 16, owns one instance for the
// whole call: it runs that instance's n CFR+ iterations with a barrier between
// depth levels (no grid barrier). How many CTAs an instance gets is chosen by
// plan_clusters from the sizes in the batch; instances of one cluster size
// are one launch, and the launches of a call run concurrently (chain_enter).
// The CTAs of a cluster share each depth's work, meet at the hardware cluster
// barrier (barrier.cluster, release/acquire) between depths, and read the
// state arrays through L2 because their L1s are not coherent. Each instance's
// arithmetic depends only on its own arrays and on (THREADS, LANES), not on
// the number of its CTAs: a solve gives bitwise the same result alone and
// inside any mix run with the same shape. Wide chance nodes are summed by one
// CTA in a fixed order.
//
// One CTA for every instance left the largest alone on one SM: a round of 64
// endgames of 1e3 to 2e5 edges (50 iterations, exploitability, strategies)
// 13.2 -> 5.0 ms; of ten of 2e5 to 1e6 edges, 8 CTAs each before, 11.9 -> 9.2.
#pragma once
#include <algorithm>
#include <queue>
#include <utility>
#include <vector>

#include "kernels.cuh"

namespace cfr {

// CTAs for every instance of a batch (host). load: the instance's nodes times
// the share of the longest run's iterations. Starting from `least` CTAs each,
// the instance with the most load per CTA takes the next cluster size while
// SMs are left for it, or its share exceeds an even one of the whole batch;
// kSplitNodes per CTA and less stay whole, because a cluster barrier costs
// more than a CTA's (about 1,600 cycles against 300 with stores in flight)
// and the state is then read through L2. Clusters above 8 CTAs need most of a
// GPC: at most six of them.
constexpr int64_t kSplitNodes = 12000;
inline std::vector<int> plan_clusters(const std::vector<int64_t> &load, int least, int sms) {
  static const int sizes[] = {1, 2, 3, 4, 6, 8, 12, 16};
  const int n = (int)load.size();
  std::vector<int> cta(n, least);
  std::priority_queue<std::pair<int64_t, int>> most;  // (load per CTA, instance)
  int64_t all = 0;
  int used = 0, wide = 0;
  for (int i = 0; i < n; ++i) {
    all += load[i];
    used += least;
    most.push({load[i] / least, -i});
  }
  while (!most.empty()) {
    const int64_t per = most.top().first;
    const int i = -most.top().second;
    most.pop();
    if (per <= kSplitNodes) break;
    int next = 0;
    for (int c : sizes)
      if (c > cta[i]) { next = c; break; }
    if (next == 0 || (next > 8 && cta[i] <= 8 && wide == 6)) continue;
    if (used + next - cta[i] > sms && per <= all / sms) break;
    if (next > 8 && used + next - cta[i] > sms) continue;
    if (next > 8 && cta[i] <= 8) ++wide;
    used += next - cta[i];
    cta[i] = next;
    most.push({load[i] / next, -i});
  }
  return cta;
}

// Everything a CTA needs about one bound instance (device pointers into the
// instance's own arena).
struct InstDesc {
  GameView g;
  void *reach;
  void *v;
  void *sigma;
  double *R;
  double *avg;
  long long *t;
  const LevelWork *lw;
  double2 *reach2;
  double2 *vb;
  double *vavg;
  double *sbs;
  double *out;      // read-out scratch of A doubles (as sbs)
  double *res;      // four results of batch_br_kernel
  long long n_iter; // iterations this call runs for the instance
  int32_t D;
  int32_t rule;
  int32_t n_sets;
  int32_t root_vs;  // the root's value slot (N - 1)
  int32_t order;    // 0 simultaneous, 1 alternating updates
  int32_t pad;
};

template <int THREADS>
__device__ __forceinline__ double cta_sum(double x, double *sm) {
  __syncthreads();
  sm[threadIdx.x] = x;
  __syncthreads();
#pragma unroll
  for (int s = THREADS / 2; s > 0; s >>= 1) {
    if ((int)threadIdx.x < s) sm[threadIdx.x] += sm[threadIdx.x + s];
    __syncthreads();
  }
  const double r = sm[0];
  __syncthreads();
  return r;
}

// Cluster geometry (1 and 0 outside a cluster launch) and the barrier
// between depths: the CTA barrier, or the cluster barrier whose release /
// acquire makes each CTA's global writes visible to the others.
__device__ __forceinline__ unsigned cluster_ncta() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ unsigned cluster_rank() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
template <bool CLUSTERED>
__device__ __forceinline__ void level_sync() {
  if constexpr (CLUSTERED)
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
  else
    __syncthreads();
}

// Wide chance node: its internal children copy its reach (thread ct of NT).
template <typename T, bool PERSIST>
__device__ __forceinline__ void cta_fwd_wide(const GameView &g, vec2_t<T> *reach, int32_t wi, int ct, int NT) {
  const int32_t ir = __ldg(g.wide_irank + wi);
  const int32_t off = __ldg(g.int_cirank + ir);
  const int32_t nch = __ldg(g.big_irank + off);
  const vec2_t<T> r = ldm<PERSIST>(reach + ir);
  for (int32_t j = ct; j < nch; j += NT) {
    const int32_t c = __ldg(g.big_irank + off + 1 + j);
    if (c >= 0) reach[c] = r;
  }
}

// Wide chance node wi inside one CTA: value = sum of the children's values.
// P64 sums left to right (thread 0); P32 uses the fixed-shape CTA tree.
template <typename T, int THREADS, bool PERSIST>
__device__ __forceinline__ void cta_bwd_wide(const GameView &g, T *v, int32_t wi, double *sm) {
  const int32_t h = __ldg(g.wide_vs + wi);
  const int32_t cb = __ldg(g.wide_vb + wi), ce = cb + __ldg(g.wide_nch + wi);
  if constexpr (sizeof(T) == 8) {
    const double s = ordered_sum<THREADS, PERSIST>(v, cb, ce);
    if (threadIdx.x == 0) v[h] = s;
  } else {
    double x = 0.0;
    for (int32_t c = cb + threadIdx.x; c < ce; c += THREADS) x += (double)ldm<PERSIST>(v + c);
    x = cta_sum<THREADS>(x, sm);
    if (threadIdx.x == 0) v[h] = (T)x;
  }
}

constexpr int kBatchLevels = 32;  // depths whose work descriptors a CTA keeps in shared memory

// FP64 kernels hold two registers a value: fewer threads, more registers. The
// FP64 pipe is full with four warps an SM.
template <typename T, int MAXA, int THREADS> constexpr int kBatchThreads = sizeof(T) == 8 && THREADS > 256 ? (MAXA <= 4 ? 512 : 256) : THREADS;

// Every launch of one call's chain may start as soon as the one before it has
// started (programmatic dependent launch: the instances are independent);
// the first CTA of each waits, once its own work is done, for the launch
// before to be complete, so the end of the last launch is the end of all.
__device__ __forceinline__ void chain_enter() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void chain_leave() {
  if (blockIdx.x == 0) asm volatile("griddepcontrol.wait;" ::: "memory");
}

// What bounds it: a small instance is a chain of dependent steps, 2 D - 1 of
// them an iteration, each a barrier and two or three dependent loads; a large
// one is latency of gathers at the occupancy of 64 registers a thread. The
// slot updates (FP64) wait until the values of all depths are known and then
// run one thread per set over the whole game: on the way up they would hold
// every depth back by a dependent chain of FP64 instructions that serve a few
// lanes each.
template <typename T, int MAXA, int LANES, int THREADS, bool CLUSTERED>
__global__ void __launch_bounds__(THREADS) batch_iterate_kernel(const InstDesc *table,
                                                                const __grid_constant__ InstDesc one, int n_inst) {
  __shared__ double sm[THREADS];
  __shared__ double s_rows[THREADS / 32][kChainDoubles<T, MAXA, LANES>];
  __shared__ LevelWork s_lw[kBatchLevels];
  chain_enter();
  const int ncta = CLUSTERED ? (int)cluster_ncta() : 1;   // CTAs sharing this instance
  const int rank = CLUSTERED ? (int)cluster_rank() : 0;
  const int inst = (int)blockIdx.x / ncta;
  if (inst >= n_inst) return;  // the whole cluster leaves together
  const int ct = rank * THREADS + (int)threadIdx.x, NT = ncta * THREADS;
  const InstDesc in = table ? table[inst] : one;
  StateView<T> st;
  st.reach = (vec2_t<T> *)in.reach;
  st.v = (T *)in.v;
  st.sigma = (T *)in.sigma;
  st.R = in.R;
  st.avg = in.avg;
  st.t = in.t;
  T *def_r = (T *)in.sbs, *def_m = (T *)in.out;  // the sets' totals (read-out scratch, idle here)
  const LevelWork *lw = in.lw;
  if (in.D <= kBatchLevels) {
    const int words = in.D * (int)(sizeof(LevelWork) / 4);
    for (int i = threadIdx.x; i < words; i += THREADS)
      reinterpret_cast<int *>(s_lw)[i] = reinterpret_cast<const int *>(in.lw)[i];
    lw = s_lw;
    __syncthreads();
  }
  const long long t0 = *in.t;
  const int lane = threadIdx.x % LANES, gid = ct / LANES;
  const int NG = NT / LANES;
  const unsigned mask = group_mask<LANES>();
  double *rows = s_rows[threadIdx.x / 32];
  const int halves = in.order ? 2 : 1;  // alternating: player 1's half, then player 2's
  for (long long it = 0; it < in.n_iter; ++it) {
    const double wt = avg_weight(t0 + it + 1, in.rule);
    for (int hf = 0; hf < halves; ++hf) {
      const int upd = in.order ? (1 << hf) : 3;
      for (int d = 0; d < in.D; ++d) {
        if (in.g.int_edge) {  // member order: depth d + 1 pulls
          if (d + 1 >= in.D) break;
          const int32_t qe = lw[d + 1].ie;
          for (int32_t q = lw[d + 1].ib + ct; q < qe; q += kPull * NT)
            fwd_pull<T, CLUSTERED>(in.g, st.sigma, st.reach, q, NT, qe);
        } else {
          const LevelWork w = lw[d];
          for (int32_t qw = w.ib + rank * THREADS + (threadIdx.x & ~31); qw < w.ie; qw += 4 * NT) {
            if (w.fan) fwd_int4<T, CLUSTERED, true>(in.g, st.sigma, st.reach, qw + (threadIdx.x & 31), NT, w.ie);
            else fwd_int4<T, CLUSTERED, false>(in.g, st.sigma, st.reach, qw + (threadIdx.x & 31), NT, w.ie);
          }
          for (int32_t i = w.wd0; i < w.wd1; ++i) cta_fwd_wide<T, CLUSTERED>(in.g, st.reach, i, ct, NT);
        }
        level_sync<CLUSTERED>();
      }
      for (int d = in.D - 1; d >= 0; --d) {
        const LevelWork w = lw[d];
        if (d == 0 && w.is0 == w.is1) break;  // a chance root's value has no reader in an iteration
        if (d > 0) {
          for (int32_t i = w.ch0 + ct; i < w.ch1; i += NT)
            bwd_chance<T, CLUSTERED>(in.g, st.v, i);
          if (rank == 0)
            for (int32_t i = w.wd0; i < w.wd1; ++i) cta_bwd_wide<T, THREADS, CLUSTERED>(in.g, st.v, i, sm);
        }
        for (int32_t I = w.is0 + gid; I < w.is1; I += NG)
          bwd_set<T, MAXA, LANES, CLUSTERED, sizeof(T) == 4, true>(in.g, st, I, I >= w.is2, lane, mask, wt, in.rule,
                                                                  upd, rows, def_r, def_m);
        level_sync<CLUSTERED>();
      }
      if (upd == 3) {
        for (int32_t I = ct; I < in.n_sets; I += NT)
          update_set<T, MAXA, CLUSTERED>(in.g, st, I, wt, in.rule, def_r, def_m);
      } else {  // one player's sets
        for (int d = 0; d < in.D; ++d) {
          const int32_t i0 = upd == 1 ? lw[d].is0 : lw[d].is2, i1 = upd == 1 ? lw[d].is2 : lw[d].is1;
          for (int32_t I = i0 + (ct + NT - i0 % NT) % NT; I < i1; I += NT)  // set I: always thread I % NT
            update_set<T, MAXA, CLUSTERED>(in.g, st, I, wt, in.rule, def_r, def_m);
        }
      }
      level_sync<CLUSTERED>();
    }
  }
  if (ct == 0) *in.t = t0 + in.n_iter;
  chain_leave();
}

// Exploitability of every instance's average strategy (FP64): normalise the
// average, forward reach under it, then both best responses by depth (the
// arithmetic of br_level_kernel). CTAs and clusters as batch_iterate_kernel.
template <int MAXA, int LANES, int THREADS, bool CLUSTERED>
__global__ void __launch_bounds__(THREADS) batch_br_kernel(const InstDesc *table, const __grid_constant__ InstDesc one,
                                                           int n_inst) {
  __shared__ double sm[THREADS];
  chain_enter();
  const int ncta = CLUSTERED ? (int)cluster_ncta() : 1;
  const int rank = CLUSTERED ? (int)cluster_rank() : 0;
  const int inst = (int)blockIdx.x / ncta;
  if (inst >= n_inst) return;
  const int ct = rank * THREADS + (int)threadIdx.x, NT = ncta * THREADS;
  const InstDesc in = table ? table[inst] : one;
  const GameView &g = in.g;
  // average strategy, normalised per set
  for (int32_t I = ct; I < in.n_sets; I += NT) {
    const int32_t sb = __ldg(g.iset_slot + I), na = __ldg(g.iset_slot + I + 1) - sb;
    double tot = 0.0;
    for (int32_t a = 0; a < na; ++a) tot += in.avg[sb + a];
    for (int32_t a = 0; a < na; ++a) in.sbs[sb + a] = tot > 0.0 ? in.avg[sb + a] / tot : 1.0 / (double)na;
  }
  level_sync<CLUSTERED>();
  for (int d = 0; d < in.D; ++d) {
    if (g.int_edge) {  // member order: depth d + 1 pulls
      if (d + 1 >= in.D) break;
      const int32_t qe = in.lw[d + 1].ie;
      for (int32_t q = in.lw[d + 1].ib + ct; q < qe; q += kPull * NT)
        fwd_pull<double, CLUSTERED>(g, in.sbs, in.reach2, q, NT, qe);
    } else {
      const LevelWork w = in.lw[d];
      for (int32_t qw = w.ib + rank * THREADS + (threadIdx.x & ~31); qw < w.ie; qw += 4 * NT) {
        if (w.fan) fwd_int4<double, CLUSTERED, true>(g, in.sbs, in.reach2, qw + (threadIdx.x & 31), NT, w.ie);
        else fwd_int4<double, CLUSTERED, false>(g, in.sbs, in.reach2, qw + (threadIdx.x & 31), NT, w.ie);
      }
      for (int32_t i = w.wd0; i < w.wd1; ++i) cta_fwd_wide<double, CLUSTERED>(g, in.reach2, i, ct, NT);
    }
    level_sync<CLUSTERED>();
  }
  const int lane = threadIdx.x % LANES, gid = ct / LANES;
  const int NG = NT / LANES;
  const unsigned mask = group_mask<LANES>();
  for (int d = in.D - 1; d >= 0; --d) {
    const LevelWork w = in.lw[d];
    for (int32_t i = w.ch0 + ct; i < w.ch1; i += NT) br_chance<CLUSTERED>(g, in.vb, in.vavg, i);
    for (int32_t i = w.wd0; i < w.wd1 && rank == 0; ++i) {
      const int32_t h = __ldg(g.wide_vs + i);
      const int32_t cb = __ldg(g.wide_vb + i), ce = cb + __ldg(g.wide_nch + i);
      double sx = 0.0, sy = 0.0, sa = 0.0;
      for (int32_t c = cb + threadIdx.x; c < ce; c += THREADS) {
        const double2 x = ldm<CLUSTERED>(in.vb + c);
        sx += x.x; sy += x.y; sa += ldm<CLUSTERED>(in.vavg + c);
      }
      sx = cta_sum<THREADS>(sx, sm);
      sy = cta_sum<THREADS>(sy, sm);
      sa = cta_sum<THREADS>(sa, sm);
      if (threadIdx.x == 0) { in.vb[h] = make_double2(sx, sy); in.vavg[h] = sa; }
    }
    for (int32_t I = w.is0 + gid; I < w.is1; I += NG)
      br_set<MAXA, LANES, CLUSTERED>(g, in.reach2, in.sbs, in.vb, in.vavg, I, I >= w.is2 ? 1 : 0, lane, mask);
    level_sync<CLUSTERED>();
  }
  if (ct == 0) {
    const double2 root = ldm<CLUSTERED>(in.vb + in.root_vs);
    in.res[0] = 0.5 * (root.x - root.y);
    in.res[1] = root.x;
    in.res[2] = root.y;
    in.res[3] = ldm<CLUSTERED>(in.vavg + in.root_vs);
  }
  chain_leave();
}

}  // namespace cfr
