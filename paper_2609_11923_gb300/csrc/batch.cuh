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
// arithmetic depends only on its own arrays and on the caller's threads and
// lanes, not on the number of its CTAs or on the other instances: a solve gives
// bitwise the same result alone and inside any mix run with the same shape.
// Wide chance nodes are summed by one CTA in a fixed order.
//
// What it gave, step by step, for a round of 64 endgames of 1e3 to 2e5 edges
// (50 iterations, exploitability, strategies) and one of ten of 2e5 to 1e6: one
// CTA each (8 for the ten) 13.2 and 11.9 ms; CTAs by size 5.0 and 9.2; small
// solves in shared memory, loads issued together, slot updates by lanes 2.9 and
// 5.4; code for two and four actions and cluster sizes by what the GPU holds 2.7
// and 4.0. An iteration of 10,400 nodes in one CTA 28 -> 10.7 us.
#pragma once
#include <algorithm>
#include <queue>
#include <utility>
#include <vector>

#include "kernels.cuh"

namespace cfr {

// How many CTAs, and clusters of 4, 8 and 16 CTAs, run at the same time at one
// CTA an SM (a cluster lies in one GPC, and how many SMs each has differs from
// one GPU to the next).
struct ClusterRoom {
  int sms = 0, four = 0, eight = 0, sixteen = 0;
};

// CTAs for every instance of a batch (host): 1, 2, 4, 8 or 16, at least
// `least`, by an estimate of an iteration's time (batch_ns). The instance that
// takes longest gets twice its CTAs, or more, as long as all of them run at the
// same time (a cluster too many waits for a whole instance: ten large endgames with
// six of 16 took 89 us an iteration, with four 64); a batch that does not run
// at the same time anyway, while it takes longer than an even share of it.
struct BatchLoad {
  int64_t nodes, sets, depths;
  int64_t chain;  // members of each depth's largest set, summed
  bool resident;  // by one CTA, from shared memory
  bool fp64;
  bool best;      // a best response (in FP64): a depth's barriers find it less ready
  double share;   // of the longest run's iterations
};

// An iteration by c CTAs in ns: what every depth costs (barriers and chains of
// loads, both ways), what the CTAs share, and the largest sets, each walked by
// one group. Least squares over 38 games alone, 1,024 threads and 8 lanes, 1 to
// 16 CTAs: endgames of 10,000 to 920,000 nodes (5 depths), random trees of 122
// to 275,000 (4 to 11), two-round card games of 2,800 to 350,000 (8), chains of
// 10 to 100 depths, sets of 300 and 3,000 members; within 20% in FP32 (7 to 10%
// on average), 36% in FP64 (13%). By nodes alone, fitted to endgames, a game of
// 300 chains of 100 depths side by side got 16 CTAs: 881 us an iteration, by
// one 696. (Best responses of 16 random trees of 3,385 nodes: by one CTA each 84
// us, by 8 or 16 100.)
inline double batch_ns(const BatchLoad &l, int c) {
  const double D = (double)l.depths, I = (double)l.sets / c, N = (double)l.nodes / c, L = (double)l.chain;
  if (l.fp64) return c > 1 ? 2500.0 + (l.best ? 6000.0 : 3300.0) * D + 68.0 * I + 3.4 * N + 200.0 * L : 1340.0 * D + 61.0 * I + 3.3 * N + 137.0 * L;
  if (c > 1) return 1800.0 + 2570.0 * D + 19.0 * I + 0.53 * N + 9.0 * L;
  return l.resident ? 1700.0 + 580.0 * D + 10.5 * I + 0.13 * N + 6.6 * L : 580.0 * D + 19.0 * I + 0.39 * N + 8.3 * L;
}

inline std::vector<int> plan_clusters(const std::vector<BatchLoad> &load, int least, const ClusterRoom &room) {
  const int n = (int)load.size();
  auto time = [&](int i, int c) { return batch_ns(load[i], c) * load[i].share; };
  auto exists = [&](int c) { return c == 16 ? room.sixteen > 0 : c == 8 ? room.eight > 0 : c == 4 ? room.four > 0 : true; };
  std::vector<int> cta(n, least);
  int count[17] = {0};  // instances by CTAs
  double work = 0.0;    // CTA ns
  std::priority_queue<std::pair<double, int>> longest;  // (ns, instance)
  for (int i = 0; i < n; ++i) {
    ++count[least];
    work += least * time(i, least);
    longest.push({time(i, least), -i});
  }
  auto fits = [&]() {
    const int eights = 2 * count[16] + count[8];
    return count[16] <= room.sixteen && eights <= room.eight && 2 * eights + count[4] <= room.four &&
           8 * eights + 4 * count[4] + 2 * count[2] + count[1] <= room.sms;
  };
  const bool waves = !fits();
  while (!longest.empty()) {
    const double t = longest.top().first;
    const int i = -longest.top().second, c = cta[i];
    longest.pop();
    int more = 2 * c;  // the next size that is faster: a cluster of two may lose more to its barriers than it shares
    while (more <= 16 && exists(more) && time(i, more) >= t) more *= 2;
    if (more > 16 || !exists(more)) continue;
    --count[c];
    ++count[more];
    if (!fits() && !(waves && t > work / room.sms)) {
      ++count[c];
      --count[more];
      continue;
    }
    work += more * time(i, more) - c * t;
    cta[i] = more;
    longest.push({time(i, more), -i});
  }
  // where the longest in the end found no room to grow, others that would take
  // no longer as they were have grown for nothing (of 40 random trees alike 11
  // got clusters: 779 us for 20 iterations instead of 679)
  int last = 0;
  for (int i = 1; i < n; ++i)
    if (time(i, cta[i]) > time(last, cta[last])) last = i;
  if (n > 0 && cta[last] == least)
    for (int i = 0; i < n; ++i)
      if (time(i, least) <= 1.02 * time(last, least)) cta[i] = least;
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
  int32_t n_nodes, n_int, n_dec, n_slots, n_chance;  // value slots, internal nodes, members, slots, narrow chance nodes
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

// Where a solve's arrays are while a batched kernel runs.
//   kSolo      one CTA, in global memory: its L1 holds what fits
//   kCluster   several CTAs: state is read through L2, L1s are not coherent
//   kResident  one CTA, copied into shared memory for the whole call
constexpr int kSolo = 0, kCluster = 1, kResident = 2;

// Threads of a CTA. The caller's 1,024 become 512 with twice the registers
// (64 spilled; results do not depend on it); FP64 holds two registers a value,
// and its pipe is full with four warps an SM.
template <typename T, int MAXA, int THREADS>
constexpr int kBatchThreads = THREADS <= 256 || (sizeof(T) == 8 && MAXA > 4) ? 256 : 512;

template <int MODE, typename X>
__device__ __forceinline__ X ldk(const X *p) {  // the compiled game: never written
  if constexpr (MODE == kResident) return *p;
  else return __ldg(p);
}

// Byte offsets of a resident solve's arrays in shared memory (16-byte
// aligned; the state that goes back to global memory is sigma, R and avg:
// reach and the inner values are recomputed by every iteration).
struct ResidentLayout {
  uint32_t iset_slot, iset_mem, iset_vb, iset_rank, mem_vs, int_edge, ch_vb, ch_nch, ch_vs;
  uint32_t reach, v, sigma, R, avg, def_r, def_m, total;
};

__host__ __device__ inline ResidentLayout resident_layout(const InstDesc &in, uint32_t T) {
  ResidentLayout L;
  uint32_t at = 0;
  auto take = [&](uint32_t n, uint32_t size) {
    const uint32_t o = at;
    at += (n * size + 15u) & ~15u;
    return o;
  };
  const uint32_t I = (uint32_t)in.n_sets, A = (uint32_t)in.n_slots;
  L.iset_slot = take(I + 1, 4);
  L.iset_mem = take(I + 1, 4);
  L.iset_vb = take(I, 4);
  L.iset_rank = take(I, 8);
  L.mem_vs = take((uint32_t)in.n_dec, 4);
  L.int_edge = take((uint32_t)in.n_int, 8);
  L.ch_vb = take((uint32_t)in.n_chance, 4);
  L.ch_nch = take((uint32_t)in.n_chance, 4);
  L.ch_vs = take((uint32_t)in.n_chance, 4);
  L.reach = take((uint32_t)in.n_int, 2 * T);
  L.v = take((uint32_t)in.n_nodes, T);
  L.sigma = take(A, T);
  L.R = take(A, 8);
  L.avg = take(A, 8);
  L.def_r = take(A, T);
  L.def_m = take(A, T);
  L.total = at;
  return L;
}

// Only games of at most this many nodes may be resident: the byte count
// decides, and the 32-bit sums of resident_layout cannot wrap below it (no
// array has more than a few elements more than the game has nodes).
constexpr int32_t kResidentNodes = 1 << 16;
constexpr uint32_t kResidentBytes = 190 * 1024;

// Bytes of shared memory that the arrays take, 0 if they do not fit (host).
inline uint32_t resident_size(const InstDesc &in, uint32_t T) {
  if (in.n_nodes > kResidentNodes) return 0;
  const uint32_t n = resident_layout(in, T).total;
  return n <= kResidentBytes ? std::max(n, 16u) : 0;
}

// The arrays that a batched iteration works on (member order).
template <typename T> struct GroupView {
  const int32_t *iset_slot, *iset_mem, *iset_vb, *mem_vs, *ch_vb, *ch_nch, *ch_vs;
  const int2 *iset_rank, *int_edge;
  vec2_t<T> *reach;
  T *v, *sigma, *def_r, *def_m;
  double *R, *avg;
};

// Internal nodes q, q + stride, ... of one depth pull their reach from their
// parents' (as fwd_pull): kPullFar in flight while that many are left, then
// two.
constexpr int kPullFar = 4;
template <typename T, int MODE>
__device__ __forceinline__ void group_pull(const GroupView<T> &g, int32_t q, int32_t stride, int32_t qe) {
  constexpr bool C = MODE == kCluster;
  if constexpr (MODE != kResident) {
    for (; q + (kPullFar - 1) * stride < qe; q += kPullFar * stride) {
      int2 e[kPullFar];
      vec2_t<T> r[kPullFar];
      T s[kPullFar];
#pragma unroll
      for (int u = 0; u < kPullFar; ++u) e[u] = ldk<MODE>(g.int_edge + q + u * stride);
#pragma unroll
      for (int u = 0; u < kPullFar; ++u) {
        r[u] = ldm<C>(g.reach + e[u].x);
        s[u] = e[u].y >= 0 ? ldm<C>(g.sigma + (e[u].y & kMask)) : T(1);
      }
#pragma unroll
      for (int u = 0; u < kPullFar; ++u) {
        if (e[u].y >= 0) {
          if (e[u].y & kP2Bit) r[u].y = r[u].y * s[u];
          else r[u].x = r[u].x * s[u];
        }
        g.reach[q + u * stride] = r[u];
      }
    }
  }
  for (; q < qe; q += 2 * stride) {
    const bool two = q + stride < qe;
    const int2 e0 = ldk<MODE>(g.int_edge + q), e1 = two ? ldk<MODE>(g.int_edge + q + stride) : e0;
    vec2_t<T> r0 = ldm<C>(g.reach + e0.x), r1 = two ? ldm<C>(g.reach + e1.x) : r0;
    const T s0 = e0.y >= 0 ? ldm<C>(g.sigma + (e0.y & kMask)) : T(1);
    const T s1 = two && e1.y >= 0 ? ldm<C>(g.sigma + (e1.y & kMask)) : T(1);
    if (e0.y >= 0) {
      if (e0.y & kP2Bit) r0.y = r0.y * s0;
      else r0.x = r0.x * s0;
    }
    if (e1.y >= 0) {
      if (e1.y & kP2Bit) r1.y = r1.y * s1;
      else r1.x = r1.x * s1;
    }
    g.reach[q] = r0;
    if (two) g.reach[q + stride] = r1;
  }
}

// The regret terms are rounded before they are added (no fused multiply-add),
// in every form of the sum below.
__device__ __forceinline__ float times(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float plus(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ double times(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ double plus(double a, double b) { return __dadd_rn(a, b); }

// FP32: sets averaging this many members at a depth take a warp each: eight
// lanes walk them in many dependent steps, and there are few of them. The
// sums are those of eight lanes, bit for bit (group_set_long).
constexpr int kLongSet = 32;

// One set by the LANES lanes of a group: its members' values, and the set's
// totals into def_r and def_m (see bwd_set, whose sums these are). Every load
// of a step is issued before the first value is used. The groups of a warp run
// in step (see warp_chains): shorter sets, and groups without a set (no
// members, no actions), idle along, adding zeros. (50 iterations of one-card poker 174 -> 156 us;
// ten in FP64 of an 80k-node random tree, whose near-root depths these are, by
// halves 1,970 -> 1,911.)
struct GroupSet {  // a set's record
  int32_t sb, na, m0, M, vb;
  int2 rk;
};
template <typename T, int MODE> __device__ __forceinline__ GroupSet group_record(const GroupView<T> &g, int32_t I) {
  GroupSet s;
  s.sb = ldk<MODE>(g.iset_slot + I);
  s.na = ldk<MODE>(g.iset_slot + I + 1) - s.sb;
  s.m0 = ldk<MODE>(g.iset_mem + I);
  s.M = ldk<MODE>(g.iset_mem + I + 1) - s.m0;
  s.vb = ldk<MODE>(g.iset_vb + I);
  s.rk = ldk<MODE>(g.iset_rank + I);
  return s;
}

template <typename T, int MAXA, int LANES, int MODE>
__device__ __forceinline__ void group_members(const GroupView<T> &g, const GroupSet &s, bool p2, int lane,
                                              int32_t longest, int upd, double *rows) {
  constexpr bool C = MODE == kCluster, CHAINS = sizeof(T) == 8;
  constexpr int U = LANES <= 8 ? 2 : 1;  // members of a lane in flight
  const int32_t sb = s.sb, na = s.na, m0 = s.m0, M = s.M, vb = s.vb;
  const int2 rk = s.rk;
  T sig[MAXA], racc[MAXA], spw = T(0);
  double acc[kChainAcc<MAXA, LANES>];
#pragma unroll
  for (int a = 0; a < MAXA; ++a) {
    sig[a] = a < na ? ldm<C>(g.sigma + sb + a) : T(0);
    racc[a] = T(0);
  }
#pragma unroll
  for (int i = 0; i < kChainAcc<MAXA, LANES>; ++i) acc[i] = 0.0;
  for (int32_t k0 = 0; k0 < longest; k0 += U * LANES) {
    int32_t h[U];
    vec2_t<T> r[U];
    T vc[U][MAXA];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int32_t k = k0 + u * LANES + lane;
      const bool in = k < M;
      h[u] = in ? ldk<MODE>(g.mem_vs + m0 + k) : -1;
      r[u].x = r[u].y = T(0);
      if (in) r[u] = ldm<C>(g.reach + rk.x + k * rk.y);
      const T *v = g.v + vb + k;
#pragma unroll
      for (int a = 0; a < MAXA; ++a) vc[u][a] = in && a < na ? ldm<C>(v + a * M) : T(0);
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (k0 + u * LANES >= longest) break;
      T vh = T(0);
#pragma unroll
      for (int a = 0; a < MAXA; ++a)
        if (a < na) vh = vh + sig[a] * vc[u][a];
      if (h[u] >= 0) g.v[h[u]] = vh;
      const T po = p2 ? r[u].x : r[u].y;  // opponent's reach (chance is inside v)
      const T pw = p2 ? r[u].y : r[u].x;  // own reach
      const T f = (p2 ? T(-1) : T(1)) * po;
      if constexpr (CHAINS) {
        T d[MAXA], mm[MAXA];
#pragma unroll
        for (int a = 0; a < MAXA; ++a) {
          d[a] = T(0);
          mm[a] = T(0);
          if (a < na) {
            d[a] = f * (vc[u][a] - vh);
            mm[a] = pw * sig[a];
          }
        }
        const int32_t left = longest - k0 - u * LANES;
        accumulate_chains<MAXA, LANES>(rows, left < LANES ? left : LANES, MAXA, 0xffffffffu, d, mm, acc);
      } else {
#pragma unroll
        for (int a = 0; a < MAXA; ++a)
          if (a < na) racc[a] = plus(racc[a], times(f, vc[u][a] - vh));  // 0 for lanes without a member
        spw += pw;
      }
    }
  }
  const bool live = upd & (p2 ? 2 : 1);  // alternating updates: the other player's sets only pass their values up
  if constexpr (CHAINS) {
#pragma unroll
    for (int i = 0; i < kChainAcc<MAXA, LANES>; ++i) {
      const int c = lane + i * LANES;
      if (live && c < na) g.def_r[sb + c] = acc[i];
      else if (live && c >= MAXA && c - MAXA < na) g.def_m[sb + c - MAXA] = acc[i];
    }
  } else {
    __syncwarp();
    spw = group_sum_butterfly<LANES>(spw, 0xffffffffu);
    group_sum_scatter<LANES, MAXA>(racc, lane, 0xffffffffu);
    if (live && na > 0 && lane == 0) g.def_m[sb] = spw;
    constexpr int STEP = MAXA <= LANES ? LANES / MAXA : 1, PER = MAXA <= LANES ? 1 : MAXA / LANES;
    if (live && lane % STEP == 0) {
#pragma unroll
      for (int i = 0; i < PER; ++i)
        if (lane / STEP * PER + i < na) g.def_r[sb + lane / STEP * PER + i] = racc[i];
    }
  }
}

// The work of a set, in games of more than four actions in code for two, four
// or MAXA: what bounds a small game is the instructions of its groups, and most
// sets of an endgame have two actions where its largest has seven (64 endgames
// of 1e3 to 2e5 edges 2,916 -> 2,591 us, ten of 2e5 to 1e6 5,774 -> 4,954; one-
// card poker and random trees, whose warps mix two to four actions, 3-6%
// slower that way).
template <typename T, int MAXA, int LANES, int MODE>
__device__ __forceinline__ void group_set(const GroupView<T> &g, int32_t I, bool in, bool p2, int lane, int upd,
                                          double *rows) {
  GroupSet s = {};
  if (in) s = group_record<T, MODE>(g, I);
  const int32_t longest = __reduce_max_sync(0xffffffffu, s.M);
  if constexpr (MAXA > 4) {
    const int most = __reduce_max_sync(0xffffffffu, s.na);
    if (most <= 2) return group_members<T, 2, LANES, MODE>(g, s, p2, lane, longest, upd, rows);
    if (most <= 4) return group_members<T, 4, LANES, MODE>(g, s, p2, lane, longest, upd, rows);
  }
  group_members<T, MAXA, LANES, MODE>(g, s, p2, lane, longest, upd, rows);
}

// The sets I0 .. I1 (from I2 on player 2's) of one depth by `all` threads,
// thread ct of them.
template <typename T, int MAXA, int LANES, int MODE>
__device__ __forceinline__ void group_sets(const GroupView<T> &g, int32_t I0, int32_t I2, int32_t I1, int ct, int all,
                                           int upd, double *rows) {
  const int sub = ct % 32 / LANES, lane = ct % LANES;
  for (int32_t W = I0 + ct / 32 * (32 / LANES); W < I1; W += all / LANES) {  // the warp's first set
    const int32_t I = W + sub;
    group_set<T, MAXA, LANES, MODE>(g, I, I < I1, I >= I2, lane, upd, rows);
  }
}

// One long set by a warp with the sums of group_set<.., 8, ..>: lane l of
// eight adds members l, l + 8, l + 16, ... in turn. The warp's lanes compute 32
// members' terms at once, then every lane adds the four of its column (its
// lane modulo 8) in that order. FP32.
template <int MAXA, int MODE>
__device__ __forceinline__ void group_members_long(const GroupView<float> &g, const GroupSet &s, bool p2, int upd) {
  constexpr bool C = MODE == kCluster;
  constexpr int U = 2;  // members of a lane in flight
  const int lane = threadIdx.x & 31, col = lane & 7;
  const int32_t sb = s.sb, na = s.na, m0 = s.m0, M = s.M, vb = s.vb;
  const int2 rk = s.rk;
  float sig[MAXA], racc[MAXA], spw = 0.f;
#pragma unroll
  for (int a = 0; a < MAXA; ++a) {
    sig[a] = a < na ? ldm<C>(g.sigma + sb + a) : 0.f;
    racc[a] = 0.f;
  }
  for (int32_t k0 = 0; k0 < M; k0 += U * 32) {
    int32_t h[U];
    float2 r[U];
    float vc[U][MAXA];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int32_t k = k0 + u * 32 + lane;
      const bool in = k < M;
      h[u] = in ? ldk<MODE>(g.mem_vs + m0 + k) : -1;
      r[u] = make_float2(0.f, 0.f);
      if (in) r[u] = ldm<C>(g.reach + rk.x + k * rk.y);
      const float *v = g.v + vb + k;
#pragma unroll
      for (int a = 0; a < MAXA; ++a) vc[u][a] = in && a < na ? ldm<C>(v + a * M) : 0.f;
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (k0 + u * 32 >= M) break;
      float vh = 0.f;
#pragma unroll
      for (int a = 0; a < MAXA; ++a)
        if (a < na) vh = vh + sig[a] * vc[u][a];
      if (h[u] >= 0) g.v[h[u]] = vh;
      const float po = p2 ? r[u].x : r[u].y, pw = p2 ? r[u].y : r[u].x;
      const float f = (p2 ? -1.f : 1.f) * po;
#pragma unroll
      for (int a = 0; a < MAXA; ++a) {
        if (a < na) {  // the same for the whole warp
          const float d = times(f, vc[u][a] - vh);
#pragma unroll
          for (int c = 0; c < 4; ++c) racc[a] = plus(racc[a], __shfl_sync(0xffffffffu, d, c * 8 + col));
        }
      }
#pragma unroll
      for (int c = 0; c < 4; ++c) spw = plus(spw, __shfl_sync(0xffffffffu, pw, c * 8 + col));
    }
  }
  if (!(upd & (p2 ? 2 : 1))) return;
  spw = group_sum_butterfly<8>(spw, 0xffffffffu);
  group_sum_scatter<8, MAXA>(racc, col, 0xffffffffu);
  if (lane == 0) g.def_m[sb] = spw;
  constexpr int STEP = 8 / MAXA;
  if (lane < 8 && lane % STEP == 0 && lane / STEP < na) g.def_r[sb + lane / STEP] = racc[0];
}

template <int MAXA, int MODE>
__device__ __forceinline__ void group_set_long(const GroupView<float> &g, int32_t I, bool p2, int upd) {
  const GroupSet s = group_record<float, MODE>(g, I);
  if constexpr (MAXA > 4) {
    if (s.na <= 2) return group_members_long<2, MODE>(g, s, p2, upd);
    if (s.na <= 4) return group_members_long<4, MODE>(g, s, p2, upd);
  }
  group_members_long<MAXA, MODE>(g, s, p2, upd);
}

// The slot updates from the sets' totals, four lanes a set, a slot each (and
// slots 4 to 7 in a second step where a set has them): FP64 instructions then
// serve most lanes of a warp, and the chain of a set is one slot's.
constexpr int kUpdateLanes = 4;
template <typename T> struct SlotTotals {
  double R, S;
  T r, m;
};

template <typename T, int MODE>
__device__ __forceinline__ SlotTotals<T> slot_totals(const GroupView<T> &g, int32_t sb, int32_t q) {
  constexpr bool C = MODE == kCluster;
  SlotTotals<T> t;
  t.R = g.R[q];
  t.S = g.avg[q];
  t.r = ldm<C>(g.def_r + q);
  if constexpr (sizeof(T) == 4) t.m = g.sigma[q] * ldm<C>(g.def_m + sb);  // this thread wrote sigma the iteration before
  else t.m = ldm<C>(g.def_m + q);
  return t;
}

template <typename T>
__device__ __forceinline__ T slot_write(const GroupView<T> &g, int32_t q, const SlotTotals<T> &t, double wt, int rule) {
  double Rn, Sn;
  const double x = slot_terms(t.R, t.S, as_double(t.r), as_double(t.m), wt, rule, Rn, Sn);
  g.R[q] = Rn;
  g.avg[q] = Sn;
  if constexpr (sizeof(T) == 8) return x;
  else return narrow_pos(x);
}

template <typename T, int MAXA, int MODE>
__device__ __forceinline__ void group_update(const GroupView<T> &g, int32_t I, bool in, int a, double wt, int rule) {
  constexpr int L = kUpdateLanes;
  constexpr unsigned full = 0xffffffffu;  // the groups of a warp run in step
  int32_t sb = 0, na = 0;
  if (in) {
    sb = ldk<MODE>(g.iset_slot + I);
    na = ldk<MODE>(g.iset_slot + I + 1) - sb;
  }
  const int32_t q = sb + a;
  T pos = T(0), more = T(0);
  if (a < na) pos = slot_write(g, q, slot_totals<T, MODE>(g, sb, q), wt, rule);
  T tot = T(0);  // positive parts in action order
#pragma unroll
  for (int b = 0; b < L; ++b) {
    const T x = __shfl_sync(full, pos, b, L);
    if (b < na) tot += x;
  }
  if (MAXA > L && __any_sync(full, na > L)) {
    if (a + L < na) more = slot_write(g, q + L, slot_totals<T, MODE>(g, sb, q + L), wt, rule);
#pragma unroll
    for (int b = 0; b < L; ++b) {
      const T x = __shfl_sync(full, more, b, L);
      if (b + L < na) tot += x;
    }
    if (a + L < na) g.sigma[q + L] = match(more, tot, na);
  }
  if (a < na) g.sigma[q] = match(pos, tot, na);
}

// The slots of sets I0 .. I1 by `all` threads, thread ct of them: set I always
// by the same threads, whatever I0 (their L1 holds its R and avg).
template <typename T, int MAXA, int MODE>
__device__ __forceinline__ void group_updates(const GroupView<T> &g, int32_t I0, int32_t I1, int ct, int all,
                                              double wt, int rule) {
  constexpr int L = kUpdateLanes;
  const int sub = ct % 32 / L, groups = all / L;
  for (int32_t W = I0 - I0 % groups + ct / 32 * (32 / L); W < I1; W += groups) {  // the warp's first set
    const int32_t I = W + sub;
    group_update<T, MAXA, MODE>(g, I, I >= I0 && I < I1, ct % L, wt, rule);
  }
}

// Every launch of one call's chain may start as soon as the one before it has
// started (programmatic dependent launch: the instances are independent);
// the first CTA of each waits, once its own work is done, for the launch
// before to be complete, so the end of the last launch is the end of all.
__device__ __forceinline__ void chain_enter() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void chain_leave() {
  if (blockIdx.x == 0) asm volatile("griddepcontrol.wait;" ::: "memory");
}

// What bounds it: a small instance is a chain of dependent steps, 2 D - 1 of
// them an iteration, each a barrier and two or three dependent loads, so the
// smallest games run from shared memory; a large one is the latency of its
// gathers. The slot updates (FP64) wait until the values of all depths are
// known and then run over the whole game at once: on the way up they would
// hold every depth back by a dependent chain of FP64 instructions that serve
// a few lanes each.
template <typename T, int MAXA, int LANES, int NT, int MODE>
__global__ void __launch_bounds__(NT, MODE == kSolo && NT <= 256 && MAXA <= 4 ? 2 : 1) batch_iterate_kernel(const InstDesc *table, const __grid_constant__ InstDesc one,
                                                           int n_inst) {
  constexpr bool CLUSTERED = MODE == kCluster;
  extern __shared__ __align__(128) unsigned char s_solve[];
  __shared__ double sm[MODE == kResident ? 1 : NT];
  __shared__ double s_rows[NT / 32][kChainDoubles<T, MAXA, LANES>];
  __shared__ LevelWork s_lw[kBatchLevels];
  __shared__ InstDesc s_in;
  __shared__ unsigned char s_long[64];  // depths (modulo 64) whose sets average kLongSet members or more
  chain_enter();
  const int ncta = CLUSTERED ? (int)cluster_ncta() : 1;   // CTAs sharing this instance
  const int rank = CLUSTERED ? (int)cluster_rank() : 0;
  const int inst = (int)blockIdx.x / ncta;
  if (inst >= n_inst) return;  // the whole cluster leaves together
  const int tid = threadIdx.x, ct = rank * NT + tid, all = ncta * NT;
  {
    const int *src = reinterpret_cast<const int *>(table ? table + inst : &one);
    for (int i = tid; i < (int)(sizeof(InstDesc) / 4); i += NT) reinterpret_cast<int *>(&s_in)[i] = src[i];
  }
  __syncthreads();
  const InstDesc &in = s_in;
  const int D = in.D, rule = in.rule;
  const LevelWork *lw = in.lw;
  if (D <= kBatchLevels) {
    const int words = D * (int)(sizeof(LevelWork) / 4);
    for (int i = tid; i < words; i += NT)
      reinterpret_cast<int *>(s_lw)[i] = reinterpret_cast<const int *>(in.lw)[i];
    lw = s_lw;
  }
  GroupView<T> g;
  if constexpr (MODE == kResident) {
    const ResidentLayout L = resident_layout(in, sizeof(T));
    auto stage = [&](uint32_t off, const void *src, uint32_t bytes) {  // arena arrays are padded to 256 bytes
      const uint32_t dst = (uint32_t)__cvta_generic_to_shared(s_solve + off);
      for (uint32_t i = tid * 16u; i < bytes; i += NT * 16u)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + i), "l"((const char *)src + i) : "memory");
      return s_solve + off;
    };
    const uint32_t I = (uint32_t)in.n_sets, A = (uint32_t)in.n_slots;
    g.iset_slot = (const int32_t *)stage(L.iset_slot, in.g.iset_slot, 4 * (I + 1));
    g.iset_mem = (const int32_t *)stage(L.iset_mem, in.g.iset_mem, 4 * (I + 1));
    g.iset_vb = (const int32_t *)stage(L.iset_vb, in.g.iset_vb, 4 * I);
    g.iset_rank = (const int2 *)stage(L.iset_rank, in.g.iset_rank, 8 * I);
    g.mem_vs = (const int32_t *)stage(L.mem_vs, in.g.mem_vs, 4 * (uint32_t)in.n_dec);
    g.int_edge = (const int2 *)stage(L.int_edge, in.g.int_edge, 8 * (uint32_t)in.n_int);
    g.ch_vb = (const int32_t *)stage(L.ch_vb, in.g.ch_vb, 4 * (uint32_t)in.n_chance);
    g.ch_nch = (const int32_t *)stage(L.ch_nch, in.g.ch_nch, 4 * (uint32_t)in.n_chance);
    g.ch_vs = (const int32_t *)stage(L.ch_vs, in.g.ch_vs, 4 * (uint32_t)in.n_chance);
    g.reach = (vec2_t<T> *)stage(L.reach, in.reach, 2 * (uint32_t)sizeof(T));  // the root's
    g.v = (T *)stage(L.v, in.v, (uint32_t)sizeof(T) * (uint32_t)in.n_nodes);
    g.sigma = (T *)stage(L.sigma, in.sigma, (uint32_t)sizeof(T) * A);
    g.R = (double *)stage(L.R, in.R, 8 * A);
    g.avg = (double *)stage(L.avg, in.avg, 8 * A);
    g.def_r = (T *)(s_solve + L.def_r);
    g.def_m = (T *)(s_solve + L.def_m);
    asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 0;" ::: "memory");
  } else {
    g.iset_slot = in.g.iset_slot;
    g.iset_mem = in.g.iset_mem;
    g.iset_vb = in.g.iset_vb;
    g.iset_rank = in.g.iset_rank;
    g.mem_vs = in.g.mem_vs;
    g.int_edge = in.g.int_edge;
    g.ch_vb = in.g.ch_vb;
    g.ch_nch = in.g.ch_nch;
    g.ch_vs = in.g.ch_vs;
    g.reach = (vec2_t<T> *)in.reach;
    g.v = (T *)in.v;
    g.sigma = (T *)in.sigma;
    g.R = in.R;
    g.avg = in.avg;
    g.def_r = (T *)in.sbs;  // the sets' totals (read-out scratch, idle here)
    g.def_m = (T *)in.out;
  }
  const long long t0 = *in.t, n_iter = in.n_iter;
  const int n_sets = in.n_sets;
  if (tid < 64) s_long[tid] = 0;
  __syncthreads();
  if (D <= 64 && tid < D) {
    const int n = lw[tid].is1 - lw[tid].is0;
    if (n > 0) s_long[tid] = in.g.iset_mem[lw[tid].is1] - in.g.iset_mem[lw[tid].is0] >= kLongSet * n;
  }
  __syncthreads();
  double *rows = s_rows[tid / 32];
  const int halves = in.order ? 2 : 1;  // alternating: player 1's half, then player 2's
  for (long long it = 0; it < n_iter; ++it) {
    const double wt = avg_weight(t0 + it + 1, rule);
    for (int hf = 0; hf < halves; ++hf) {
      const int upd = halves == 2 ? (1 << hf) : 3;
      for (int d = 1; d < D; ++d) {
        group_pull<T, MODE>(g, lw[d].ib + ct, all, lw[d].ie);
        level_sync<CLUSTERED>();
      }
      for (int d = D - 1; d >= 0; --d) {
        const LevelWork &w = lw[d];
        const int is0 = w.is0, is2 = w.is2, is1 = w.is1;
        if (d == 0 && is0 == is1) break;  // a chance root's value has no reader in an iteration
        if (d > 0) {
          for (int32_t i = w.ch0 + ct; i < w.ch1; i += all) {  // narrow chance nodes: left to right
            const int32_t cb = ldk<MODE>(g.ch_vb + i), n = ldk<MODE>(g.ch_nch + i);
            T s = T(0);
            for (int32_t c = 0; c < n; ++c) s = s + ldm<CLUSTERED>(g.v + cb + c);
            g.v[ldk<MODE>(g.ch_vs + i)] = s;
          }
          if constexpr (MODE != kResident) {
            if (rank == 0)
              for (int32_t i = w.wd0; i < w.wd1; ++i) cta_bwd_wide<T, NT, CLUSTERED>(in.g, g.v, i, sm);
          }
        }
        bool by_warp = false;
        if constexpr (sizeof(T) == 4 && LANES == 8) {
          by_warp = s_long[d & 63] != 0;
          if (by_warp)
            for (int32_t I = is0 + ct / 32; I < is1; I += all / 32) group_set_long<MAXA, MODE>(g, I, I >= is2, upd);
        }
        if (!by_warp) group_sets<T, MAXA, LANES, MODE>(g, is0, is2, is1, ct, all, upd, rows);
        level_sync<CLUSTERED>();
      }
      if (upd == 3) {
        group_updates<T, MAXA, MODE>(g, 0, n_sets, ct, all, wt, rule);
      } else {  // one player's sets
        for (int d = 0; d < D; ++d)
          group_updates<T, MAXA, MODE>(g, upd == 1 ? lw[d].is0 : lw[d].is2, upd == 1 ? lw[d].is2 : lw[d].is1, ct, all,
                                       wt, rule);
      }
      level_sync<CLUSTERED>();
    }
  }
  if constexpr (MODE == kResident) {
    for (int q = tid; q < in.n_slots; q += NT) {
      ((T *)in.sigma)[q] = g.sigma[q];
      in.R[q] = g.R[q];
      in.avg[q] = g.avg[q];
    }
  }
  if (ct == 0) *in.t = t0 + n_iter;
  chain_leave();
}

// Breadth-first and value-slot reach orders (layout options): the same
// iteration with the pushing forward of kernels.cuh.
template <typename T, int MAXA, int LANES, int NT, int MODE>
__global__ void __launch_bounds__(NT) batch_iterate_push_kernel(const InstDesc *table,
                                                                const __grid_constant__ InstDesc one, int n_inst) {
  constexpr bool CLUSTERED = MODE == kCluster;
  __shared__ double sm[NT];
  __shared__ double s_rows[NT / 32][kChainDoubles<T, MAXA, LANES>];
  chain_enter();
  const int ncta = CLUSTERED ? (int)cluster_ncta() : 1;
  const int rank = CLUSTERED ? (int)cluster_rank() : 0;
  const int inst = (int)blockIdx.x / ncta;
  if (inst >= n_inst) return;
  const int ct = rank * NT + (int)threadIdx.x, all = ncta * NT;
  const InstDesc &in = table ? table[inst] : one;
  StateView<T> st;
  st.reach = (vec2_t<T> *)in.reach;
  st.v = (T *)in.v;
  st.sigma = (T *)in.sigma;
  st.R = in.R;
  st.avg = in.avg;
  st.t = in.t;
  const long long t0 = *in.t;
  const int lane = threadIdx.x % LANES, gid = ct / LANES, ngroups = all / LANES;
  const unsigned mask = group_mask<LANES>();
  double *rows = s_rows[threadIdx.x / 32];
  const int halves = in.order ? 2 : 1;
  for (long long it = 0; it < in.n_iter; ++it) {
    const double wt = avg_weight(t0 + it + 1, in.rule);
    for (int hf = 0; hf < halves; ++hf) {
      const int upd = in.order ? (1 << hf) : 3;
      for (int d = 0; d < in.D; ++d) {
        const LevelWork w = in.lw[d];
        for (int32_t qw = w.ib + rank * NT + (threadIdx.x & ~31); qw < w.ie; qw += 4 * all) {
          if (w.fan) fwd_int4<T, CLUSTERED, true>(in.g, st.sigma, st.reach, qw + (threadIdx.x & 31), all, w.ie);
          else fwd_int4<T, CLUSTERED, false>(in.g, st.sigma, st.reach, qw + (threadIdx.x & 31), all, w.ie);
        }
        for (int32_t i = w.wd0; i < w.wd1; ++i) cta_fwd_wide<T, CLUSTERED>(in.g, st.reach, i, ct, all);
        level_sync<CLUSTERED>();
      }
      for (int d = in.D - 1; d >= 0; --d) {
        const LevelWork w = in.lw[d];
        if (d > 0) {
          for (int32_t i = w.ch0 + ct; i < w.ch1; i += all) bwd_chance<T, CLUSTERED>(in.g, st.v, i);
          if (rank == 0)
            for (int32_t i = w.wd0; i < w.wd1; ++i) cta_bwd_wide<T, NT, CLUSTERED>(in.g, st.v, i, sm);
        }
        for (int32_t I = w.is0 + gid; I < w.is1; I += ngroups)
          bwd_set<T, MAXA, LANES, CLUSTERED>(in.g, st, I, I >= w.is2, lane, mask, wt, in.rule, upd, rows);
        level_sync<CLUSTERED>();
      }
    }
  }
  if (ct == 0) *in.t = t0 + in.n_iter;
  chain_leave();
}

// Exploitability of every instance's average strategy (FP64): normalise the
// average, forward reach under it, then both best responses by depth (the
// arithmetic of br_level_kernel). CTAs and clusters as batch_iterate_kernel.
// wide_parts: partial sums of a wide chance node, the caller's and not the
// CTA's threads (which games of more than four actions in the call lower): the
// second half of them is the first step of the tree of twice the threads.
template <int MAXA, int LANES, int THREADS, bool CLUSTERED>
__global__ void __launch_bounds__(THREADS, 1) batch_br_kernel(const InstDesc *table, const __grid_constant__ InstDesc one,
                                                           int n_inst, int wide_parts) {
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
    for (int32_t a = 0; a < na; ++a) in.sbs[sb + a] = match(in.avg[sb + a], tot, na);
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
      for (int part = threadIdx.x; part < wide_parts; part += THREADS) {  // one or two a thread
        double px = 0.0, py = 0.0, pa = 0.0;
        for (int32_t c = cb + part; c < ce; c += wide_parts) {
          const double2 x = ldm<CLUSTERED>(in.vb + c);
          px += x.x; py += x.y; pa += ldm<CLUSTERED>(in.vavg + c);
        }
        sx = part < THREADS ? px : sx + px;
        sy = part < THREADS ? py : sy + py;
        sa = part < THREADS ? pa : sa + pa;
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
