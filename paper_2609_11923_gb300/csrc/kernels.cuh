// kernels.cuh — sm_103a kernels of one CFR+ iteration over the compiled game.
//
// Stage (a), forward reach (eq. (opfwd) on both lanes, eq. (lanes)): reach
//   is stored for internal nodes only (terminal reach is never read), by
//   internal rank. Member order (the default): each thread takes four
//   internal nodes of depth d + 1, and each reads its parent's reach through
//   its edge record and writes its own (fwd_pull). Breadth-first and
//   value-slot orders: each thread takes four internal nodes of depth d and
//   writes both reach lanes of their internal children (fwd_int4). The
//   acting player's lane is multiplied by sigma(I, a); the other lane and
//   chance edges copy through (the paper's sentinel multiplier 1 becomes a
//   branch on the edge's slot word).
// Stage (b), terminal utility: the value array holds pi_c(z) u(z) in every
//   terminal's value slot from bind time on (eq. (template)); no kernel
//   writes it again, which removes the per-iteration template copy.
// Stages (c) + (d), backward (eqs. (opbwd), (instregret), (regret), (rm)):
//   values live in value slots: the children of one set's members form one
//   contiguous block, and every node writes its own value into its parent's
//   block. Per depth, chance nodes sum their children's values (one thread
//   each; a chance root is skipped, nothing reads its value) and every
//   information set of that depth is handled by one group of LANES lanes,
//   which reads its members' reach as one run in member order: members' values v(h) = sum_a sigma(I,a) v(h.a), the regret terms
//   s * pi_{-i}(h) * (v(h.a) - v(h)) and the average terms pi_i(h) sigma(I,a)
//   are summed over members in a fixed order (no atomics), then
//   R <- max(R + r, 0) (CFR+), avg += t * m, and sigma^{t+1}(I,.) = RM(R) is
//   written in place (nothing reads sigma(I,.) again in this iteration).
//   P64 sums members strictly in ascending node order (lane order within each
//   chunk of LANES members), the order of the recursive definition; P32 keeps
//   per-lane partial sums and finishes with an xor butterfly (fixed shape,
//   deterministic run to run).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace cfr {

template <typename T> struct Vec2;
template <> struct Vec2<float> { using type = float2; };
template <> struct Vec2<double> { using type = double2; };
template <typename T> using vec2_t = typename Vec2<T>::type;

constexpr int kThreads = 256;
constexpr int32_t kP2Bit = 1 << 30;
constexpr int32_t kMask = kP2Bit - 1;

// Loads of arrays that a persistent kernel rewrites between grid barriers go
// around L1 (ld.global.cg): L1 is not coherent across SMs.
template <bool PERSIST, typename X>
__device__ __forceinline__ X ldm(const X *p) {
  if constexpr (PERSIST) return __ldcg(p);
  else return *p;
}

// Programmatic dependent launch between the per-level kernels: every such
// kernel first waits until the launch before it has completed and its
// writes are visible (griddepcontrol.wait; a no-op without a programmatic
// dependency), then lets the next launch start being scheduled
// (launch_dependents), so the next kernel's launch and block scheduling
// overlap this kernel's tail instead of following it.
__device__ __forceinline__ void pdl_enter() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// Loads that a kernel issues before that wait ("early"): the compiled game,
// and state that the launch before does not write. The launches before that
// one have completed by then (each waits before it lets its successor start).
// A launch of a small depth is a chain of dependent loads behind the wait;
// early ones leave one of them there: an iteration of a 81k-node card game
// 33.2 -> 29.2 us, of the 2.8M-node random tree 84.5 -> 79.3 (with the loads of
// a member issued before their first use), of the 27M-node card game 174 -> 165.

constexpr int32_t kWideNode = 1024;   // chance nodes above this fan-out go by chunks
constexpr int32_t kWideChunkK = 2048; // children per chunk of a wide node

struct GameView {
  const int32_t *__restrict__ iset_slot;
  const int32_t *__restrict__ iset_mem;
  // value slots: a set's members' children form one block starting at
  // iset_vb[I] (action-major: child a of member k at iset_vb[I] + a * M +
  // (k - first member), M members); every node writes its own value to the
  // slot its parent reads (mem_vs, ch_vs, wide_vs)
  const int32_t *__restrict__ iset_vb;
  const int32_t *__restrict__ mem_vs;
  const int32_t *__restrict__ ch_vb;       // narrow chance nodes: children's block,
  const int32_t *__restrict__ ch_nch;      //   child count,
  const int32_t *__restrict__ ch_vs;       //   own value slot
  const int32_t *__restrict__ wide_vb;     // wide chance nodes: the same
  const int32_t *__restrict__ wide_nch;
  const int32_t *__restrict__ wide_vs;
  const int32_t *__restrict__ wide_chunk;  // prefix of their chunk counts
  double *wide_part;                       // [3 * chunks] partial sums
  unsigned *wide_cnt;                      // [wide nodes] chunks finished (reset by the last one)
  // compact index space of the internal nodes (reach is stored only there)
  const int32_t *__restrict__ int_slot;    // slot word of each internal node
  const uint32_t *__restrict__ int_mask;   // internal children (bit a), or kBigBit
  const int32_t *__restrict__ int_cirank;  // rank of the first internal child, or big_irank offset
  const int32_t *__restrict__ big_irank;   // [nch, child ranks...] of nodes with > 31 children
  const int2 *__restrict__ int_edge;       // member order: each internal node's (parent rank, slot word of
                                           //   its edge or -1 under chance); else null
  const int32_t *__restrict__ mem_irank;   // internal rank of each member (null in member order)
  const int2 *__restrict__ iset_rank;      // member order: per set, rank of member 0 and the stride
                                           //   of its members' ranks (else null)
  const int32_t *__restrict__ wide_irank;  // internal rank of each wide node
};

constexpr uint32_t kBigBit = 0x80000000u;

template <typename T> struct StateView {
  vec2_t<T> *reach;
  T *v;
  T *sigma;
  double *R;
  double *avg;
  long long *t;  // completed iterations; iteration t+1 uses weight w = t+1
};

struct LevelWork {
  int32_t ib, ie;         // internal ranks of depth d
  int32_t lb, le;         // nodes of depth d
  int32_t ch0, ch1;       // narrow chance nodes of depth d (ch_* arrays)
  int32_t is0, is2, is1;  // sets of depth d: player 1 [is0, is2), player 2 [is2, is1)
  int32_t wd0, wd1;       // wide chance nodes of depth d (wide_* arrays)
  int32_t wc0, wc1;       // their chunks
  int32_t fan;            // 1 if a chance node of depth d has more than kFanLight internal children
};

// Where set I's members keep their reach: member k (global member index) has
// rank kb + k * rg (member order), or the rank table's entry (kb = rg = 0).
struct MemberRanks {
  int32_t kb, rg;
};

__device__ __forceinline__ MemberRanks member_ranks(const GameView &g, int32_t I, int32_t m0) {
  MemberRanks mr{0, 0};
  if (g.iset_rank) {
    const int2 x = __ldg(g.iset_rank + I);
    mr.rg = x.y;
    mr.kb = x.x - m0 * x.y;
  }
  return mr;
}

// The wide node owning chunk q (binary search over the level's prefix).
__device__ __forceinline__ int32_t wide_of_chunk(const GameView &g, const LevelWork &w, int32_t q) {
  int32_t lo = w.wd0, hi = w.wd1 - 1;
  while (lo < hi) {
    const int32_t mid = (lo + hi + 1) >> 1;
    if (__ldg(g.wide_chunk + mid) <= q) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// Fixed-shape block reduction of N values at once (all threads call it; the
// results are valid in thread 0): butterflies within the warps, then one
// across them.
template <int N>
__device__ __forceinline__ void block_sum(double (&x)[N]) {
  __shared__ double sm[N][kThreads / 32];
  const int warp = threadIdx.x / 32, lane = threadIdx.x & 31;
#pragma unroll
  for (int off = 16; off > 0; off >>= 1)
#pragma unroll
    for (int i = 0; i < N; ++i) x[i] += __shfl_xor_sync(0xffffffffu, x[i], off);
  __syncthreads();  // the array may still be read from the call before
  if (lane == 0)
#pragma unroll
    for (int i = 0; i < N; ++i) sm[i][warp] = x[i];
  __syncthreads();
  if (warp == 0) {
#pragma unroll
    for (int i = 0; i < N; ++i) x[i] = lane < kThreads / 32 ? sm[i][lane] : 0.0;
#pragma unroll
    for (int off = kThreads / 64; off > 0; off >>= 1)
#pragma unroll
      for (int i = 0; i < N; ++i) x[i] += __shfl_xor_sync(0xffffffffu, x[i], off);
  }
}

// The sum of v[cb, ce) strictly left to right (the FP64 parity order), for
// one block of N threads that all call it: the block stages N values at a
// time in shared memory, and thread 0 adds one batch while the others load
// the next. The result is valid in thread 0.
template <int N, bool PERSIST, typename T>
__device__ __forceinline__ double ordered_sum(const T *v, int32_t cb, int32_t ce) {
  __shared__ double buf[2 * N];
  const int tid = threadIdx.x;
  double s = 0.0;
  if (cb + tid < ce) buf[tid] = (double)ldm<PERSIST>(v + cb + tid);
  __syncthreads();
  int b = 0;
  for (int32_t c0 = cb; c0 < ce; c0 += N) {
    if (c0 + N + tid < ce) buf[(b ^ 1) * N + tid] = (double)ldm<PERSIST>(v + c0 + N + tid);
    if (tid == 0) {
      const int n = ce - c0 < N ? ce - c0 : N;
      for (int j = 0; j < n; ++j) s = s + buf[b * N + j];
    }
    __syncthreads();
    b ^= 1;
  }
  return s;
}

// ------------------------------------------------------------ forward reach
// reach of child a of an internal node with slot word s and reach r
template <typename T, bool PERSIST>
__device__ __forceinline__ vec2_t<T> child_reach(const T *sigma, int32_t s, vec2_t<T> r, int a) {
  if (s >= 0) {
    const T sa = ldm<PERSIST>(sigma + (s & kMask) + a);
    if (s & kP2Bit) r.y = r.y * sa;
    else r.x = r.x * sa;
  }
  return r;
}

// Writes the reach of the internal children of one internal node: children
// flagged in the mask get consecutive internal ranks from cir on; nodes with
// more than 31 children list their children's ranks in big_irank (terminal
// children -1, never written: nothing reads a terminal's reach).
template <typename T, bool PERSIST>
__device__ __forceinline__ void fwd_write(const GameView &g, const T *sigma, vec2_t<T> *reach, int32_t s,
                                          uint32_t mask, int32_t cir, vec2_t<T> r) {
  if (mask & kBigBit) {
    const int32_t nch = __ldg(g.big_irank + cir);
    if (nch > kWideNode) return;  // wide: done by chunks
    for (int32_t a = 0; a < nch; ++a) {
      const int32_t q = __ldg(g.big_irank + cir + 1 + a);
      if (q >= 0) reach[q] = child_reach<T, PERSIST>(sigma, s, r, a);
    }
  } else {
    int32_t q = cir;
    while (mask) {
      const int a = __ffs(mask) - 1;
      mask &= mask - 1;
      reach[q++] = child_reach<T, PERSIST>(sigma, s, r, a);
    }
  }
}

constexpr int kFanLight = 4;  // chance nodes with more internal children are written by the whole warp

// Four internal nodes q, q+stride, q+2 stride, q+3 stride per thread: their
// records and reach are read together (coalesced), then their children's
// reach is written. A chance node's internal children all copy its reach, so
// a chance node with many of them (a card dealt mid-game) is written by the
// whole warp as one coalesced run instead of by its own thread alone. All 32
// lanes of the warp call this together (q = warp base + lane; a lane whose
// nodes lie past qe still takes part in the warp-wide writes).
template <typename T, bool PERSIST, bool FAN>
__device__ __forceinline__ void fwd_int4(const GameView &g, const T *sigma, vec2_t<T> *reach, int32_t q,
                                         int32_t stride, int32_t qe) {
  int32_t sl[4], ci[4];
  uint32_t mk[4];
  vec2_t<T> r[4];
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int32_t x = q + u * stride;
    mk[u] = 0u; sl[u] = -1; ci[u] = 0;
    r[u].x = T(0); r[u].y = T(0);
    if (x < qe) {
      sl[u] = __ldg(g.int_slot + x);
      mk[u] = __ldg(g.int_mask + x);
      ci[u] = __ldg(g.int_cirank + x);
      r[u] = ldm<PERSIST>(reach + x);
    }
  }
  if constexpr (!FAN) {  // depths without chance nodes of many internal children
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (mk[u]) fwd_write<T, PERSIST>(g, sigma, reach, sl[u], mk[u], ci[u], r[u]);
    return;
  }
  bool hvy[4], any = false;
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    hvy[u] = sl[u] < 0 && mk[u] != 0u && ((mk[u] & kBigBit) || __popc(mk[u]) > kFanLight);
    any = any || hvy[u];
  }
  if (!__any_sync(0xffffffffu, any)) {  // the common case: every node of the warp is light
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (mk[u]) fwd_write<T, PERSIST>(g, sigma, reach, sl[u], mk[u], ci[u], r[u]);
    return;
  }
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const bool heavy = hvy[u];
    unsigned hv = __ballot_sync(0xffffffffu, heavy);
    if (mk[u] && !heavy) fwd_write<T, PERSIST>(g, sigma, reach, sl[u], mk[u], ci[u], r[u]);
    while (hv) {
      const int j = __ffs(hv) - 1;
      hv &= hv - 1;
      const uint32_t m = __shfl_sync(0xffffffffu, mk[u], j);
      const int32_t c0 = __shfl_sync(0xffffffffu, ci[u], j);
      vec2_t<T> rr;
      rr.x = __shfl_sync(0xffffffffu, r[u].x, j);
      rr.y = __shfl_sync(0xffffffffu, r[u].y, j);
      if (m & kBigBit) {
        const int32_t nch = __ldg(g.big_irank + c0);
        if (nch <= kWideNode)  // wide nodes go by chunks
          for (int32_t a = lane; a < nch; a += 32) {
            const int32_t c = __ldg(g.big_irank + c0 + 1 + a);
            if (c >= 0) reach[c] = rr;
          }
      } else {
        const int n = __popc(m);
        for (int i = lane; i < n; i += 32) reach[c0 + i] = rr;
      }
    }
  }
}

// One chunk of a wide chance node: its internal children copy its reach.
template <typename T, bool PERSIST>
__device__ __forceinline__ void fwd_wide_chunk(const GameView &g, const LevelWork &w, vec2_t<T> *reach, int32_t q) {
  const int32_t wi = wide_of_chunk(g, w, q);
  const int32_t ir = __ldg(g.wide_irank + wi);
  const int32_t off = __ldg(g.int_cirank + ir);
  const int32_t nch = __ldg(g.big_irank + off);
  const int32_t j0 = (q - __ldg(g.wide_chunk + wi)) * kWideChunkK;
  const int32_t j1 = min(nch, j0 + kWideChunkK);
  const vec2_t<T> r = ldm<PERSIST>(reach + ir);
  for (int32_t j = j0 + threadIdx.x; j < j1; j += blockDim.x) {
    const int32_t c = __ldg(g.big_irank + off + 1 + j);
    if (c >= 0) reach[c] = r;
  }
}

// Grid: nb_nodes blocks over the internal nodes of depth d, then one block
// per wide chunk.
template <typename T, bool FAN>
__global__ void __launch_bounds__(kThreads) fwd_level_kernel(GameView g, const T *sigma, vec2_t<T> *reach,
                                                            LevelWork w, int nb_nodes) {
  pdl_enter();
  if ((int)blockIdx.x >= nb_nodes) {
    fwd_wide_chunk<T, false>(g, w, reach, w.wc0 + (int32_t)blockIdx.x - nb_nodes);
    return;
  }
  const int32_t stride = nb_nodes * blockDim.x;
  const int lane = threadIdx.x & 31;
  for (int32_t qw = w.ib + blockIdx.x * blockDim.x + (threadIdx.x & ~31); qw < w.ie; qw += 4 * stride)
    fwd_int4<T, false, FAN>(g, sigma, reach, qw + lane, stride, w.ie);
}

// Member order: each internal node of ranks [qb, qe) (one depth) pulls its
// reach from its parent's, times the strategy of its edge in the acting
// player's lane (a chance edge copies it). kPull nodes per thread in flight.
constexpr int kPull = 4;
struct PullEdges {
  int2 e[kPull];
};

__device__ __forceinline__ void pull_edges(const GameView &g, int32_t q, int32_t stride, int32_t qe, PullEdges &p) {
#pragma unroll
  for (int u = 0; u < kPull; ++u) {
    const int32_t x = q + u * stride;
    p.e[u] = make_int2(-1, -1);
    if (x < qe) p.e[u] = __ldg(g.int_edge + x);
  }
}

template <typename T, bool PERSIST>
__device__ __forceinline__ void pull_sigma(const T *sigma, const PullEdges &p, T (&sa)[kPull]) {
#pragma unroll
  for (int u = 0; u < kPull; ++u)
    sa[u] = p.e[u].x >= 0 && p.e[u].y >= 0 ? ldm<PERSIST>(sigma + (p.e[u].y & kMask)) : T(1);
}

template <typename T, bool PERSIST>
__device__ __forceinline__ void pull_write(vec2_t<T> *reach, int32_t q, int32_t stride, const PullEdges &p,
                                           const T (&sa)[kPull]) {
  vec2_t<T> r[kPull];
#pragma unroll
  for (int u = 0; u < kPull; ++u) {
    r[u].x = T(0); r[u].y = T(0);
    if (p.e[u].x >= 0) r[u] = ldm<PERSIST>(reach + p.e[u].x);
  }
#pragma unroll
  for (int u = 0; u < kPull; ++u) {
    if (p.e[u].x < 0) continue;
    if (p.e[u].y >= 0) {
      if (p.e[u].y & kP2Bit) r[u].y = r[u].y * sa[u];
      else r[u].x = r[u].x * sa[u];
    }
    reach[q + u * stride] = r[u];
  }
}

template <typename T, bool PERSIST>
__device__ __forceinline__ void fwd_pull(const GameView &g, const T *sigma, vec2_t<T> *reach, int32_t q,
                                         int32_t stride, int32_t qe) {
  PullEdges p;
  T sa[kPull];
  pull_edges(g, q, stride, qe, p);
  pull_sigma<T, PERSIST>(sigma, p, sa);
  pull_write<T, PERSIST>(reach, q, stride, p, sa);
}

// early: the launch before writes no strategy (it is a forward launch).
template <typename T>
__global__ void __launch_bounds__(kThreads) fwd_pull_kernel(GameView g, const T *sigma, vec2_t<T> *reach,
                                                            int32_t qb, int32_t qe, int early) {
  const int32_t stride = gridDim.x * blockDim.x;
  int32_t q = qb + blockIdx.x * blockDim.x + threadIdx.x;
  PullEdges p;
  T sa[kPull];
  pull_edges(g, q, stride, qe, p);
  if (early) {
    pull_sigma<T, false>(sigma, p, sa);
    pdl_enter();
  } else {
    pdl_enter();
    pull_sigma<T, false>(sigma, p, sa);
  }
  if (q < qe) pull_write<T, false>(reach, q, stride, p, sa);
  for (q += kPull * stride; q < qe; q += kPull * stride) fwd_pull<T, false>(g, sigma, reach, q, stride, qe);
}

// ------------------------------------------------------------ group helpers
template <int LANES>
__device__ __forceinline__ unsigned group_mask() {
  if constexpr (LANES == 32) return 0xffffffffu;
  else return ((1u << LANES) - 1u) << (((threadIdx.x & 31) / LANES) * LANES);
}

template <int LANES, typename X>
__device__ __forceinline__ X group_sum_butterfly(X x, unsigned mask) {
#pragma unroll
  for (int off = LANES / 2; off > 0; off >>= 1) x += __shfl_xor_sync(mask, x, off, LANES);
  return x;
}

// V values (a power of two) summed over the group by the butterfly's tree,
// the values shared out on the way: after the step over lane distance off a
// lane keeps the half of the values that its bit of off names, so the sums
// take V - 1 + log2(LANES / V) shuffles instead of V * log2(LANES), and value
// i ends in lanes i * LANES / V ... (V <= LANES) or in x[i % (V / LANES)] of
// lane i / (V / LANES). The same bits as V butterflies.
template <int LANES, int V, typename X>
__device__ __forceinline__ void group_sum_scatter(X (&x)[V], int lane, unsigned mask) {
  int n = V;
#pragma unroll
  for (int off = LANES / 2; off > 0; off >>= 1) {
    if (n > 1) {
      const bool up = lane & off;
      n >>= 1;
#pragma unroll
      for (int i = 0; i < V / 2; ++i) {
        if (i < n) {
          const X mine = up ? x[n + i] : x[i], other = up ? x[i] : x[n + i];
          x[i] = mine + __shfl_xor_sync(mask, other, off, LANES);
        }
      }
    } else {
      x[0] += __shfl_xor_sync(mask, x[0], off, LANES);
    }
  }
}

// ------------------------------------------------------------- update rules
// CFR+ clamps the cumulative regret at zero; vanilla CFR does not; PCFR+
// clamps like CFR+ and matches the next strategy against R + r, the
// iteration's instantaneous regret serving as the prediction (Section 3,
// update rules).
constexpr int kRuleCfrPlus = 0, kRuleCfr = 1, kRulePcfrPlus = 2;

// Averaging weight of iteration t (1-based): t, or t^2 under PCFR+.
__device__ __forceinline__ double avg_weight(long long t, int rule) {
  const double x = (double)t;
  return rule == kRulePcfrPlus ? x * x : x;
}

// Conversions and comparisons of doubles in integer arithmetic. GB300's FP64
// pipe takes one warp instruction every 16-19 cycles per SM whatever the
// number of active lanes (an instruction whose predicate is off in all of
// them included), and conversions (cvt.f64.f32, cvt.f32.f64) and compares
// (setp.f64) run there too, with 100 cycles of latency each (measured; 64
// for an add). The slot update is a chain of them on a few lanes of a warp, so
// only its add and its multiply-add stay on that pipe, and what is rarely
// needed is a function of its own, or the compiler runs it always, predicated
// off: a round of 16 warps 2,372 -> 609 cycles, of one warp 645 -> 304. Same
// results bit for bit (NaNs stay NaNs).
__device__ __forceinline__ double widen(float x) {  // (double)x
  const uint32_t e = (__float_as_uint(x) >> 23) & 255u;
  const bool sub = e == 0u;  // zero or subnormal: scaled into the normal range first
  const uint32_t u = __float_as_uint(sub ? x * 18446744073709551616.f : x);
  uint32_t hi = ((u & 0x7fffffffu) >> 3) + (sub ? 0x34000000u : 0x38000000u) + (e == 255u ? 0x38000000u : 0u);
  if ((u << 1) == 0u) hi = 0u;
  return __hiloint2double((int)((u & 0x80000000u) | hi), (int)(u << 29));
}

static __device__ __noinline__ float narrow_rare(double x) { return (float)x; }

__device__ __forceinline__ float narrow_pos(double x) {  // (float)x of x >= 0, to nearest, ties to even
  const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
  const uint32_t e = (hi >> 20) - 896u;
  const uint32_t m = (e << 23) | ((hi & 0xfffffu) << 3) | (lo >> 29);
  const uint32_t rest = lo & 0x1fffffffu;  // bits below the last place
  const bool zero = (hi | lo) == 0u;
  float y = zero ? 0.f : __uint_as_float(m + (rest > 0x10000000u - (m & 1u) ? 1u : 0u));
  if (!zero && e - 1u >= 254u) y = narrow_rare(x);  // to a subnormal or infinite float
  return y;
}

__device__ __forceinline__ double positive_part(double x) {  // x > 0.0 ? x : 0.0 (NaN and -0 give 0)
  const long long b = __double_as_longlong(x);
  return b > 0 && b <= 0x7ff0000000000000ll ? x : 0.0;
}

// A set total as a double: FP32 totals are widened.
__device__ __forceinline__ double as_double(float x) { return widen(x); }
__device__ __forceinline__ double as_double(double x) { return x; }

// PCFR+ matches against R + r.
static __device__ __noinline__ double predicted(double R, double r) { return R + r; }

// sigma of a slot from its positive part and the set's sum of them (uniform
// where the sum is zero), with one division.
__device__ __forceinline__ float match(float pos, float tot, int32_t na) {
  const bool some = tot > 0.f;
  return (some ? pos : 1.f) / (some ? tot : (float)na);
}
__device__ __forceinline__ double match(double pos, double tot, int32_t na) {
  const long long b = __double_as_longlong(tot);
  const bool some = b > 0 && b <= 0x7ff0000000000000ll;
  return (some ? pos : 1.0) / (some ? tot : widen((float)na));
}

// One slot's update from its set's totals (instantaneous regret r, average
// term m) and its cumulative regret R and average sum S: Rn = R + r (clamped
// at 0 except under vanilla CFR) and Sn = S + wt * m. Returns what regret
// matching takes the positive part of: the new R, or R + r under PCFR+.
__device__ __forceinline__ double slot_terms(double R, double S, double r, double m, double wt, int rule, double &Rn,
                                             double &Sn) {
  Rn = R + r;
  if (rule != kRuleCfr) Rn = positive_part(Rn);
  Sn = S + wt * m;
  double x = Rn;
  if (rule == kRulePcfrPlus) x = predicted(Rn, r);
  return positive_part(x);
}

// The same on the slot's entries in memory.
__device__ __forceinline__ double slot_update(double *R, double *avg, int32_t q, double r, double m, double wt,
                                              int rule) {
  double Rn, Sn;
  const double pos = slot_terms(R[q], avg[q], r, m, wt, rule, Rn, Sn);
  R[q] = Rn;
  avg[q] = Sn;
  return pos;
}

// ------------------------------------------------------------- backward
// Narrow chance node i: the sum of its children's values (left to right).
template <typename T, bool PERSIST>
__device__ __forceinline__ void bwd_chance(const GameView &g, T *v, int32_t i) {
  const int32_t cb = __ldg(g.ch_vb + i), ce = cb + __ldg(g.ch_nch + i);
  T s = T(0);
  for (int32_t c = cb; c < ce; ++c) s = s + ldm<PERSIST>(v + c);
  v[__ldg(g.ch_vs + i)] = s;
}

// One chunk of a wide chance node's value sum. P32: every chunk block sums
// its children (fixed shape), and the block that finishes last adds the
// chunk partials in chunk order (an integer ticket decides who is last; no
// float atomics). P64: the first chunk's block sums all children strictly
// left to right, the order of the recursive definition.
template <typename T, bool PERSIST>
__device__ __forceinline__ void bwd_wide_chunk(const GameView &g, const LevelWork &w, T *v, int32_t q) {
  const int32_t wi = wide_of_chunk(g, w, q);
  const int32_t h = __ldg(g.wide_vs + wi);  // the node's own value slot
  const int32_t cb = __ldg(g.wide_vb + wi), ce = cb + __ldg(g.wide_nch + wi);
  const int32_t q0 = __ldg(g.wide_chunk + wi), nq = __ldg(g.wide_chunk + wi + 1) - q0;
  if constexpr (sizeof(T) == 8) {
    if (q == q0) {  // block-uniform: the whole block stages the children
      const double s = ordered_sum<kThreads, PERSIST>(v, cb, ce);
      if (threadIdx.x == 0) v[h] = s;
    }
    return;
  } else {
    const int32_t c0 = cb + (q - q0) * kWideChunkK, c1 = min(ce, c0 + kWideChunkK);
    double x[1] = {0.0};
    for (int32_t c = c0 + threadIdx.x; c < c1; c += blockDim.x) x[0] += (double)ldm<PERSIST>(v + c);
    block_sum(x);
    __shared__ unsigned s_ticket;
    if (threadIdx.x == 0) {
      g.wide_part[q] = x[0];
      __threadfence();
      s_ticket = atomicAdd(g.wide_cnt + wi, 1u);
    }
    __syncthreads();
    if (s_ticket == (unsigned)(nq - 1)) {  // the last chunk's block adds the partials (fixed shape)
      __threadfence();
      double y[1] = {0.0};
      for (int32_t k = threadIdx.x; k < nq; k += blockDim.x) y[0] += __ldcg(g.wide_part + q0 + k);
      block_sum(y);
      if (threadIdx.x == 0) {
        v[h] = (T)y[0];
        g.wide_cnt[wi] = 0u;
      }
    }
  }
}

// A member's two indices (member order: coalesced reads): its own value slot
// and its internal rank (where its reach lives; in member order the rank
// follows from the member index and the set's rank base and stride). Past
// the set's end: -1.
__device__ __forceinline__ int32_t member_rank(const GameView &g, int32_t k, MemberRanks mr) {
  return g.mem_irank ? __ldg(g.mem_irank + k) : mr.kb + k * mr.rg;
}

__device__ __forceinline__ void member_idx(const GameView &g, int32_t k, int32_t m1, MemberRanks mr, int32_t &ps,
                                           int32_t &ir) {
  ps = -1;
  ir = -1;
  if (k < m1) {
    ps = __ldg(g.mem_vs + k);
    ir = member_rank(g, k, mr);
  }
}

// Loads and per-member terms of one member (k < m1) whose indices are
// already known, or zeros. The member's child a is slot vb + a * M + (k -
// m0) of the set's block (M = m1 - m0 members): for each action the group's
// lanes read consecutive members' children as one run. The average-strategy terms are
// pw * sigma(a), each added, in member order in FP64, as the definition does.
template <typename T, int MAXA, bool PERSIST>
__device__ __forceinline__ void member_data(const GameView &g, const StateView<T> &st, int32_t k, int32_t m0,
                                            int32_t m1, int32_t vb, int32_t na, bool p2, const T (&sig)[MAXA],
                                            int32_t h, int32_t ir, T (&d)[MAXA], T (&mm)[MAXA]) {
#pragma unroll
  for (int a = 0; a < MAXA; ++a) { d[a] = T(0); mm[a] = T(0); }
  if (k >= m1) return;
  const int32_t cb = vb + (k - m0), M = m1 - m0;
  const vec2_t<T> r = ldm<PERSIST>(st.reach + ir);
  T vc[MAXA];
#pragma unroll
  for (int a = 0; a < MAXA; ++a)  // every load before the first use
    vc[a] = a < na ? ldm<PERSIST>(st.v + cb + a * M) : T(0);
  T vh = T(0);
#pragma unroll
  for (int a = 0; a < MAXA; ++a)
    if (a < na) vh = vh + sig[a] * vc[a];
  st.v[h] = vh;
  const T po = p2 ? r.x : r.y;  // opponent's reach (chance is inside v)
  const T pw = p2 ? r.y : r.x;  // own reach
  const T f = (p2 ? T(-1) : T(1)) * po;
#pragma unroll
  for (int a = 0; a < MAXA; ++a) {
    if (a < na) {
      d[a] = f * (vc[a] - vh);
      mm[a] = pw * sig[a];
    }
  }
}

// Indices, loads and per-member terms of one member (k < m1), or zeros.
template <typename T, int MAXA, bool PERSIST>
__device__ __forceinline__ void member_terms(const GameView &g, const StateView<T> &st, int32_t k, int32_t m0,
                                             int32_t m1, MemberRanks mr, int32_t vb, int32_t na, bool p2,
                                             const T (&sig)[MAXA], T (&d)[MAXA], T (&mm)[MAXA]) {
  int32_t h, ir;
  member_idx(g, k, m1, mr, h, ir);
  member_data<T, MAXA, PERSIST>(g, st, k, m0, m1, vb, na, p2, sig, h, ir, d, mm);
}

// FP64 sums of a set run in the order of the definition, one dependent chain
// of adds for every slot's regret term and every slot's average term. On
// GB300 a warp instruction of the FP64 pipe costs the SM 16-19 cycles
// however few lanes it serves, so a chain belongs to one lane: chain c < MAXA
// is the regret sum of action c, chain MAXA + a the average sum of action a,
// and lane c % LANES of the group adds chain c's terms member by member from
// the warp's rows in shared memory. (Every lane adding every chain took
// 2 * na adds a member where this takes one or two.) One FP64 iteration of the
// 11M-node card game, autotuned: 701 -> 488 us; of an 80k-node random tree in
// two half passes: 367 -> 266 us. (A short last chunk in unrolled code,
// predicated off past its members: 40 sets of one member by 32 lanes in the
// persistent form 197 us an iteration instead of 139, a random tree of 10,400
// nodes in a batch 59 instead of 54.)
template <typename T, int MAXA, int LANES>
constexpr bool kChains = sizeof(T) == 8 && LANES >= 4 && LANES <= 32 && MAXA <= 8;
template <int MAXA, int LANES> constexpr int kChainAcc = (2 * MAXA + LANES - 1) / LANES;  // chains of a lane
constexpr int kChainRow = 33;  // doubles of a chain's row: a term of each lane, and one that spreads the banks
template <typename T, int MAXA, int LANES>
constexpr int kChainDoubles = kChains<T, MAXA, LANES> ? 2 * MAXA * kChainRow : 1;  // a warp's rows

template <int MAXA, int LANES>
__device__ __forceinline__ void accumulate_chains(double *rows, int32_t cnt, int32_t na, unsigned mask,
                                                  const double (&d)[MAXA], const double (&mm)[MAXA],
                                                  double (&acc)[kChainAcc<MAXA, LANES>]) {
  const int wl = threadIdx.x & 31, lane = wl & (LANES - 1), g0 = wl - lane;
#pragma unroll
  for (int a = 0; a < MAXA; ++a) {
    if (a < na) {
      rows[a * kChainRow + wl] = d[a];
      rows[(MAXA + a) * kChainRow + wl] = mm[a];
    }
  }
  __syncwarp(mask);
  auto add = [&](int j) {
#pragma unroll
    for (int i = 0; i < kChainAcc<MAXA, LANES>; ++i) {
      const int c = lane + i * LANES;  // rows of actions >= na hold stale terms: their sums are never used
      if (c < 2 * MAXA) acc[i] = acc[i] + rows[c * kChainRow + g0 + j];
    }
  };
  if (cnt >= LANES) {
#pragma unroll
    for (int j = 0; j < LANES; ++j) add(j);
  } else {  // no more instructions than members: one that is predicated off takes its turn on the FP64 pipe too
#pragma unroll 1
    for (int j = 0; j < cnt; ++j) add(j);
  }
  __syncwarp(mask);
}

// Adds one chunk's member terms to the group totals. P64 without chains:
// lane order (the members' ascending order), every lane ends with the same
// totals. P32: per-lane partial sums (finished by a butterfly).
template <typename T, int MAXA, int LANES>
__device__ __forceinline__ void accumulate_chunk(int32_t cnt, int32_t na, unsigned mask, const T (&d)[MAXA],
                                                 const T (&mm)[MAXA], T (&racc)[MAXA], T (&macc)[MAXA]) {
  if constexpr (sizeof(T) == 8) {
    for (int j = 0; j < cnt; ++j) {
#pragma unroll
      for (int a = 0; a < MAXA; ++a) {
        if (a < na) {
          racc[a] = racc[a] + __shfl_sync(mask, d[a], j, LANES);
          macc[a] = macc[a] + __shfl_sync(mask, mm[a], j, LANES);
        }
      }
    }
  } else {
#pragma unroll
    for (int a = 0; a < MAXA; ++a) {
      racc[a] += d[a];
      macc[a] += mm[a];
    }
  }
}

// One information set, processed by the LANES lanes of one group. Members go
// in chunks of LANES (two chunks per step for narrow groups); each step loads
// the next step's member indices while its own reach and child values are in
// flight, so a step waits for one memory round trip, not two. The update of
// the set's slots runs one lane per action.
template <typename T, int MAXA> struct SetHead {  // what a set's pass reads that no backward launch of another depth writes
  int32_t sb, na, m0, m1, vb;
  MemberRanks mr;
  T sig[MAXA];
  double R, S;  // lane a's slot (groups of at least MAXA lanes)
};

template <typename T, int MAXA, int LANES, bool PERSIST>
__device__ __forceinline__ void load_head(const GameView &g, const StateView<T> &st, int32_t I, int lane,
                                          SetHead<T, MAXA> &h) {
  h.sb = __ldg(g.iset_slot + I);
  h.na = __ldg(g.iset_slot + I + 1) - h.sb;
  h.m0 = __ldg(g.iset_mem + I);
  h.m1 = __ldg(g.iset_mem + I + 1);
  h.vb = __ldg(g.iset_vb + I);
  h.mr = member_ranks(g, I, h.m0);
#pragma unroll
  for (int a = 0; a < MAXA; ++a) h.sig[a] = a < h.na ? ldm<PERSIST>(st.sigma + h.sb + a) : T(0);
  h.R = h.S = 0.0;
  if (LANES >= MAXA && lane < h.na) {
    h.R = st.R[h.sb + lane];
    h.S = st.avg[h.sb + lane];
  }
}

// A warp's sets in step: its 32 / LANES groups run one set each through the
// same instructions, shorter sets (and groups without a set: na = 0, no
// members) idle along. With a loop and sync masks of each group's own the
// groups of a warp drifted apart and every instruction was issued once per
// group, which an FP64 pipe that takes 16-19 cycles for a warp instruction
// feels most. FP64 sets of two and three actions have code of their own
// where all of a warp's are (the pipe takes as long for a predicated
// instruction as for another). One iteration: the 11M-node card game in FP64
// 568 -> 404 us (autotuned 464 -> 350), an 80k-node random tree in two half
// passes 236 -> 195; in FP32 a 2.8M-node random tree 72 -> 66, a card game of
// 81k nodes 29.0 -> 26.9.

// FP64: the members of each group's set, none of more than NA actions: their
// values, and in r[i] and m[i] the totals of slot lane + i * LANES, summed in
// member order. Members past a set's end add zeros.
template <int MAXA, int LANES, int NA, int PER>
__device__ __forceinline__ void warp_chains(const GameView &g, const StateView<double> &st,
                                            const SetHead<double, MAXA> &hd, bool p2, int lane, int32_t longest,
                                            double *rows, double (&r)[PER], double (&m)[PER]) {
  constexpr int C = 2 * NA, ACC = (C + LANES - 1) / LANES;  // chains: regret, then average, by action
  constexpr int U = LANES <= 8 ? 2 : 1;                     // chunks in flight
  constexpr bool EXACT = NA < MAXA;                         // every set of the warp has NA actions (or none)
  const int wl = threadIdx.x & 31, g0 = wl - lane;
  const int32_t m0 = hd.m0, m1 = hd.m1, M = m1 - m0;
  double acc[ACC];
#pragma unroll
  for (int i = 0; i < ACC; ++i) acc[i] = 0.0;
  int32_t ps[U], ir[U];
#pragma unroll
  for (int u = 0; u < U; ++u) member_idx(g, m0 + u * LANES + lane, m1, hd.mr, ps[u], ir[u]);
  for (int32_t k0 = 0; k0 < longest; k0 += U * LANES) {
    int32_t qs[U], jr[U];  // the next step's indices
#pragma unroll
    for (int u = 0; u < U; ++u) member_idx(g, m0 + k0 + (U + u) * LANES + lane, m1, hd.mr, qs[u], jr[u]);
    double2 re[U];
    double vc[U][NA], d[U][NA], mm[U][NA];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const bool in = ps[u] >= 0;
      const int32_t cb = hd.vb + k0 + u * LANES + lane;
      re[u] = make_double2(0.0, 0.0);
      if (in) re[u] = st.reach[ir[u]];
#pragma unroll
      for (int a = 0; a < NA; ++a) vc[u][a] = in && (EXACT || a < hd.na) ? st.v[cb + a * M] : 0.0;
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      double vh = hd.sig[0] * vc[u][0];
#pragma unroll
      for (int a = 1; a < NA; ++a) vh = vh + hd.sig[a] * vc[u][a];
      if (ps[u] >= 0) st.v[ps[u]] = vh;
      const double f = p2 ? -re[u].x : re[u].y;  // opponent's reach, the regret's sign
      const double pw = p2 ? re[u].y : re[u].x;
#pragma unroll
      for (int a = 0; a < NA; ++a) {
        d[u][a] = f * (vc[u][a] - vh);
        mm[u][a] = pw * hd.sig[a];
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int32_t cnt = longest - k0 - u * LANES;
      if (cnt <= 0) break;
#pragma unroll
      for (int a = 0; a < NA; ++a) {
        rows[a * kChainRow + wl] = d[u][a];
        rows[(NA + a) * kChainRow + wl] = mm[u][a];
      }
      __syncwarp();
      const double *row = rows + lane * kChainRow + g0;
      if (cnt >= LANES) {
#pragma unroll
        for (int j = 0; j < LANES; ++j)
#pragma unroll
          for (int i = 0; i < ACC; ++i)
            if (lane + i * LANES < C) acc[i] = acc[i] + row[i * LANES * kChainRow + j];
      } else {
#pragma unroll 1
        for (int j = 0; j < cnt; ++j)
#pragma unroll
          for (int i = 0; i < ACC; ++i)
            if (lane + i * LANES < C) acc[i] = acc[i] + row[i * LANES * kChainRow + j];
      }
      __syncwarp();
    }
#pragma unroll
    for (int u = 0; u < U; ++u) { ps[u] = qs[u]; ir[u] = jr[u]; }
  }
#pragma unroll
  for (int p = 0; p < PER; ++p) {
    r[p] = p < ACC ? acc[p] : 0.0;
    m[p] = 0.0;
#pragma unroll
    for (int i = 0; i < ACC; ++i) {  // chain NA + lane + p * LANES
      const int c = NA + lane + p * LANES;
      const double x = __shfl_sync(0xffffffffu, acc[i], c % LANES, LANES);
      if (c / LANES == i) m[p] = x;
    }
  }
}

template <typename T, int MAXA, int LANES>
constexpr bool kInStep = MAXA <= 8 && LANES >= 4 && LANES <= 32;

template <typename T, int MAXA, int LANES>
__device__ __forceinline__ void bwd_sets(const GameView &g, const StateView<T> &st, const SetHead<T, MAXA> &hd,
                                         bool p2, int lane, double wt, int rule, int upd, double *rows) {
  constexpr unsigned full = 0xffffffffu;
  constexpr int PER = (MAXA + LANES - 1) / LANES;  // slots of a lane: lane, lane + LANES, ...
  const int32_t sb = hd.sb, na = hd.na;
  const int most = __reduce_max_sync(full, na);
  T r[PER], m[PER];
  if constexpr (sizeof(T) == 8) {
    const int32_t longest = __reduce_max_sync(full, hd.m1 - hd.m0);
    if (most == 2 && __all_sync(full, na == 2 || na == 0))
      warp_chains<MAXA, LANES, 2, PER>(g, st, hd, p2, lane, longest, rows, r, m);
    else if (most == 3 && __all_sync(full, na == 3 || na == 0))
      warp_chains<MAXA, LANES, 3, PER>(g, st, hd, p2, lane, longest, rows, r, m);
    else
      warp_chains<MAXA, LANES, MAXA, PER>(g, st, hd, p2, lane, longest, rows, r, m);
  } else {
    const int32_t m0 = hd.m0, m1 = hd.m1, vb = hd.vb;
    T racc[MAXA], macc[MAXA];
#pragma unroll
    for (int a = 0; a < MAXA; ++a) racc[a] = macc[a] = T(0);
    auto add = [&](const T(&d)[MAXA], const T(&mm)[MAXA]) {
#pragma unroll
      for (int a = 0; a < MAXA; ++a) {
        racc[a] += d[a];
        macc[a] += mm[a];
      }
    };
    constexpr int U = LANES <= 8 ? 2 : 1;  // chunks in flight
    int32_t ps[U], ir[U];
#pragma unroll
    for (int u = 0; u < U; ++u) member_idx(g, m0 + u * LANES + lane, m1, hd.mr, ps[u], ir[u]);
    for (int32_t k0 = m0; k0 < m1; k0 += U * LANES) {
      int32_t qs[U], jr[U];  // the next step's indices
#pragma unroll
      for (int u = 0; u < U; ++u) member_idx(g, k0 + (U + u) * LANES + lane, m1, hd.mr, qs[u], jr[u]);
      T d[U][MAXA], mm[U][MAXA];
#pragma unroll
      for (int u = 0; u < U; ++u)
        member_data<T, MAXA, false>(g, st, k0 + u * LANES + lane, m0, m1, vb, na, p2, hd.sig, ps[u], ir[u], d[u], mm[u]);
#pragma unroll
      for (int u = 0; u < U; ++u) add(d[u], mm[u]);
#pragma unroll
      for (int u = 0; u < U; ++u) { ps[u] = qs[u]; ir[u] = jr[u]; }
    }
    __syncwarp();
#pragma unroll
    for (int a = 0; a < MAXA; ++a) {
      if (a < most) {
        racc[a] = group_sum_butterfly<LANES>(racc[a], full);
        macc[a] = group_sum_butterfly<LANES>(macc[a], full);
      }
    }
#pragma unroll
    for (int p = 0; p < PER; ++p) {
      r[p] = m[p] = T(0);
#pragma unroll
      for (int a = 0; a < MAXA; ++a)
        if (a == lane + p * LANES) { r[p] = racc[a]; m[p] = macc[a]; }
    }
  }
  // alternating updates: the other player's sets only pass their values up
  const bool live = upd & (p2 ? 2 : 1);
  T pos[PER];
#pragma unroll
  for (int p = 0; p < PER; ++p) {
    const int a = lane + p * LANES;
    double x = 0.0;
    if (live && a < na) {
      if constexpr (LANES >= MAXA) {
        double Rn, Sn;
        x = slot_terms(hd.R, hd.S, as_double(r[p]), as_double(m[p]), wt, rule, Rn, Sn);
        st.R[sb + a] = Rn;
        st.avg[sb + a] = Sn;
      } else {
        x = slot_update(st.R, st.avg, sb + a, as_double(r[p]), as_double(m[p]), wt, rule);
      }
    }
    if constexpr (sizeof(T) == 8) pos[p] = x;
    else pos[p] = narrow_pos(x);
  }
  T tot = T(0);  // in action order; slots past the set's add zero
#pragma unroll
  for (int a = 0; a < MAXA; ++a)
    if (a < most) tot += __shfl_sync(full, pos[a / LANES], a % LANES, LANES);
#pragma unroll
  for (int p = 0; p < PER; ++p) {
    const int a = lane + p * LANES;
    if (live && a < na) st.sigma[sb + a] = match(pos[p], tot, na);
  }
}

template <typename T, int MAXA, int LANES, bool PERSIST>
__device__ __forceinline__ void bwd_set(const GameView &g, const StateView<T> &st, const SetHead<T, MAXA> &hd, bool p2,
                                        int lane, unsigned mask, double wt, int rule, int upd, double *rows) {
  const int32_t sb = hd.sb, na = hd.na, m0 = hd.m0, m1 = hd.m1, vb = hd.vb;
  const MemberRanks mr = hd.mr;
  const T(&sig)[MAXA] = hd.sig;
  T racc[MAXA], macc[MAXA];
#pragma unroll
  for (int a = 0; a < MAXA; ++a) {
    racc[a] = T(0);
    macc[a] = T(0);
  }
  constexpr bool CHAINS = kChains<T, MAXA, LANES>;
  double acc[kChainAcc<MAXA, LANES>];  // CHAINS: this lane's chains instead of racc, macc
#pragma unroll
  for (int i = 0; i < kChainAcc<MAXA, LANES>; ++i) acc[i] = 0.0;
  auto add_chunk = [&](int32_t cnt, const T(&d)[MAXA], const T(&mm)[MAXA]) {
    if constexpr (CHAINS) accumulate_chains<MAXA, LANES>(rows, cnt, na, mask, d, mm, acc);
    else accumulate_chunk<T, MAXA, LANES>(cnt, na, mask, d, mm, racc, macc);
  };
  constexpr bool TWO = MAXA <= 8 && LANES <= 8;  // narrow groups keep two chunks in flight
  int32_t k0 = m0;
  if constexpr (TWO) {
    if (k0 + LANES < m1) {
      int32_t ps0, ir0, ps1, ir1;
      member_idx(g, k0 + lane, m1, mr, ps0, ir0);
      member_idx(g, k0 + LANES + lane, m1, mr, ps1, ir1);
      for (; k0 + LANES < m1; k0 += 2 * LANES) {
        int32_t qs0, jr0, qs1, jr1;  // the next step's indices
        member_idx(g, k0 + 2 * LANES + lane, m1, mr, qs0, jr0);
        member_idx(g, k0 + 3 * LANES + lane, m1, mr, qs1, jr1);
        T d0[MAXA], mm0[MAXA], d1[MAXA], mm1[MAXA];
        member_data<T, MAXA, PERSIST>(g, st, k0 + lane, m0, m1, vb, na, p2, sig, ps0, ir0, d0, mm0);
        member_data<T, MAXA, PERSIST>(g, st, k0 + LANES + lane, m0, m1, vb, na, p2, sig, ps1, ir1, d1, mm1);
        add_chunk(LANES, d0, mm0);
        const int32_t c1 = (m1 - k0 - LANES) < LANES ? (m1 - k0 - LANES) : LANES;
        add_chunk(c1, d1, mm1);
        ps0 = qs0; ir0 = jr0; ps1 = qs1; ir1 = jr1;
      }
    }
  }
  if constexpr (TWO) {  // the last chunk
    for (; k0 < m1; k0 += LANES) {
      T d[MAXA], mm[MAXA];
      member_terms<T, MAXA, PERSIST>(g, st, k0 + lane, m0, m1, mr, vb, na, p2, sig, d, mm);
      const int32_t cnt = (m1 - k0) < LANES ? (m1 - k0) : LANES;
      add_chunk(cnt, d, mm);
    }
  } else {
    int32_t ps, ir;
    member_idx(g, k0 + lane, m1, mr, ps, ir);
    for (; k0 < m1; k0 += LANES) {
      int32_t qs, jr;  // the next step's indices
      member_idx(g, k0 + LANES + lane, m1, mr, qs, jr);
      T d[MAXA], mm[MAXA];
      member_data<T, MAXA, PERSIST>(g, st, k0 + lane, m0, m1, vb, na, p2, sig, ps, ir, d, mm);
      const int32_t cnt = (m1 - k0) < LANES ? (m1 - k0) : LANES;
      add_chunk(cnt, d, mm);
      ps = qs; ir = jr;
    }
  }
  // alternating updates: the other player's sets only pass their values up
  if (!(upd & (p2 ? 2 : 1))) return;
  if constexpr (sizeof(T) == 4) {
#pragma unroll
    for (int a = 0; a < MAXA; ++a) {
      if (a < na) {
        racc[a] = group_sum_butterfly<LANES>(racc[a], mask);
        macc[a] = group_sum_butterfly<LANES>(macc[a], mask);
      }
    }
  }
  // every lane now holds the set's totals racc[a], macc[a] (CHAINS: its own
  // chains' totals)
  if constexpr (CHAINS && LANES < MAXA) {  // more actions than lanes are possible: every lane takes all totals
#pragma unroll
    for (int a = 0; a < MAXA; ++a) {
      racc[a] = __shfl_sync(mask, acc[a / LANES], a % LANES, LANES);
      macc[a] = __shfl_sync(mask, acc[(MAXA + a) / LANES], (MAXA + a) % LANES, LANES);
    }
  }
  if (na <= LANES) {
    // lane a updates slot a (slot_update), then sigma^{t+1} = RM; the sum of
    // positive parts runs in action order
    T r = T(0), m = T(0);
    if constexpr (CHAINS && LANES >= MAXA) {
      r = acc[0];
      if constexpr (MAXA % LANES == 0) m = acc[MAXA / LANES];
      else m = __shfl_sync(mask, acc[0], (lane + MAXA) & (LANES - 1), LANES);
    } else {
#pragma unroll
      for (int a = 0; a < MAXA; ++a)
        if (a == lane) { r = racc[a]; m = macc[a]; }
    }
    double pos = 0.0;
    if (LANES >= MAXA) {
      if (lane < na) {
        double Rn, Sn;
        pos = slot_terms(hd.R, hd.S, as_double(r), as_double(m), wt, rule, Rn, Sn);
        st.R[sb + lane] = Rn;
        st.avg[sb + lane] = Sn;
      }
    } else if (lane < na) {
      pos = slot_update(st.R, st.avg, sb + lane, as_double(r), as_double(m), wt, rule);
    }
    if constexpr (sizeof(T) == 8) {
      double tot = 0.0;
      for (int a = 0; a < na; ++a) tot += __shfl_sync(mask, pos, a, LANES);
      if (lane < na) st.sigma[sb + lane] = match(pos, tot, na);
    } else {
      const float pf = narrow_pos(pos);
      float tot = 0.f;
      for (int a = 0; a < na; ++a) tot += __shfl_sync(mask, pf, a, LANES);
      if (lane < na) st.sigma[sb + lane] = match(pf, tot, na);
    }
  } else if (lane == 0) {
    T pos[MAXA];
    T tot = T(0);
#pragma unroll
    for (int a = 0; a < MAXA; ++a) {
      if (a < na) {
        const double x = slot_update(st.R, st.avg, sb + a, as_double(racc[a]), as_double(macc[a]), wt, rule);
        if constexpr (sizeof(T) == 8) pos[a] = x;
        else pos[a] = narrow_pos(x);
        tot += pos[a];
      }
    }
#pragma unroll
    for (int a = 0; a < MAXA; ++a)
      if (a < na) st.sigma[sb + a] = match(pos[a], tot, na);
  }
}

template <typename T, int MAXA, int LANES, bool PERSIST>
__device__ __forceinline__ void bwd_set(const GameView &g, const StateView<T> &st, int32_t I, bool p2, int lane,
                                        unsigned mask, double wt, int rule, int upd, double *rows) {
  SetHead<T, MAXA> hd;
  load_head<T, MAXA, LANES, PERSIST>(g, st, I, lane, hd);
  bwd_set<T, MAXA, LANES, PERSIST>(g, st, hd, p2, lane, mask, wt, rule, upd, rows);
}

// One information set per block, for depths with few sets of hundreds of
// members each: all kThreads threads load members tid, tid + kThreads, ...
// at once. P64: each chunk's member terms are staged in shared memory and
// thread a adds column a in ascending member order, the order the group form
// uses, so the result is bitwise the same; P32: per-thread partial sums
// finished by a fixed-shape tree. The slot update runs one thread per action.
template <typename T, int MAXA>
__device__ __forceinline__ void bwd_set_block(const GameView &g, const StateView<T> &st, int32_t I, bool p2,
                                              double wt, int rule, int upd) {
  __shared__ T s_d[kThreads * MAXA], s_m[kThreads * MAXA];  // [member][action]
  __shared__ double s_pos[MAXA];
  const int tid = threadIdx.x;
  const int32_t sb = __ldg(g.iset_slot + I);
  const int32_t na = __ldg(g.iset_slot + I + 1) - sb;
  const int32_t m0 = __ldg(g.iset_mem + I), m1 = __ldg(g.iset_mem + I + 1);
  const int32_t vb = __ldg(g.iset_vb + I);
  const MemberRanks mr = member_ranks(g, I, m0);
  T sig[MAXA], racc[MAXA], macc[MAXA];
#pragma unroll
  for (int a = 0; a < MAXA; ++a) {
    sig[a] = a < na ? st.sigma[sb + a] : T(0);
    racc[a] = T(0);
    macc[a] = T(0);
  }
  T r = T(0), m = T(0);  // P64: r is chain tid's running sum (tid < 2 MAXA)
  int32_t ps, ir;
  member_idx(g, m0 + tid, m1, mr, ps, ir);
  for (int32_t k0 = m0; k0 < m1; k0 += kThreads) {
    int32_t qs, jr;  // the next chunk's indices
    member_idx(g, k0 + kThreads + tid, m1, mr, qs, jr);
    T d[MAXA], mm[MAXA];
    member_data<T, MAXA, false>(g, st, k0 + tid, m0, m1, vb, na, p2, sig, ps, ir, d, mm);
    ps = qs;
    ir = jr;
    if constexpr (sizeof(T) == 8) {
#pragma unroll
      for (int a = 0; a < MAXA; ++a) {
        s_d[tid * MAXA + a] = d[a];
        s_m[tid * MAXA + a] = mm[a];
      }
      __syncthreads();
      if (tid < 2 * MAXA) {  // one chain a thread: the regret columns, then the average columns
        const int cnt = (m1 - k0) < kThreads ? (m1 - k0) : kThreads;
        const T *col = tid < MAXA ? s_d + tid : s_m + (tid - MAXA);
        for (int j = 0; j < cnt; ++j) r = r + col[j * MAXA];
      }
      __syncthreads();
    } else {
#pragma unroll
      for (int a = 0; a < MAXA; ++a) {
        racc[a] += d[a];
        macc[a] += mm[a];
      }
    }
  }
  if (!(upd & (p2 ? 2 : 1))) return;  // alternating updates: values only (uniform over the block)
  if constexpr (sizeof(T) == 4) {
#pragma unroll
    for (int a = 0; a < MAXA; ++a) {
      s_d[tid * MAXA + a] = racc[a];
      s_m[tid * MAXA + a] = macc[a];
    }
    __syncthreads();
    for (int off = kThreads / 2; off > 0; off >>= 1) {
      if (tid < off) {
#pragma unroll
        for (int a = 0; a < MAXA; ++a) {
          s_d[tid * MAXA + a] += s_d[(tid + off) * MAXA + a];
          s_m[tid * MAXA + a] += s_m[(tid + off) * MAXA + a];
        }
      }
      __syncthreads();
    }
    if (tid < na) {
      r = s_d[tid];
      m = s_m[tid];
    }
  }
  if constexpr (sizeof(T) == 8) {  // thread a takes its average chain's total
    __syncthreads();
    if (tid >= MAXA && tid < 2 * MAXA) s_m[tid - MAXA] = r;
    __syncthreads();
    if (tid < na) m = s_m[tid];
  }
  // thread a updates slot a (slot_update), then sigma^{t+1} = RM with the
  // positive parts summed in action order
  double pos = 0.0;
  if (tid < na) {
    pos = slot_update(st.R, st.avg, sb + tid, as_double(r), as_double(m), wt, rule);
    s_pos[tid] = pos;
  }
  __syncthreads();
  if (tid < na) {
    if constexpr (sizeof(T) == 8) {
      double tot = 0.0;
      for (int a = 0; a < na; ++a) tot += s_pos[a];
      st.sigma[sb + tid] = match(pos, tot, na);
    } else {
      float tot = 0.f;
      for (int a = 0; a < na; ++a) tot += narrow_pos(s_pos[a]);
      st.sigma[sb + tid] = match(narrow_pos(pos), tot, na);
    }
  }
  __syncthreads();  // shared arrays are reused by the block's next set
}

// Grid: nb_chance blocks over narrow chance nodes, then one block per wide
// chunk, then the information-set groups (LANES == kThreads: one set per
// block). early: the first set of every group is read up before waiting for
// the launch before, which writes nothing of this depth but its children's
// values or its members' reach. spread: the depth has fewer warps of sets than
// blocks could hold, and each block takes one warp's sets before any takes two
// (in FP64 eight warps on an SM wait for its one FP64 pipe: a depth of
// 153 sets of 120 members 34 us -> 25).
constexpr int kBwdEarly = 1, kBwdSpread = 2;
template <typename T, int MAXA, int LANES>
__global__ void __launch_bounds__(kThreads, MAXA > 8 ? 1 : (MAXA <= 4 ? 4 : 3) - (sizeof(T) == 8 ? 1 : 0)) bwd_level_kernel(GameView g, StateView<T> st, LevelWork w,
                                                            int nb_chance, int rule, int upd, int bump_t,
                                                            int flags) {
  const bool early = flags & kBwdEarly;
  const int nb_wide = w.wc1 - w.wc0;
  if ((int)blockIdx.x < nb_chance) {
    pdl_enter();
    const int32_t stride = nb_chance * blockDim.x;
    for (int32_t i = w.ch0 + blockIdx.x * blockDim.x + threadIdx.x; i < w.ch1; i += stride)
      bwd_chance<T, false>(g, st.v, i);
  } else if ((int)blockIdx.x < nb_chance + nb_wide) {
    pdl_enter();
    bwd_wide_chunk<T, false>(g, w, st.v, w.wc0 + (int32_t)blockIdx.x - nb_chance);
  } else if constexpr (LANES == kThreads) {
    pdl_enter();
    const int first = nb_chance + nb_wide;
    const double wt = avg_weight(*st.t + 1, rule);
    for (int32_t I = w.is0 + ((int)blockIdx.x - first); I < w.is1; I += (int)gridDim.x - first)
      bwd_set_block<T, MAXA>(g, st, I, I >= w.is2, wt, rule, upd);
  } else {
    constexpr int GPB = kThreads / LANES;
    const int first = nb_chance + nb_wide;
    const int blk = (int)blockIdx.x - first, nblk = (int)gridDim.x - first;
    const int gid = flags & kBwdSpread
                        ? ((int)threadIdx.x / 32 * nblk + blk) * (32 / LANES) + (int)(threadIdx.x % 32) / LANES
                        : blk * GPB + (int)threadIdx.x / LANES;
    const int ngroups = nblk * GPB;
    const int lane = threadIdx.x % LANES;
    const unsigned mask = group_mask<LANES>();
    __shared__ double s_rows[kThreads / 32][kChainDoubles<T, MAXA, LANES>];
    int32_t I = w.is0 + gid;
    int32_t Iw = I;  // in step: every lane stays while the warp's first set is one
    if constexpr (kInStep<T, MAXA, LANES>) Iw = I - (int)(threadIdx.x % 32) / LANES;
    SetHead<T, MAXA> hd = {};
    if (!early) pdl_enter();
    if (I < w.is1) load_head<T, MAXA, LANES, false>(g, st, I, lane, hd);
    if (early) pdl_enter();
    const double wt = avg_weight(*st.t + 1, rule);
    while (Iw < w.is1) {
      if constexpr (kInStep<T, MAXA, LANES>)
        bwd_sets<T, MAXA, LANES>(g, st, hd, I >= w.is2, lane, wt, rule, upd, s_rows[threadIdx.x / 32]);
      else
        bwd_set<T, MAXA, LANES, false>(g, st, hd, I >= w.is2, lane, mask, wt, rule, upd, s_rows[threadIdx.x / 32]);
      I += ngroups;
      Iw += ngroups;
      if (kInStep<T, MAXA, LANES>) hd = {};
      if (I < w.is1) load_head<T, MAXA, LANES, false>(g, st, I, lane, hd);
    }
  }
  if (bump_t) {  // depth 0 holds only the root: no other block reads t here
    __syncthreads();
    if (blockIdx.x == 0 && threadIdx.x == 0) *st.t += 1;
  }
}

static __global__ void bump_t_kernel(long long *t, long long n) { *t += n; }

// ------------------------------------------------------- persistent form
__device__ __forceinline__ unsigned ld_acquire_gpu(const unsigned *p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_release_gpu(unsigned *p, unsigned v) {
  asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

struct Barrier {
  unsigned *count;     // arrivals at the current barrier
  unsigned *gen;       // generation, bumped by the last arrival
  int *err;            // set to 1 when a wait gives up
  long long spin_limit;
  unsigned expected;   // arrivals that complete a barrier (gridDim.x normally)
};

// Grid-wide barrier with a bounded wait: returns false (and sets *err) when
// the spin budget runs out, or when another block has reported an error.
__device__ __forceinline__ bool grid_sync(const Barrier &b) {
  __shared__ int s_ok;
  __syncthreads();
  if (gridDim.x == 1 && b.expected == 1) return true;
  if (threadIdx.x == 0) {
    __threadfence();
    const unsigned g0 = ld_acquire_gpu(b.gen);
    const unsigned arrived = atomicAdd(b.count, 1u) + 1u;
    int ok = 1;
    if (arrived == b.expected) {
      atomicExch(b.count, 0u);
      __threadfence();
      st_release_gpu(b.gen, g0 + 1u);
    } else {
      long long spins = 0;
      while (ld_acquire_gpu(b.gen) == g0) {
        if (++spins > b.spin_limit) {
          atomicExch(b.err, 1);
          ok = 0;
          break;
        }
        __nanosleep(64);
      }
    }
    if (ok && *(volatile int *)b.err != 0) ok = 0;
    __threadfence();
    s_ok = ok;
  }
  __syncthreads();
  return s_ok != 0;
}

template <typename T> struct PersistArgs {
  GameView g;
  StateView<T> st;
  const LevelWork *lw;
  int D;
  int rule;
  int order;  // 0 simultaneous, 1 alternating (two half-iterations)
  long long n_iter;
  Barrier bar;
};

// All n iterations in one launch; depth levels separated by grid barriers
// (2D barriers per iteration, 4D under alternating updates). The grid is
// co-resident (cooperative launch).
template <typename T, int MAXA, int LANES>
__global__ void __launch_bounds__(kThreads) persistent_kernel(PersistArgs<T> a) {
  const long long t0 = __ldcg(a.st.t);
  const int tid = blockIdx.x * blockDim.x + threadIdx.x;
  const int nthr = gridDim.x * blockDim.x;
  const int gid = tid / LANES, ngroups = nthr / LANES, lane = tid % LANES;
  const unsigned mask = group_mask<LANES>();
  const int halves = a.order ? 2 : 1;  // alternating: player 1's half, then player 2's
  __shared__ double s_rows[kThreads / 32][kChainDoubles<T, MAXA, LANES>];
  for (long long it = 0; it < a.n_iter; ++it) {
    const double wt = avg_weight(t0 + it + 1, a.rule);
    for (int hf = 0; hf < halves; ++hf) {
      const int upd = a.order ? (1 << hf) : 3;
      for (int d = 0; d < a.D; ++d) {
        const LevelWork w = a.lw[d];
        if (a.g.int_edge) {  // member order: depth d + 1 pulls
          if (d + 1 < a.D) {
            const int32_t qe = a.lw[d + 1].ie;
            for (int32_t q = a.lw[d + 1].ib + tid; q < qe; q += kPull * nthr)
              fwd_pull<T, true>(a.g, a.st.sigma, a.st.reach, q, nthr, qe);
          }
        } else {
          for (int32_t qw = w.ib + (tid & ~31); qw < w.ie; qw += 4 * nthr) {
            if (w.fan) fwd_int4<T, true, true>(a.g, a.st.sigma, a.st.reach, qw + (tid & 31), nthr, w.ie);
            else fwd_int4<T, true, false>(a.g, a.st.sigma, a.st.reach, qw + (tid & 31), nthr, w.ie);
          }
          for (int32_t q = w.wc0 + blockIdx.x; q < w.wc1; q += gridDim.x) fwd_wide_chunk<T, true>(a.g, w, a.st.reach, q);
        }
        if (!grid_sync(a.bar)) return;
      }
      for (int d = a.D - 1; d >= 0; --d) {
        const LevelWork w = a.lw[d];
        if (d > 0) {  // a chance root's value has no reader in an iteration
          for (int32_t i = w.ch0 + tid; i < w.ch1; i += nthr) bwd_chance<T, true>(a.g, a.st.v, i);
          for (int32_t q = w.wc0 + blockIdx.x; q < w.wc1; q += gridDim.x) bwd_wide_chunk<T, true>(a.g, w, a.st.v, q);
        }
        for (int32_t I = w.is0 + gid; I < w.is1; I += ngroups)
          bwd_set<T, MAXA, LANES, true>(a.g, a.st, I, I >= w.is2, lane, mask, wt, a.rule, upd, s_rows[threadIdx.x / 32]);
        if (!grid_sync(a.bar)) return;
      }
    }
  }
  if (tid == 0) *a.st.t = t0 + a.n_iter;
}

// ---------------------------------------------------------- state set-up
template <typename T>
__global__ void init_state_kernel(const int32_t *iset_slot, int32_t n_sets, T *sigma, double *R, double *avg,
                                  int32_t A, long long *t, vec2_t<T> *reach, double2 *reach2) {
  const int32_t stride = gridDim.x * blockDim.x;
  const int32_t tid = blockIdx.x * blockDim.x + threadIdx.x;
  for (int32_t q = tid; q < A; q += stride) { R[q] = 0.0; avg[q] = 0.0; }
  for (int32_t I = tid; I < n_sets; I += stride) {
    const int32_t sb = iset_slot[I], na = iset_slot[I + 1] - sb;
    const T u = T(1) / (T)na;  // RM of zero regret
    for (int32_t a = 0; a < na; ++a) sigma[sb + a] = u;
  }
  if (tid == 0) {
    *t = 0;
    vec2_t<T> one;
    one.x = T(1); one.y = T(1);
    reach[0] = one;  // root reach of both lanes (never overwritten)
    reach2[0] = make_double2(1.0, 1.0);
  }
}

// Every value slot from the template in slot order: terminals get
// pi_c(z) u(z) (eq. (template)), internal nodes 0 (overwritten by every
// backward pass before their parents read them).
template <typename T>
__global__ void init_values_kernel(const double *tmpl_vs, int32_t N, T *v, double2 *vb, double *vavg) {
  const int32_t stride = gridDim.x * blockDim.x;
  for (int32_t h = blockIdx.x * blockDim.x + threadIdx.x; h < N; h += stride) {
    const double x = tmpl_vs[h];
    v[h] = (T)x;
    vb[h] = make_double2(x, x);
    vavg[h] = x;
  }
}

// sigma from R by regret matching (used after a state upload)
template <typename T>
__global__ void rm_kernel(const int32_t *iset_slot, int32_t n_sets, const double *R, T *sigma) {
  const int32_t stride = gridDim.x * blockDim.x;
  for (int32_t I = blockIdx.x * blockDim.x + threadIdx.x; I < n_sets; I += stride) {
    const int32_t sb = iset_slot[I], na = iset_slot[I + 1] - sb;
    double tot = 0.0;
    for (int32_t a = 0; a < na; ++a) tot += R[sb + a] > 0.0 ? R[sb + a] : 0.0;
    for (int32_t a = 0; a < na; ++a) {
      const double p = R[sb + a] > 0.0 ? R[sb + a] : 0.0;
      sigma[sb + a] = (T)(tot > 0.0 ? p / tot : 1.0 / (double)na);
    }
  }
}

// ------------------------------------------------------------- read-out
// The average strategy of every set (uniform where its sum is zero) into
// out[to[q]] for slot q, or out[q] without `to`. A lane a slot: what bounds it
// is the FP64 division (137 cycles a warp and SM), so each slot has one. LANES
// = 1: one thread a set, for sets of more than 8 actions.
template <int LANES>
__global__ void __launch_bounds__(kThreads) avg_strategy_kernel(const int32_t *iset_slot, int32_t n_sets,
                                                                const double *avg, const int32_t *to, double *out) {
  const int32_t groups = gridDim.x * blockDim.x / LANES;
  const int lane = threadIdx.x % LANES;
  for (int32_t I = (blockIdx.x * blockDim.x + threadIdx.x) / LANES; I < n_sets; I += groups) {
    const int32_t sb = iset_slot[I], na = iset_slot[I + 1] - sb;
    if constexpr (LANES > 1) {
      const double x = lane < na ? avg[sb + lane] : 0.0;
      double tot = 0.0;  // in action order
#pragma unroll
      for (int a = 0; a < LANES; ++a) {
        const double y = __shfl_sync(group_mask<LANES>(), x, a, LANES);
        if (a < na) tot += y;
      }
      if (lane < na) out[to ? to[sb + lane] : sb + lane] = match(x, tot, na);
    } else {
      double tot = 0.0;
      for (int32_t a = 0; a < na; ++a) tot += avg[sb + a];
      for (int32_t a = 0; a < na; ++a) out[to ? to[sb + a] : sb + a] = match(avg[sb + a], tot, na);
    }
  }
}

// The current strategy in spec slot order: out[to[q]] = sigma[q].
template <typename T>
__global__ void __launch_bounds__(kThreads) current_strategy_kernel(const T *sigma, const int32_t *to, double *out,
                                                                    int32_t A) {
  const int32_t stride = gridDim.x * blockDim.x;
  for (int32_t q = blockIdx.x * blockDim.x + threadIdx.x; q < A; q += stride) out[to[q]] = as_double(sigma[q]);
}

// ------------------------------------------------ exact best response (FP64)
// Lane x of vb: player 1 best-responds (maximises), player 2 plays the
// average. Lane y: player 2 best-responds (minimises player 1's payoff),
// player 1 plays the average. vavg: both play the average. All values are
// chance-weighted (eq. (template)), so the counterfactual weight of a member
// is the opponent's reach under the average strategy alone.
// Wide chance node, best-response values: chunk partials of (x, y, avg),
// finished in chunk order by the last block (as bwd_wide_chunk).
__device__ __forceinline__ void br_wide_chunk(const GameView &g, const LevelWork &w, double2 *vb, double *vavg,
                                              int32_t q) {
  const int32_t wi = wide_of_chunk(g, w, q);
  const int32_t h = __ldg(g.wide_vs + wi);
  const int32_t cb = __ldg(g.wide_vb + wi), ce = cb + __ldg(g.wide_nch + wi);
  const int32_t q0 = __ldg(g.wide_chunk + wi), nq = __ldg(g.wide_chunk + wi + 1) - q0;
  const int32_t c0 = cb + (q - q0) * kWideChunkK, c1 = min(ce, c0 + kWideChunkK);
  double x[3] = {0.0, 0.0, 0.0};
  for (int32_t c = c0 + threadIdx.x; c < c1; c += blockDim.x) {
    const double2 y = vb[c];
    x[0] += y.x; x[1] += y.y; x[2] += vavg[c];
  }
  block_sum(x);
  __shared__ unsigned s_ticket;
  if (threadIdx.x == 0) {
    g.wide_part[3 * q] = x[0]; g.wide_part[3 * q + 1] = x[1]; g.wide_part[3 * q + 2] = x[2];
    __threadfence();
    s_ticket = atomicAdd(g.wide_cnt + wi, 1u);
  }
  __syncthreads();
  if (s_ticket == (unsigned)(nq - 1)) {  // the last chunk's block adds the partials (fixed shape)
    __threadfence();
    double y[3] = {0.0, 0.0, 0.0};
    for (int32_t k = threadIdx.x; k < nq; k += blockDim.x)
#pragma unroll
      for (int i = 0; i < 3; ++i) y[i] += __ldcg(g.wide_part + 3 * (q0 + k) + i);
    block_sum(y);
    if (threadIdx.x == 0) {
      vb[h] = make_double2(y[0], y[1]);
      vavg[h] = y[2];
      g.wide_cnt[wi] = 0u;
    }
  }
}

// A double's place in the order of its values as an integer (both zeros the
// same): FP64 compares run on the slow FP64 pipe.
__device__ __forceinline__ long long order_key(double x) {
  const long long b = __double_as_longlong(x);
  return (b << 1) == 0 ? 0 : b ^ ((b >> 63) & 0x7fffffffffffffffll);
}

// Narrow chance node i, best-response values: left to right.
template <bool PERSIST>
__device__ __forceinline__ void br_chance(const GameView &g, double2 *vb, double *vavg, int32_t i) {
  const int32_t h = __ldg(g.ch_vs + i);
  const int32_t cb = __ldg(g.ch_vb + i), ce = cb + __ldg(g.ch_nch + i);
  double sx = 0.0, sy = 0.0, sa = 0.0;
  for (int32_t c = cb; c < ce; ++c) {
    const double2 x = ldm<PERSIST>(vb + c);
    sx += x.x; sy += x.y; sa += ldm<PERSIST>(vavg + c);
  }
  vb[h] = make_double2(sx, sy);
  vavg[h] = sa;
}

// One information set's best response, by the LANES lanes of one group. The
// FP64 pipe (a warp instruction every 16-19 cycles an SM) bounds it: every
// member and action takes three fused multiply-adds, each lane sums its own
// members' action values, and the group's sums are finished by a shared-out
// butterfly, so nothing is added twice. A lane keeps its last kBrKeep members'
// action values in registers until the best action is known and writes both
// of a member's values at once; members before those write the other lane's
// value on the way and take a second pass over the best action's children.
// Best responses to a strategy of the 11M-node card game: 893 -> 269 us (every
// lane used to add every member's value, and the launches to wait for one
// another's end; 285 with one member kept).
template <int MAXA> constexpr int kBrKeep = MAXA <= 4 ? 4 : (MAXA <= 8 ? 2 : 1);

template <int MAXA, int LANES, bool PERSIST>
__device__ __forceinline__ void br_set(const GameView &g, const double2 *reach2, const double *sbs, double2 *vb,
                                       double *vavg, int32_t I, int p, int lane, unsigned mask) {
  constexpr int KEEP = kBrKeep<MAXA>;
  const int32_t sb = __ldg(g.iset_slot + I), na = __ldg(g.iset_slot + I + 1) - sb;
  const int32_t m0 = __ldg(g.iset_mem + I), M = __ldg(g.iset_mem + I + 1) - m0;
  const MemberRanks mr = member_ranks(g, I, m0);
  const int32_t vb0 = __ldg(g.iset_vb + I);
  double sg[MAXA], Q[MAXA];
#pragma unroll
  for (int a = 0; a < MAXA; ++a) { sg[a] = a < na ? ldm<PERSIST>(sbs + sb + a) : 0.0; Q[a] = 0.0; }
  // one member (k < M): its value slot, the other lane's value, and its own
  // player's values of the actions
  auto member = [&](int32_t k, double (&own)[MAXA], double &oth) {
    const int32_t h = __ldg(g.mem_vs + m0 + k);
    const double2 r = ldm<PERSIST>(reach2 + member_rank(g, m0 + k, mr));
    constexpr int W = MAXA <= 8 ? MAXA : 4;  // actions whose loads are issued together
    const double po = p ? r.x : r.y;
    double va = 0.0;
    oth = 0.0;
#pragma unroll
    for (int a0 = 0; a0 < MAXA; a0 += W) {
      double2 x[W];
      double y[W];
#pragma unroll
      for (int j = 0; j < W; ++j) {
        if (a0 + j < na) {
          x[j] = ldm<PERSIST>(vb + vb0 + k + (a0 + j) * M);
          y[j] = ldm<PERSIST>(vavg + vb0 + k + (a0 + j) * M);
        }
      }
#pragma unroll
      for (int j = 0; j < W; ++j) {
        const int a = a0 + j;
        if (a < na) {
          own[a] = p ? x[j].y : x[j].x;
          Q[a] = fma(po, own[a], Q[a]);
          oth = fma(sg[a], p ? x[j].x : x[j].y, oth);
          va = fma(sg[a], y[j], va);
        }
      }
    }
    vavg[h] = va;
    return h;
  };
  const int32_t chunks = (M + LANES - 1) / LANES;
  const int32_t kept = chunks > KEEP ? (chunks - KEEP) * LANES : 0;  // first member that is kept
  for (int32_t k = lane; k < kept; k += LANES) {
    double own[MAXA], oth;
    const int32_t h = member(k, own, oth);
    reinterpret_cast<double *>(vb + h)[1 - p] = oth;
  }
  double own[KEEP][MAXA], oth[KEEP];
  int32_t h[KEEP];
#pragma unroll
  for (int c = 0; c < KEEP; ++c) {
    const int32_t k = kept + c * LANES + lane;
    h[c] = -1;
    if (k < M) h[c] = member(k, own[c], oth[c]);
  }
  int best = 0;
  if constexpr (MAXA <= 8) {
    group_sum_scatter<LANES, MAXA>(Q, lane, mask);
    constexpr int STEP = MAXA <= LANES ? LANES / MAXA : 1, PER = MAXA <= LANES ? 1 : MAXA / LANES;
    long long top = 0;
#pragma unroll
    for (int a = 0; a < MAXA; ++a) {
      long long q = __shfl_sync(mask, order_key(Q[a % PER]), a / PER * STEP, LANES);
      if (p) q = -q;
      if (a == 0 || (a < na && q > top)) { top = q; best = a; }
    }
  } else {
    long long top = 0;
#pragma unroll
    for (int a = 0; a < MAXA; ++a) {
      if (a < na) {
        long long q = order_key(group_sum_butterfly<LANES>(Q[a], mask));
        if (p) q = -q;
        if (a == 0 || q > top) { top = q; best = a; }
      }
    }
  }
  // the group's lanes hold the same sums, so best agrees across it
  for (int32_t k = lane; k < kept; k += LANES) {
    const int32_t hk = __ldg(g.mem_vs + m0 + k);
    const double2 x = ldm<PERSIST>(vb + vb0 + k + best * M);
    reinterpret_cast<double *>(vb + hk)[p] = p ? x.y : x.x;
  }
#pragma unroll
  for (int c = 0; c < KEEP; ++c) {
    if (h[c] >= 0) {
      double mine = own[c][0];
#pragma unroll
      for (int a = 1; a < MAXA; ++a)
        if (a == best) mine = own[c][a];
      vb[h[c]] = p ? make_double2(oth[c], mine) : make_double2(mine, oth[c]);
    }
  }
}

template <int MAXA, int LANES>
__global__ void __launch_bounds__(kThreads) br_level_kernel(GameView g, const double2 *reach2, const double *sbs,
                                                           double2 *vb, double *vavg, LevelWork w, int nb_chance) {
  pdl_enter();
  const int nb_wide = w.wc1 - w.wc0;
  if ((int)blockIdx.x >= nb_chance && (int)blockIdx.x < nb_chance + nb_wide) {
    br_wide_chunk(g, w, vb, vavg, w.wc0 + (int32_t)blockIdx.x - nb_chance);
    return;
  }
  if ((int)blockIdx.x < nb_chance) {
    const int32_t stride = nb_chance * blockDim.x;
    for (int32_t i = w.ch0 + blockIdx.x * blockDim.x + threadIdx.x; i < w.ch1; i += stride)
      br_chance<false>(g, vb, vavg, i);
    return;
  }
  constexpr int GPB = kThreads / LANES;
  const int first = nb_chance + nb_wide;
  const int gid = ((int)blockIdx.x - first) * GPB + (int)threadIdx.x / LANES;
  const int ngroups = ((int)gridDim.x - first) * GPB;
  const int lane = threadIdx.x % LANES;
  const unsigned mask = group_mask<LANES>();
  for (int32_t I = w.is0 + gid; I < w.is1; I += ngroups)
    br_set<MAXA, LANES, false>(g, reach2, sbs, vb, vavg, I, I >= w.is2 ? 1 : 0, lane, mask);
}

// The root's best-response values as one record: exploitability, both best
// responses, the value of the average strategies.
static __global__ void br_result_kernel(const double2 *vb, const double *vavg, int32_t root, double *out) {
  pdl_enter();
  const double2 x = vb[root];
  out[0] = 0.5 * (x.x - x.y);
  out[1] = x.x;
  out[2] = x.y;
  out[3] = vavg[root];
}

}  // namespace cfr
