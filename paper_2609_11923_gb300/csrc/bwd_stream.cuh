// bwd_stream.cuh — the FP32 backward pass of one depth with its inputs
// streamed into shared memory by the bulk-copy (TMA) engine.
//
// Same arithmetic as bwd_set (eqs. (opbwd), (instregret), (regret), (rm), the
// CFR+ clamp; Algorithm 1), different data movement. In member order the
// information sets of a depth are a contiguous range and so is everything a
// run of consecutive sets reads: their members' reach (one run, tiles
// interleaved inside it), their members' children's values (one run of value
// slots), their members' own value slots, their slots' strategy, regret and
// average, and their set descriptors. The host cuts each depth's sets into
// chunks of whole groups (a tile of four sets, or one untiled set); the
// depth's narrow chance nodes follow as chance chunks (consecutive nodes,
// whose children are one run of value slots, and their entries of the chance
// arrays). A CTA's warps form teams (StreamShape), and every team walks its
// own chunks through its own ring of kStreamStages stages: as soon as its
// threads are done with a chunk, one of its warps starts the cp.async.bulk
// copies of the next chunk but one into the same stage. No team waits for
// another, so the copies of some teams are in flight while others compute;
// the loads in flight cost no registers; the one scattered access left is
// each member's value write into its parent set's block.
//
// What bounds it: the largest depths are near what DRAM gives (a depth of 3.7M
// members, 93 MB: 31 us -> 26 with 8 warps on one group -> with teams), the
// others spend their time in the latencies of a group's few hundred
// instructions, which only independent warps hide. A set of 153 members is 5
// steps of one warp (19 for a tile of four); over eight warps it was one step
// that most lanes sat out, and the sums' shuffles cost more than the members.
// All depths of the 27M-node card game: an iteration of 230 us -> 131 (202 by
// lane groups, 161 with the best form of each depth); of the 11M-node one
// 110 by lane groups, 80 here.
//
// Work inside a chunk: the team takes one group at a time: thread t serves
// set j = t % G of the group (G = 4 for a tile, 1 otherwise) and members
// q = t / G, t / G + n / G, ... of that set (n threads in the team), so a
// warp reads a tile's reach as one contiguous run. Per-thread FP32 partial
// sums are finished by a fixed-shape butterfly within the warp and, in the
// warp whose turn the group is, a sum over the team's warps in order
// (deterministic run to run); that warp then updates the group's slots (one lane per slot) and
// writes sigma^{t+1}. The form pays where sets are long.
#pragma once
#include <algorithm>

#include "kernels.cuh"

namespace cfr {

constexpr int kStreamLanes = 512;                 // lanes_per_set code of this form
constexpr int kStreamStages = 2;                  // a team's ring
constexpr int kStreamStageBytes = 48 * 1024;      // bytes one chunk may stage at most
constexpr int kStreamPackBytes = 6 * 1024;        // groups are packed into a chunk up to this size,
constexpr int kStreamSpread = 16 * 152;           // as long as the depth makes this many chunks (one for each warp of a GB300's
                                                  // 152 SMs; games are compiled on hosts without a GPU to ask)
constexpr int kStreamChanceBytes = 1024;          // chance nodes are packed up to this size in any case
constexpr int kStreamSideBytes = 2048;            // bytes of a chunk's R, average sums and descriptors: bounds its sets (32 of
                                                  // two actions), which a team updates one group after another
constexpr int kStreamMaxWarps = 16;               // warps of a streaming CTA (one CTA per SM)
constexpr int kStreamMinWarps = 6;                // of a CTA of one-warp teams
constexpr int kStreamDynSmem = 216 * 1024;        // bytes of all teams' rings
constexpr int kStreamMinMembers = 32;             // mean members per set below which the autotuner does not try it
// Mean members per set from which a depth streams by default: of an untiled
// depth, and of a tiled one, which lane groups read worse. Iterations by lane
// groups / streamed from fewer members on: card games of 36 members a set
// 39 / 46 us, of 66-78 untiled 54 / 64, of 78 (tiled in the large depths) 62 /
// 54 with those depths streamed, of 105-120 105 / 80, of 153-171 202 / 131; an
// endgame of 97-99 33 / 27.
constexpr int kStreamAutoMembers = 96, kStreamAutoTiled = 64;
constexpr int kStreamChanceMax = 1024;            // chance nodes per chance chunk at most

// Per information set (member order), 32 bytes, read by the streaming form.
struct SetInfo {
  int32_t sb, na;        // first slot, actions
  int32_t m0, nm;        // first member, member count
  int32_t vb;            // first value slot of the block of its members' children
  int32_t rank0, rstep;  // reach rank of member 0 and the stride of its members' ranks
  int32_t flags;         // bits 0-2: G (sets in the group it starts: 1 or 4; 0 inside a tile); bit 8: player 2
};

// One chunk and the element ranges it stages, widened to 16-byte
// boundaries. A set chunk (kind kChunkSets): consecutive sets [I0, I1),
// reach ranks [ra, ra + nra) (even), value slots [va, va + nva), members
// [ka, ka + nka), slots [sa, sa + nsa) (multiples of 4). A chance chunk
// (kind kChunkChance): consecutive narrow chance nodes [I0, I1) of the
// depth, their children's value slots [va, va + nva) and their entries
// [ka, ka + nka) of the chance arrays (first child slot, child count, own
// value slot); ra = nra = sa = nsa = 0.
constexpr int32_t kChunkSets = 0, kChunkChance = 1;
struct StreamChunk {
  int32_t I0, I1;
  int32_t ra, nra;
  int32_t va, nva;
  int32_t ka, nka;
  int32_t sa, nsa;
  int32_t kind;
  int32_t pad[5];
};

static_assert(sizeof(SetInfo) == 32, "SetInfo is staged in 32-byte records");
static_assert(sizeof(StreamChunk) == 64, "StreamChunk is 64 bytes");

// Byte offsets of the staged arrays: what the members' work reads, then
// (from total on) what the slot updates read besides: R, then the average
// sums, 8 bytes a slot each. (s_*: the latter's sizes together with the
// descriptors', which kStreamSideBytes bounds; nothing is laid out by them.)
struct StreamLayout {
  uint32_t reach, val, mem, info, sig, total;
  uint32_t s_info, s_R, s_avg, s_total;
};

__host__ __device__ inline StreamLayout stream_layout(const StreamChunk &c) {
  StreamLayout L;
  const uint32_t nset = (uint32_t)sizeof(SetInfo) * (uint32_t)(c.I1 - c.I0);
  L.reach = 0;
  L.val = L.reach + 8u * (uint32_t)c.nra;
  L.mem = L.val + 4u * (uint32_t)c.nva;
  L.info = L.mem + 4u * (uint32_t)c.nka;
  L.sig = L.info + nset;
  L.total = L.sig + 4u * (uint32_t)c.nsa;
  L.s_info = 0;
  L.s_R = nset;
  L.s_avg = L.s_R + 8u * (uint32_t)c.nsa;
  L.s_total = L.s_avg + 8u * (uint32_t)c.nsa;
  return L;
}

__host__ __device__ inline bool stream_fits(const StreamLayout &L) {
  return L.total <= (uint32_t)kStreamStageBytes && L.s_total <= (uint32_t)kStreamSideBytes;
}

// Bytes of a set chunk's stage.
__host__ __device__ inline uint32_t stream_bytes(const StreamChunk &c) {
  return stream_layout(c).total + 16u * (uint32_t)c.nsa;
}

// A chance chunk's stage: the children's values, then its entries of the
// three chance arrays.
struct ChanceLayout {
  uint32_t vb, nch, vs, total;  // offsets of ch_vb, ch_nch, ch_vs entries; bytes
};

__host__ __device__ inline ChanceLayout chance_layout(const StreamChunk &c) {
  ChanceLayout L;
  L.vb = 4u * (uint32_t)c.nva;
  L.nch = L.vb + 4u * (uint32_t)c.nka;
  L.vs = L.nch + 4u * (uint32_t)c.nka;
  L.total = L.vs + 4u * (uint32_t)c.nka;
  return L;
}

__host__ __device__ inline bool chance_fits(const StreamChunk &c) {
  return c.nva > 0 && c.nka > 0 && c.I1 > c.I0 && chance_layout(c).total <= (uint32_t)kStreamStageBytes;
}

__device__ __forceinline__ uint32_t smem_u32(const void *p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}

// 1-D bulk copy global -> shared (16-byte aligned addresses, size a multiple
// of 16), completing `bytes` on the mbarrier.
__device__ __forceinline__ void bulk_g2s(uint32_t dst, const void *src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "l"(src), "r"(bytes), "r"(bar)
               : "memory");
}

// Bounded wait for the phase of the given parity: false when it gave up
// (about a second of polling).
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity) {
  long long t0 = 0;
  for (int it = 0; it < (1 << 26); ++it) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    if (ok) return true;
    if (it == 0) t0 = clock64();
    if (clock64() - t0 > 2000000000ll) break;  // about a second at the boost clock
  }
  return false;
}

__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

// How a depth's teams are laid out: teams of `warps` warps, `teams` of them in
// a CTA, stages of `bytes` bytes (at least the depth's largest chunk).
struct StreamShape {
  int32_t teams, warps, bytes;
};

// The stages take kStreamDynSmem bytes at most: as many teams as they hold, of
// one warp where that makes kStreamMinWarps and else of as many as a CTA's
// warps allow; larger teams too where the depth has too few chunks to give
// every team one. (Iterations: seven teams of one warp 131 us, of two 132, at
// depths of 13 KB tiles; three of five 488, two of eight 526, at 26 KB tiles
// of a 129M-node card game; at 33 KB of the 264M-node one 951 and 935. One
// warp doing all of a team's updates: 994 there. Groups packed into chunks of
// 6 KB at depths with fewer chunks than teams: 35 us instead of 27 for an
// endgame of a million edges.)
inline StreamShape stream_shape(int64_t largest, int64_t chunks, int sms) {
  StreamShape z;
  z.bytes = (int32_t)((largest + 127) / 128 * 128);
  z.teams = std::max(1, std::min(kStreamMaxWarps, kStreamDynSmem / (kStreamStages * z.bytes)));
  z.warps = z.teams >= kStreamMinWarps ? 1 : std::min(8, kStreamMaxWarps / z.teams);
  while (z.warps < 8 && z.teams > 1 && chunks <= (int64_t)sms * (z.teams / 2)) {
    z.teams /= 2;
    z.warps = std::min(8, kStreamMaxWarps / z.teams);
  }
  return z;
}

// What lane `lane` of a team's first warp copies of every chunk: copy lane of
// the stage, in the stage's order (set chunks: reach, values, members,
// descriptors, strategy, R, average sums; chance chunks: values, first slots,
// child counts, own slots). w: the chunk's words with the first element and
// the count (the descriptors': the end); shift: log2 of an element's bytes.
struct StreamCopy {
  const void *base;
  int32_t w, shift;
};

constexpr int kIssueRest = 1, kIssueValues = 2, kIssueAll = 3;

// Issues the copies of a chunk into a stage, by all lanes of one warp, each of
// which passes word `lane` of the chunk and its copy of a set and of a chance
// chunk. Returns false (and issues nothing) if the chunk does not fit. parts:
// kIssueRest the expected byte count and every copy but the children's
// values, kIssueValues the children's values (of everything a backward launch
// reads, the one input the backward launch before it writes).
__device__ __forceinline__ bool stream_issue(int32_t word, const StreamCopy &sets, const StreamCopy &chance,
                                             unsigned char *stage, uint32_t bytes, uint32_t bar, int parts) {
  const int lane = threadIdx.x & 31;
  const int32_t kind = __shfl_sync(0xffffffffu, word, 10);
  const StreamCopy c = kind == kChunkChance ? chance : sets;
  const int32_t e = __shfl_sync(0xffffffffu, word, c.w), x = __shfl_sync(0xffffffffu, word, c.w + 1);
  const int32_t cnt = c.w == 0 ? x - e : x;
  const uint32_t n = c.base ? (uint32_t)cnt << c.shift : 0u;
  uint32_t end = n;  // of this copy in the stage
#pragma unroll
  for (int off = 1; off < 8; off <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, end, off);
    if (lane >= off) end += y;
  }
  const uint32_t total = __shfl_sync(0xffffffffu, end, 7);
  if ((kind != kChunkSets && kind != kChunkChance) || __any_sync(0xffffffffu, c.base && cnt <= 0) || total > bytes)
    return false;
  if (lane == 0 && (parts & kIssueRest)) mbar_expect_tx(bar, total);
  __syncwarp();
  if (n > 0 && (parts & (lane == (kind == kChunkChance ? 0 : 1) ? kIssueValues : kIssueRest)))
    bulk_g2s(smem_u32(stage) + end - n, static_cast<const unsigned char *>(c.base) + ((size_t)e << c.shift), n, bar);
  return true;
}

__device__ __forceinline__ StreamChunk stream_chunk(int32_t word) {  // from its words, one a lane
  StreamChunk d;
  int32_t *w = reinterpret_cast<int32_t *>(&d);
#pragma unroll
  for (int i = 0; i < 11; ++i) w[i] = __shfl_sync(0xffffffffu, word, i);
  return d;
}

// The members q0, q0 + step, ... of one staged set of NA actions (0: na, at
// most MAXA): writes their values and adds their terms to racc (the regret
// sums, player 2's with the sign still to be turned) and own (the sum of the
// set's own reach, which times the strategy is the average sum). Two members
// a step, every load before the first use.
template <int MAXA, int NA>
__device__ __forceinline__ void stream_sum(const float2 *sr, int32_t rstep, const int32_t *sm, const float *sv,
                                           const float (&sig)[MAXA], int32_t nm, int32_t na, bool p2, int32_t q0,
                                           int32_t step, float *v, float (&racc)[MAXA], float &own) {
  constexpr int A = NA ? NA : MAXA;
  auto member = [&](const float2 &r, int32_t h, const float(&vc)[A]) {
    float vh = 0.f;
#pragma unroll
    for (int a = 0; a < A; ++a)
      if (NA || a < na) vh = vh + sig[a] * vc[a];
    v[h] = vh;
    const float po = p2 ? r.x : r.y;  // opponent's reach (chance is inside v)
    own += p2 ? r.y : r.x;
#pragma unroll
    for (int a = 0; a < A; ++a)
      if (NA || a < na) racc[a] += po * (vc[a] - vh);
  };
  int32_t q = q0;
  for (; q + step < nm; q += 2 * step) {
    const float2 r0 = sr[q * rstep], r1 = sr[(q + step) * rstep];
    const int32_t h0 = sm[q], h1 = sm[q + step];
    float c0[A], c1[A];
#pragma unroll
    for (int a = 0; a < A; ++a) {
      c0[a] = NA || a < na ? sv[q + a * nm] : 0.f;  // an action-major block
      c1[a] = NA || a < na ? sv[q + step + a * nm] : 0.f;
    }
    member(r0, h0, c0);
    member(r1, h1, c1);
  }
  if (q < nm) {
    const float2 r0 = sr[q * rstep];
    const int32_t h0 = sm[q];
    float c0[A];
#pragma unroll
    for (int a = 0; a < A; ++a) c0[a] = NA || a < na ? sv[q + a * nm] : 0.f;
    member(r0, h0, c0);
  }
}

// The member work of one group of sets (G = 1 or 4) of a staged chunk by the
// n threads of a team: thread t serves set j = t % G and members t / G,
// t / G + n / G, ...; writes each member's value and leaves the thread's
// partial sums, finished by a butterfly over the warp's lanes that serve the
// same set, in racc (regret) and own (own reach). Sets of two or three
// actions, as all of a warp's usually are, take code of their own: predicates
// over MAXA actions doubled a member's instructions, and the members'
// instructions are what a large depth's time goes into.
template <int MAXA>
__device__ __forceinline__ void stream_members(const StreamChunk &d, const StreamLayout &L, const unsigned char *stage,
                                               int32_t I, int G, int t, int n, float *v, float (&racc)[MAXA],
                                               float &own) {
  const SetInfo *sinfo = reinterpret_cast<const SetInfo *>(stage + L.info);
  const int gs = G == 4 ? 2 : 0;
  const SetInfo si = sinfo[I + (t & (G - 1)) - d.I0];
  const bool p2 = (si.flags >> 8) & 1;
  const float2 *sr = reinterpret_cast<const float2 *>(stage + L.reach) + (si.rank0 - d.ra);
  const float *sv = reinterpret_cast<const float *>(stage + L.val) + (si.vb - d.va);
  const int32_t *sm = reinterpret_cast<const int32_t *>(stage + L.mem) + (si.m0 - d.ka);
  const float *ss = reinterpret_cast<const float *>(stage + L.sig) + (si.sb - d.sa);
  float sig[MAXA];
#pragma unroll
  for (int a = 0; a < MAXA; ++a) {
    sig[a] = a < si.na ? ss[a] : 0.f;
    racc[a] = 0.f;
  }
  own = 0.f;
  const int32_t q0 = t >> gs, step = n >> gs;
  int na = MAXA;
  if (__all_sync(0xffffffffu, si.na == 2)) {
    na = 2;
    stream_sum<MAXA, 2>(sr, si.rstep, sm, sv, sig, si.nm, 2, p2, q0, step, v, racc, own);
  } else if (__all_sync(0xffffffffu, si.na == 3)) {
    na = 3;
    stream_sum<MAXA, 3>(sr, si.rstep, sm, sv, sig, si.nm, 3, p2, q0, step, v, racc, own);
  } else {
    stream_sum<MAXA, 0>(sr, si.rstep, sm, sv, sig, si.nm, si.na, p2, q0, step, v, racc, own);
  }
  __syncwarp();
  for (int off = G; off < 32; off <<= 1) {
    own += __shfl_xor_sync(0xffffffffu, own, off);
#pragma unroll
    for (int a = 0; a < MAXA; ++a)
      if (a < na) racc[a] += __shfl_xor_sync(0xffffffffu, racc[a], off);
  }
}

// What lane a * G + j of the updating warp needs of slot a of set j; read
// before the stage is refilled.
struct StreamSlot {
  double R, S;
  float sig, sign;  // the strategy; of the regret terms
  int32_t q, na;    // the slot, the set's actions
  bool live;
};

__device__ __forceinline__ StreamSlot stream_slot(const StreamChunk &d, const StreamLayout &L,
                                                  const unsigned char *stage, int32_t I, int G, int maxa, int upd) {
  const int lane = threadIdx.x & 31;
  const int gs = G == 4 ? 2 : 0;
  const int j = lane & (G - 1), a = lane >> gs;
  const SetInfo si = reinterpret_cast<const SetInfo *>(stage + L.info)[I + j - d.I0];
  StreamSlot z;
  z.na = si.na;
  z.q = si.sb + a;
  z.live = a < maxa && a < si.na && (upd & ((si.flags >> 8) & 1 ? 2 : 1));
  z.R = z.S = 0.0;
  z.sig = 0.f;
  z.sign = (si.flags >> 8) & 1 ? -1.f : 1.f;
  if (z.live) {
    const double *sR = reinterpret_cast<const double *>(stage + L.total);
    z.sig = reinterpret_cast<const float *>(stage + L.sig)[z.q - d.sa];
    z.R = sR[z.q - d.sa];
    z.S = sR[d.nsa + z.q - d.sa];
  }
  return z;
}

// The slot update of one group by one warp: lane = a * G + j updates slot a of
// set j with its regret total r and the set's own reach, then writes sigma^{t+1} of the group's sets.
template <int MAXA>
__device__ __forceinline__ void stream_update(const StreamSlot &z, int G, float r, float own, float *sigma, double *Rg,
                                              double *avgg, double wt, int rule) {
  const int j = threadIdx.x & (G - 1);
  float pf = 0.f;
  if (z.live) {
    double Rn, Sn;
    pf = narrow_pos(slot_terms(z.R, z.S, widen(z.sign * r), widen(own * z.sig), wt, rule, Rn, Sn));
    Rg[z.q] = Rn;
    avgg[z.q] = Sn;
  }
  float tot = 0.f;  // positive parts in action order
#pragma unroll
  for (int b = 0; b < MAXA; ++b) {
    const float x = __shfl_sync(0xffffffffu, pf, (b * G + j) & 31);
    if (b < z.na) tot += x;
  }
  if (z.live) sigma[z.q] = match(pf, tot, z.na);
}

// A team's work on a staged chance chunk: its thread t of n sums the children
// of nodes I0 + t, I0 + t + n, ... left to right (as bwd_chance does: the same
// value bit for bit) and writes the node's value.
__device__ __forceinline__ void stream_chance_chunk(const StreamChunk &d, const unsigned char *stage, int t, int n,
                                                    float *v) {
  const ChanceLayout C = chance_layout(d);
  const float *sv = reinterpret_cast<const float *>(stage);
  const int32_t *svb = reinterpret_cast<const int32_t *>(stage + C.vb);
  const int32_t *snc = reinterpret_cast<const int32_t *>(stage + C.nch);
  const int32_t *svs = reinterpret_cast<const int32_t *>(stage + C.vs);
  for (int32_t i = d.I0 + t; i < d.I1; i += n) {
    const int32_t k = i - d.ka;
    const float *p = sv + (svb[k] - d.va);
    const int32_t nc = snc[k];
    float sum = 0.f;
    for (int32_t c = 0; c < nc; ++c) sum = sum + p[c];
    v[svs[k]] = sum;
  }
}

// Grid: CTAs of shape.teams teams over chunks [c0, c1) of this depth (its set
// chunks, then its chance chunks; a depth with wide chance nodes does not
// stream). Chunk i of a team uses stage i % kStreamStages. Barriers of a team
// (every wait bounded):
//   full[s]  the copies of the chunk in stage s have landed (bytes counted)
//   sync     teams of several warps: all threads are done with a group (or a
//            chance chunk) and have left their partial sums in red
// A stage is refilled only after every thread of the team is done with its
// chunk, so a phase cannot complete twice before its waiters see it. red is
// double-buffered: the warp whose turn a group is has read red[p] before it
// arrives at the next group's sync, which the others pass before they write
// red[p] again.
template <int MAXA>
__global__ void __launch_bounds__(32 * kStreamMaxWarps, 1)
    bwd_stream_kernel(GameView g, StateView<float> st, const SetInfo *info, const StreamChunk *chunks, int32_t c0,
                      int32_t c1, int rule, int upd, int *err, int early, StreamShape shape) {
  constexpr int S = kStreamStages;
  static_assert(S == 2, "the descriptors in flight are the current chunk's, the next one's and the one's after");
  extern __shared__ __align__(128) unsigned char s_stage[];  // [team][stage]
  __shared__ __align__(8) uint64_t s_full[kStreamMaxWarps][S], s_sync[kStreamMaxWarps];
  __shared__ float s_red[2][kStreamMaxWarps][4][MAXA + 1];
  if (!early) pdl_enter();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int team = warp / shape.warps, tw = warp - team * shape.warps;  // warp tw of the team
  const int n = 32 * shape.warps, t = 32 * tw + lane;                   // thread t of n
  const int32_t stride = (int32_t)gridDim.x * shape.teams;
  const int32_t first = c0 + (int32_t)blockIdx.x + team * (int32_t)gridDim.x;
  const uint32_t full0 = smem_u32(&s_full[team][0]), sync = smem_u32(&s_sync[team]);
  unsigned char *ring = s_stage + (size_t)team * S * shape.bytes;
  if ((smem_u32(s_stage) & 15u) != 0u) {  // bulk copies need 16-byte aligned destinations
    if (threadIdx.x == 0) atomicExch(err, 1);
    return;
  }
  if (t == 0) {
    for (int s = 0; s < S; ++s) mbar_init(full0 + 8 * s, 1);
    mbar_init(sync, n);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  __syncthreads();  // barriers initialised (the only CTA-wide barrier)
  auto word = [&](int32_t c) {  // word `lane` of chunk c
    return lane < 16 && c < c1 ? __ldg(reinterpret_cast<const int32_t *>(chunks + c) + lane) : 0;
  };
  StreamCopy sets{nullptr, 0, 0}, chance{nullptr, 0, 0};  // this lane's copies
  if (lane == 0) { sets = {st.reach, 2, 3}; chance = {st.v, 4, 2}; }
  if (lane == 1) { sets = {st.v, 4, 2}; chance = {g.ch_vb, 6, 2}; }
  if (lane == 2) { sets = {g.mem_vs, 6, 2}; chance = {g.ch_nch, 6, 2}; }
  if (lane == 3) { sets = {info, 0, 5}; chance = {g.ch_vs, 6, 2}; }
  if (lane == 4) sets = {st.sigma, 8, 2};
  if (lane == 5) sets = {st.R, 8, 3};
  if (lane == 6) sets = {st.avg, 8, 3};
  auto issue = [&](int32_t i, int32_t w, int parts) {
    return stream_issue(w, sets, chance, ring + (i % S) * shape.bytes, (uint32_t)shape.bytes, full0 + 8 * (i % S),
                        parts);
  };
  int32_t w0 = word(first), w1 = word(first + stride);
  // fault-injection hook (err[1], set on the host): issue no copy after the
  // first ones, so that the waits for the next chunk run out
  const bool stall = reinterpret_cast<volatile const int *>(err)[1] != 0;
  bool ok = true;
  // the first chunks of the team. early: the launch before this one is the
  // backward launch of the next depth, which writes only values of this
  // depth's children (and its own slots), so everything else is copied before
  // waiting for that launch to finish (programmatic dependent launch), and
  // the children's values after
  if (tw == 0) {
    for (int i = 0; i < S && ok && first + i * stride < c1; ++i) {
      ok = issue(i, i ? w1 : w0, early ? kIssueRest : kIssueAll);  // a chunk larger than a stage: the waits give up
    }
  }
  if (early) {
    pdl_enter();
    if (tw == 0)
      for (int i = 0; i < S && ok && first + i * stride < c1; ++i) issue(i, i ? w1 : w0, kIssueValues);
  }
  const double wt = avg_weight(*st.t + 1, rule);
  uint32_t phase = 0;  // of sync: groups and chance chunks done
  int32_t i = 0;
  for (; ok; ++i) {
    const int32_t c = first + i * stride;
    if (c >= c1) break;
    const int32_t w2 = word(c + 2 * stride);  // its latency overlaps this chunk's work
    const int s = i % S;
    ok = __all_sync(0xffffffffu, mbar_wait(full0 + 8 * s, (uint32_t)((i / S) & 1)));
    if (!ok) break;
    const StreamChunk d = stream_chunk(w0);
    const unsigned char *stage = ring + s * shape.bytes;
    auto refill = [&](bool turn) {  // every thread of the team is done with the stage
      if (turn && c + 2 * stride < c1 && !stall) {
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        ok = issue(i + S, w2, kIssueAll);
      }
    };
    auto team_sync = [&]() {
      __syncwarp();
      if (shape.warps > 1) {
        mbar_arrive(sync);
        ok = __all_sync(0xffffffffu, mbar_wait(sync, phase & 1));
        ++phase;
      }
    };
    if (d.kind == kChunkChance) {
      stream_chance_chunk(d, stage, t, n, st.v);
      team_sync();
      if (ok) refill(tw == 0);
    } else {
      const StreamLayout L = stream_layout(d);
      const SetInfo *sinfo = reinterpret_cast<const SetInfo *>(stage + L.info);
      for (int32_t I = d.I0; I < d.I1 && ok;) {
        const int G = sinfo[I - d.I0].flags & 7;
        float racc[MAXA], own;
        stream_members<MAXA>(d, L, stage, I, G, t, n, st.v, racc, own);
        // the team's warps take turns at the slot updates and the refills
        const bool turn = shape.warps == 1 || (int)(phase % (uint32_t)shape.warps) == tw;
        StreamSlot z;
        if (turn) z = stream_slot(d, L, stage, I, G, MAXA, upd);
        const int a = lane >> (G == 4 ? 2 : 0), j = lane & (G - 1);
        float r = 0.f;
        if (shape.warps > 1) {
          float(*red)[4][MAXA + 1] = s_red[phase & 1];
          if (lane < G) {
#pragma unroll
            for (int b = 0; b < MAXA; ++b) red[warp][lane][b] = racc[b];
            red[warp][lane][MAXA] = own;
          }
          team_sync();
          if (ok && turn && a < MAXA) {
            own = 0.f;
            for (int w = 0; w < shape.warps; ++w) {  // warps in order
              r += red[warp - tw + w][j][a];
              own += red[warp - tw + w][j][MAXA];
            }
          }
        } else {
          __syncwarp();
#pragma unroll
          for (int b = 0; b < MAXA; ++b)
            if (a == b) r = racc[b];
        }
        if (!ok) break;
        I += G;
        if (I >= d.I1) refill(turn);
        if (turn) stream_update<MAXA>(z, G, r, own, st.sigma, st.R, st.avg, wt, rule);
      }
    }
    w0 = w1;
    w1 = w2;
  }
  if (!ok) {
    atomicExch(err, 1);
    // let the team's copies in flight land before the warp leaves (bounded)
    for (int32_t k = i; k < i + S && first + k * stride < c1; ++k)
      mbar_wait(full0 + 8 * (k % S), (uint32_t)((k / S) & 1));
  }
}

}  // namespace cfr
