// mlp_fused.cu — the warm-start network of three hidden layers of 256 as a few
// kernels on the 5th-generation tensor cores (tcgen05, accumulators in TMEM).
//
// mlp_rows_kernel takes tiles of 128 rows through the whole network: the
// rows' features, then each layer's activations, stay in shared memory as the
// BF16 A operand, the layers' weights stream past them from packed images (a
// ring of 32 KB blocks filled by bulk copies), and the epilogue of one layer
// (bias, ReLU, BF16 rounding) writes the next layer's operand. A training
// pass goes on with the softmax's gradient and the products with the
// transposed weights in the same tile, and leaves the activations and the
// gradients of every layer, transposed, as 64-row operand blocks for
// mlp_wgrad_kernel: the weight gradients are products over the rows, split
// over CTAs, and mlp_reduce_kernel adds the splits in order.
//
// Every operand block is what a bulk copy can put into shared memory as it
// is: rows of 64 BF16 values along the contraction (128 bytes), their 16-byte
// pieces exchanged within 8 rows by the 128-byte swizzle that the tensor
// cores' K-major operand descriptor names.
//
// Numerics are those of mlp_gemm layer by layer: operands rounded to BF16,
// products summed in FP32, bias, ReLU, softmax, bias gradients and weight
// gradients in FP32.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <cmath>
#include <string>

#include "../../include/mlp.h"
#include "bwd_stream.cuh"

namespace mlpf {

using cfr::bulk_g2s;
using cfr::mbar_arrive;
using cfr::mbar_expect_tx;
using cfr::mbar_init;
using cfr::mbar_wait;
using cfr::smem_u32;

constexpr int kH = 256;                       // hidden width
constexpr int kOut = 8;                       // logits
constexpr int kTile = 128;                    // rows of a tile
constexpr int kBlkK = 64;                     // contraction elements of a block
constexpr uint32_t kWBlk = 256 * 128;         // bytes of a block of 256 rows
constexpr uint32_t kABlk = kTile * 128;       // bytes of a block of a tile's rows
constexpr uint32_t kOBlk = 16 * 128;          // bytes of a block of the output layer (8 logits and 8 rows of zeros)
// Tiles of a CTA in flight and weight blocks in flight (64 KB of activations a
// tile, 32 KB a block).
template <int PIPES> constexpr int kRing = PIPES == 1 ? 4 : 2;
constexpr int kEpi = 256;                     // epilogue threads: 8 warps
constexpr int kThreads = kEpi + 64;           // and a loading and an issuing warp
constexpr int kStagesPredict = 4, kStagesTrain = 7;
// One 64-row operand group of a training pass: X, h1, h2, h3, d1, d2, d3
// (256 rows each) and the logits' gradient (16 rows).
constexpr uint32_t kGroup = 7 * kWBlk + kOBlk;
// Row splits of the weight gradients: 4 x 16 CTAs fill under half the SMs, but
// every split writes and the reduction reads 0.7 MB.
constexpr int kMaxSplits = 16;

// Byte offset of element (row, k) in an operand block (128-byte swizzle).
__host__ __device__ __forceinline__ uint32_t blk_off(uint32_t row, uint32_t k) {
  return row * 128u + ((((k >> 3) ^ row) & 7u) << 4) + (k & 7u) * 2u;
}

// Offsets of the layers' images in the packed weights. Forward images hold
// W^T (a row per output, the inputs along the contraction), backward images W
// (a row per input); in_blocks = blocks of the first layer's inputs.
struct Images {
  uint32_t fwd[4], bwd[4], bytes;
};
__host__ __device__ inline Images images(int in_blocks) {
  Images im;
  uint32_t at = 0;
  im.fwd[0] = at; at += (uint32_t)in_blocks * kWBlk;
  im.fwd[1] = at; at += 4 * kWBlk;
  im.fwd[2] = at; at += 4 * kWBlk;
  im.fwd[3] = at; at += 4 * kOBlk;
  im.bwd[0] = 0;  // the features' gradient is not needed
  im.bwd[1] = at; at += 4 * kWBlk;
  im.bwd[2] = at; at += 4 * kWBlk;
  im.bwd[3] = at; at += kWBlk;
  im.bytes = at;
  return im;
}

struct RowArgs {
  const float *X;
  const unsigned char *img;
  const float *b[4];
  const int32_t *nact;
  const float *target, *weight;
  float *prob;               // predict
  float *loss_rows;          // train
  unsigned char *groups;     // train: operand groups of 64 rows
  float *colsum;             // train: [tile][4][256] bias gradients of the tile
  int *err;
  int B, in_dim, in_blocks, tiles, vec;
};

// ------------------------------------------------------------------ tcgen05
// K-major operand, 128-byte swizzle: start address, 1,024 bytes between
// groups of 8 rows, descriptor version 1 (bit 46), swizzle mode 2 (bits 61-63).
__device__ __forceinline__ uint64_t op_desc(uint32_t addr) {
  return (uint64_t)((addr >> 4) & 0x3fffu) | (1ull << 16) | (64ull << 32) | (1ull << 46) | (2ull << 61);
}

// BF16 operands, FP32 accumulators, both operands K-major.
__host__ __device__ constexpr uint32_t op_idesc(int m, int n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(m >> 4) << 24);
}

__device__ __forceinline__ void mma_f16(uint32_t acc, uint64_t a, uint64_t b, uint32_t idesc, uint32_t add) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(acc),
      "l"(a), "l"(b), "r"(idesc), "r"(add)
      : "memory");
}

__device__ __forceinline__ void mma_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ void tmem_alloc(uint32_t dst, uint32_t cols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(dst), "r"(cols) : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ void tmem_free(uint32_t addr, uint32_t cols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(addr), "r"(cols) : "memory");
}

__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// A wait gave up. The word may be page-locked host memory: a plain store.
__device__ __forceinline__ void report(int *err) { *reinterpret_cast<volatile int *>(err) = 1; }

// Bounded wait of a thread that other threads meet at named barriers: when it
// gives up (or another thread has) it says so and goes on without waiting, so
// that every such barrier is still reached by all.
__device__ __forceinline__ void wait_or_go_on(uint32_t bar, uint32_t parity, volatile int *stop, int *err) {
  if (*stop == 0 && !mbar_wait(bar, parity)) {
    *stop = 1;
    report(err);
  }
}

// 32 columns of this thread's accumulator row (a warp reads its 32 lanes).
__device__ __forceinline__ void tmem_ld32(uint32_t addr, float (&x)[32]) {
  uint32_t r[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,"
      "%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
        "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
        "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(addr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 32; ++i) x[i] = __uint_as_float(r[i]);
}

__device__ __forceinline__ void tmem_ld8(uint32_t addr, float (&x)[8]) {
  uint32_t r[8];
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(addr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 8; ++i) x[i] = __uint_as_float(r[i]);
}

__device__ __forceinline__ uint32_t pack2(float lo, float hi) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t *>(&v);
}

// ---------------------------------------------------------- rows of a batch
// Stages of a tile: 0-2 hidden layers, 3 logits, and in training 4-6 the
// gradients of h3, h2, h1.
template <bool TRAIN> struct Stage {
  static constexpr int kCount = TRAIN ? kStagesTrain : kStagesPredict;
  // ring entries of a stage, and the image offset and bytes of each
  __device__ static int entries(int s, int in_blocks) { return s == 0 ? in_blocks : (s == 3 || s == 4) ? 1 : 4; }
  __device__ static uint32_t offset(const Images &im, int s, int e) {
    if (s < 3) return im.fwd[s] + (uint32_t)e * kWBlk;
    if (s == 3) return im.fwd[3];
    return im.bwd[7 - s] + (uint32_t)e * kWBlk;
  }
  __device__ static uint32_t bytes(int s) { return s == 3 ? 4 * kOBlk : kWBlk; }
};

struct RowSmem {  // after the operand blocks
  uint64_t full[4], empty[4], acc[2], act[2];
  uint32_t tmem;
  int stop;
  float bias[4][kH];
  float col[4][kH];  // column sums of the tile's four 32-row parts
};

// What bounds it: at 200,000 rows the tensor cores' 74 GFLOP (40 us) and the
// epilogues between dependent layers, which one tile a CTA does not overlap; the rows'
// features are the only traffic to speak of (160 MB; the layers one after
// another with FP32 activations moved ten times that). 200,000 rows: 2,781 us
// as one mma.sync product a layer, 166 here with one tile a CTA, 128 with two.
// A training step of 4,096 rows: 2,500 us as 30 launches, 159 here with the
// host's share.
//
// PIPES = 2 (inference with more tiles than SMs): two tiles a CTA in turn, the
// epilogue of one under the products of the other. Each has its own operand
// blocks, accumulators and four epilogue warps; every layer's weights are
// loaded once for each.
template <bool TRAIN, int PIPES>
__global__ void __launch_bounds__(kThreads, 1) mlp_rows_kernel(const RowArgs a) {
  static_assert(!TRAIN || PIPES == 1, "a training tile takes all epilogue warps");
  extern __shared__ __align__(1024) unsigned char s_dyn[];
  using S = Stage<TRAIN>;
  constexpr int R = kRing<PIPES>, PT = kEpi / PIPES;  // ring blocks, epilogue threads of a tile
  unsigned char *s_ring = s_dyn + PIPES * 4 * kABlk;
  RowSmem &sm = *reinterpret_cast<RowSmem *>(s_ring + R * kWBlk);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (tid == 0) {
    for (int i = 0; i < R; ++i) {
      mbar_init(smem_u32(&sm.full[i]), 1);
      mbar_init(smem_u32(&sm.empty[i]), 1);
    }
    for (int p = 0; p < PIPES; ++p) {
      mbar_init(smem_u32(&sm.acc[p]), 1);
      mbar_init(smem_u32(&sm.act[p]), PT);
    }
    sm.stop = (smem_u32(s_dyn) & 1023u) != 0u;  // the swizzle needs 1,024-byte aligned blocks
    if (sm.stop) report(a.err);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    fence_smem();
  }
  if (warp == 8) tmem_alloc(smem_u32(&sm.tmem), 256 * PIPES);
  for (int i = tid; i < 4 * kH; i += kThreads) {
    const int l = i / kH, c = i % kH;
    sm.bias[l][c] = l < 3 || c < kOut ? a.b[l][c] : 0.f;
  }
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = sm.tmem;
  volatile int *stop = &sm.stop;
  const Images im = images(a.in_blocks);

  if (*stop == 0) {
    if (warp == 8) {
      // the loading thread: every tile's weight blocks in the order of use
      if (lane == 0) {
        int n = 0;  // ring entries issued
        bool ok = true;
        for (int t = blockIdx.x; t < a.tiles && ok; t += PIPES * gridDim.x)
          for (int sp = 0; sp < S::kCount * PIPES && ok; ++sp) {
            const int s = sp / PIPES, p = sp % PIPES;
            if (t + p * (int)gridDim.x >= a.tiles) continue;
            for (int e = 0; e < S::entries(s, a.in_blocks); ++e, ++n) {
              const int slot = n % R;
              if (n >= R && !mbar_wait(smem_u32(&sm.empty[slot]), (uint32_t)((n / R - 1) & 1))) { ok = false; break; }
              if (*stop) { ok = false; break; }
              const uint32_t bytes = S::bytes(s);
              mbar_expect_tx(smem_u32(&sm.full[slot]), bytes);
              bulk_g2s(smem_u32(s_ring + slot * kWBlk), a.img + S::offset(im, s, e), bytes, smem_u32(&sm.full[slot]));
            }
          }
        if (!ok) {
          *stop = 1;
          report(a.err);
        }
        for (int i = n > R ? n - R : 0; i < n; ++i)  // no copy is in flight when the CTA leaves
          mbar_wait(smem_u32(&sm.full[i % R]), (uint32_t)((i / R) & 1));
      }
    } else if (warp == 9) {
      // the issuing thread
      if (lane == 0) {
        int n = 0, turn[2] = {0, 0};
        bool ok = true;
        for (int t = blockIdx.x; t < a.tiles && ok; t += PIPES * gridDim.x)
          for (int sp = 0; sp < S::kCount * PIPES && ok; ++sp) {
            const int s = sp / PIPES, p = sp % PIPES;
            if (t + p * (int)gridDim.x >= a.tiles) continue;
            if (!mbar_wait(smem_u32(&sm.act[p]), (uint32_t)(turn[p] & 1)) || *stop) { ok = false; break; }
            ++turn[p];
            fence_after();
            const uint32_t idesc = s == 3 ? op_idesc(kTile, 16) : op_idesc(kTile, kH);
            for (int e = 0; e < S::entries(s, a.in_blocks); ++e, ++n) {
              const int slot = n % R;
              if (!mbar_wait(smem_u32(&sm.full[slot]), (uint32_t)((n / R) & 1)) || *stop) { ok = false; break; }
              fence_after();
              const uint32_t wb = smem_u32(s_ring + slot * kWBlk), ab = smem_u32(s_dyn + p * 4 * kABlk);
              // 16 elements of the contraction (32 bytes of a row) an instruction
              const int steps = s == 3 ? 16 : s == 4 ? 1 : 4;
              for (int k = 0; k < steps; ++k) {
                const uint32_t blk = s == 3 ? (uint32_t)(k >> 2) : (uint32_t)e, in = (uint32_t)(k & 3) * 32u;
                const uint64_t da = op_desc(ab + blk * kABlk + in);
                const uint64_t db = op_desc(wb + (s == 3 ? blk * kOBlk : 0u) + in);
                mma_f16(tmem + (uint32_t)p * 256u, da, db, idesc, (e | k) ? 1u : 0u);
              }
              mma_commit(smem_u32(&sm.empty[slot]));
            }
            if (ok) mma_commit(smem_u32(&sm.acc[p]));
          }
        if (!ok) {
          *stop = 1;
          report(a.err);
        }
      }
    } else {
      // epilogue: thread = row of the tile; with one tile the warpgroups share
      // the columns, with two each has its own tile
      const int p = PIPES == 2 ? warp >> 2 : 0, wg = PIPES == 2 ? 0 : warp >> 2;
      const int part = warp & 3, row = part * 32 + lane, ptid = tid % PT;
      unsigned char *s_act = s_dyn + p * 4 * kABlk;
      const uint32_t acc = tmem + (uint32_t)p * 256u + ((uint32_t)(part * 32) << 16);
      const uint32_t in_pad = (uint32_t)a.in_blocks * kBlkK;
      int turn = 0;
      for (int t = blockIdx.x + p * gridDim.x; t < a.tiles; t += PIPES * gridDim.x) {
        const int r0 = t * kTile;
        unsigned char *grp = TRAIN ? a.groups + (size_t)(2 * t + (row >> 6)) * kGroup : nullptr;
        const uint32_t gk = (uint32_t)(row & 63);  // this row's place in its group's contraction
        // the tile's features, rounded to BF16 (rows past the batch and
        // columns past the features are zeros)
        if (a.vec) {
          const int nv = (int)in_pad / 4, items = kTile * nv;
          for (int i0 = ptid; i0 < items; i0 += 8 * PT) {
            float4 x[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
              const int i = i0 + u * PT, r = i / nv, c = i % nv * 4;
              x[u] = make_float4(0.f, 0.f, 0.f, 0.f);
              if (i < items && r0 + r < a.B && c < a.in_dim)
                x[u] = __ldg(reinterpret_cast<const float4 *>(a.X + (size_t)(r0 + r) * a.in_dim + c));
            }
#pragma unroll
            for (int u = 0; u < 8; ++u) {
              const int i = i0 + u * PT, r = i / nv, c = i % nv * 4;
              if (i < items) {
                uint2 w;
                w.x = pack2(x[u].x, x[u].y);
                w.y = pack2(x[u].z, x[u].w);
                *reinterpret_cast<uint2 *>(s_act + (c / kBlkK) * kABlk + blk_off((uint32_t)r, (uint32_t)(c % kBlkK))) = w;
              }
            }
          }
        } else {
          const int items = kTile * (int)in_pad;
          for (int i = ptid; i < items; i += PT) {
            const int r = i / (int)in_pad, c = i % (int)in_pad;
            const float x = r0 + r < a.B && c < a.in_dim ? a.X[(size_t)(r0 + r) * a.in_dim + c] : 0.f;
            *reinterpret_cast<__nv_bfloat16 *>(s_act + (c / kBlkK) * kABlk + blk_off((uint32_t)r, (uint32_t)(c % kBlkK))) =
                __float2bfloat16_rn(x);
          }
        }
        fence_smem();
        mbar_arrive(smem_u32(&sm.act[p]));
        if constexpr (TRAIN) {  // the features' operand block: every epilogue thread has to have written its part
          asm volatile("bar.sync 1, 256;" ::: "memory");
          for (uint32_t c = (uint32_t)wg * 8u; c < in_pad; c += 16u) {  // 8 columns at a time
            const uint4 v = *reinterpret_cast<const uint4 *>(s_act + (c / kBlkK) * kABlk + blk_off((uint32_t)row, c % kBlkK));
            const __nv_bfloat16 *h = reinterpret_cast<const __nv_bfloat16 *>(&v);
#pragma unroll
            for (uint32_t j = 0; j < 8; ++j) *reinterpret_cast<__nv_bfloat16 *>(grp + blk_off(c + j, gk)) = h[j];
          }
          asm volatile("bar.sync 1, 256;" ::: "memory");  // read by all before the first layer's values replace it
        }
        uint32_t live[3][4];  // which of this thread's hidden values are positive
#pragma unroll
        for (int s = 0; s < S::kCount; ++s) {
          wait_or_go_on(smem_u32(&sm.acc[p]), (uint32_t)(turn & 1), stop, a.err);
          ++turn;
          fence_after();
          if (s == 3) {
            if (wg == 0) {
              float z[kOut];
              tmem_ld8(acc, z);
              const bool in = r0 + row < a.B;
              const int na = in ? a.nact[r0 + row] : 0;
              float mx = -INFINITY;
#pragma unroll
              for (int j = 0; j < kOut; ++j) {
                z[j] += sm.bias[3][j];
                if (j < na) mx = fmaxf(mx, z[j]);
              }
              float sum = 0.f;
#pragma unroll
              for (int j = 0; j < kOut; ++j)
                if (j < na) sum += __expf(z[j] - mx);
              const float lse = mx + __logf(sum);
              // inference after a wait that gave up: no row passes for a result
              const float failed = !TRAIN && *stop != 0 ? __int_as_float(0x7fc00000) : 0.f;
              float p[kOut];
#pragma unroll
              for (int j = 0; j < kOut; ++j) p[j] = (j < na ? __expf(z[j] - lse) : 0.f) + failed;
              if constexpr (!TRAIN) {
                if (in) {
                  float4 *o = reinterpret_cast<float4 *>(a.prob + (size_t)(r0 + row) * kOut);
                  o[0] = make_float4(p[0], p[1], p[2], p[3]);
                  o[1] = make_float4(p[4], p[5], p[6], p[7]);
                }
              } else {
                float g[kOut];
                float loss = 0.f;
                const float w = in && a.weight ? a.weight[r0 + row] : 1.f;
#pragma unroll
                for (int j = 0; j < kOut; ++j) {
                  g[j] = 0.f;
                  if (j < na) {
                    const float y = a.target[(size_t)(r0 + row) * kOut + j];
                    loss -= y * (z[j] - lse);
                    g[j] = (p[j] - y) * w / (float)a.B;
                  }
                }
                if (in) a.loss_rows[r0 + row] = loss * w;
                uint4 v;
                v.x = pack2(g[0], g[1]);
                v.y = pack2(g[2], g[3]);
                v.z = pack2(g[4], g[5]);
                v.w = pack2(g[6], g[7]);
                *reinterpret_cast<uint4 *>(s_act + blk_off((uint32_t)row, 0)) = v;
                *reinterpret_cast<uint4 *>(s_act + blk_off((uint32_t)row, 8)) = make_uint4(0u, 0u, 0u, 0u);
                const __nv_bfloat16 *h = reinterpret_cast<const __nv_bfloat16 *>(&v);
#pragma unroll
                for (uint32_t j = 0; j < 8; ++j)
                  *reinterpret_cast<__nv_bfloat16 *>(grp + 7 * kWBlk + blk_off(j, gk)) = h[j];
#pragma unroll
                for (int j = 0; j < kOut; ++j) {
                  float x = g[j];
                  for (int off = 16; off > 0; off >>= 1) x += __shfl_xor_sync(0xffffffffu, x, off);
                  if (lane == 0) sm.col[part][j] = x;
                }
                asm volatile("bar.sync 2, 128;" ::: "memory");
                if (tid < kOut)
                  a.colsum[((size_t)t * 4 + 3) * kH + tid] = sm.col[0][tid] + sm.col[1][tid] + sm.col[2][tid] + sm.col[3][tid];
                asm volatile("bar.sync 2, 128;" ::: "memory");  // before the columns are used again
              }
            }
          } else {
            const int l = s < 3 ? s : 6 - s;  // the hidden layer this stage writes (its values, or their gradient)
            for (int q = 0; q < 4 * PIPES; ++q) {
              const uint32_t c0 = (uint32_t)(wg * 128 + q * 32);
              float x[32];
              tmem_ld32(acc + c0, x);
              if (s < 3) {
                uint32_t m = 0;
#pragma unroll
                for (int j = 0; j < 32; ++j) {
                  x[j] += sm.bias[l][c0 + j];
                  if (x[j] > 0.f) m |= 1u << j;
                  else x[j] = 0.f;
                }
                if constexpr (TRAIN) {
#pragma unroll
                  for (int u = 0; u < 4; ++u)
                    if (u == q) live[l][u] = m;
                }
              } else {
                uint32_t m = 0;
#pragma unroll
                for (int u = 0; u < 4; ++u)
                  if (u == q) m = live[l][u];
#pragma unroll
                for (int j = 0; j < 32; ++j)
                  if (!(m >> j & 1u)) x[j] = 0.f;
              }
              uint32_t w[16];
#pragma unroll
              for (int j = 0; j < 16; ++j) w[j] = pack2(x[2 * j], x[2 * j + 1]);
              if (s != S::kCount - 1) {
                unsigned char *blk = s_act + (c0 / kBlkK) * kABlk;
#pragma unroll
                for (int j = 0; j < 4; ++j)
                  *reinterpret_cast<uint4 *>(blk + blk_off((uint32_t)row, c0 % kBlkK + 8u * j)) =
                      make_uint4(w[4 * j], w[4 * j + 1], w[4 * j + 2], w[4 * j + 3]);
              }
              if constexpr (TRAIN) {
                // h_l is operand l + 1 of the group, d_l operand l + 4
                unsigned char *op = grp + (size_t)(s < 3 ? l + 1 : l + 4) * kWBlk;
#pragma unroll
                for (int j = 0; j < 32; ++j)
                  *reinterpret_cast<uint16_t *>(op + blk_off(c0 + j, gk)) = (uint16_t)(w[j / 2] >> (16 * (j & 1)));
                if (s > 3) {
                  cfr::group_sum_scatter<32, 32>(x, lane, 0xffffffffu);  // lane j: column c0 + j over the warp's rows
                  sm.col[part][c0 + lane] = x[0];
                }
              }
            }
            if (TRAIN && s > 3) {
              asm volatile("bar.sync %0, 128;" ::"r"(2 + wg) : "memory");
              const int c = wg * 128 + (tid & 127);
              a.colsum[((size_t)t * 4 + l) * kH + c] = sm.col[0][c] + sm.col[1][c] + sm.col[2][c] + sm.col[3][c];
              asm volatile("bar.sync %0, 128;" ::"r"(2 + wg) : "memory");
            }
          }
          fence_before();
          if (s != S::kCount - 1) {
            fence_smem();
            mbar_arrive(smem_u32(&sm.act[p]));
          }
        }
      }
    }
  } else if constexpr (!TRAIN) {
    for (int t = blockIdx.x; t < a.tiles; t += gridDim.x)
      for (int i = tid; i < kTile * kOut; i += kThreads)
        if (t * kTile + i / kOut < a.B) a.prob[(size_t)t * kTile * kOut + i] = __int_as_float(0x7fc00000);
  }
  __syncwarp();
  fence_before();
  __syncthreads();
  fence_after();
  if (warp == 8) tmem_free(tmem, 256 * PIPES);
}

// ------------------------------------------------------- weight gradients
// gW_l = h_l^T d_l over the rows of one split: A = the features or a hidden
// layer (256 operand rows, as two accumulators of 128), B = the gradient of
// the next layer. Grid (splits, 4).
constexpr int kGradRing = 3;
constexpr uint32_t kGradSlot = 2 * kWBlk;
struct GradSmem {
  uint64_t full[kGradRing], empty[kGradRing], acc;
  uint32_t tmem;
  int stop;
};

__global__ void __launch_bounds__(kThreads, 1) mlp_wgrad_kernel(const unsigned char *groups, int n_groups, int per_split,
                                                                int in_dim, float *part, size_t split_stride, int *err) {
  extern __shared__ __align__(1024) unsigned char s_dyn[];
  GradSmem &sm = *reinterpret_cast<GradSmem *>(s_dyn + kGradRing * kGradSlot);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int l = blockIdx.y, split = blockIdx.x;
  const int g0 = split * per_split, g1 = min(n_groups, g0 + per_split);
  const int N = l < 3 ? kH : 16;
  const uint32_t b_bytes = l < 3 ? kWBlk : kOBlk;
  if (tid == 0) {
    for (int i = 0; i < kGradRing; ++i) {
      mbar_init(smem_u32(&sm.full[i]), 1);
      mbar_init(smem_u32(&sm.empty[i]), 1);
    }
    mbar_init(smem_u32(&sm.acc), 1);
    sm.stop = (smem_u32(s_dyn) & 1023u) != 0u;
    if (sm.stop) report(err);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    fence_smem();
  }
  if (warp == 8) tmem_alloc(smem_u32(&sm.tmem), 512);
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = sm.tmem;
  volatile int *stop = &sm.stop;
  if (*stop == 0 && g0 < g1) {
    if (warp == 8) {
      if (lane == 0) {
        int n = 0;
        bool ok = true;
        for (int g = g0; g < g1; ++g, ++n) {
          const int slot = n % kGradRing;
          if ((n >= kGradRing && !mbar_wait(smem_u32(&sm.empty[slot]), (uint32_t)((n / kGradRing - 1) & 1))) || *stop) { ok = false; break; }
          const unsigned char *src = groups + (size_t)g * kGroup;
          mbar_expect_tx(smem_u32(&sm.full[slot]), kWBlk + b_bytes);
          bulk_g2s(smem_u32(s_dyn + slot * kGradSlot), src + (size_t)l * kWBlk, kWBlk, smem_u32(&sm.full[slot]));
          bulk_g2s(smem_u32(s_dyn + slot * kGradSlot + kWBlk), src + (size_t)(l + 4) * kWBlk, b_bytes,
                   smem_u32(&sm.full[slot]));
        }
        if (!ok) {
          *stop = 1;
          report(err);
        }
        for (int i = n > kGradRing ? n - kGradRing : 0; i < n; ++i)
          mbar_wait(smem_u32(&sm.full[i % kGradRing]), (uint32_t)((i / kGradRing) & 1));
      }
    } else if (warp == 9) {
      if (lane == 0) {
        bool ok = true;
        const uint32_t idesc = op_idesc(128, N);
        for (int g = g0, n = 0; g < g1; ++g, ++n) {
          const int slot = n % kGradRing;
          if (!mbar_wait(smem_u32(&sm.full[slot]), (uint32_t)((n / kGradRing) & 1)) || *stop) { ok = false; break; }
          fence_after();
          const uint32_t ab = smem_u32(s_dyn + slot * kGradSlot), bb = ab + kWBlk;
          for (uint32_t k = 0; k < 4; ++k) {
            const uint64_t db = op_desc(bb + k * 32u);
            mma_f16(tmem, op_desc(ab + k * 32u), db, idesc, (n | (int)k) ? 1u : 0u);
            mma_f16(tmem + 256u, op_desc(ab + kABlk + k * 32u), db, idesc, (n | (int)k) ? 1u : 0u);
          }
          mma_commit(smem_u32(&sm.empty[slot]));
        }
        if (ok) mma_commit(smem_u32(&sm.acc));
        else {
          *stop = 1;
          report(err);
        }
      }
    } else {
      const int wg = warp >> 2, i = wg * 128 + (warp & 3) * 32 + lane;  // this thread's input feature
      if (!mbar_wait(smem_u32(&sm.acc), 0) || *stop) {
        *stop = 1;
        report(err);
      } else {
        fence_after();
        const uint32_t acc = tmem + (uint32_t)wg * 256u + ((uint32_t)((warp & 3) * 32) << 16);
        const int rows = l == 0 ? in_dim : kH;
        float *out = part + (size_t)split * split_stride +
                     (l == 0 ? 0 : (size_t)in_dim * kH + (size_t)(l - 1) * kH * kH);
        if (l < 3) {
          for (int c0 = 0; c0 < kH; c0 += 32) {
            float x[32];
            tmem_ld32(acc + (uint32_t)c0, x);
            if (i < rows) {
              float4 *o = reinterpret_cast<float4 *>(out + (size_t)i * kH + c0);
#pragma unroll
              for (int j = 0; j < 8; ++j) o[j] = make_float4(x[4 * j], x[4 * j + 1], x[4 * j + 2], x[4 * j + 3]);
            }
          }
        } else {
          float x[8];
          tmem_ld8(acc, x);
          float4 *o = reinterpret_cast<float4 *>(out + (size_t)i * kOut);
          o[0] = make_float4(x[0], x[1], x[2], x[3]);
          o[1] = make_float4(x[4], x[5], x[6], x[7]);
        }
      }
    }
  }
  __syncwarp();
  fence_before();
  __syncthreads();
  fence_after();
  if (warp == 8) tmem_free(tmem, 512);
}

// The splits' sums in order (weights), the tiles' column sums in order
// (biases), and the rows' losses (one block, fixed shape): out[0] the sum.
struct ReduceArgs {
  const float *part, *colsum, *loss_rows;
  float *gW[4], *gb[4];
  float *loss;
  size_t split_stride;
  int splits, tiles, B, in_dim;
};

__global__ void __launch_bounds__(256) mlp_reduce_kernel(const ReduceArgs a) {
  const int nw = (int)(a.split_stride / 4), nb_w = (nw + 255) / 256;
  const int b = blockIdx.x;
  if (b < nb_w) {
    const int i = b * 256 + threadIdx.x;
    if (i >= nw) return;
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 4
    for (int k = 0; k < a.splits; ++k) {
      const float4 x = __ldg(reinterpret_cast<const float4 *>(a.part + (size_t)k * a.split_stride) + i);
      s.x += x.x; s.y += x.y; s.z += x.z; s.w += x.w;
    }
    size_t e = (size_t)i * 4, n0 = (size_t)a.in_dim * kH;
    int l = 0;
    if (e >= n0) {
      e -= n0;
      l = 1 + (int)(e / (kH * kH));
      e -= (size_t)(l - 1) * kH * kH;
    }
    reinterpret_cast<float4 *>(a.gW[l])[e / 4] = s;
    return;
  }
  if (b < nb_w + 4) {
    const int l = b - nb_w, c = threadIdx.x, n = l < 3 ? kH : kOut;
    if (c >= n) return;
    float s = 0.f;
#pragma unroll 4
    for (int t = 0; t < a.tiles; ++t) s += __ldg(a.colsum + ((size_t)t * 4 + l) * kH + c);
    a.gb[l][c] = s;
    return;
  }
  __shared__ float sh[256];
  float s = 0.f;
  for (int i = threadIdx.x; i < a.B; i += 256) s += a.loss_rows[i];
  sh[threadIdx.x] = s;
  __syncthreads();
  for (int off = 128; off > 0; off >>= 1) {
    if (threadIdx.x < off) sh[threadIdx.x] += sh[threadIdx.x + off];
    __syncthreads();
  }
  if (threadIdx.x == 0) a.loss[0] = sh[0];
}

// ------------------------------------------------------------ Adam, packing
// All of a network's tensors in one launch: tensor 2 l = W_l, 2 l + 1 = b_l.
// Writes the BF16 copy of the weights and, with img, their packed images.
struct AdamArgs {
  float *w[8];
  const float *g[8];
  float *m[8], *v[8];
  __nv_bfloat16 *wb[4];
  unsigned char *img;
  int n[8], first[9];  // elements, first block
  int fi[4], fo[4], in_blocks;
  float lr, b1, b2, eps, bc1, bc2;
  int update;          // 0: only the copies
};

__global__ void __launch_bounds__(256) mlp_adam_all_kernel(const AdamArgs a) {
  int t = 0;
  while (t < 7 && (int)blockIdx.x >= a.first[t + 1]) ++t;
  const int i = ((int)blockIdx.x - a.first[t]) * 256 + (int)threadIdx.x;
  if (i >= a.n[t]) return;
  float x = a.w[t][i];
  if (a.update) {
    const float gi = a.g[t][i];
    const float mi = a.b1 * a.m[t][i] + (1.f - a.b1) * gi;
    const float vi = a.b2 * a.v[t][i] + (1.f - a.b2) * gi * gi;
    a.m[t][i] = mi;
    a.v[t][i] = vi;
    x = x - a.lr * (mi / a.bc1) / (sqrtf(vi / a.bc2) + a.eps);
    a.w[t][i] = x;
  }
  if (t & 1) return;
  const int l = t >> 1;
  const __nv_bfloat16 h = __float2bfloat16_rn(x);
  a.wb[l][i] = h;
  if (!a.img) return;
  const Images im = images(a.in_blocks);
  const uint32_t in = (uint32_t)(i / a.fo[l]), out = (uint32_t)(i % a.fo[l]);
  const uint32_t rows = l < 3 ? kWBlk : kOBlk;
  *reinterpret_cast<__nv_bfloat16 *>(a.img + im.fwd[l] + (in / kBlkK) * rows + blk_off(out, in % kBlkK)) = h;
  if (l > 0)
    *reinterpret_cast<__nv_bfloat16 *>(a.img + im.bwd[l] + (out / kBlkK) * kWBlk + blk_off(in, out % kBlkK)) = h;
}

// Workspace of a training pass over `rows` rows (byte offsets, 256-byte aligned).
struct Work {
  size_t groups, part, colsum, loss_rows, loss, bytes;
  size_t split_stride;
  int tiles, n_groups, per_split, splits;
};
static Work work_of(int in_dim, int rows) {
  Work w;
  w.tiles = (rows + kTile - 1) / kTile;
  w.n_groups = 2 * w.tiles;
  w.per_split = (w.n_groups + kMaxSplits - 1) / kMaxSplits;
  w.splits = (w.n_groups + w.per_split - 1) / w.per_split;
  w.split_stride = (size_t)in_dim * kH + 2 * (size_t)kH * kH + (size_t)kH * kOut;
  size_t at = 0;
  auto take = [&](size_t n) {
    const size_t o = at;
    at += (n + 255) & ~size_t(255);
    return o;
  };
  w.groups = take((size_t)w.n_groups * kGroup);
  w.part = take((size_t)w.splits * w.split_stride * 4);
  w.colsum = take((size_t)w.tiles * 4 * kH * 4);
  w.loss_rows = take((size_t)rows * 4);
  w.loss = take(8);  // the summed loss, then the error word
  w.bytes = at;
  return w;
}

template <int PIPES> constexpr size_t kRowSmem = PIPES * 4 * (size_t)kABlk + kRing<PIPES> * (size_t)kWBlk + sizeof(RowSmem);
constexpr size_t kGradSmem = kGradRing * (size_t)kGradSlot + sizeof(GradSmem);

static thread_local std::string g_err;
static int fail(int code, const std::string &what) {
  g_err = what;
  return code;
}

}  // namespace mlpf

using namespace mlpf;

#define NET_CK(x)                                                                                   \
  do {                                                                                              \
    const cudaError_t e_ = (x);                                                                     \
    if (e_ != cudaSuccess) return fail(-7, std::string(__func__) + ": " + cudaGetErrorString(e_)); \
  } while (0)

static bool aligned16(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }
static bool net_shape(int in_dim) { return in_dim >= 4 && in_dim <= kH && in_dim % 4 == 0; }
static int sm_count(int *n) {
  int dev = 0;
  NET_CK(cudaGetDevice(&dev));
  NET_CK(cudaDeviceGetAttribute(n, cudaDevAttrMultiProcessorCount, dev));
  return 0;
}

static int row_args(RowArgs &a, const float *X, int in_dim, int rows, const void *img, const float *const *b,
                    const int32_t *nact, int *err) {
  if (!X || !img || !b || !nact || !err || rows <= 0 || !net_shape(in_dim))
    return fail(-1, "mlp_net: bad argument");
  if (!aligned16(img)) return fail(-1, "mlp_net: img must be 16-byte aligned");  // bulk copies
  a = RowArgs{};
  a.X = X;
  a.img = (const unsigned char *)img;
  for (int l = 0; l < 4; ++l) a.b[l] = b[l];
  a.nact = nact;
  a.err = err;
  a.B = rows;
  a.in_dim = in_dim;
  a.in_blocks = (in_dim + kBlkK - 1) / kBlkK;
  a.tiles = (rows + kTile - 1) / kTile;
  a.vec = aligned16(X);
  return 0;
}

extern "C" {

const char *mlp_net_last_error(void) { return g_err.c_str(); }

size_t mlp_net_image_bytes(int in_dim) { return net_shape(in_dim) ? images((in_dim + kBlkK - 1) / kBlkK).bytes : 0; }

size_t mlp_net_work_bytes(int in_dim, int rows) { return net_shape(in_dim) && rows > 0 ? work_of(in_dim, rows).bytes : 0; }

int mlp_net_predict(const float *X, int in_dim, int rows, const void *img, const float *const *b, const int32_t *nact,
                    float *prob, int *err, void *stream) {
  RowArgs a;
  int rc = row_args(a, X, in_dim, rows, img, b, nact, err), sms = 0;
  if (rc) return rc;
  if (!prob || !aligned16(prob)) return fail(-1, "mlp_net_predict: prob must be 16-byte aligned");
  if ((rc = sm_count(&sms))) return rc;
  a.prob = prob;
  // more tiles than SMs: two in turn on each
  const bool two = a.tiles > sms;
  auto kern = two ? mlp_rows_kernel<false, 2> : mlp_rows_kernel<false, 1>;
  const size_t smem = two ? kRowSmem<2> : kRowSmem<1>;
  NET_CK(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  kern<<<a.tiles < sms ? a.tiles : sms, mlpf::kThreads, smem, (cudaStream_t)stream>>>(a);
  NET_CK(cudaGetLastError());
  return 0;
}

int mlp_net_grad(const float *X, int in_dim, int rows, const void *img, const float *const *b, const int32_t *nact,
                 const float *target, const float *weight, float *const *gW, float *const *gb, void *work,
                 size_t work_bytes, float **loss, void *stream) {
  if (!target || !gW || !gb || !work || !loss || rows <= 0 || !net_shape(in_dim)) return fail(-1, "mlp_net_grad: bad argument");
  const Work w = work_of(in_dim, rows);
  if (work_bytes < w.bytes) return fail(-1, "mlp_net_grad: the workspace is too small");
  if (!aligned16(work)) return fail(-1, "mlp_net_grad: work must be 16-byte aligned");
  for (int l = 0; l < 4; ++l)
    if (!aligned16(gW[l])) return fail(-1, "mlp_net_grad: the weight gradients must be 16-byte aligned");
  unsigned char *ws = (unsigned char *)work;
  RowArgs a;
  int rc = row_args(a, X, in_dim, rows, img, b, nact, (int *)(ws + w.loss + 4)), sms = 0;
  if (rc) return rc;
  if ((rc = sm_count(&sms))) return rc;
  cudaStream_t s = (cudaStream_t)stream;
  a.target = target;
  a.weight = weight;
  a.loss_rows = (float *)(ws + w.loss_rows);
  a.groups = ws + w.groups;
  a.colsum = (float *)(ws + w.colsum);
  *loss = (float *)(ws + w.loss);
  NET_CK(cudaFuncSetAttribute(mlp_rows_kernel<true, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kRowSmem<1>));
  NET_CK(cudaFuncSetAttribute(mlp_wgrad_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kGradSmem));
  NET_CK(cudaMemsetAsync(ws + w.loss, 0, 8, s));
  mlp_rows_kernel<true, 1><<<a.tiles < sms ? a.tiles : sms, mlpf::kThreads, kRowSmem<1>, s>>>(a);
  NET_CK(cudaGetLastError());
  float *part = (float *)(ws + w.part);
  mlp_wgrad_kernel<<<dim3((unsigned)w.splits, 4), mlpf::kThreads, kGradSmem, s>>>(a.groups, w.n_groups, w.per_split, in_dim,
                                                                            part, w.split_stride, a.err);
  NET_CK(cudaGetLastError());
  ReduceArgs r;
  r.part = part;
  r.colsum = a.colsum;
  r.loss_rows = a.loss_rows;
  for (int l = 0; l < 4; ++l) {
    r.gW[l] = gW[l];
    r.gb[l] = gb[l];
  }
  r.loss = *loss;
  r.split_stride = w.split_stride;
  r.splits = w.splits;
  r.tiles = w.tiles;
  r.B = rows;
  r.in_dim = in_dim;
  const int nb = (int)((w.split_stride / 4 + 255) / 256) + 5;
  mlp_reduce_kernel<<<nb, 256, 0, s>>>(r);
  NET_CK(cudaGetLastError());
  return 0;
}

int mlp_net_adam(float *const *w, const float *const *g, float *const *m, float *const *v, void *const *wb, void *img,
                 int in_dim, float lr, float b1, float b2, float eps, long step, void *stream) {
  if (!w || !wb || !net_shape(in_dim) || (step > 0 && (!g || !m || !v))) return fail(-1, "mlp_net_adam: bad argument");
  AdamArgs a{};
  const int dims[5] = {in_dim, kH, kH, kH, kOut};
  int blk = 0;
  for (int l = 0; l < 4; ++l) {
    a.fi[l] = dims[l];
    a.fo[l] = dims[l + 1];
    a.wb[l] = (__nv_bfloat16 *)wb[l];
    for (int q = 0; q < 2; ++q) {
      const int t = 2 * l + q;
      a.n[t] = q == 0 ? dims[l] * dims[l + 1] : dims[l + 1];
      a.first[t] = blk;
      blk += (a.n[t] + 255) / 256;
      a.w[t] = w[t];
      if (step > 0) {
        a.g[t] = g[t];
        a.m[t] = m[t];
        a.v[t] = v[t];
      }
    }
  }
  a.first[8] = blk;
  a.img = (unsigned char *)img;
  a.in_blocks = (in_dim + kBlkK - 1) / kBlkK;
  a.update = step > 0;
  a.lr = lr;
  a.b1 = b1;
  a.b2 = b2;
  a.eps = eps;
  a.bc1 = step > 0 ? 1.f - powf(b1, (float)step) : 1.f;
  a.bc2 = step > 0 ? 1.f - powf(b2, (float)step) : 1.f;
  mlp_adam_all_kernel<<<blk, 256, 0, (cudaStream_t)stream>>>(a);
  NET_CK(cudaGetLastError());
  return 0;
}

}  // extern "C"
