// nw_embed.cu -- embeddings of a word set: the character CNN's whole forward pass
// (embedding, three convolutions, mean, linear layer) in one kernel, on the
// fifth-generation tensor cores.  Training runs layer by layer (nw_conv.cu): its
// backward pass reads the activations.
//
// Layer by layer, the float32 activations of 128 channels a position went
// through memory between the products (600k words: 2.5 GB written and three
// times that read), through registers into shared memory, and 128 x 128 tiles of
// K = 96 or 384 were too short to hide it: 9.3 ms, 7 % of the tensor pipe.
// Here a position's activations never leave the SM: 600k words 9.3 -> 1.63 ms; 200k
// words 3.20 -> 0.60 ms (0.54 in the kernel, tensor pipe 35 %; the products alone
// are 0.19 at the measured bf16 rate).  What is left is the chain of a block's
// layers, pooling and linear layer, which the other block's products hide in part.
//
//   * Rows.  A block is 128 rows of one word length L: each word's L positions
//     followed by one zero row, floor(129 / (L + 1)) words (at most 64).  The
//     zero rows are the convolutions' padding, for both neighbours.
//   * Activations are kept as bf16 in the canonical K-major layout without
//     swizzle, in chunks of 8 channels: row r of a chunk at 16 (r + 1).  Rows are
//     then 16 bytes apart everywhere, so the operand of the tap at t - 1, t or
//     t + 1 is the same matrix from 0, 16 or 32 bytes in: no im2col copies.
//     Every value is rounded to bf16 (nearest even) once, when it becomes an
//     operand, as in the layer-by-layer products, and the products of an output
//     are added in the same order, so the embeddings are the same bit for bit.
//   * A CTA (one per SM, persistent) works on two blocks at a time, a layer of
//     one and then the same layer of the other: each 24 KiB piece of weights
//     (K = 96), streamed from L2 through a ring that holds one layer, feeds the
//     products of both, and the products of one block run under the other's
//     epilogue.  Eight worker warps a block (two for each row, half the channels
//     each: four leave every warp waiting on its own chain, 0.97 ms for 200k
//     words) stage the embeddings, turn each layer's accumulator (tensor memory)
//     into the next operand in place (bias, ReLU, zero rows), sum the last
//     layer's positions in their order, and write the linear layer's outputs; one
//     thread streams weights, one issues products.
// Every wait is bounded; when one runs out the CTA sets kErrWait, waits (bounded)
// for the copies and products it issued, frees its tensor memory and returns.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "nw_cnn.h"
#include "nw_internal.cuh"
#include "nw_tc.cuh"

namespace nw {
namespace cnn {
namespace {

constexpr int kRows = 128;                   // rows of a block
constexpr int kChunkA = (kRows + 2) * 16;    // bytes of an activation chunk: rows -1 .. 128
constexpr int kActBytes = (kCh / 8) * kChunkA;  // activations of a block
constexpr int kPieceBytes = 24576;           // K = 96 of a convolution's weights
constexpr int kPieceSteps = 6;               // products of K = 16 in it
constexpr int kLinBytes = kCh * kOut * 2;    // the linear layer's weights: one shorter piece
constexpr int kPieces2 = 4;                  // layers 2 and 3; layer 1 and the linear layer have one each
constexpr int kPiecesTile = 2 + 2 * kPieces2;
constexpr int kRing = kPieces2;              // a whole layer: both blocks read a piece before it is replaced
constexpr int kHalf = 128;                   // worker threads of half a block's channels
constexpr int kWorkers = 4 * kHalf / 32;     // worker warps
constexpr int kThreads = kWorkers * 32 + 64;
constexpr int kMaxWords = 64;                // words of a block
constexpr int kSliceStride = kRows + 1;      // pooling: floats between two channels of a 32-channel slice
constexpr int kOffRing = 0;
constexpr int kOffAct = kOffRing + kRing * kPieceBytes;  // two blocks
// after the last convolution a block's activations give way to a slice of its
// outputs and to the pooled operand, 64 rows (the product's other 64 rows read
// what lies behind; their outputs are not used)
constexpr int kOffPooled = 32 * kSliceStride * 4;
constexpr int kPooledChunk = kMaxWords * 16;
constexpr int kOffBias = kOffAct + 2 * kActBytes;        // b1, b2, b3, bl
constexpr int kOffFirst = kOffBias + (3 * kCh + kOut) * 4;  // EmbedArgs::first, 64 entries
constexpr int kOffBars = kOffFirst + 64 * 4;
constexpr int kOffSlice = kOffBars + (2 * kRing + 4) * 8;   // the second halves' slices
constexpr int kOffTable = kOffSlice + 2 * 32 * kSliceStride * 4;  // embeddings in bf16
constexpr int kMaxAlphabet = 256;            // of a model
constexpr int kTableRow = 5;                 // 16-byte units of an embedding (four, and one against bank conflicts)
constexpr int kSmem = kOffTable + kMaxAlphabet * kTableRow * 16;
static_assert(kOffPooled % 16 == 0 && kOffTable % 16 == 0 && kOffPooled + (kCh / 8) * kPooledChunk <= kActBytes, "the pooled operand fits");
static_assert(kOffPooled + (kCh / 8) * kPooledChunk + 1024 <= kActBytes + (kSmem - kOffBias), "its unused rows are shared memory");
static_assert(kMaxLen <= kRows && kBuckets <= 63, "a word fits a block; lengths in two ballots");
static_assert(kSmem <= 227 * 1024 && kEmb == 32 && kCh == 128 && kOut == 64, "one CTA per SM, fixed shapes");
constexpr long long kWaitCycles = 2000000000ll;  // about a second
constexpr uint32_t kIdesc = tc::idesc_bf16(kRows, kCh), kIdescL = tc::idesc_bf16(kRows, kOut);
constexpr uint32_t kTmemCols = 512;  // a block's accumulator at 128 b, its linear layer's at 256 + 64 b

// the weights as the products read them, in the order of use: chunks of 8 K
// values, [row][8] each (W1 12 chunks, W2 and W3 48, Wl 16 of 64 rows)
constexpr size_t kPackBytes = (size_t)(kPiecesTile - 1) * kPieceBytes + kLinBytes;

__global__ void __launch_bounds__(256) pack_weights_kernel(const float* __restrict__ W, Layout L, __nv_bfloat16* out) {
  const int x = blockIdx.x * 256 + threadIdx.x;
  if (x >= (int)(kPackBytes / 2)) return;
  constexpr int n1 = kCh * 3 * kEmb, n2 = kCh * 3 * kCh;
  const float* src;
  int K, rows, at;
  if (x < n1) {
    src = W + L.W1; K = 3 * kEmb; rows = kCh; at = x;
  } else if (x < n1 + n2) {
    src = W + L.W2; K = 3 * kCh; rows = kCh; at = x - n1;
  } else if (x < n1 + 2 * n2) {
    src = W + L.W3; K = 3 * kCh; rows = kCh; at = x - n1 - n2;
  } else {
    src = W + L.Wl; K = kCh; rows = kOut; at = x - n1 - 2 * n2;
  }
  const int chunk = at / (rows * 8), r = at / 8 % rows, k = chunk * 8 + at % 8;
  out[x] = __float2bfloat16_rn(src[(size_t)r * K + k]);
}

struct EmbedArgs {
  const float* params;
  Layout L;
  const __nv_bfloat16* pack;
  const uint32_t* sym;   // the set's symbols (a_enc) and original indices by sorted position
  const uint32_t* perm;
  uint32_t shift, alphabet;
  uint32_t nblocks;
  // by length: first block, words, first sorted position, first symbol
  uint32_t first[kBuckets + 1], count[kBuckets], start[kBuckets], base[kBuckets];
  float* out;            // n x kOut, original order
  uint32_t* err;
};

struct Block {
  uint32_t L, words, pos, sym;  // length, words, first sorted position, first symbol
};

__host__ __device__ constexpr uint32_t block_words(uint32_t L) {
  return 129u / (L + 1u) < (uint32_t)kMaxWords ? 129u / (L + 1u) : (uint32_t)kMaxWords;
}

// block b, by a whole warp; `first` is EmbedArgs::first padded to 64 entries
__device__ __forceinline__ Block block_of(const EmbedArgs& P, const uint32_t* first, uint32_t b) {
  Block k{0u, 0u, 0u, 0u};
  if (b >= P.nblocks) return k;
  const int lane = threadIdx.x & 31;
  const uint32_t L = (uint32_t)__popc(__ballot_sync(~0u, b >= first[lane + 1])) +
                     (uint32_t)__popc(__ballot_sync(~0u, lane < 31 && b >= first[(lane + 33) & 63]));
  const uint32_t w0 = (b - first[L]) * block_words(L);
  k.L = L;
  k.words = min(block_words(L), P.count[L] - w0);
  k.pos = P.start[L] + w0;
  k.sym = P.base[L] + w0 * L;
  return k;
}

// a block's worker threads agree on `ok`; a half's threads meet
__device__ __forceinline__ bool block_and(int blk, bool ok) {
  uint32_t r;
  asm volatile(
      "{\n .reg .pred p, q;\n setp.ne.u32 p, %1, 0;\n barrier.cta.red.and.pred.aligned q, %2, %3, p;\n"
      " selp.u32 %0, 1, 0, q;\n}\n"
      : "=r"(r)
      : "r"((uint32_t)ok), "r"(1 + blk), "n"(2 * kHalf)
      : "memory");
  return r != 0u;
}
__device__ __forceinline__ void half_sync(int blk, int half) {
  asm volatile("barrier.cta.sync.aligned %0, %1;\n" ::"r"(3 + 2 * blk + half), "n"(kHalf) : "memory");
}

__device__ __forceinline__ uint32_t pack2(float a, float b) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<const uint32_t*>(&v);
}
// ReLU of two sums rounded to bf16 (rounding keeps the order, so after it), or 0 (`keep` 0)
__device__ __forceinline__ uint32_t relu2(float a, float b, uint32_t keep) {
  const __nv_bfloat162 v = __hmax2(__floats2bfloat162_rn(a, b), __floats2bfloat162_rn(0.f, 0.f));
  return *reinterpret_cast<const uint32_t*>(&v) & keep;
}

__global__ void __launch_bounds__(kThreads, 1) embed_kernel(const __grid_constant__ EmbedArgs P) {
  extern __shared__ __align__(1024) unsigned char smem[];
  __shared__ uint32_t s_tmem;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  float* s_bias = reinterpret_cast<float*>(smem + kOffBias);
  const uint32_t bar0 = tc::smem_u32(smem + kOffBars);
  auto full_bar = [&](uint32_t s) { return bar0 + 8u * s; };
  auto empty_bar = [&](uint32_t s) { return bar0 + 8u * (kRing + s); };
  // by block: an operand is staged (its warps); a layer's products are done
  auto ready_bar = [&](uint32_t b) { return bar0 + 8u * (2 * kRing + b); };
  auto acc_bar = [&](uint32_t b) { return bar0 + 8u * (2 * kRing + 2 + b); };
  uint32_t* s_first = reinterpret_cast<uint32_t*>(smem + kOffFirst);
  const uint32_t tiles = (P.nblocks + 1u) / 2u;
  const float* W = P.params;
  for (int x = tid; x < kCh; x += kThreads) {
    s_bias[x] = W[P.L.b1 + x];
    s_bias[kCh + x] = W[P.L.b2 + x];
    s_bias[2 * kCh + x] = W[P.L.b3 + x];
    if (x < kOut) s_bias[3 * kCh + x] = W[P.L.bl + x];
    if (x < 64) s_first[x] = x <= kBuckets ? P.first[x] : ~0u;
  }
  uint4* s_table = reinterpret_cast<uint4*>(smem + kOffTable);
  for (uint32_t x = tid; x < P.alphabet * 4u; x += kThreads) {
    const float4* e = reinterpret_cast<const float4*>(W + P.L.emb) + 2u * x;
    const float4 a = __ldg(e), b = __ldg(e + 1);
    s_table[(x >> 2) * kTableRow + (x & 3u)] = make_uint4(pack2(a.x, a.y), pack2(a.z, a.w), pack2(b.x, b.y), pack2(b.z, b.w));
  }
  if (tid == 0) {
    for (uint32_t s = 0; s < (uint32_t)kRing; ++s) {
      tc::mbar_init(full_bar(s), 1);
      tc::mbar_init(empty_bar(s), 1);
    }
    for (uint32_t b = 0; b < 2u; ++b) {
      tc::mbar_init(ready_bar(b), kWorkers / 2);
      tc::mbar_init(acc_bar(b), 1);
    }
    tc::mbar_init_fence();
  }
  if (warp == 0) tc::tmem_alloc(tc::smem_u32(&s_tmem), kTmemCols);
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  const uint32_t tbase = s_tmem;

  if (warp == kWorkers) {
    // ---- weights: every tile's pieces, in order, through the ring
    if (lane == 0) {
      uint32_t u = 0;  // pieces issued
      bool ok = true;
      for (uint32_t t = blockIdx.x; ok && t < tiles; t += gridDim.x)
        for (uint32_t p = 0; p < (uint32_t)kPiecesTile; ++p, ++u) {
          const uint32_t s = u % kRing;
          if (u >= (uint32_t)kRing && !tc::mbar_wait(empty_bar(s), (u / kRing - 1u) & 1u, kWaitCycles)) {
            atomicOr(P.err, kErrWait);
            ok = false;
            break;
          }
          const uint32_t bytes = p + 1u < (uint32_t)kPiecesTile ? kPieceBytes : kLinBytes;
          tc::mbar_expect_tx(full_bar(s), bytes);
          tc::bulk_g2s(tc::smem_u32(smem + kOffRing + s * kPieceBytes),
                       reinterpret_cast<const unsigned char*>(P.pack) + (size_t)p * kPieceBytes, bytes, full_bar(s));
        }
      // every copy issued has landed before the CTA exits (bounded)
      for (uint32_t v = u > (uint32_t)kRing ? u - kRing : 0u; v < u; ++v)
        if (!tc::mbar_wait(full_bar(v % kRing), (v / kRing) & 1u, kWaitCycles)) {
          atomicOr(P.err, kErrWait);
          break;
        }
    }
  } else if (warp == kWorkers + 1) {
    // ---- products.  One thread issues them all, so its own instructions are on
    // the critical path: descriptors are constants added to four bases.
    if (lane == 0) {
      uint32_t u = 0, layers = 0;  // pieces of finished layers, finished layers
      bool ok = true;
      const uint64_t wdesc = tc::smem_desc(tc::smem_u32(smem + kOffRing), 2048u, 128u, 0u);
      const uint64_t ldesc = tc::smem_desc(tc::smem_u32(smem + kOffRing), 1024u, 128u, 0u);
      auto piece_full = [&](uint32_t x) { return tc::mbar_wait(full_bar(x % kRing), (x / kRing) & 1u, kWaitCycles); };
      for (uint32_t t = blockIdx.x; ok && t < tiles; t += gridDim.x)
#pragma unroll 1
        for (uint32_t layer = 0; ok && layer < 4u; ++layer) {
#pragma unroll 1
          for (uint32_t b = 0; b < 2u; ++b) {
            const uint32_t act = tc::smem_u32(smem + kOffAct + b * kActBytes);
            const uint64_t adesc = tc::smem_desc(act, (uint32_t)kChunkA, 128u, 0u);
            const uint32_t acc = tbase + b * (uint32_t)kCh;
            ok = ok && tc::mbar_wait(ready_bar(b), layers & 1u, kWaitCycles);
            if (layer == 0u) {
              if (b == 0u) ok = ok && piece_full(u);
              if (ok) {
                tc::fence_after();
                const uint64_t wd = wdesc + (uint64_t)((u % kRing) * (kPieceBytes / 16));
#pragma unroll
                for (int ks = 0; ks < kPieceSteps; ++ks)  // two a tap
                  tc::mma(acc, adesc + (uint64_t)((ks >> 1) + (ks & 1) * 2 * (kChunkA / 16)), wd + (uint64_t)(ks * 256), kIdesc,
                          ks > 0 ? 1u : 0u);
                if (b == 1u) tc::commit(empty_bar(u % kRing));
              }
            } else if (layer < 3u) {
#pragma unroll
              for (int p = 0; p < kPieces2; ++p) {
                if (b == 0u) ok = ok && piece_full(u + p);
                if (ok) {
                  tc::fence_after();
                  const uint64_t wd = wdesc + (uint64_t)(((u + p) % kRing) * (kPieceBytes / 16));
#pragma unroll
                  for (int ks = 0; ks < kPieceSteps; ++ks) {
                    const int step = p * kPieceSteps + ks;  // eight a tap
                    tc::mma(acc, adesc + (uint64_t)((step >> 3) + (step & 7) * 2 * (kChunkA / 16)), wd + (uint64_t)(ks * 256),
                            kIdesc, step > 0 ? 1u : 0u);
                  }
                  if (b == 1u) tc::commit(empty_bar((u + p) % kRing));
                }
              }
            } else {
              if (b == 0u) ok = ok && piece_full(u);
              if (ok) {
                tc::fence_after();
                const uint64_t wd = ldesc + (uint64_t)((u % kRing) * (kPieceBytes / 16));
                const uint64_t pd = tc::smem_desc(act + (uint32_t)kOffPooled, (uint32_t)kPooledChunk, 128u, 0u);
#pragma unroll
                for (int ks = 0; ks < kCh / 16; ++ks)
                  tc::mma(tbase + 256u + b * (uint32_t)kOut, pd + (uint64_t)(ks * 2 * (kPooledChunk / 16)), wd + (uint64_t)(ks * 128),
                          kIdescL, ks > 0 ? 1u : 0u);
                if (b == 1u) tc::commit(empty_bar(u % kRing));
              }
            }
            // after a wait that ran out too, so that the exit can wait for what was issued
            tc::commit(acc_bar(b));
          }
          u += layer == 1u || layer == 2u ? kPieces2 : 1;
          ++layers;
        }
      if (!ok) atomicOr(P.err, kErrWait);
      // the products issued have completed before tensor memory is freed
      if (layers)
        for (uint32_t b = 0; b < 2u; ++b)
          if (!tc::mbar_wait(acc_bar(b), (layers - 1u) & 1u, kWaitCycles)) atomicOr(P.err, kErrWait);
    }
  } else {
    // ---- workers: thread = row `r` of block `blk`, half its channels
    const int blk = warp >> 3, half = (warp >> 2) & 1, r = tid & (kHalf - 1);
    unsigned char* act = smem + kOffAct + blk * kActBytes;
    float* slice = reinterpret_cast<float*>(half ? smem + kOffSlice + blk * (32 * kSliceStride * 4) : act);
    const uint32_t lane_base = tbase + ((uint32_t)((warp & 3) * 32) << 16);
    uint32_t layers = 0;
    bool ok = true;
    auto publish = [&]() {  // this warp's part of an operand, for the tensor cores
      tc::fence_proxy_async();
      tc::fence_before();
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(ready_bar((uint32_t)blk));
    };
    auto products_done = [&]() {
      const bool got = tc::mbar_wait(acc_bar((uint32_t)blk), layers & 1u, kWaitCycles);
      ++layers;
      ok = block_and(blk, got);
      if (!ok && r == 0) atomicOr(P.err, kErrWait);
      tc::fence_after();
      return ok;
    };
    // the row of block (t, blk): whether it holds a symbol, and the symbol
    Block k;
    uint32_t sym = 0u;
    auto row_of = [&](uint32_t t) {
      k = block_of(P, s_first, 2u * t + (uint32_t)blk);
      const uint32_t w = (uint32_t)r / (k.L + 1u), at = (uint32_t)r % (k.L + 1u);
      const bool have = w < k.words && at < k.L;
      if (have) sym = __ldg(P.sym + k.sym + w * k.L + at);
      return have;
    };
    bool real = row_of(blockIdx.x);
    for (uint32_t t = blockIdx.x; t < tiles; t += gridDim.x) {
      const uint32_t keep = real ? ~0u : 0u;
      // embeddings, and the rows around the block (pooling has overwritten them)
      {
        uint4 q[2] = {make_uint4(0u, 0u, 0u, 0u), make_uint4(0u, 0u, 0u, 0u)};
        if (real) {
          const uint32_t code = (sym & 0xffffu) >> P.shift;
          if (code >= P.alphabet) {
            atomicOr(P.err, kErrInput);
          } else {
            q[0] = s_table[code * kTableRow + 2u * half];
            q[1] = s_table[code * kTableRow + 2u * half + 1u];
          }
        }
#pragma unroll
        for (int c = 0; c < 2; ++c) *reinterpret_cast<uint4*>(act + (2 * half + c) * kChunkA + (r + 1) * 16) = q[c];
        if (half == 0 && r < 2 * (kCh / 8))
          *reinterpret_cast<uint4*>(act + (r >> 1) * kChunkA + (r & 1) * (kRows + 1) * 16) = make_uint4(0u, 0u, 0u, 0u);
      }
      publish();
      // layers 1 and 2: the accumulator becomes the next operand, in place
#pragma unroll 1
      for (int layer = 0; layer < 2; ++layer) {
        if (!products_done()) break;
        const float4* bias = reinterpret_cast<const float4*>(s_bias + layer * kCh);
#pragma unroll 1
        for (int c = half * (kCh / 2); c < (half + 1) * (kCh / 2); c += 32) {
          uint32_t v[32];
          tc::tmem_ld32(lane_base + (uint32_t)(blk * kCh + c), v);
          tc::tmem_wait(v);
#pragma unroll
          for (int j = 0; j < 32; j += 8) {
            const float4 b0 = bias[(c + j) >> 2], b1 = bias[((c + j) >> 2) + 1];
            auto f = [&](int x) { return __uint_as_float(v[j + x]); };
            *reinterpret_cast<uint4*>(act + ((c + j) >> 3) * kChunkA + (r + 1) * 16) =
                make_uint4(relu2(f(0) + b0.x, f(1) + b0.y, keep), relu2(f(2) + b0.z, f(3) + b0.w, keep),
                           relu2(f(4) + b1.x, f(5) + b1.y, keep), relu2(f(6) + b1.z, f(7) + b1.w, keep));
          }
        }
        publish();
      }
      // layer 3: 32 channels at a time to shared memory, each word's positions
      // added in their order (lane = channel), the mean as the linear layer's operand
      if (!ok || !products_done()) break;
      const Block kb = k;  // the next tile's row is read ahead
      if (t + gridDim.x < tiles) real = row_of(t + gridDim.x);
#pragma unroll 1
      for (int c = half * (kCh / 2); c < (half + 1) * (kCh / 2); c += 32) {
        uint32_t v[32];
        tc::tmem_ld32(lane_base + (uint32_t)(blk * kCh + c), v);
        tc::tmem_wait(v);
        const float4* bias = reinterpret_cast<const float4*>(s_bias + 2 * kCh + c);
#pragma unroll
        for (int j = 0; j < 32; j += 4) {
          const float4 b = bias[j >> 2];
          slice[j * kSliceStride + r] = fmaxf(__uint_as_float(v[j]) + b.x, 0.f);
          slice[(j + 1) * kSliceStride + r] = fmaxf(__uint_as_float(v[j + 1]) + b.y, 0.f);
          slice[(j + 2) * kSliceStride + r] = fmaxf(__uint_as_float(v[j + 2]) + b.z, 0.f);
          slice[(j + 3) * kSliceStride + r] = fmaxf(__uint_as_float(v[j + 3]) + b.w, 0.f);
        }
        half_sync(blk, half);
        const int ch = c + lane;
        unsigned char* dst = act + kOffPooled + (ch >> 3) * kPooledChunk + (ch & 7) * 2;
        // four words at a time: four independent chains
#pragma unroll 1
        for (uint32_t x = (uint32_t)(warp & 3); x < kb.words; x += 16u) {
          const float* y[4];
          float acc[4];
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            y[i] = slice + lane * kSliceStride + (int)(min(x + 4u * i, kb.words - 1u) * (kb.L + 1u));
            acc[i] = 0.f;
          }
#pragma unroll 2
          for (uint32_t p = 0; p < kb.L; ++p) {
#pragma unroll
            for (int i = 0; i < 4; ++i) acc[i] += y[i][p];
          }
#pragma unroll
          for (int i = 0; i < 4; ++i)
            if (x + 4u * i < kb.words)
              *reinterpret_cast<__nv_bfloat16*>(dst + (x + 4u * i) * 16u) =
                  __float2bfloat16_rn(kb.L > 0u ? acc[i] / (float)kb.L : 0.f);
        }
        half_sync(blk, half);
      }
      publish();
      if (!products_done()) break;
      if (r < kMaxWords) {  // thread = word: 32 of its 64 outputs
        const bool have = (uint32_t)r < kb.words;
        uint32_t v[32];
        tc::tmem_ld32(lane_base + 256u + (uint32_t)(blk * kOut + half * 32), v);
        tc::tmem_wait(v);
        if (have) {
          float* dst = P.out + (size_t)__ldg(P.perm + kb.pos + (uint32_t)r) * kOut + half * 32;
#pragma unroll
          for (int j = 0; j < 32; j += 4) {
            const float4 b = *reinterpret_cast<const float4*>(s_bias + 3 * kCh + half * 32 + j);
            *reinterpret_cast<float4*>(dst + j) =
                make_float4(__uint_as_float(v[j]) + b.x, __uint_as_float(v[j + 1]) + b.y, __uint_as_float(v[j + 2]) + b.z,
                            __uint_as_float(v[j + 3]) + b.w);
          }
        }
        __syncwarp();
      }
    }
  }
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  if (warp == 0) tc::tmem_dealloc(tbase, kTmemCols);
}

}  // namespace

size_t fwd_pack_bytes() { return kPackBytes; }

cudaError_t pack_fwd(const float* params, const Layout& L, void* pack, cudaStream_t s) {
  pack_weights_kernel<<<(unsigned)((kPackBytes / 2 + 255) / 256), 256, 0, s>>>(params, L, static_cast<__nv_bfloat16*>(pack));
  return cudaGetLastError();
}

cudaError_t embed_words(const float* params, const Layout& L, uint32_t alphabet, const Buckets& bk, const uint32_t* sym,
                        const uint32_t* perm, uint32_t shift, void* pack, float* out, uint32_t* err, int sms,
                        cudaStream_t s) {
  EmbedArgs P{};
  P.params = params;
  P.L = L;
  P.pack = static_cast<const __nv_bfloat16*>(pack);
  P.sym = sym;
  P.perm = perm;
  P.shift = shift;
  P.alphabet = alphabet;
  P.out = out;
  P.err = err;
  for (int len = 0; len < kBuckets; ++len) {
    P.first[len] = P.nblocks;
    P.count[len] = bk.count[len];
    P.start[len] = bk.start[len];
    P.base[len] = bk.aenc_base[len];
    P.nblocks += (bk.count[len] + block_words((uint32_t)len) - 1) / block_words((uint32_t)len);
  }
  P.first[kBuckets] = P.nblocks;
  if (P.nblocks == 0) return cudaSuccess;
  cudaError_t e = pack_fwd(params, L, pack, s);
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(embed_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem);
  if (e != cudaSuccess) return e;
  embed_kernel<<<std::min<unsigned>((P.nblocks + 1u) / 2u, (unsigned)sms), kThreads, kSmem, s>>>(P);
  return cudaGetLastError();
}

}  // namespace cnn
}  // namespace nw
