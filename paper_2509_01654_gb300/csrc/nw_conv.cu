// nw_conv.cu -- the convolutions of a training batch on the fifth-generation
// tensor cores: conv_fwd (one layer's products, bias and ReLU) and conv_bwd (one
// layer's weight, bias and input gradients from a single read of the output
// gradient and of the layer's input).
//
// As separate products (forward with gathered windows; dW split over rows with
// atomics, dX, column sums) each read the 128 float32 channels of every row
// again, three times for the taps, through registers: 64 us a layer forward and
// 364 us backward for 132k rows, where moving each operand once is 135 MB
// (20 us) and 200 MB (30 us).  Here: 28 to 39 us a layer forward, 42 to 79
// backward; a CTA's reads, products and stores of a tile overlap only in part.
//
//   * Rows are taken in padded order (Packed::prow): every word's rows, then one
//     zero row.  A tile is 128 padded rows and one on either side.  With the zero
//     rows in place a tap is a shift by one row for every word at once.
//   * Operands lie in shared memory as bf16 (rounded to nearest even from float32
//     as they are read, once), in chunks of 8 channels: row r of a chunk at
//     16 (r + 1).  Read with rows as M and channels as K (K-major), a shifted
//     start address gives the layer's windows, and the output gradient gives
//     dX = sum over taps of its rows moved by 1 - tap against the layer's weights.
//     Read with channels as M and rows as K (MN-major), the same bytes give dW,
//     with the input's rows moved by tap - 1.  No operand is transposed or copied
//     for a tap.
//   * A CTA (one per SM, persistent) keeps the layer's weights in shared memory
//     and dW (128 x 3 Ci) in tensor memory over all its tiles; dW is added to
//     memory once, four floats a reduction.  The next tile's rows are read into
//     registers, all loads of a tile in flight together, while the tensor cores
//     work on this one.
//   * Results leave 32 bytes a lane pair (store_row): 16 bytes a lane are half
//     sectors.
// Every wait is bounded; when one runs out the CTA sets kErrWait, waits
// (bounded) for what it issued, frees its tensor memory and returns.
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

constexpr int kRows = 128;                     // padded rows of a tile
constexpr int kChunk = (kRows + 2) * 16;       // bytes of a chunk of 8 channels: rows -1 .. 128
constexpr int kAct = (kCh / 8) * kChunk;       // bytes of 128 channels
constexpr int kThreads = 512, kWarps = kThreads / 32;
constexpr int kK = kTaps * kCh;                // dX: K = (tap, output channel)
constexpr int kOffDy = kK * kCh * 2;           // behind the weights
constexpr int kOffX = kOffDy + kAct;
constexpr int kOffGate = kOffX + kAct;         // [row][channel / 8]: bit i set where the input's channel i is positive
constexpr int kOffRow = kOffGate + kRows * (kCh / 8);  // the tile's packed rows, by row slot
constexpr int kOffBars = kOffRow + (kRows + 8) * 4;
constexpr int kSmem = kOffBars + 3 * 8 + 8;
constexpr uint32_t kDxCol = 384;               // tensor memory: dW at 0, dX here
constexpr int kPiece = 24576;                  // weights: bytes a copy
constexpr long long kWaitCycles = 2000000000ll;  // about a second
static_assert(kSmem <= 227 * 1024 && kCh == 128 && kTaps == 3, "fixed shapes");
static_assert(kWarps * 2 * 4 == kRows && kWarps * kCh * 4 <= kAct, "four rows a thread; bias sums fit the operand");

struct BwdArgs {
  const float* dY;      // output gradient, or (top layer) null:
  const float* Ytop;    //   the layer's output, its gradient the mean's: Y > 0 ? dP[word] : 0
  const float* dP;
  const int* rword;
  const float* X;       // the layer's input
  const int* prow;
  const int* Tp;        // padded rows, at most cap
  int cap;
  const __nv_bfloat16* wpack;
  float* dX;            // x (X > 0) for 128 input channels
  float* dW;
  float* db;
  uint32_t* err;
};

__device__ __forceinline__ uint32_t pack2(float a, float b) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<const uint32_t*>(&v);
}
__device__ __forceinline__ uint4 pack8(float4 a, float4 b) {
  return make_uint4(pack2(a.x, a.y), pack2(a.z, a.w), pack2(b.x, b.y), pack2(b.z, b.w));
}
__device__ __forceinline__ uint32_t positive8(float4 a, float4 b) {
  return (a.x > 0.f ? 1u : 0u) | (a.y > 0.f ? 2u : 0u) | (a.z > 0.f ? 4u : 0u) | (a.w > 0.f ? 8u : 0u) |
         (b.x > 0.f ? 16u : 0u) | (b.y > 0.f ? 32u : 0u) | (b.z > 0.f ? 64u : 0u) | (b.w > 0.f ? 128u : 0u);
}

// A row's 32 values of a warp's rows (lane = row), whose pointers are `dst` (null: no
// row): lanes 2 i and 2 i + 1 exchange halves of 8 values, so that one store of the
// pair covers 32 bytes of one row.
__device__ __forceinline__ void store_row(float* dst, const float (&v)[32]) {
  const bool odd = threadIdx.x & 1;
  float* other = reinterpret_cast<float*>(__shfl_xor_sync(~0u, reinterpret_cast<unsigned long long>(dst), 1));
  float* even_row = odd ? other : dst;
  float* odd_row = odd ? dst : other;
#pragma unroll
  for (int j = 0; j < 32; j += 8) {
    float mine[4], got[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      mine[i] = odd ? v[j + 4 + i] : v[j + i];
      got[i] = __shfl_xor_sync(~0u, odd ? v[j + i] : v[j + 4 + i], 1);
    }
    // even lane: its own values j .. j + 3, the odd row's j .. j + 3; odd lane: j + 4 .. j + 7 of both
    const float4 e = odd ? make_float4(got[0], got[1], got[2], got[3]) : make_float4(mine[0], mine[1], mine[2], mine[3]);
    const float4 o = odd ? make_float4(mine[0], mine[1], mine[2], mine[3]) : make_float4(got[0], got[1], got[2], got[3]);
    if (even_row) *reinterpret_cast<float4*>(even_row + j + (odd ? 4 : 0)) = e;
    if (odd_row) *reinterpret_cast<float4*>(odd_row + j + (odd ? 4 : 0)) = o;
  }
}

// W[128][3][Ci] as the (tap, output) x input operand: chunks of 8 outputs, [ci][8]
__global__ void __launch_bounds__(256) pack_bwd_kernel(const float* __restrict__ W, Layout L, __nv_bfloat16* out) {
  const int x = blockIdx.x * 256 + threadIdx.x;
  constexpr int n3 = kK * kCh, n1 = kK * kEmb;
  if (x >= 2 * n3 + n1) return;
  const int layer = x < n3 ? 3 : (x < 2 * n3 ? 2 : 1);
  const int at = layer == 3 ? x : (layer == 2 ? x - n3 : x - 2 * n3);
  const int Ci = layer == 1 ? kEmb : kCh;
  const float* w = W + (layer == 3 ? L.W3 : (layer == 2 ? L.W2 : L.W1));
  const int ci = at / 8 % Ci, k = at / (8 * Ci) * 8 + at % 8;
  out[x] = __float2bfloat16_rn(w[((size_t)(k % kCh) * kTaps + k / kCh) * Ci + ci]);
}

template <int Ci, bool kTop>
__global__ void __launch_bounds__(kThreads, 1) conv_bwd_kernel(const __grid_constant__ BwdArgs P) {
  constexpr uint32_t kDxIdesc = tc::idesc_bf16(kRows, Ci);
  constexpr uint32_t kDwIdesc = tc::idesc_bf16(kRows, Ci) | (1u << 15) | (1u << 16);  // both MN-major
  constexpr int kXq = Ci == kCh ? 5 : 2;  // input chunks a thread reads ahead (the last: two row slots' only)
  extern __shared__ __align__(1024) unsigned char smem[];
  __shared__ uint32_t s_tmem;
  const int Tp = min(*P.Tp, P.cap);
  const int tiles = (Tp + kRows - 1) / kRows;
  if ((int)blockIdx.x >= tiles) return;  // block-uniform, before any barrier or allocation
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  unsigned char* s_dy = smem + kOffDy;
  unsigned char* s_x = smem + kOffX;
  const uint32_t bar0 = tc::smem_u32(smem + kOffBars);
  const uint32_t w_bar = bar0, dx_bar = bar0 + 8u, dw_bar = bar0 + 16u;
  if (tid == 0) {
    tc::mbar_init(w_bar, 1);
    tc::mbar_init(dx_bar, 1);
    tc::mbar_init(dw_bar, 1);
    tc::mbar_init_fence();
  }
  if (warp == 0) tc::tmem_alloc(tc::smem_u32(&s_tmem), 512u);
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  const uint32_t tbase = s_tmem;
  if (tid == 0) {
    tc::mbar_expect_tx(w_bar, kK * Ci * 2);
    for (int o = 0; o < kK * Ci * 2; o += kPiece)
      tc::bulk_g2s(tc::smem_u32(smem + o), reinterpret_cast<const unsigned char*>(P.wpack) + o, kPiece, w_bar);
  }

  // 128 channels: eight lanes of a warp hold 4 chunks of 2 rows (their 16-byte
  // stores meet no bank twice), a chunk's 32 bytes come from one sector; row
  // slots 0 .. 129 are rows -1 .. 128, four a thread and two of warp 0.
  // 32 channels: thread = (row slot, chunk), and eight of warp 0.
  const int ch = (lane & 3) + 4 * (lane >> 3);
  auto slot_of = [&](int q) { return 2 * (warp + kWarps * q) + ((lane >> 2) & 1); };
  auto packed_row = [&](int tile, int slot) {
    const int p = tile * kRows + slot - 1;
    return slot < kRows + 2 && p >= 0 && p < Tp ? __ldg(P.prow + p) : -1;
  };
  auto xslot_of = [&](int q) { return Ci == kCh ? slot_of(q) : (tid + kThreads * q) >> 2; };
  const int xch = Ci == kCh ? ch : tid & 3;
  int* s_row = reinterpret_cast<int*>(smem + kOffRow);
  float db[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) db[i] = 0.f;
  int row[5], nrow[5];  // packed rows of this thread's slots: the tile being read, the one after
  uint4 ndy[5], nx[kXq];
  uint32_t ngate[kXq];
  auto rows_of = [&](int tile) {
#pragma unroll
    for (int q = 0; q < 5; ++q) nrow[q] = tile < tiles ? packed_row(tile, slot_of(q)) : -1;
  };
  auto add_dy = [&](int q, float4 a, float4 b) {
    const int slot = slot_of(q);
    if (slot >= 1 && slot <= kRows) {  // the neighbours' rows are other tiles'
      db[0] += a.x; db[1] += a.y; db[2] += a.z; db[3] += a.w;
      db[4] += b.x; db[5] += b.y; db[6] += b.z; db[7] += b.w;
    }
    ndy[q] = pack8(a, b);
  };
  const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
  // the rows of `tile`, whose packed rows are in nrow; then the next tile's packed rows
  auto read_tile = [&](int tile) {
#pragma unroll
    for (int q = 0; q < 5; ++q) row[q] = nrow[q];
    if (kTop) {
      int word[5];
#pragma unroll
      for (int q = 0; q < 5; ++q) word[q] = row[q] >= 0 ? __ldg(P.rword + row[q]) : 0;
#pragma unroll
      for (int q0 = 0; q0 < 5; q0 += 3) {  // (three rows of both operands at a time: registers)
        float4 y[6], d[6];
#pragma unroll
        for (int i = 0; i < 3 && q0 + i < 5; ++i) {
          const float4* yp = reinterpret_cast<const float4*>(P.Ytop + (size_t)max(row[q0 + i], 0) * kCh + ch * 8);
          const float4* dp = reinterpret_cast<const float4*>(P.dP + (size_t)word[q0 + i] * kCh + ch * 8);
          const bool in = row[q0 + i] >= 0;
          y[2 * i] = in ? __ldg(yp) : zero;
          y[2 * i + 1] = in ? __ldg(yp + 1) : zero;
          d[2 * i] = in ? __ldg(dp) : zero;
          d[2 * i + 1] = in ? __ldg(dp + 1) : zero;
        }
#pragma unroll
        for (int i = 0; i < 3 && q0 + i < 5; ++i) {
          const float4 ya = y[2 * i], yb = y[2 * i + 1], da = d[2 * i], e = d[2 * i + 1];
          auto f = [](float yv, float dv) { return yv > 0.f ? dv : 0.f; };
          add_dy(q0 + i, make_float4(f(ya.x, da.x), f(ya.y, da.y), f(ya.z, da.z), f(ya.w, da.w)),
                 make_float4(f(yb.x, e.x), f(yb.y, e.y), f(yb.z, e.z), f(yb.w, e.w)));
        }
      }
    } else {
      float4 y[10];
#pragma unroll
      for (int q = 0; q < 5; ++q) {
        const float4* yp = reinterpret_cast<const float4*>(P.dY + (size_t)max(row[q], 0) * kCh + ch * 8);
        y[2 * q] = row[q] >= 0 ? __ldg(yp) : zero;
        y[2 * q + 1] = row[q] >= 0 ? __ldg(yp + 1) : zero;
      }
#pragma unroll
      for (int q = 0; q < 5; ++q) add_dy(q, y[2 * q], y[2 * q + 1]);
    }
    float4 x[2 * kXq];
#pragma unroll
    for (int q = 0; q < kXq; ++q) {
      const int t = Ci == kCh ? row[q] : packed_row(tile, xslot_of(q));
      const float4* xp = reinterpret_cast<const float4*>(P.X + (size_t)max(t, 0) * Ci + xch * 8);
      x[2 * q] = t >= 0 ? __ldg(xp) : zero;
      x[2 * q + 1] = t >= 0 ? __ldg(xp + 1) : zero;
    }
    rows_of(tile + (int)gridDim.x);
#pragma unroll
    for (int q = 0; q < kXq; ++q) {
      nx[q] = pack8(x[2 * q], x[2 * q + 1]);
      ngate[q] = positive8(x[2 * q], x[2 * q + 1]);
    }
  };
  auto put_tile = [&]() {
#pragma unroll
    for (int q = 0; q < 5; ++q) {
      const int slot = slot_of(q);
      if (slot >= kRows + 2) continue;
      *reinterpret_cast<uint4*>(s_dy + ch * kChunk + slot * 16) = ndy[q];
      if (ch == 0) s_row[slot] = row[q];
    }
#pragma unroll
    for (int q = 0; q < kXq; ++q) {
      const int slot = xslot_of(q);
      if (slot >= kRows + 2) continue;
      *reinterpret_cast<uint4*>(s_x + xch * kChunk + slot * 16) = nx[q];
      if (Ci == kCh && slot >= 1 && slot <= kRows) smem[kOffGate + (slot - 1) * (kCh / 8) + xch] = (unsigned char)ngate[q];
    }
  };

  rows_of(blockIdx.x);
  read_tile(blockIdx.x);
  put_tile();
  bool ok = true, issued = false;
  uint32_t n = 0;
  for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x, ++n) {
    tc::fence_proxy_async();  // the operands, for the tensor cores
    tc::fence_before();       // last tile's dX has been read
    __syncthreads();
    if (tid == 0 && (n > 0 || tc::mbar_wait(w_bar, 0u, kWaitCycles))) {
      tc::fence_after();
      const uint64_t a = tc::smem_desc(tc::smem_u32(s_dy), (uint32_t)kChunk, 128u, 0u);
      const uint64_t b = tc::smem_desc(tc::smem_u32(smem), (uint32_t)(Ci * 16), 128u, 0u);
#pragma unroll 8
      for (int ks = 0; ks < kK / 16; ++ks)  // eight a tap
        tc::mma(tbase + kDxCol, a + (uint64_t)(2 - (ks >> 3) + (ks & 7) * 2 * (kChunk / 16)), b + (uint64_t)(ks * 2 * Ci),
                kDxIdesc, ks > 0 ? 1u : 0u);
      tc::commit(dx_bar);
      // MN-major: 8 channels to the next at the stride offset, 8 rows to the next at the leading offset
      const uint64_t at = tc::smem_desc(tc::smem_u32(s_dy), 128u, (uint32_t)kChunk, 0u);
      const uint64_t bt = tc::smem_desc(tc::smem_u32(s_x), 128u, (uint32_t)kChunk, 0u);
#pragma unroll 1
      for (int tap = 0; tap < kTaps; ++tap)
#pragma unroll
        for (int ks = 0; ks < kRows / 16; ++ks)
          tc::mma(tbase + (uint32_t)(tap * Ci), at + (uint64_t)(1 + ks * 16), bt + (uint64_t)(tap + ks * 16), kDwIdesc,
                  n > 0 || ks > 0 ? 1u : 0u);
      tc::commit(dw_bar);
      issued = true;
    }
    const int next = tile + (int)gridDim.x;
    if (next < tiles) read_tile(next);  // in flight while the products run
    ok = __syncthreads_and(tc::mbar_wait(dx_bar, n & 1u, kWaitCycles)) != 0;
    if (!ok) break;
    tc::fence_after();
    if (warp < 4 * (Ci / 32)) {  // thread = row, 32 input channels
      const int r = (warp & 3) * 32 + lane, c = (warp >> 2) * 32;
      uint32_t v[32];
      tc::tmem_ld32(tbase + ((uint32_t)((warp & 3) * 32) << 16) + kDxCol + (uint32_t)c, v);
      tc::tmem_wait(v);
      const int t = s_row[r + 1];
      const uint32_t gate =
          Ci == kCh ? *reinterpret_cast<const uint32_t*>(smem + kOffGate + r * (kCh / 8) + (warp >> 2) * 4) : ~0u;
      float o[32];
#pragma unroll
      for (int j = 0; j < 32; ++j) o[j] = gate >> j & 1u ? __uint_as_float(v[j]) : 0.f;
      store_row(t >= 0 ? P.dX + (size_t)t * Ci + c : nullptr, o);
    }
    ok = __syncthreads_and(tc::mbar_wait(dw_bar, n & 1u, kWaitCycles)) != 0;
    if (!ok) break;
    if (next < tiles) put_tile();
  }
  if (ok) {
    tc::fence_after();
    // dW: lane = output channel, 32 columns a load; CTAs start at different columns
    const int o = (warp & 3) * 32 + lane;
    constexpr int kGroups = kTaps * Ci / 32;
#pragma unroll 1
    for (int x = warp >> 2; x < kGroups; x += kWarps / 4) {
      const int c = (x + (int)blockIdx.x) % kGroups * 32;
      uint32_t v[32];
      tc::tmem_ld32(tbase + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)c, v);
      tc::tmem_wait(v);
      float4* dst = reinterpret_cast<float4*>(P.dW + (size_t)o * (kTaps * Ci) + c);
#pragma unroll
      for (int j = 0; j < 8; ++j)
        atomicAdd(dst + j, make_float4(__uint_as_float(v[4 * j]), __uint_as_float(v[4 * j + 1]), __uint_as_float(v[4 * j + 2]),
                                       __uint_as_float(v[4 * j + 3])));
    }
    // db: two rows of a warp, then the warps
    float* s_db = reinterpret_cast<float*>(s_dy);
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      db[i] += __shfl_xor_sync(~0u, db[i], 4);
      if (!(lane & 4)) s_db[warp * kCh + ch * 8 + i] = db[i];
    }
    __syncthreads();
    if (tid < kCh) {
      float sum = 0.f;
#pragma unroll
      for (int w = 0; w < kWarps; ++w) sum += s_db[w * kCh + tid];
      atomicAdd(P.db + tid, sum);
    }
  } else if (tid == 0) {
    atomicOr(P.err, kErrWait);
    // what was issued has completed before tensor memory is freed (bounded)
    tc::mbar_wait(w_bar, 0u, kWaitCycles);
    if (issued) tc::mbar_wait(dw_bar, n & 1u, kWaitCycles);
  }
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  if (warp == 0) tc::tmem_dealloc(tbase, 512u);
}

struct FwdArgs {
  const float* X;
  const int* prow;
  const int* Tp;        // padded rows, at most cap
  int cap;
  const __nv_bfloat16* wpack;  // chunks of 8 of K = (tap, input channel), [output][8]
  const float* bias;
  float* Y;
  uint32_t* err;
};

template <int Ci>
__global__ void __launch_bounds__(kThreads, 1) conv_fwd_kernel(const __grid_constant__ FwdArgs P) {
  constexpr int kKf = kTaps * Ci;
  constexpr int kChunks = Ci / 8;                      // of a row
  constexpr int kQ = ((kRows + 2) * kChunks + kThreads - 1) / kThreads;  // chunks a thread reads
  constexpr uint32_t kIdesc = tc::idesc_bf16(kRows, kCh);
  extern __shared__ __align__(1024) unsigned char smem[];
  __shared__ uint32_t s_tmem;
  const int Tp = min(*P.Tp, P.cap);
  const int tiles = (Tp + kRows - 1) / kRows;
  if ((int)blockIdx.x >= tiles) return;  // block-uniform, before any barrier or allocation
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  unsigned char* s_x = smem + kOffX;
  float* s_bias = reinterpret_cast<float*>(smem + kOffGate);
  const uint32_t w_bar = tc::smem_u32(smem + kOffBars), y_bar = w_bar + 8u;
  if (tid == 0) {
    tc::mbar_init(w_bar, 1);
    tc::mbar_init(y_bar, 1);
    tc::mbar_init_fence();
  }
  if (tid < kCh) s_bias[tid] = __ldg(P.bias + tid);
  if (warp == 0) tc::tmem_alloc(tc::smem_u32(&s_tmem), kCh);
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  const uint32_t tbase = s_tmem;
  if (tid == 0) {
    tc::mbar_expect_tx(w_bar, kKf * kCh * 2);
    for (int o = 0; o < kKf * kCh * 2; o += kPiece)
      tc::bulk_g2s(tc::smem_u32(smem + o), reinterpret_cast<const unsigned char*>(P.wpack) + o, kPiece, w_bar);
  }
  // as in the backward kernel: eight lanes store 4 chunks of 2 rows
  const int ch = Ci == kCh ? (lane & 3) + 4 * (lane >> 3) : tid & 3;
  auto slot_of = [&](int q) {
    return Ci == kCh ? 2 * (warp + kWarps * q) + ((lane >> 2) & 1) : (tid + kThreads * q) >> 2;
  };
  int* s_row = reinterpret_cast<int*>(smem + kOffRow);
  int row[kQ], nrow[kQ];
  uint4 nx[kQ];
  auto rows_of = [&](int tile) {
#pragma unroll
    for (int q = 0; q < kQ; ++q) {
      const int slot = slot_of(q), p = tile * kRows + slot - 1;
      nrow[q] = tile < tiles && slot < kRows + 2 && p >= 0 && p < Tp ? __ldg(P.prow + p) : -1;
    }
  };
  auto read_tile = [&](int tile) {
    float4 x[2 * kQ];
#pragma unroll
    for (int q = 0; q < kQ; ++q) {
      row[q] = nrow[q];
      const float4* xp = reinterpret_cast<const float4*>(P.X + (size_t)max(row[q], 0) * Ci + ch * 8);
      x[2 * q] = row[q] >= 0 ? __ldg(xp) : make_float4(0.f, 0.f, 0.f, 0.f);
      x[2 * q + 1] = row[q] >= 0 ? __ldg(xp + 1) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    rows_of(tile + (int)gridDim.x);
#pragma unroll
    for (int q = 0; q < kQ; ++q) nx[q] = pack8(x[2 * q], x[2 * q + 1]);
  };
  auto put_tile = [&]() {
#pragma unroll
    for (int q = 0; q < kQ; ++q) {
      const int slot = slot_of(q);
      if (slot >= kRows + 2) continue;
      *reinterpret_cast<uint4*>(s_x + ch * kChunk + slot * 16) = nx[q];
      if (ch == 0) s_row[slot] = row[q];
    }
  };
  rows_of(blockIdx.x);
  read_tile(blockIdx.x);
  put_tile();
  bool ok = true, issued = false;
  uint32_t n = 0;
  for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x, ++n) {
    tc::fence_proxy_async();
    tc::fence_before();
    __syncthreads();
    if (tid == 0 && (n > 0 || tc::mbar_wait(w_bar, 0u, kWaitCycles))) {
      tc::fence_after();
      const uint64_t a = tc::smem_desc(tc::smem_u32(s_x), (uint32_t)kChunk, 128u, 0u);
      const uint64_t b = tc::smem_desc(tc::smem_u32(smem), 2048u, 128u, 0u);
#pragma unroll 6
      for (int ks = 0; ks < kKf / 16; ++ks) {
        const int tap = ks / (Ci / 16), at = ks % (Ci / 16);
        tc::mma(tbase, a + (uint64_t)(tap + at * 2 * (kChunk / 16)), b + (uint64_t)(ks * 256), kIdesc, ks > 0 ? 1u : 0u);
      }
      tc::commit(y_bar);
      issued = true;
    }
    const int next = tile + (int)gridDim.x;
    const int t = s_row[(warp & 3) * 32 + lane + 1];  // thread = row, 32 channels
    if (next < tiles) read_tile(next);  // in flight while the products run
    ok = __syncthreads_and(tc::mbar_wait(y_bar, n & 1u, kWaitCycles)) != 0;
    if (!ok) break;
    if (next < tiles) put_tile();  // the products have read this tile's rows, the threads their packed rows
    tc::fence_after();
    const int c = (warp >> 2) * 32;
    uint32_t v[32];
    tc::tmem_ld32(tbase + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)c, v);
    tc::tmem_wait(v);
    float o[32];
#pragma unroll
    for (int j = 0; j < 32; ++j) o[j] = fmaxf(__uint_as_float(v[j]) + s_bias[c + j], 0.f);
    store_row(t >= 0 ? P.Y + (size_t)t * kCh + c : nullptr, o);
  }
  if (!ok && tid == 0) {
    atomicOr(P.err, kErrWait);
    // what was issued has completed before tensor memory is freed (bounded)
    tc::mbar_wait(w_bar, 0u, kWaitCycles);
    if (issued) tc::mbar_wait(y_bar, n & 1u, kWaitCycles);
  }
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  if (warp == 0) tc::tmem_dealloc(tbase, kCh);
}

template <int Ci>
cudaError_t launch_fwd(const FwdArgs& P, int sms, cudaStream_t s) {
  const int tiles = (P.cap + kRows - 1) / kRows;
  if (tiles <= 0) return cudaSuccess;
  cudaError_t e = cudaFuncSetAttribute(conv_fwd_kernel<Ci>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem);
  if (e != cudaSuccess) return e;
  conv_fwd_kernel<Ci><<<std::min(tiles, sms), kThreads, kSmem, s>>>(P);
  return cudaGetLastError();
}

template <int Ci, bool kTop>
cudaError_t launch(const BwdArgs& P, int sms, cudaStream_t s) {
  const int tiles = (P.cap + kRows - 1) / kRows;
  if (tiles <= 0) return cudaSuccess;
  cudaError_t e = cudaFuncSetAttribute(conv_bwd_kernel<Ci, kTop>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem);
  if (e != cudaSuccess) return e;
  conv_bwd_kernel<Ci, kTop><<<std::min(tiles, sms), kThreads, kSmem, s>>>(P);
  return cudaGetLastError();
}

}  // namespace

size_t bwd_pack_bytes() { return (size_t)kK * (2 * kCh + kEmb) * 2; }

cudaError_t pack_bwd(const float* params, const Layout& L, void* pack, cudaStream_t s) {
  pack_bwd_kernel<<<(unsigned)((bwd_pack_bytes() / 2 + 255) / 256), 256, 0, s>>>(params, L, static_cast<__nv_bfloat16*>(pack));
  return cudaGetLastError();
}

cudaError_t conv_fwd(int layer, const float* X, const Packed& pk, const void* pack, const float* bias, float* Y,
                     uint32_t* err, int sms, cudaStream_t s) {
  // the packed weights are in the order of the layers, W1 of 96 x 128
  FwdArgs P{X, pk.prow, pk.Tp, pk.Tmax + pk.Bw, static_cast<const __nv_bfloat16*>(pack), bias, Y, err};
  if (layer == 1) return launch_fwd<kEmb>(P, sms, s);
  P.wpack += (size_t)kTaps * kEmb * kCh + (size_t)(layer - 2) * kK * kCh;
  return launch_fwd<kCh>(P, sms, s);
}

cudaError_t conv_bwd(int layer, const float* dY, const float* Ytop, const float* dP, const float* X, const Packed& pk,
                     const void* pack, float* dX, float* dW, float* db, uint32_t* err, int sms, cudaStream_t s) {
  BwdArgs P{};
  P.dY = dY;
  P.Ytop = Ytop;
  P.dP = dP;
  P.rword = pk.rword;
  P.X = X;
  P.prow = pk.prow;
  P.Tp = pk.Tp;
  P.cap = pk.Tmax + pk.Bw;
  P.wpack = static_cast<const __nv_bfloat16*>(pack) + (size_t)(3 - layer) * kK * kCh;
  P.dX = dX;
  P.dW = dW;
  P.db = db;
  P.err = err;
  if (layer == 3) return launch<kCh, true>(P, sms, s);
  if (layer == 2) return launch<kCh, false>(P, sms, s);
  return launch<kEmb, false>(P, sms, s);
}

}  // namespace cnn
}  // namespace nw
