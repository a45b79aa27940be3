// nw_conv_bwd.cu -- backward pass of one convolution of the proposal network in
// one kernel: weight gradient, bias gradient and input gradient from a single
// read of the output gradient and of the layer's input.
//
// As separate products (dW split over rows with atomics, dX, column sums) each
// read the 128 float32 channels of every row again, through registers, and ran
// on the warp-level tensor path: 364 us a layer for 164k rows, where reading
// both operands and writing dX once is 250 MB, about 37 us.
//
//   * Rows are taken in padded order (Packed::prow): every word's rows, then one
//     zero row.  A tile is 128 padded rows and one on either side.  With the zero
//     rows in place a tap is a shift by one row for every word at once.
//   * Both operands lie in shared memory as bf16 (rounded to nearest even from
//     float32 as they are read, once), in chunks of 8 channels: row r of a chunk
//     at 16 (r + 1).  Read with rows as M and channels as K (K-major) the output
//     gradient gives dX = sum over taps of its rows moved by 1 - tap against the
//     layer's weights; read with channels as M and rows as K (MN-major) the same
//     bytes give dW, with the input's rows moved by tap - 1.  No operand is
//     transposed or copied for a tap.
//   * dW (128 x 3 Ci) stays in tensor memory over all tiles of a CTA (one per
//     SM, persistent) and is added to memory once, four floats a reduction; the
//     layer's weights stay in shared memory.  The next tile's rows are read into
//     registers while the tensor cores work on this one.
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
constexpr int kOffBars = kOffGate + kRows * (kCh / 8);
constexpr int kSmem = kOffBars + 3 * 8 + 8;
constexpr uint32_t kDxCol = 384;               // tensor memory: dW at 0, dX here
constexpr int kPiece = 24576;                  // weights: bytes a copy
constexpr long long kWaitCycles = 2000000000ll;  // about a second
static_assert(kSmem <= 227 * 1024 && kCh == 128 && kTaps == 3, "fixed shapes");
static_assert(kWarps * 2 * 4 == kRows && kWarps * kCh * 4 <= kAct, "four rows a thread; bias sums fit the operand");

struct BwdArgs {
  const float* dY;      // output gradient, or (top layer) null:
  const float* Ytop;    //   the layer's output, its gradient the mean's: Y > 0 ? dP[word] / length : 0
  const float* dP;
  const int* rinfo;
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
  float db[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) db[i] = 0.f;
  auto read_dy = [&](int tile, int slot) {
    const int t = packed_row(tile, slot);
    if (t < 0) return make_uint4(0u, 0u, 0u, 0u);
    float4 a, b;
    if (kTop) {
      const float4* y = reinterpret_cast<const float4*>(P.Ytop + (size_t)t * kCh + ch * 8);
      const float4* d = reinterpret_cast<const float4*>(P.dP + (size_t)__ldg(P.rword + t) * kCh + ch * 8);
      const float4 ya = __ldg(y), yb = __ldg(y + 1), da = __ldg(d), e = __ldg(d + 1);
      const float len = (float)(__ldg(P.rinfo + t) & 255);
      a = make_float4(ya.x > 0.f ? da.x / len : 0.f, ya.y > 0.f ? da.y / len : 0.f, ya.z > 0.f ? da.z / len : 0.f,
                      ya.w > 0.f ? da.w / len : 0.f);
      b = make_float4(yb.x > 0.f ? e.x / len : 0.f, yb.y > 0.f ? e.y / len : 0.f, yb.z > 0.f ? e.z / len : 0.f,
                      yb.w > 0.f ? e.w / len : 0.f);
    } else {
      const float4* y = reinterpret_cast<const float4*>(P.dY + (size_t)t * kCh + ch * 8);
      a = __ldg(y);
      b = __ldg(y + 1);
    }
    if (slot >= 1 && slot <= kRows) {  // the neighbours' rows are other tiles'
      db[0] += a.x; db[1] += a.y; db[2] += a.z; db[3] += a.w;
      db[4] += b.x; db[5] += b.y; db[6] += b.z; db[7] += b.w;
    }
    return pack8(a, b);
  };
  auto read_x = [&](int tile, int slot, int c, uint32_t& gate) {
    const int t = packed_row(tile, slot);
    gate = 0u;
    if (t < 0) return make_uint4(0u, 0u, 0u, 0u);
    const float4* x = reinterpret_cast<const float4*>(P.X + (size_t)t * Ci + c * 8);
    const float4 a = __ldg(x), b = __ldg(x + 1);
    gate = positive8(a, b);
    return pack8(a, b);
  };
  auto put_x = [&](int slot, int c, uint4 v, uint32_t gate) {
    *reinterpret_cast<uint4*>(s_x + c * kChunk + slot * 16) = v;
    if (Ci == kCh && slot >= 1 && slot <= kRows) smem[kOffGate + (slot - 1) * (kCh / 8) + c] = (unsigned char)gate;
  };
  uint4 ndy[5], nx[kXq];
  uint32_t ngate[kXq];
  auto xslot_of = [&](int q) { return Ci == kCh ? slot_of(q) : (tid + kThreads * q) >> 2; };
  const int xch = Ci == kCh ? ch : tid & 3;
  auto read_tile = [&](int tile) {
#pragma unroll
    for (int q = 0; q < 5; ++q) ndy[q] = read_dy(tile, slot_of(q));
#pragma unroll
    for (int q = 0; q < kXq; ++q) nx[q] = read_x(tile, xslot_of(q), xch, ngate[q]);
  };
  auto put_tile = [&]() {
#pragma unroll
    for (int q = 0; q < 5; ++q)
      if (slot_of(q) < kRows + 2) *reinterpret_cast<uint4*>(s_dy + ch * kChunk + slot_of(q) * 16) = ndy[q];
#pragma unroll
    for (int q = 0; q < kXq; ++q)
      if (xslot_of(q) < kRows + 2) put_x(xslot_of(q), xch, nx[q], ngate[q]);
  };

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
      const int t = packed_row(tile, r + 1);
      if (t >= 0) {
        const uint32_t gate =
            Ci == kCh ? *reinterpret_cast<const uint32_t*>(smem + kOffGate + r * (kCh / 8) + (warp >> 2) * 4) : ~0u;
        float* dst = P.dX + (size_t)t * Ci + c;
#pragma unroll
        for (int j = 0; j < 32; j += 4)
          *reinterpret_cast<float4*>(dst + j) =
              make_float4(gate >> j & 1u ? __uint_as_float(v[j]) : 0.f, gate >> (j + 1) & 1u ? __uint_as_float(v[j + 1]) : 0.f,
                          gate >> (j + 2) & 1u ? __uint_as_float(v[j + 2]) : 0.f,
                          gate >> (j + 3) & 1u ? __uint_as_float(v[j + 3]) : 0.f);
      }
      __syncwarp();
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

cudaError_t conv_bwd(int layer, const float* dY, const float* Ytop, const float* dP, const float* X, const Packed& pk,
                     const void* pack, float* dX, float* dW, float* db, uint32_t* err, int sms, cudaStream_t s) {
  BwdArgs P{};
  P.dY = dY;
  P.Ytop = Ytop;
  P.dP = dP;
  P.rinfo = pk.rinfo;
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
