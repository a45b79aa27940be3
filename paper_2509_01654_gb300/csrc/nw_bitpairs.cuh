// nw_bitpairs.cuh -- bit-parallel scores (nw_bitrow.cuh) of explicit pairs, and
// of a row word against its proposal candidates with the k best selected.
#pragma once

#include <limits.h>

#include "nw_bitrow.cuh"
#include "nw_launch.h"

namespace nw {

template <class W>
__device__ __forceinline__ W cols_below(int n);  // columns 0 .. n - 1
template <>
__device__ __forceinline__ B32 cols_below<B32>(int n) {
  return {n >= 32 ? 0xffffffffu : (1u << n) - 1u};
}
template <>
__device__ __forceinline__ B64 cols_below<B64>(int n) {
  const uint64_t v = (1ull << n) - 1ull;  // n <= kMaxLen
  return {(uint32_t)v, (uint32_t)(v >> 32)};
}
// the columns of a mask as C: all of them, or the first 32
template <class C>
__device__ __forceinline__ C cols_of(B32 x) {
  return x;
}
template <class C>
__device__ __forceinline__ C cols_of(B64 x) {
  if constexpr (sizeof(C) == 4) return {x.lo};
  else return x;
}
__device__ __forceinline__ int cols_count(B32 x) { return __popc(x.lo); }
__device__ __forceinline__ int cols_count(B64 x) { return __popc(x.lo) + __popc(x.hi); }
// sets column j of a mask in shared memory that only this thread touches (an
// addition without a return value: a read-modify-write would wait for its load)
__device__ __forceinline__ void set_col(B32* x, int j) { atomicOr(&x->lo, 1u << j); }
__device__ __forceinline__ void set_col(B64* x, int j) { atomicOr(j < 32 ? &x->lo : &x->hi, 1u << (j & 31)); }

// A word's 16-byte record: byte 0 its length, then up to 15 codes; a longer
// word has its offset in the symbols in the second 32 bits and that of its pair
// record, with its half, in the third.
constexpr int kRecCodes = 15;
__device__ __forceinline__ uint32_t rec_byte(const uint4& r, int b) {  // b a compile-time constant
  const uint32_t w = b < 4 ? r.x : (b < 8 ? r.y : (b < 12 ? r.z : r.w));
  return (w >> (8 * (b & 3))) & 0xffu;
}

// Sixteen codes of a word, a byte each, from its first on.
struct Codes16 {
  uint32_t w[4];
};
__device__ __forceinline__ Codes16 rec_codes(const uint4& r) {
  return {{__funnelshift_r(r.x, r.y, 8), __funnelshift_r(r.y, r.z, 8), __funnelshift_r(r.z, r.w, 8), r.w >> 8}};
}
// The same for symbols at .. at + 15 (at a multiple of 16) of a word of len symbols in
// the pair records (`word`: brec_w of it): four symbols a load, all loads in flight.
__device__ __forceinline__ Codes16 brec_codes(const uint32_t* __restrict__ b_rec, uint32_t word, uint32_t shift, int at,
                                              int len) {
  const uint4* src = reinterpret_cast<const uint4*>(b_rec + (word & ~3u) + at);
  uint4 v[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) v[q] = at + 4 * q < len ? __ldg(src + q) : make_uint4(0u, 0u, 0u, 0u);
  const uint32_t sh = (word & 1u) * 16u + shift, mask = 0x7fu;  // (alphabets of up to 128)
  Codes16 c;
#pragma unroll
  for (int q = 0; q < 4; ++q)
    c.w[q] = ((~v[q].x >> sh) & mask) | (((~v[q].y >> sh) & mask) << 8) | (((~v[q].z >> sh) & mask) << 16) |
           (((~v[q].w >> sh) & mask) << 24);
  return c;
}
__device__ __forceinline__ uint32_t code_at(const Codes16& c, int x) {  // x a compile-time constant
  return (c.w[x >> 2] >> (8 * (x & 3))) & 0xffu;
}
__device__ __forceinline__ uint32_t next_code(Codes16& c) {  // takes the first code off
  const uint32_t code = c.w[0] & 0xffu;
#pragma unroll
  for (int q = 0; q < 3; ++q) c.w[q] = __funnelshift_r(c.w[q], c.w[q + 1], 8);
  c.w[3] >>= 8;
  return code;
}

// ---- explicit pairs: one thread per pair, the longer word in the thread's
// columns (W: 32 columns while the dictionary's words fit, else 64), the
// shorter one streamed.  The match masks sit in the thread's own column of a
// shared table (entry code * blockDim + thread: no two lanes share a bank),
// set from the longer word and cleared again after the pair.  A thread loops
// over its own word lengths, so a warp of mixed lengths runs one code path;
// the DPX kernel it replaces ran one unrolled body per length present in the
// warp.  Every lane reads other words, so a load takes 32 tag look-ups whatever its
// width.  With the words' records (P.rec) a pair of words of up to 15 symbols takes
// two 16-byte loads; other words are read 16 symbols at a time from the pair records,
// four a load, and a pair's first loads are issued together.  (Symbol by symbol a word
// of 24 took 72 loads.)  With records its own instructions bound it (ALU pipe 63 %, L1
// 47 %), without them L1 (70 %): 31 and 51 us in the kernel.  1,000,003 random
// pairs of 100k words, whole calls: lengths N(8, 3) 397 us DPX, 62 with records, 76
// without; all of 16 symbols 126, 67 (symbol by symbol 300); of 24, 164, 90 (412); of
// 40, 398, 174.
template <int MM, int XX, class W>
__global__ void __launch_bounds__(kBitPairsBlock) bit_pairs_kernel(const PairsParams P) {
  extern __shared__ __align__(16) unsigned char s_pairs[];
  W* tab = reinterpret_cast<W*>(s_pairs) + threadIdx.x;
  const uint32_t pitch = blockDim.x;
  const uint64_t step = (uint64_t)gridDim.x * pitch;
  uint64_t p = (uint64_t)blockIdx.x * pitch + threadIdx.x, next = 0;
  uint32_t i = 0u, j = 0u, ni = 0u, nj = 0u;  // this pair, and the next one read ahead
  if (p < P.m) {
    i = P.pi[p];
    j = P.pj[p];
  }
  for (uint32_t c = 0; c < P.alphabet; ++c) tab[c * pitch] = W{};
  for (; p < P.m; p = next, i = ni, j = nj) {
    next = p + step;
    if (next < P.m) {
      ni = P.pi[next];
      nj = P.pj[next];
    }
    if (i >= P.n || j >= P.n) {
      atomicOr(P.err, kErrInput);
      P.out[p] = INT16_MIN;
      continue;
    }
    uint4 ra = make_uint4(0u, 0u, 0u, 0u), rb = ra;  // the shorter word's record, the longer one's
    int la, lb;
    if (P.rec) {
      ra = __ldg(P.rec + i);
      rb = __ldg(P.rec + j);
      la = (int)(ra.x & 0xffu);
      lb = (int)(rb.x & 0xffu);
    } else {  // few pairs: the pair records' offsets, as for words too long for a record
      const uint32_t pa = __ldg(P.rank + i), pb = __ldg(P.rank + j);
      la = __ldg(P.slen + pa);
      lb = __ldg(P.slen + pb);
      ra.z = __ldg(P.brec_w + pa);
      rb.z = __ldg(P.brec_w + pb);
    }
    if (la > lb) {
      const uint4 t = ra;
      ra = rb;
      rb = t;
      const int l = la;
      la = lb;
      lb = l;
    }
    int g = 0;
    if (la > 0) {
      auto first = [&](const uint4& r, int len) {
        return P.rec && len <= kRecCodes ? rec_codes(r) : brec_codes(P.b_rec, r.z, P.shift, 0, len);
      };
      const Codes16 b0 = first(rb, lb);
      Codes16 c = first(ra, la);
      auto each_column = [&](auto f) {
#pragma unroll
        for (int x = 0; x < 16; ++x)
          if (x < lb) f(tab + code_at(b0, x) * pitch, x);
#pragma unroll 1
        for (int at = 16; at < lb; at += 16) {
          const Codes16 b = brec_codes(P.b_rec, rb.z, P.shift, at, lb);
#pragma unroll
          for (int x = 0; x < 16; ++x)
            if (at + x < lb) f(tab + code_at(b, x) * pitch, at + x);
        }
      };
      each_column([](W* t, int x) { set_col(t, x); });
      auto rows = [&](auto kind) {
        using V = decltype(kind);
        constexpr bool kSplit = sizeof(V) == 4;  // (64 columns: a word may straddle bit 32)
        auto next_mask = [&]() { return cols_of<V>(tab[next_code(c) * pitch]); };
        const V NL = cols_below<V>(lb - 1);
        V H[bit_planes(MM, XX)];
        bit_first<MM, XX, kSplit>(H, next_mask(), NL);
#pragma unroll 1
        for (int r = 1;;) {
          const int end = la < (r | 15) + 1 ? la : (r | 15) + 1;
#pragma unroll 1
          for (; r < end; ++r) bit_next<MM, XX, kSplit>(H, next_mask(), NL);
          if (r == la) break;
          c = brec_codes(P.b_rec, ra.z, P.shift, r, la);  // r a multiple of 16
        }
        V D[bit_digits(MM)];
        bit_digit_planes<MM, XX>(H, D);
        const V F = cols_below<V>(lb);
#pragma unroll
        for (int d = 0; d < bit_digits(MM); ++d) g += cols_count(D[d] & F) << d;
      };
      if constexpr (sizeof(W) == 8) {
        if (__any_sync(__activemask(), lb > 32)) rows(B64{});
        else rows(B32{});  // (a list in order of length)
      } else {
        rows(B32{});
      }
      each_column([](W* t, int) { *t = W{}; });
    }
    P.out[p] = (int16_t)(g * P.coef + P.gap * (la + lb));
  }
}

// ---- rescoring: one warp per row word.  The row's word streams; a lane holds
// K candidates in its columns, as in the all-pairs kernel.  Candidates are
// taken in three classes of length (up to 8 and 16 columns and the rest: K = 8,
// 4, 1), each lane building the masks of its own candidates in its own column
// of the warp's table.  Scores become list keys (score above the reversed
// index) in shared memory, and the k best come off by warp-wide maxima.  It
// replaces a length sort per row, a grouping of candidate pairs by width, a
// launch per width and a selection, which moved every candidate and score
// through memory several times: 100k rows, C = 512, k = 10: 2.7 -> 1.15 ms.  The
// loops over candidates and words are kept rolled: unrolled, the warps of an SM
// waited for instructions half of the time (1.9 ms).
// A candidate costs one 16-byte record instead of a chain of four loads.
struct RescoreBits {
  const uint32_t* cand;    // rows x C: indices of D's words (UINT32_MAX: none)
  uint32_t rows, C, k, nd;
  bool self;               // rows and candidates are one set: a word may not be its own candidate
  const uint4* rec;        // nd records of D's words, by original index
  const uint32_t* d_sym;
  const uint32_t* r_rank;  // the row words
  const uint8_t* r_slen;
  const uint32_t* r_aoff;
  const uint32_t* r_sym;
  uint32_t shift, alphabet, coef;
  int32_t gap, key_lo;     // key = ((s - key_lo) << ib) | (imask - index)
  uint32_t ib, imask;
  uint32_t* out_idx;
  int16_t* out_score;
  uint32_t* err;
};

// one class: the candidates s_cand[beg, end), K per lane at a pitch of 64 / K
template <int MM, int XX, int K>
__device__ __forceinline__ void rescore_class(const RescoreBits& P, uint32_t beg, uint32_t end, int la,
                                              const uint16_t* s_row, const uint32_t* s_cand, uint32_t* s_key,
                                              uint32_t* tab, int lane) {
  constexpr int PITCH = 64 / K;
  constexpr bool kSplit = PITCH <= 32;
#pragma unroll 1
  for (uint32_t base = beg; base < end; base += 32u * K) {
    __syncwarp();
    for (uint32_t x = (uint32_t)lane; x < P.alphabet * 16u; x += 32u)
      reinterpret_cast<uint4*>(tab)[x] = make_uint4(0u, 0u, 0u, 0u);
    __syncwarp();
    uint64_t fm = 0, nl = 0;
#pragma unroll 1
    for (int w = 0; w < K; ++w) {
      const uint32_t at = base + 32u * (uint32_t)w + (uint32_t)lane;
      if (at >= end) break;
      const uint4 r = __ldg(P.rec + s_cand[at]);
      const int len = (int)(r.x & 0xffu);
      // the masks are the lane's own column, so the additions never collide
      uint32_t* col = tab + 2u * (uint32_t)lane;
      if (PITCH == 8 || len <= kRecCodes) {
        uint32_t* half = col + ((w * PITCH) >> 5);
        const uint32_t first = 1u << ((w * PITCH) & 31);
#pragma unroll
        for (int j = 0; j < (PITCH < kRecCodes ? PITCH : kRecCodes); ++j)
          if (j < len) atomicOr(half + rec_byte(r, j + 1) * 64u, first << j);
      } else {
        const uint32_t* src = P.d_sym + r.y;
#pragma unroll 1
        for (int j = 0; j < len; ++j) {
          const int bit = w * PITCH + j;
          atomicOr(col + ((__ldg(src + j) & 0xffffu) >> P.shift) * 64u + (bit >> 5), 1u << (bit & 31));
        }
      }
      const uint64_t f = (1ull << len) - 1ull;  // len <= kMaxLen < 64
      fm |= f << (w * PITCH);
      nl |= (f >> 1) << (w * PITCH);
    }
    const B64 FM{(uint32_t)fm, (uint32_t)(fm >> 32)}, NL{(uint32_t)nl, (uint32_t)(nl >> 32)};
    B64 H[bit_planes(MM, XX)];
#pragma unroll
    for (int x = 0; x < bit_planes(MM, XX); ++x) H[x] = B64{};
    if (la > 0) {
      auto mask = [&](int r) {
        const uint2 v = *reinterpret_cast<const uint2*>(tab + s_row[r] * 64u + 2u * lane);
        return B64{v.x, v.y};
      };
      B64 M = mask(0);
      bit_first<MM, XX, kSplit>(H, M, NL);
      if (la > 1) M = mask(1);
#pragma unroll 1
      for (int r = 1; r < la; ++r) {
        const B64 cur = M;
        if (r + 1 < la) M = mask(r + 1);
        bit_next<MM, XX, kSplit>(H, cur, NL);
      }
    }
    B64 D[bit_digits(MM)];
    bit_digit_planes<MM, XX>(H, D);
    int gv[K];
    bit_scores<MM, K, 0, PITCH>(D, FM, (int)P.coef, gv);
    int ln[K];
    field_lengths<K, 0, PITCH>(FM, ln);
#pragma unroll
    for (int w = 0; w < K; ++w) {
      const uint32_t at = base + 32u * w + (uint32_t)lane;
      if (at < end)
        s_key[at] = ((uint32_t)(gv[w] + P.gap * (la + ln[w]) - P.key_lo) << P.ib) | (P.imask - s_cand[at]);
    }
  }
}

constexpr int kRescoreWarps = 2;
constexpr int kRescoreMaxC = 512;
// shared memory of a warp: match masks, candidates by class, keys, the row's codes
__host__ __device__ constexpr size_t rescore_warp_bytes(uint32_t alphabet, uint32_t C) {
  return (size_t)alphabet * 256u + 2u * ((C + 3u) & ~3u) * sizeof(uint32_t) + 96u;
}

template <int MM, int XX>
__global__ void __launch_bounds__(kRescoreWarps * 32) bit_rescore_kernel(const __grid_constant__ RescoreBits P) {
  extern __shared__ __align__(16) unsigned char s_res[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  unsigned char* mine = s_res + (size_t)warp * rescore_warp_bytes(P.alphabet, P.C);
  uint32_t* tab = reinterpret_cast<uint32_t*>(mine);
  uint32_t* s_cand = tab + P.alphabet * 64u;
  uint32_t* s_key = s_cand + ((P.C + 3u) & ~3u);
  uint16_t* s_row = reinterpret_cast<uint16_t*>(s_key + ((P.C + 3u) & ~3u));
  const unsigned below = (1u << lane) - 1u;
  for (uint32_t i = blockIdx.x * kRescoreWarps + warp; i < P.rows; i += gridDim.x * kRescoreWarps) {
    __syncwarp();
    const uint32_t ri = __ldg(P.r_rank + i);
    const int la = __ldg(P.r_slen + ri);
    const uint32_t ao = __ldg(P.r_aoff + ri);
    for (int x = lane; x < la; x += 32) s_row[x] = (uint16_t)((__ldg(P.r_sym + ao + x) & 0xffffu) >> P.shift);
    // the candidates by class of length: up to 8 symbols from the front, 9 to 16
    // from the back, the rest behind the first ones (through the key area)
    uint32_t n8 = 0u, n16 = 0u, nx = 0u;
    const uint32_t* row = P.cand + (size_t)i * P.C;
#pragma unroll 1
    for (uint32_t x0 = 0; x0 < P.C; x0 += 128u) {
      uint32_t j[4], len[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const uint32_t at = x0 + 32u * q + (uint32_t)lane;
        j[q] = at < P.C ? __ldg(row + at) : 0xffffffffu;
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        if (j[q] != 0xffffffffu && (j[q] >= P.nd || (P.self && j[q] == i))) {
          atomicOr(P.err, kErrInput);
          j[q] = 0xffffffffu;
        }
        len[q] = j[q] != 0xffffffffu ? __ldg(&P.rec[j[q]].x) & 0xffu : 0xffu;
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const bool a8 = len[q] <= 8u, a16 = !a8 && len[q] <= 16u, ax = len[q] > 16u && len[q] != 0xffu;
        const unsigned m8 = __ballot_sync(0xffffffffu, a8), m16 = __ballot_sync(0xffffffffu, a16),
                       mx = __ballot_sync(0xffffffffu, ax);
        if (a8) s_cand[n8 + __popc(m8 & below)] = j[q];
        if (a16) s_cand[P.C - 1u - n16 - __popc(m16 & below)] = j[q];
        if (ax) s_key[nx + __popc(mx & below)] = j[q];
        n8 += (uint32_t)__popc(m8);
        n16 += (uint32_t)__popc(m16);
        nx += (uint32_t)__popc(mx);
      }
    }
    __syncwarp();
    for (uint32_t x = (uint32_t)lane; x < nx; x += 32u) s_cand[n8 + x] = s_key[x];
    __syncwarp();
    for (uint32_t x = (uint32_t)lane; x < P.C; x += 32u) s_key[x] = 0u;
    __syncwarp();
    rescore_class<MM, XX, 8>(P, 0u, n8, la, s_row, s_cand, s_key, tab, lane);
    rescore_class<MM, XX, 4>(P, P.C - n16, P.C, la, s_row, s_cand, s_key, tab, lane);
    rescore_class<MM, XX, 1>(P, n8, n8 + nx, la, s_row, s_cand, s_key, tab, lane);
    __syncwarp();
    // the k best keys: each lane keeps its own best, the warp's best comes off
    uint32_t key[kRescoreMaxC / 32], best = 0u;
#pragma unroll
    for (int q = 0; q < kRescoreMaxC / 32; ++q) {
      const uint32_t at = 32u * q + (uint32_t)lane;
      key[q] = at < P.C ? s_key[at] : 0u;
      best = key[q] > best ? key[q] : best;
    }
    uint32_t hold = 0u;  // result r of this lane, r % 32 == lane
    for (uint32_t r = 0; r < P.k; ++r) {
      const uint32_t top = __reduce_max_sync(0xffffffffu, best);
      if ((r & 31u) == (uint32_t)lane) hold = top;
      if (top != 0u && best == top) {  // keys are distinct: one lane
        best = 0u;
#pragma unroll
        for (int q = 0; q < kRescoreMaxC / 32; ++q) {
          if (key[q] == top) key[q] = 0u;
          best = key[q] > best ? key[q] : best;
        }
      }
      if ((r & 31u) == 31u || r + 1u == P.k) {
        const uint32_t o = (r & ~31u) + (uint32_t)lane;
        if (o < P.k) {
          const size_t at = (size_t)i * P.k + o;
          P.out_idx[at] = hold ? P.imask - (hold & P.imask) : 0xffffffffu;
          P.out_score[at] = hold ? (int16_t)((int32_t)(hold >> P.ib) + P.key_lo) : (int16_t)INT16_MIN;
        }
        hold = 0u;
      }
    }
  }
}

}  // namespace nw
