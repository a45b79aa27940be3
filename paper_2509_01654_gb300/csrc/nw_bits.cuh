// nw_bits.cuh -- the bit-parallel alignment kernel (sm_103a): for match /
// mismatch scorings whose shifted recurrence has few steps (below), 64 cells
// of Algorithm 1's matrix advance per group of logic instructions.
//
// Recurrence.  With G[i][j] = H[i][j] - p*(i + j) (see nw_dp.cuh)
//     G[i][j] = max(G[i-1][j-1] + s, G[i-1][j], G[i][j-1]),  G[i][0] = G[0][j] = 0,
// s = s'_m on equal symbols and s'_x+ = max(s'_x, 0) otherwise.  Dividing by
// g = gcd(s'_m, s'_x+) leaves steps (m, x).  The horizontal and vertical
// differences h = G[i][j] - G[i][j-1] and v = G[i][j] - G[i-1][j] lie in
// 0 .. m, and one cell maps the difference h' above it and the difference v'
// to its left to
//     c = max(s, h', v'),   v = c - h',   h = c - v'
// (divide the cell's three terms by G[i-1][j-1]).  This is the bit-vector
// formulation of alignment by difference encoding (Myers, "A fast bit-vector
// algorithm for approximate string matching", J. ACM 1999; Loving, Hernandez
// and Benson, "BitPAl", Bioinformatics 2014, for general integer scorings);
// the equations used here are derived below from the cell map itself.
//
// Encoding.  A row's differences are held as m bit planes H[a], a = 1..m, bit
// j set when h_j >= a (a thermometer code); M has the bits whose column
// symbol equals the row's symbol.  U[a] has the bits with v' >= a, i.e. the
// plane of v >= a moved up by one column.  From the cell map:
//     v >= a  <=>  M and h' <= m - a,  or  x - h' >= a,  or  v' - h' >= a
//             =    (M & ~H[m-a+1]) | ~H[x-a+1] (if a <= x)
//                  | OR over b >= 0 of (~H[b+1] & U[a+b])
// and the same with H and U exchanged gives the new H.  The term b = 0 refers
// to the plane being computed.  For a <= x it is contained in ~H[x-a+1];
// for a > x it is a run that continues while h' = 0: with g the set of bits
// that start a run and z = ~H[1], the carries of (g | z) + g are exactly
// the runs, and the carry INTO bit j is v' >= a at j: U[a] = P ^ g ^ (P + g),
// P = g | z.  m - x additions and O(m^2) three-input logic operations a row.
//
// Packing.  A lane's 64 bits hold up to eight words of the same length b side
// by side, K = words_per_lane(b) of them at a pitch of K's own (a compile-time
// constant), so a warp's task covers 32 K words.  No separator bits: clearing
// the last column of every word (mask NL) in P and g keeps a carry from
// leaving its word, and a plane moved up by one column has the last column
// cleared first.
//
// Match masks.  A block (four warps) keeps the masks of its B words in shared
// memory, masks[code][lane] (256 bytes a code), built once per task; the
// warps share them and take 16 A words at a time each.  A row costs one
// broadcast read of the A symbol's table offset and one conflict-free 8-byte
// read.
//
// Score.  G = g * (sum of the word's h) = g * (sum of the planes' bit counts);
// for m >= 3 the planes are first recoded to binary digits, so that a word
// takes two or three bit counts.
#pragma once

#include "nw_dp.cuh"

namespace nw {

// The bit planes of 64 columns.
struct B64 {
  uint32_t lo, hi;
};
__device__ __forceinline__ B64 operator&(B64 a, B64 b) { return {a.lo & b.lo, a.hi & b.hi}; }
__device__ __forceinline__ B64 operator|(B64 a, B64 b) { return {a.lo | b.lo, a.hi | b.hi}; }
__device__ __forceinline__ B64 operator^(B64 a, B64 b) { return {a.lo ^ b.lo, a.hi ^ b.hi}; }
__device__ __forceinline__ B64 operator~(B64 a) { return {~a.lo, ~a.hi}; }

// a + b: with Split (no word straddles bit 32) the halves are independent
template <bool Split>
__device__ __forceinline__ B64 add64(B64 a, B64 b) {
  if constexpr (Split) {
    return {a.lo + b.lo, a.hi + b.hi};
  } else {
    const uint64_t s = (((uint64_t)a.hi << 32) | a.lo) + (((uint64_t)b.hi << 32) | b.lo);
    return {(uint32_t)s, (uint32_t)(s >> 32)};
  }
}

// One row: H[1..m] (index a - 1) of row i - 1 becomes row i.
template <int MM, int XX, bool Split>
__device__ __forceinline__ void bit_row(B64 (&H)[MM], const B64 M, const B64 NL) {
  B64 U[MM + 1];  // U[a], a = 1..m (v' >= a)
  const B64 z = ~H[0] & NL;
  // (M | U[m]) and (M | H[m]) stand in for M: where v' = m the cell is a
  // match's anyway (v' - h' = m - h'), which saves the last term of each sum
#pragma unroll
  for (int a = MM; a >= 1; --a) {
    if (a > XX) {
      B64 g;
      if (a == MM) {
        g = M & z;
      } else {
        B64 t = M;  // M & ~H[m-a+1], joined by U[m] (b = m - a) under the same mask
        t = (t | U[MM]) & ~H[MM - a];
#pragma unroll
        for (int b = 1; b < MM - a; ++b) t = t | (~H[b] & U[a + b]);
        g = t & NL;
        // g may hold bits with H[1] = 0 and set: they are run starts too
      }
      const B64 P = g | z;
      const B64 s = add64<Split>(P, g);
      U[a] = P ^ g ^ s;
    } else {
      B64 t = a == MM ? (M & ~H[0]) : ((M | U[MM]) & ~H[MM - a]);
#pragma unroll
      for (int b = XX - a + 1 > 1 ? XX - a + 1 : 1; b < MM - a; ++b) t = t | (~H[b] & U[a + b]);
      t = (t | ~H[XX - a]) & NL;
      U[a] = add64<Split>(t, t);
    }
  }
  B64 N[MM];
  const B64 q = M | H[MM - 1];
#pragma unroll
  for (int a = 1; a <= MM; ++a) {
    B64 t = q & ~U[MM - a + 1];
    const int b0 = a <= XX ? XX - a + 1 : 0;
#pragma unroll
    for (int b = b0; b < MM - a; ++b) t = t | (~U[b + 1] & H[a + b - 1]);
    if (a <= XX) t = t | ~U[XX - a + 1];
    N[a - 1] = t;
  }
#pragma unroll
  for (int a = 0; a < MM; ++a) H[a] = N[a];
}

// The planes recoded to binary digits: h = sum over d of 2^d * D[d].
__host__ __device__ constexpr int bit_digits(int m) { return m == 1 ? 1 : (m <= 3 ? 2 : 3); }
template <int MM>
__device__ __forceinline__ void bit_digit_planes(const B64 (&H)[MM], B64 (&D)[bit_digits(MM)]) {
  if constexpr (MM == 1) {
    D[0] = H[0];
  } else if constexpr (MM == 2) {
    D[0] = H[0] & ~H[1];
    D[1] = H[1];
  } else if constexpr (MM == 3) {
    D[0] = H[0] ^ H[1] ^ H[2];
    D[1] = H[1];
  } else if constexpr (MM == 4) {
    D[0] = (H[0] ^ H[1] ^ H[2]) & ~H[3];
    D[1] = H[1] & ~H[3];
    D[2] = H[3];
  } else {
    D[0] = H[0] ^ H[1] ^ H[2] ^ H[3] ^ H[4];
    D[1] = H[1] & ~H[3];
    D[2] = H[3];
  }
}

// bits of a word's field [w * pitch, (w + 1) * pitch) in the two halves
__host__ __device__ constexpr uint32_t field_lo(int w, int pitch) {
  uint32_t m = 0;
  for (int j = w * pitch; j < (w + 1) * pitch && j < 32; ++j) m |= 1u << j;
  return m;
}
__host__ __device__ constexpr uint32_t field_hi(int w, int pitch) {
  uint32_t m = 0;
  for (int j = w * pitch; j < (w + 1) * pitch && j < 64; ++j)
    if (j >= 32) m |= 1u << (j - 32);
  return m;
}
template <int W, int PITCH>
__device__ __forceinline__ int field_count(B64 x, B64 FM) {
  constexpr uint32_t ml = field_lo(W, PITCH), mh = field_hi(W, PITCH);
  int c = 0;
  if constexpr (ml != 0u) c += __popc(x.lo & FM.lo & ml);
  if constexpr (mh != 0u) c += __popc(x.hi & FM.hi & mh);
  return c;
}

// G of words 0..K-1 (real units: coef = g)
template <int MM, int K, int W = 0>
__device__ __forceinline__ void bit_scores(const B64 (&D)[bit_digits(MM)], B64 FM, int coef, int (&g)[K]) {
  if constexpr (W < K) {
    constexpr int P = bit_pitch(K);
    int v = 0;
#pragma unroll
    for (int d = 0; d < bit_digits(MM); ++d) v += field_count<W, P>(D[d], FM) * (coef << d);
    g[W] = v;
    bit_scores<MM, K, W + 1>(D, FM, coef, g);
  }
}

// value i of a register array by a run-time index
template <int N>
__device__ __forceinline__ uint32_t pick(const uint32_t (&v)[N], int i) {
  uint32_t r = v[0];
#pragma unroll
  for (int x = 1; x < N; ++x) r = x == i ? v[x] : r;
  return r;
}

// what a task's warps share
struct BitTask {
  TaskGeom g;
  int K;                  // words per lane
  int la, lb, mx;         // mx: the longer of the two
  uint32_t a_base;        // index of A word g.a0's first symbol in T.a_sym
  uint32_t b_base;        // index of B word g.b0's first symbol in T.b_sym
  bool check;             // same bucket, chunks overlap: test a < b
};

// The A words of one task against the lane's K words (b = b0 + 32 w + lane).
template <int MM, int XX, int EPI, int K>
__device__ __forceinline__ void bit_task(const BitParams& P, const BitTerms& T, const BitTask& Q,
                                         const unsigned char* masks, uint32_t* wh, uint32_t* sA, uint32_t& inserts,
                                         int max_iters) {
  constexpr int PITCH = bit_pitch(K);
  constexpr bool kSplit = PITCH == 8 || PITCH == 16 || PITCH == 32;
  constexpr bool kLists = EPI != kEpiMatrix;
  constexpr bool kHist = EPI == kEpiListsLaneHist;
  constexpr int KP = (K + 1) / 2;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const TaskGeom& g = Q.g;
  const int pconst = T.gap * (Q.la + Q.lb);  // score = G + pconst
  const bool listsA = kLists && T.A.slots != nullptr;
  const bool listsB = kLists && T.B.slots != nullptr;
  const bool serialA = !kHist && listsA && T.serial_a != 0u;
  const int la = Q.la;

  // columns of the lane's words: all of them, and all but each word's last
  B64 FM{0u, 0u}, NL{0u, 0u};
  {
    const uint64_t f = Q.lb >= 64 ? ~0ull : ((1ull << Q.lb) - 1ull);
    uint64_t fm = 0, nl = 0;
#pragma unroll
    for (int w = 0; w < K; ++w) {
      fm |= f << (w * PITCH);
      nl |= (f >> 1) << (w * PITCH);
    }
    FM = {(uint32_t)fm, (uint32_t)(fm >> 32)};
    NL = {(uint32_t)nl, (uint32_t)(nl >> 32)};
  }
  uint32_t vmask = 0u;  // bit w: word w exists
#pragma unroll
  for (int w = 0; w < K; ++w) vmask |= (g.b0 + 32u * w + lane < g.bend ? 1u : 0u) << w;
  const bool full = __all_sync(0xffffffffu, vmask == (1u << K) - 1u) && !Q.check;

  // B-side list bounds in G, packed for the prefilter (see neg_bound16)
  uint32_t nB2[KP];
#pragma unroll
  for (int i = 0; i < KP; ++i) {
    int t[2] = {INT_MAX, INT_MAX};
#pragma unroll
    for (int h = 0; h < 2; ++h)
      if (listsB && ((vmask >> (2 * i + h)) & 1u))
        t[h] = g_bound(P, T, __ldcg(T.B.thr + g.b0 + 32u * (2 * i + h) + lane), Q.mx, pconst);
    nB2[i] = neg_bound2(t[0], t[1]);
  }
  uint32_t ob[EPI == kEpiMatrix ? K : 1];
  if constexpr (EPI == kEpiMatrix) {
#pragma unroll
    for (int w = 0; w < K; ++w) ob[w] = (vmask >> w) & 1u ? __ldg(T.B.perm + g.b0 + 32u * w + lane) : 0u;
  }
  // histogram column of the lane, shifted so that its index is G
  uint32_t* hcol = wh + (ptrdiff_t)lane + (ptrdiff_t)(pconst - P.hist_lo) * 32;

  const int coef = (int)T.coef;
  const uint32_t sub = P.sub;
  for (uint32_t c0 = g.a0 + (uint32_t)warp * sub; c0 < g.a1; c0 += kBitWarps * sub) {
    const uint32_t nA = g.a1 - c0 < sub ? g.a1 - c0 : sub;
    // the symbols of nA consecutive A words are one run of T.a_sym: stage
    // their table offsets (two zero entries beyond for the reads ahead)
    __syncwarp();
    const uint32_t total = nA * (uint32_t)la;
    const uint32_t* src = T.a_sym + Q.a_base + (size_t)(c0 - g.a0) * (uint32_t)la;
    const uint32_t shift = T.shift;
    for (uint32_t i = lane; i < total + 2u; i += 32u)
      sA[i] = i < total ? ((__ldg(src + i) & 0xffffu) >> shift) * kMaskRow : 0u;
    const uint32_t my_a = c0 + (uint32_t)lane;
    const bool have = (uint32_t)lane < nA;
    const uint32_t my_orig = (EPI == kEpiMatrix && have) ? __ldg(T.A.perm + my_a) : 0u;
    uint32_t my_nA2 = 0u;
    if constexpr (kLists) {
      const int t = listsA && have ? g_bound(P, T, __ldcg(T.A.thr + my_a), Q.mx, pconst) : INT_MAX;
      my_nA2 = neg_bound2(t, t);
    }
    __syncwarp();

    const unsigned char* mrow = masks + lane * 8;
    const uint32_t* sp = sA;
    uint2 mv = *reinterpret_cast<const uint2*>(mrow + sp[0]);
    uint32_t o1 = sp[1];
    for (uint32_t w0 = 0; w0 < nA; ++w0) {
      const uint32_t a = c0 + w0;
      B64 H[MM];
#pragma unroll
      for (int x = 0; x < MM; ++x) H[x] = {0u, 0u};
      if (la > 0) {
        // the first row (H = 0) folds to a few operations
        {
          const B64 M{mv.x, mv.y};
          mv = *reinterpret_cast<const uint2*>(mrow + o1);
          o1 = sp[2];
          ++sp;
          bit_row<MM, XX, kSplit>(H, M, NL);
        }
#pragma unroll 2
        for (int r = 1; r < la; ++r) {
          const B64 M{mv.x, mv.y};
          mv = *reinterpret_cast<const uint2*>(mrow + o1);
          o1 = sp[2];
          ++sp;
          bit_row<MM, XX, kSplit>(H, M, NL);
        }
      }
      B64 D[bit_digits(MM)];
      bit_digit_planes<MM>(H, D);
      int gv[K];
      bit_scores<MM, K>(D, FM, coef, gv);

      if constexpr (EPI == kEpiMatrix) {
        const uint32_t oa = __shfl_sync(0xffffffffu, my_orig, (int)w0);
#pragma unroll
        for (int w = 0; w < K; ++w) {
          if (!((vmask >> w) & 1u) || (Q.check && a >= g.b0 + 32u * w + lane)) continue;
          const uint64_t i = oa < ob[w] ? oa : ob[w], j = oa < ob[w] ? ob[w] : oa;
          const uint64_t off = upper_offset(i, j, P.n);
          if (off >= P.mat_lo && off < P.mat_hi) P.mat[off] = (int8_t)(gv[w] + pconst);
        }
      } else {
        if constexpr (kHist) {
          if (full) {
#pragma unroll
            for (int w = 0; w < K; ++w) hcol[32 * gv[w]] += 1u;
          } else {
#pragma unroll
            for (int w = 0; w < K; ++w)
              if (((vmask >> w) & 1u) && (!Q.check || a < g.b0 + 32u * w + lane)) hcol[32 * gv[w]] += 1u;
          }
        } else if (EPI == kEpiLists && P.hist_mode != kHistNone) {
#pragma unroll
          for (int w = 0; w < K; ++w)
            if (((vmask >> w) & 1u) && (!Q.check || a < g.b0 + 32u * w + lane))
              hist_add(P, wh, lane, gv[w] + pconst - P.hist_lo);
        }
        uint32_t res[KP];
#pragma unroll
        for (int i = 0; i < KP; ++i) res[i] = (uint32_t)gv[2 * i] + (2 * i + 1 < K ? (uint32_t)gv[2 * i + 1 < K ? 2 * i + 1 : 0] * 65536u : 0u);
        const uint32_t nA2 = __shfl_sync(0xffffffffu, my_nA2, (int)w0);
        uint32_t any = 0u;
#pragma unroll
        for (int i = 0; i < KP; ++i) any |= __viaddmax_s16x2_relu(res[i], __vmaxs2(nB2[i], nA2), 0u);
        uint32_t amask = 0u;  // words this lane offers to the A word's list (serial offers)
        if (any) {
          const uint32_t thrA = listsA ? __ldcg(T.A.thr + a) : 0u;
          const uint32_t oa = __ldg(T.A.perm + a);
          for (int w = 0; w < K; ++w) {
            const uint32_t b = g.b0 + 32u * (uint32_t)w + (uint32_t)lane;
            if (!((vmask >> w) & 1u) || (Q.check && a >= b)) continue;
            const uint32_t rv = pick<KP>(res, w >> 1), nv = pick<KP>(nB2, w >> 1);
            const int G = (int)((w & 1) ? rv >> 16 : rv & 0xffffu);
            const int nb = (int)(int16_t)((w & 1) ? nv >> 16 : nv & 0xffffu);
            const int s = G + pconst;
            if (listsB && G + nb > 0) {  // word b takes the A word as a neighbour
              const uint32_t key = list_key(P, T, s, Q.mx, oa);
              uint32_t nm = __ldcg(T.B.thr + b);
              if (key > nm)
                nm = list_offer(T.B.slots + (size_t)b * P.k, T.B.thr + b, P.k, key, P.err, inserts, max_iters);
              const uint32_t nn = neg_bound16(g_bound(P, T, nm, Q.mx, pconst));
              const uint32_t keep = (w & 1) ? (nv & 0xffffu) | (nn << 16) : (nv & 0xffff0000u) | nn;
#pragma unroll
              for (int i = 0; i < KP; ++i)
                if (i == (w >> 1)) nB2[i] = keep;
            }
            if (listsA) {  // the A word takes word b as a neighbour
              const uint32_t ob1 = __ldg(T.B.perm + b);
              const uint32_t key = list_key(P, T, s, Q.mx, ob1);
              if (key > thrA) {
                if (serialA) amask |= 1u << w;
                else list_offer(T.A.slots + (size_t)a * P.k, T.A.thr + a, P.k, key, P.err, inserts, max_iters);
              }
            }
          }
        }
        if (serialA) {
          // many lanes may hold keys for the same A word's list: the warp
          // offers them one at a time from the best down, each against the
          // bound the previous offer returned (the lanes never race on that
          // list, and a list that is already full costs one offer)
          uint32_t thrW = 0u;
          while (__any_sync(0xffffffffu, amask != 0u)) {
            uint32_t best = 0u;
            int bw = -1;
            for (int w = 0; w < K; ++w)
              if ((amask >> w) & 1u) {
                const uint32_t rv = pick<KP>(res, w >> 1);
                const int s = (int)((w & 1) ? rv >> 16 : rv & 0xffffu) + pconst;
                const uint32_t key = list_key(P, T, s, Q.mx, __ldg(T.B.perm + g.b0 + 32u * (uint32_t)w + lane));
                if (key <= thrW) amask &= ~(1u << w);
                else if (key > best) { best = key; bw = w; }
              }
            const uint32_t m = __reduce_max_sync(0xffffffffu, best);
            if (m == 0u) break;  // every key fell below the list's bound
            const int src = __ffs(__ballot_sync(0xffffffffu, best == m)) - 1;
            uint32_t nm = 0u;
            if (lane == src) {
              nm = list_offer(T.A.slots + (size_t)a * P.k, T.A.thr + a, P.k, m, P.err, inserts, max_iters);
              amask &= ~(1u << bw);
            }
            nm = __shfl_sync(0xffffffffu, nm, src);
            thrW = nm > thrW ? nm : thrW;
          }
        }
      }
    }
  }
}

// blocks per SM the kernel is compiled for
constexpr int kBitMinBlocks = 6;

template <int MM, int XX, int EPI>
__global__ void __launch_bounds__(kBitBlock, kBitMinBlocks) nw_bit_kernel(const BitParams P) {
  extern __shared__ __align__(16) unsigned char s_bits[];
  __shared__ unsigned long long s_task[2];
  __shared__ uint32_t s_seg[2];
  // the task's terms and geometry live in shared memory: most of them are
  // read on the rare paths only, and registers are what bounds the block count
  __shared__ BitTerms T;
  __shared__ BitTask Q;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  constexpr bool kHist = EPI == kEpiListsLaneHist;
  const bool smem_hist = kHist || (EPI == kEpiLists && P.hist_mode == kHistSmem);
  const uint32_t wstride = kHist ? P.nbins * 32u : (smem_hist ? P.nbins : 0u);
  unsigned char* masks = s_bits;
  uint32_t* wh = reinterpret_cast<uint32_t*>(s_bits + P.mask_bytes) + (size_t)warp * wstride;
  uint32_t* sA = reinterpret_cast<uint32_t*>(s_bits + P.mask_bytes) + (size_t)kBitWarps * wstride +
                 (size_t)warp * P.stage_words;
  if (smem_hist)
    for (uint32_t q = lane; q < wstride; q += 32) wh[q] = 0u;
  uint64_t wpairs = 0;
  uint32_t inserts = 0;
  const int max_iters = P.dbg_insert_limit ? (int)(P.dbg_insert_limit - 1u) : kInsertMaxIters;
  auto fetch = [&](int buf) {  // thread 0: the next task and its segment
    const unsigned long long t = atomicAdd(P.counter, 1ull);
    s_task[buf] = t;
    s_seg[buf] = t < P.ntasks ? find_seg(P.segs, P.nsegs, t) : 0u;
  };
  if (tid == 0) fetch(0);
  for (int buf = 0;; buf ^= 1) {
    __syncthreads();  // the task is known, and the masks are no longer in use
    const unsigned long long t = s_task[buf];
    if (t >= P.ntasks) break;
    const Seg* S = P.segs + s_seg[buf];
    {
      const uint32_t d = S->dict;
      const uint32_t* src = reinterpret_cast<const uint32_t*>(EPI == kEpiBatchLists ? P.terms + d : P.local + d);
      if (tid < (int)(sizeof(BitTerms) / 4)) reinterpret_cast<uint32_t*>(&T)[tid] = src[tid];
    }
    if (tid == kBitBlock - 1) {
      const int K = bit_words_per_lane((int)S->lb);
      Q.g = task_geom(*S, t, P.TA, 32u * (uint32_t)K);
      Q.K = K;
      Q.la = S->la;
      Q.lb = (int)S->lb;
      Q.mx = Q.la > Q.lb ? Q.la : Q.lb;
      Q.a_base = S->aenc_base + (Q.g.a0 - S->a_beg) * (uint32_t)Q.la;
      Q.b_base = S->brec_base + (Q.g.b0 - S->b_beg) * (uint32_t)Q.lb;
      Q.check = Q.g.tri && Q.g.a1 > Q.g.b0;
    }
    if (tid == 0) fetch(buf ^ 1);  // read after the barrier at the next task's start
    __syncthreads();
    const int K = Q.K;

    // match masks of the task's B words
    uint4* mz = reinterpret_cast<uint4*>(masks);
    for (int q = tid; q < (int)(T.alphabet * (kMaskRow / 16)); q += kBitBlock) mz[q] = make_uint4(0u, 0u, 0u, 0u);
    __syncthreads();
    {
      const int pitch = bit_pitch(K);
      for (int w = warp; w < K; w += kBitWarps) {
        const uint32_t b = Q.g.b0 + 32u * (uint32_t)w + (uint32_t)lane;
        if (b < Q.g.bend) {
          const int lb = Q.lb, at = w * pitch;
          const uint32_t shift = T.shift;
          const uint32_t* src = T.b_sym + Q.b_base + (32u * (uint32_t)w + (uint32_t)lane) * (uint32_t)lb;
#pragma unroll 4
          for (int j = 0; j < lb; ++j) {
            const uint32_t c = (__ldg(src + j) & 0xffffu) >> shift;
            const int bit = at + j;
            atomicOr(reinterpret_cast<uint32_t*>(masks + c * (uint32_t)kMaskRow) + lane * 2 + (bit >> 5), 1u << (bit & 31));
          }
        }
      }
    }
    if ((EPI == kEpiLists || kHist) && P.hist_mode != kHistNone) {
      // every bin this task can produce lies inside the histogram (proven
      // bounds; the launch's plan holds only length pairs that the bins cover)
      int lo, hi;
      pair_score_bounds(T.match, T.mismatch, T.gap, Q.la < Q.lb ? Q.la : Q.lb, Q.mx, lo, hi);
      if (lo < P.hist_lo || hi - P.hist_lo >= (int)P.nbins) {
        if (tid == 0) atomicOr(P.err, kErrHistRange);
        continue;  // block-uniform
      }
    }
    __syncthreads();
    switch (K) {
      case 8: bit_task<MM, XX, EPI, 8>(P, T, Q, masks, wh, sA, inserts, max_iters); break;
      case 7: bit_task<MM, XX, EPI, 7>(P, T, Q, masks, wh, sA, inserts, max_iters); break;
      case 6: bit_task<MM, XX, EPI, 6>(P, T, Q, masks, wh, sA, inserts, max_iters); break;
      case 5: bit_task<MM, XX, EPI, 5>(P, T, Q, masks, wh, sA, inserts, max_iters); break;
      case 4: bit_task<MM, XX, EPI, 4>(P, T, Q, masks, wh, sA, inserts, max_iters); break;
      case 3: bit_task<MM, XX, EPI, 3>(P, T, Q, masks, wh, sA, inserts, max_iters); break;
      case 2: bit_task<MM, XX, EPI, 2>(P, T, Q, masks, wh, sA, inserts, max_iters); break;
      default: bit_task<MM, XX, EPI, 1>(P, T, Q, masks, wh, sA, inserts, max_iters); break;
    }
    if (smem_hist) {  // 32-bit shared counters: flush long before they could wrap
      wpairs += (uint64_t)(Q.g.a1 - Q.g.a0) * (32u * (uint32_t)K);
      if (wpairs >= (1ull << 30)) {
        hist_flush(P, wh, lane);
        wpairs = 0;
      }
    }
  }
  if (smem_hist) hist_flush(P, wh, lane);
  if (P.stats) {
    for (int o = 16; o > 0; o >>= 1) inserts += __shfl_xor_sync(0xffffffffu, inserts, o);
    if (lane == 0 && inserts) atomicAdd(P.stats, (unsigned long long)inserts);
  }
}

}  // namespace nw
