// nw_dp.cuh -- the DPX alignment kernel (sm_103a), whose inner loop is unrolled
// for the length LB of the longer word of a pair, and the list and histogram
// updates it shares with the bit-parallel kernel (nw_bits.cuh).  It scores
// substitution-matrix dictionaries, the match / mismatch scorings that the
// bit-parallel kernel does not take, and the long words of its dearest classes
// (take_long).
//
// Recurrence.  Algorithm 1 of the paper fills H[i][j] = max(H[i-1][j-1] +
// sim(A[i-1], B[j-1]), H[i-1][j] + p, H[i][j-1] + p) from H[i][0] = p*i and
// H[0][j] = p*j and returns H[la][lb].  With G[i][j] = H[i][j] - p*(i + j)
// the same recurrence reads
//     G[i][j] = max(G[i-1][j-1] + s'(a, b), G[i-1][j], G[i][j-1]),
//     G[i][0] = G[0][j] = 0,   s'(a, b) = sim(a, b) - 2p,
// so the gap terms vanish, every G is >= 0 and the score is
// G[la][lb] + p*(la + lb).  This is an exact rewrite (same maximising paths).
//
// Packing.  A lane holds two B words of length LB (lo and hi 16-bit halves
// of each register) and their DP row G[i][1..LB] in LB registers; the warp
// streams one A word at a time (the same symbol in both halves), so each
// packed instruction advances two alignments by one cell.  Per packed cell:
//     xt = a2 ^ b2[j]                    per half: -1 - (e(a) ^ e(b))
//     f  = viaddmax(xt, s'_m + 1, s'_x+) per half: s'_m if a == b else s'_x+
//     d  = diag + f                      plain 32-bit add (both halves >= 0)
//     h  = vimax3(d, up, left)           max(G[i-1][j-1] + s', G[i-1][j], G[i][j-1])
// The codes are stored shifted (e(c) = c << shift, 2^shift >= match -
// mismatch), so for different codes e(a) ^ e(b) >= match - mismatch and
// s'_m - (e(a) ^ e(b)) <= s'_x: the max with s'_x then selects the mismatch
// value.  s'_x+ = max(s'_x, 0): G is non-decreasing along rows and columns,
// so G[i-1][j-1] + s'_x < 0 + G[i-1][j-1] <= G[i-1][j] whenever s'_x < 0 and
// raising the mismatch term to 0 changes no maximum; it keeps f >= 0, so the
// packed add never carries between halves (G + f <= s'_m * LB < 2^15).
// Per two cells: one LOP3, one add and two DPX instructions.
//
// Substitution-matrix scoring (TAB): the lane holds its B words' codes
// (lo / hi halves) and the per-cell term is read from the table row of the A
// symbol, f = s'+(a, b_lo) | s'+(a, b_hi) << 16 with s'+ = max(s', 0) (the
// same argument as above makes the clamp exact and keeps the add carry-free).
#pragma once

#include <cuda_runtime.h>
#include <limits.h>

#include "nw_internal.cuh"

namespace nw {

template <int LB>
struct BRow {
  uint32_t v[LB > 0 ? LB : 1];
};

// the packed per-cell term of symbol pair column j
template <int LB, bool TAB>
__device__ __forceinline__ uint32_t cell_term(uint32_t a2, const BRow<LB>& b, int j, uint32_t C1, uint32_t C2,
                                              const uint16_t* trow) {
  if constexpr (TAB) {
    const uint32_t bv = b.v[j];
    return (uint32_t)trow[bv & 0xffffu] | ((uint32_t)trow[bv >> 16] << 16);
  } else {
    return __viaddmax_s16x2(a2 ^ b.v[j], C1, C2);
  }
}

// the table row of A symbol a2 (codes stored unshifted in TAB dictionaries)
template <bool TAB>
__device__ __forceinline__ const uint16_t* tab_row(const uint16_t* tab, uint32_t a2) {
  if constexpr (TAB) return tab + ((a2 & 0xffffu) * (uint32_t)kTabDim);
  return nullptr;
}

// One row of the shifted recurrence: G[1..LB] of row i-1 becomes row i.
template <int LB, bool TAB = false>
__device__ __forceinline__ void dp_row(uint32_t (&G)[LB], uint32_t a2, const BRow<LB>& b, uint32_t C1,
                                       uint32_t C2, const uint16_t* tab = nullptr) {
  const uint16_t* trow = tab_row<TAB>(tab, a2);
  uint32_t diag = 0u, left = 0u;
#pragma unroll
  for (int j = 0; j < LB; ++j) {
    const uint32_t f = cell_term<LB, TAB>(a2, b, j, C1, C2, trow);
    const uint32_t up = G[j];
    const uint32_t h = __vimax3_s16x2(diag + f, up, left);
    diag = up;
    G[j] = h;
    left = h;
  }
}

// The first row (i = 1): diag and up are G[0][*] = 0 and f, left >= 0, so
// the cell is max(f, left) and no row of zeros needs setting up.
template <int LB, bool TAB = false>
__device__ __forceinline__ void dp_row_first(uint32_t (&G)[LB], uint32_t a2, const BRow<LB>& b, uint32_t C1,
                                             uint32_t C2, const uint16_t* tab = nullptr) {
  const uint16_t* trow = tab_row<TAB>(tab, a2);
  uint32_t left = 0u;
#pragma unroll
  for (int j = 0; j < LB; ++j) {
    const uint32_t f = cell_term<LB, TAB>(a2, b, j, C1, C2, trow);
    left = __vimax_s16x2_relu(f, left);
    G[j] = left;
  }
}

// DP over the la rows of one A word against the lane's two B words; returns
// the packed G[la][LB] (0 when la == 0 or LB == 0).
template <int LB, bool TAB = false>
__device__ __forceinline__ uint32_t dp_word(const uint32_t* __restrict__ arow, int la,
                                            const BRow<LB>& b, uint32_t C1, uint32_t C2,
                                            const uint16_t* tab = nullptr) {
  if constexpr (LB == 0) {
    return 0u;
  } else {
    uint32_t G[LB];
#pragma unroll
    for (int j = 0; j < LB; ++j) G[j] = 0u;
    int i = 0;
#pragma unroll 1
    for (; i + 1 < la; i += 2) {
      const uint32_t a0 = __ldg(arow + i);
      const uint32_t a1 = __ldg(arow + i + 1);
      dp_row<LB, TAB>(G, a0, b, C1, C2, tab);
      dp_row<LB, TAB>(G, a1, b, C1, C2, tab);
    }
    if (i < la) dp_row<LB, TAB>(G, __ldg(arow + i), b, C1, C2, tab);
    return G[LB - 1];
  }
}

// The same DP with the A word's symbols in shared memory, symbol i at
// acol[32 * i] (the staging layout of the all-pairs kernel; every lane reads
// the same address, so each load is a broadcast).  One row per iteration: a
// body of R rows is about 64 R LB bytes of instructions, and the warps of an
// SM sub-partition are at different places of it.  With four rows, LB = 31..40
// spent 10 of 13 stall cycles per issue waiting for instructions; 4, 2 and 1
// rows took 10.7, 9.5 and 8.9 ms for a batch of 16 dictionaries (lengths
// 1..40), and 1 row was also the fastest for 20k and 200k words of 1..25.
template <int LB, bool TAB = false>
__device__ __forceinline__ uint32_t dp_word_staged(const uint32_t* acol, int la, const BRow<LB>& b, uint32_t C1,
                                                   uint32_t C2, const uint16_t* tab = nullptr) {
  if constexpr (LB == 0) {
    return 0u;
  } else {
    if (la == 0) return 0u;
    uint32_t G[LB];
    dp_row_first<LB, TAB>(G, acol[0], b, C1, C2, tab);
#pragma unroll 1
    for (int i = 1; i < la; ++i) dp_row<LB, TAB>(G, acol[32 * i], b, C1, C2, tab);
    return G[LB - 1];
  }
}

template <int LB>
__device__ __forceinline__ void load_brow(const uint4* __restrict__ rec, BRow<LB>& b) {
  if constexpr (LB > 0) {
    constexpr int Q = ceil4(LB) / 4;
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      const uint4 v = __ldg(rec + q);
      if (4 * q + 0 < LB) b.v[4 * q + 0] = v.x;
      if (4 * q + 1 < LB) b.v[4 * q + 1] = v.y;
      if (4 * q + 2 < LB) b.v[4 * q + 2] = v.z;
      if (4 * q + 3 < LB) b.v[4 * q + 3] = v.w;
    }
  }
}

// Offers `key` to a word's list of k slots.  The slots always hold the k
// largest keys offered so far (0 = empty); keys of one list are distinct.
// The smallest slot is replaced by compare-and-swap; a failed swap means
// another thread changed that slot, so the scan repeats (bounded).  Slots only
// grow, so a stale read can only make the swap fail, never corrupt the set.
// Returns a lower bound of the list's current smallest key and raises it in
// *thr.
template <bool kAhead = false>
__device__ __forceinline__ uint32_t list_offer(uint32_t* row, uint32_t* thr, uint32_t k,
                                               uint32_t key, uint32_t* err, uint32_t& inserts, int max_iters) {
  for (int it = 0; it < max_iters; ++it) {
    uint32_t m1 = 0xffffffffu, m2 = 0xffffffffu, mi = 0;
    auto slot = [&](uint32_t s, uint32_t v) {
      if (v < m1) { m2 = m1; m1 = v; mi = s; }
      else if (v < m2) { m2 = v; }
    };
    if constexpr (kAhead) {
      for (uint32_t s0 = 0; s0 < k; s0 += 8u) {  // eight slots' reads in flight
        uint32_t v[8];
#pragma unroll
        for (uint32_t q = 0; q < 8u; ++q) v[q] = s0 + q < k ? __ldcg(row + s0 + q) : 0xffffffffu;
#pragma unroll
        for (uint32_t q = 0; q < 8u; ++q) slot(s0 + q, v[q]);
      }
    } else {
      for (uint32_t s = 0; s < k; ++s) slot(s, __ldcg(row + s));
    }
    if (key <= m1) {
      atomicMax(thr, m1);
      return m1;
    }
    if (atomicCAS(row + mi, m1, key) == m1) {
      const uint32_t nm = m2 < key ? m2 : key;
      atomicMax(thr, nm);
      ++inserts;
      return nm;
    }
  }
  atomicOr(err, kErrRetry);
  return 0xffffffffu;
}

// Offers the lanes' keys (0: none) to one list of k <= 32 slots, the warp together:
// lane s holds slot s, the largest key takes the place of the smallest slot until none
// is larger, and each slot that changed is swapped in memory.  A failed swap means that
// another warp changed that slot: its key is offered again (bounded).  With j slots
// m_1 < .. < m_j given up, the j keys taken and the k - j slots left (slots only grow)
// are k keys above m_j, so each of them is rightly dropped whatever the other swaps do;
// a key is rejected only against k slots above it.
__device__ __forceinline__ void list_offer_warp(uint32_t* row, uint32_t* thr, uint32_t k, uint32_t key, uint32_t* err,
                                                uint32_t& inserts, int max_iters) {
  const uint32_t lane = threadIdx.x & 31u;
  for (int it = 0; it < max_iters; ++it) {
    const uint32_t old = lane < k ? __ldcg(row + lane) : 0xffffffffu;
    uint32_t now = old, low;
    for (;;) {
      low = __reduce_min_sync(0xffffffffu, now);
      const uint32_t top = __reduce_max_sync(0xffffffffu, key);
      if (top <= low) break;
      if ((uint32_t)(__ffs(__ballot_sync(0xffffffffu, now == low)) - 1) == lane) now = top;
      if (key == top) key = 0u;  // (keys of one list are distinct)
    }
    key = 0u;
    if (now != old) {
      if (atomicCAS(row + lane, old, now) == old) ++inserts;
      else key = now;
    }
    if (!__any_sync(0xffffffffu, key != 0u)) {
      if (lane == 0u) atomicMax(thr, low);
      return;
    }
  }
  if (lane == 0u) atomicOr(err, kErrRetry);
}

// global -> shared 4-byte asynchronous copy (cp.async.ca; 4-byte aligned)
__device__ __forceinline__ void cp_async4(uint32_t* dst, const uint32_t* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"((uint32_t)__cvta_generic_to_shared(dst)),
               "l"(src)
               : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

__device__ __forceinline__ uint64_t upper_offset(uint64_t i, uint64_t j, uint64_t n) {
  // pair (i, j), i < j, in the row-major upper triangle: S(i-1) + (j - i - 1)
  return i * (2 * n - i - 1) / 2 + (j - i - 1);
}

// Histogram accumulation.  kHistLane: every lane owns a column of the block's
// shared array (bin b of lane l at b*32 + l), so the shared additions of a
// warp never collide; kHistSmem: one shared array per warp; kHistGlobal:
// global atomics.  `bin` is the score minus the histogram's lowest score.
__device__ __forceinline__ void hist_add(const AlignParams& P, uint32_t* wh, int bin) {
  const uint32_t bi = (uint32_t)bin;
  if (bi >= P.nbins) { atomicOr(P.err, kErrHistRange); return; }
  if (P.hist_mode == kHistSmem) atomicAdd(wh + bi, 1u);
  else atomicAdd(P.hist + bi, 1ull);
}

// Moves the shared counters (lane columns, or a warp's array) to the
// histogram, taking each by exchange: other warps may be adding meanwhile.
__device__ __forceinline__ void hist_flush(const AlignParams& P, uint32_t* wh, int lane) {
  if (P.hist_mode == kHistLane) {
    for (uint32_t b = lane; b < P.nbins; b += 32) {
      uint32_t c = 0;
      for (int l = 0; l < 32; ++l) c += atomicExch(wh + b * 32u + (uint32_t)((l + lane) & 31), 0u);  // rotated: no bank conflicts
      if (c) atomicAdd(P.hist + b, (unsigned long long)c);
    }
  } else {
    for (uint32_t b = lane; b < P.nbins; b += 32) {
      const uint32_t c = atomicExch(wh + b, 0u);
      if (c) atomicAdd(P.hist + b, (unsigned long long)c);
    }
  }
}
// A warp flushes after this many of its pairs: eight warps' pairs, all in one
// lane column and bin, still fit the 32-bit counters and their 32-lane sum.
constexpr uint64_t kHistFlushPairs = 1ull << 28;

// Lowest and highest score any pair of lengths la <= lb can reach: the
// all-gap alignment and the alignment with min(la, lb) diagonal columns bound
// the optimum from below, and no alignment beats the diagonal one with every
// diagonal column a match from above (for gap <= 0; with gap > 0 the all-gap
// alignment is the larger).
__device__ __forceinline__ void pair_score_bounds(int match, int mismatch, int gap, int la, int lb, int& lo,
                                                  int& hi) {
  const int allgap = (la + lb) * gap;
  const int diag_lo = la * mismatch + (lb - la) * gap;
  const int diag_hi = la * match + (lb - la) * gap;
  lo = allgap > diag_lo ? allgap : diag_lo;
  hi = allgap > diag_hi ? allgap : diag_hi;
}

// Every bin a task can produce lies inside the histogram (checked once per
// task against the proven score bounds instead of per pair).
__device__ __forceinline__ bool hist_covers(const AlignParams& P, const Terms& T, const AlignTask& Q) {
  int lo, hi;
  pair_score_bounds(T.match, T.mismatch, T.gap, Q.la < Q.lb ? Q.la : Q.lb, Q.mx, lo, hi);
  return lo >= P.hist_lo && hi - P.hist_lo < (int)P.nbins;
}

// List key of a pair with score s whose longer word has m symbols: the raw
// score, or the rank of s/m in the normalised ranking, above the partner's
// reversed index (higher key = better neighbour).
__device__ __forceinline__ uint32_t list_key(const AlignParams& P, const Terms& T, int s, int m, uint32_t partner) {
  const uint32_t v = P.norm_rank ? (uint32_t)P.norm_rank[(s - P.norm_lo) * kBuckets + m] + 1u
                                 : (uint32_t)(s - T.key_lo);
  return (v << T.ib) | (T.imask - partner);
}

// G-space candidate bound of a list whose smallest key is >= thr_key, for
// pairs whose longer word has m symbols: a pair can enter the list only if its
// G value (score - pconst) reaches this bound.  With raw keys that is the
// threshold's own score; with normalised keys, the smallest score whose s/m
// has the threshold's rank (a lower rank makes a key below any key of that
// rank, whatever the partner).
__device__ __forceinline__ int g_bound(const AlignParams& P, const Terms& T, uint32_t thr_key, int m, int pconst) {
  if (thr_key == 0u) return INT_MIN;
  if (P.norm_rank) return (int)P.norm_smin[((thr_key >> T.ib) - 1u) * kBuckets + m] - pconst;
  return (int)(thr_key >> T.ib) + T.key_lo - pconst;
}

// Packed candidate prefilter.  A G-space bound t (a pair is a candidate for
// a list when G >= t) is held as 1 - t, clamped so that t = 0 admits every G
// (G >= 0) and t = 0x7fff none (G <= 819 * 40 < 0x7fff: the host bounds
// s'_m * NW_MAX_WORD_LEN by 32767).  For two results packed in res,
// viaddmax_relu(res, 1 - t, 0) is non-zero in a half exactly when G >= t there.
__device__ __forceinline__ uint32_t neg_bound16(int t) {
  const int c = t < 0 ? 0 : (t > 0x7fff ? 0x7fff : t);
  return (uint32_t)(1 - c) & 0xffffu;
}
__device__ __forceinline__ uint32_t neg_bound2(int t_lo, int t_hi) {
  return neg_bound16(t_lo) | (neg_bound16(t_hi) << 16);
}

// Candidate queue.  A pair that may enter a list is rare late in a launch and
// common early, and filing it takes several dependent trips to L2.  The lanes
// only append such pairs to their warp's queue; once 32 are waiting, each lane
// files one, so the trips overlap 32-fold.  (Filing each pair in the lane that
// found it took 126 of 584 ms at 600k words in the bit-parallel kernel, and
// half of its time at 100k.)  An entry: G << 16 | A word (from g.a0) << 8 |
// B word (from g.b0); G < 2^15, a task has at most 256 words on either side.
//
// Files n <= 32 queued pairs in their words' lists; returns the lane's inserts.
// kAhead: the slots of a list are read eight at a time, and where only A words
// have lists (queries) a warp's candidates for one list are offered together
// (list_offer_warp; above 32 slots one by one, the best first): a list that starts
// empty takes k candidates of each of the first warps, and one by one each was four
// trips to L2.  One by one, 16 queries of 12 symbols against 2,000 words took 388 us
// on the DPX kernel (269 before the queue) and 672 with a similarity matrix, whose
// kernels had no such epilogue (296); together 199 and 206.  Bit-parallel: one query against
// 600k words 196 -> 139 us, 4,096 11.8 -> 10.8 ms.  The all-pairs kernels, whose lists
// belong to both sides, lose by reading ahead at 600k words (390 -> 418 ms with
// histogram, 380 -> 410 normalised): there it is compiled out.
template <int EPI>
constexpr bool kFileAhead = EPI == kEpiOtherLists;
template <bool kAhead>
__device__ __forceinline__ uint32_t file_candidates_inline(const AlignParams& P, const Terms& T, const AlignTask& Q,
                                                    const uint32_t* queue, uint32_t n) {
  const uint32_t lane = threadIdx.x & 31u;
  const int max_iters = P.dbg_insert_limit ? (int)(P.dbg_insert_limit - 1u) : kInsertMaxIters;
  const bool have = lane < n;
  const uint32_t e = have ? queue[lane] : 0u;
  const uint32_t a = Q.g.a0 + ((e >> 8) & 0xffu), b = Q.g.b0 + (e & 0xffu);
  const int s = (int)(e >> 16) + T.gap * (Q.la + Q.lb);
  const uint32_t oa = have ? __ldg(T.A.perm + a) : 0u, ob = have ? __ldg(T.B.perm + b) : 0u;
  uint32_t inserts = 0u;
  if (T.B.slots && have) {  // word b takes the A word as a neighbour
    const uint32_t key = list_key(P, T, s, Q.mx, oa);
    if (key > __ldcg(T.B.thr + b))
      list_offer<kAhead>(T.B.slots + (size_t)b * P.k, T.B.thr + b, P.k, key, P.err, inserts, max_iters);
  }
  if (T.A.slots) {
    // the A word takes word b.  Several lanes may hold the same A word: one
    // lane of each such group offers at a time and the others are tested again
    // against the bound it leaves, so the lanes never race on one list
    uint32_t key = 0u;
    if (have) {
      key = list_key(P, T, s, Q.mx, ob);
      if (key <= __ldcg(T.A.thr + a)) key = 0u;
    }
    uint32_t todo;
    if (kAhead && !T.B.slots && P.k <= 32u) {  // one list at a time, its candidates together
      while ((todo = __ballot_sync(0xffffffffu, key != 0u)) != 0u) {
        const uint32_t a0 = __shfl_sync(0xffffffffu, a, __ffs(todo) - 1);
        const bool mine = key != 0u && a == a0;
        list_offer_warp(T.A.slots + (size_t)a0 * P.k, T.A.thr + a0, P.k, mine ? key : 0u, P.err, inserts, max_iters);
        if (mine) key = 0u;
      }
      return inserts;
    }
    const uint32_t group = __match_any_sync(0xffffffffu, a);
    while ((todo = __ballot_sync(0xffffffffu, key != 0u)) != 0u) {
      bool lead = (uint32_t)(__ffs(todo & group) - 1) == lane;
      if constexpr (kAhead) {
        if (!T.B.slots && __all_sync(0xffffffffu, key == 0u || (todo & group) == todo))  // one list: its best first
          lead = key == __reduce_max_sync(0xffffffffu, key);
      }
      if (lead) {
        list_offer<kAhead>(T.A.slots + (size_t)a * P.k, T.A.thr + a, P.k, key, P.err, inserts, max_iters);
        key = 0u;
      }
      __syncwarp();
      if (key != 0u && key <= __ldcg(T.A.thr + a)) key = 0u;
    }
  }
  return inserts;
}

// Out of line with kAhead: inline, every length's body of a DPX kernel held three
// copies (16 dictionaries 8.5 ms, out of line 7.7; queries the same within 2 %).  The
// all-pairs kernels file inline.
template <bool kAhead>
__device__ __noinline__ uint32_t file_candidates_call(const AlignParams& P, const Terms& T, const AlignTask& Q,
                                                      const uint32_t* queue, uint32_t n) {
  return file_candidates_inline<kAhead>(P, T, Q, queue, n);
}
template <bool kAhead>
__device__ __forceinline__ uint32_t file_candidates(const AlignParams& P, const Terms& T, const AlignTask& Q,
                                                    const uint32_t* queue, uint32_t n) {
  if constexpr (kAhead) return file_candidates_call<true>(P, T, Q, queue, n);
  else return file_candidates_inline<false>(P, T, Q, queue, n);
}

// Appends the lanes' candidates (`have`) to the queue and files the first 32
// once as many are waiting; true if it filed (the lists' bounds have moved).
template <bool kAhead>
__device__ __forceinline__ bool queue_candidate(const AlignParams& P, const Terms& T, const AlignTask& Q,
                                                uint32_t* queue, uint32_t& waiting, uint32_t& inserts, bool have,
                                                uint32_t entry) {
  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t m = __ballot_sync(0xffffffffu, have);
  if (have) queue[waiting + __popc(m & ((1u << lane) - 1u))] = entry;
  waiting += __popc(m);
  if (waiting < 32u) return false;
  __syncwarp();
  inserts += file_candidates<kAhead>(P, T, Q, queue, 32u);
  waiting -= 32u;
  const uint32_t v = lane < waiting ? queue[32 + lane] : 0u;
  __syncwarp();
  queue[lane] = v;
  __syncwarp();
  return true;
}

// One task: the A words of a chunk against the lane's two B words of length
// LB.  TAB selects substitution-matrix scoring; EPI the per-pair epilogue:
// kEpiMatrix writes the int8 upper triangle, kEpiLists updates neighbour lists
// (and a shared or global histogram), kEpiListsLaneHist lists and the lane
// columns of the shared histogram, kEpiOtherLists the lists of queries and of
// batches (named by the segment's terms in a launch spanning dictionaries).
template <int LB, int EPI, bool TAB>
__device__ __forceinline__ void dp_task(const AlignParams& P, const Terms& T, const AlignTask& Q, uint32_t* wh,
                                        uint32_t* sA, const uint16_t* sTab, uint32_t* queue, uint32_t& inserts) {
  constexpr bool kLists = EPI != kEpiMatrix;
  const int lane = threadIdx.x & 31;
  const TaskGeom g = Q.g;
  const int la = Q.la;
  const int pconst = T.gap * (la + LB);  // score = G + pconst
  const bool check = Q.check;
  const uint32_t C1 = T.C1, C2 = T.C2;
  const uint32_t blo = g.b0 + 2u * lane, bhi = blo + 1u;
  const bool vlo = blo < g.bend, vhi = bhi < g.bend;

  BRow<LB> brow;
  if constexpr (LB > 0) {
#pragma unroll
    for (int j = 0; j < LB; ++j) brow.v[j] = 0xffffffffu;
    if (vlo) load_brow<LB>(T.b_rec + Q.b_base + (size_t)lane * (ceil4(LB) / 4), brow);
    if constexpr (TAB) {
      // records hold ~code per half (unshifted codes): back to codes, and
      // code 0 for halves without a word (their results are discarded)
      const uint32_t keep = (vlo ? 0x0000ffffu : 0u) | (vhi ? 0xffff0000u : 0u);
#pragma unroll
      for (int j = 0; j < LB; ++j) brow.v[j] = ~brow.v[j] & keep;
    }
  }
  uint32_t ob_lo = 0u, ob_hi = 0u;
  if constexpr (EPI == kEpiMatrix) {
    ob_lo = vlo ? __ldg(T.B.perm + blo) : 0u;
    ob_hi = vhi ? __ldg(T.B.perm + bhi) : 0u;
  }
  uint32_t* hcol = wh + (ptrdiff_t)lane + (ptrdiff_t)(pconst - P.hist_lo) * 32;  // lane column shifted so bin = G

  // packed list bounds of the lane's words, and of A word c0 + lane
  uint32_t nB2 = 0u, my_nA2 = 0u, waiting = 0u;
  auto load_bounds_B = [&]() {
    nB2 = neg_bound2(T.B.slots && vlo ? g_bound(P, T, __ldcg(T.B.thr + blo), LB, pconst) : INT_MAX,
                     T.B.slots && vhi ? g_bound(P, T, __ldcg(T.B.thr + bhi), LB, pconst) : INT_MAX);
  };
  auto load_bound_A = [&](uint32_t c0, uint32_t nA) {
    const int t = T.A.slots && (uint32_t)lane < nA ? g_bound(P, T, __ldcg(T.A.thr + c0 + lane), LB, pconst) : INT_MAX;
    my_nA2 = neg_bound2(t, t);
  };
  if constexpr (kLists) load_bounds_B();

  for (uint32_t c0 = g.a0; c0 < g.a1; c0 += 32u) {
    // Stage 32 A words: lane l copies word c0 + l (la symbols); the warp then
    // reads symbols as shared-memory broadcasts and the G-space bound by shuffle.
    const uint32_t nA = g.a1 - c0 < 32u ? g.a1 - c0 : 32u;
    const bool have = (uint32_t)lane < nA;
    const uint32_t my_orig = (EPI == kEpiMatrix && have) ? __ldg(T.A.perm + c0 + lane) : 0u;
    if constexpr (kLists) load_bound_A(c0, nA);
    __syncwarp();
    if (have) {
      // asynchronous 4-byte copies: the word's symbol loads are in flight together
      const uint32_t* src = T.a_sym + Q.a_base + (size_t)(c0 - g.a0 + (uint32_t)lane) * (uint32_t)la;
      for (int i = 0; i < la; ++i) cp_async4(sA + 32 * i + lane, src + i);
    }
    cp_async_wait_all();
    __syncwarp();

    for (uint32_t w = 0; w < nA; ++w) {
      const uint32_t a = c0 + w;
      const uint32_t res = dp_word_staged<LB, TAB>(sA + w, la, brow, C1, C2, sTab);
      const int g_lo = (int)(res & 0xffffu);  // G >= 0
      const int g_hi = (int)(res >> 16);
      const bool ok_lo = vlo && (!check || a < blo), ok_hi = vhi && (!check || a < bhi);
      if constexpr (EPI == kEpiMatrix) {
        const uint32_t oa = __shfl_sync(0xffffffffu, my_orig, (int)w);
        if (ok_lo) {
          const uint64_t i = oa < ob_lo ? oa : ob_lo, j = oa < ob_lo ? ob_lo : oa;
          const uint64_t off = upper_offset(i, j, P.n);
          if (off >= P.mat_lo && off < P.mat_hi) P.mat[off] = (int8_t)(g_lo + pconst);
        }
        if (ok_hi) {
          const uint64_t i = oa < ob_hi ? oa : ob_hi, j = oa < ob_hi ? ob_hi : oa;
          const uint64_t off = upper_offset(i, j, P.n);
          if (off >= P.mat_lo && off < P.mat_hi) P.mat[off] = (int8_t)(g_hi + pconst);
        }
      } else {
        if constexpr (EPI == kEpiListsLaneHist) {
          if (ok_lo) atomicAdd(hcol + 32 * g_lo, 1u);
          if (ok_hi) atomicAdd(hcol + 32 * g_hi, 1u);
        } else if (EPI == kEpiLists && P.hist_mode != kHistNone) {
          if (ok_lo) hist_add(P, wh, g_lo + pconst - P.hist_lo);
          if (ok_hi) hist_add(P, wh, g_hi + pconst - P.hist_lo);
        }
        // both halves against the lower of their two lists' bounds
        const uint32_t n2 = __vmaxs2(nB2, __shfl_sync(0xffffffffu, my_nA2, (int)w));
        if (__any_sync(0xffffffffu, __viaddmax_s16x2_relu(res, n2, 0u) != 0u)) {
          const uint32_t at = ((a - g.a0) << 8) | (2u * (uint32_t)lane);
          bool filed = false;
#pragma unroll 1
          for (int h = 0; h < 2; ++h) {
            const int G = h ? g_hi : g_lo, nb = h ? (int)n2 >> 16 : (int)(int16_t)n2;
            const bool in = (h ? ok_hi : ok_lo) && G + nb > 0;
            if (!__any_sync(0xffffffffu, in)) continue;
            filed |= queue_candidate<kFileAhead<EPI>>(P, T, Q, queue, waiting, inserts, in, ((uint32_t)G << 16) | (at + (uint32_t)h));
          }
          if (filed) {
            load_bounds_B();
            load_bound_A(c0, nA);
          }
        }
      }
    }
  }
  if constexpr (kLists) {
    if (waiting) {
      __syncwarp();
      inserts += file_candidates<kFileAhead<EPI>>(P, T, Q, queue, waiting);
    }
  }
}

template <int LB, int HI, int EPI, bool TAB>
__device__ __forceinline__ void dp_dispatch(int lb, const AlignParams& P, const Terms& T, const AlignTask& Q,
                                            uint32_t* wh, uint32_t* sA, const uint16_t* sTab, uint32_t* queue,
                                            uint32_t& inserts) {
  if (lb == LB) {
    dp_task<LB, EPI, TAB>(P, T, Q, wh, sA, sTab, queue, inserts);
  } else if constexpr (LB < HI) {
    dp_dispatch<LB + 1, HI, EPI, TAB>(lb, P, T, Q, wh, sA, sTab, queue, inserts);
  }
}

// All pairs of a plan whose longer word has LO .. HI symbols.  Warps pull
// tasks from one counter and work on their own.  One launch covers ten lengths
// (a launch per length left most SMs idle for small dictionaries: every
// launch ended in a tail of single long tasks).
template <int LO, int HI, int EPI, bool TAB = false>
__global__ void __launch_bounds__(kBlock, dp_min_blocks(HI)) nw_dp_kernel(const __grid_constant__ AlignParams P) {
  extern __shared__ uint32_t s_dyn[];
  __shared__ Terms s_terms[kWarpsPerBlock];
  __shared__ AlignTask s_tasks[kWarpsPerBlock];
  __shared__ uint32_t s_queue[kWarpsPerBlock][kQueueEntries];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  constexpr bool kHist = EPI == kEpiListsLaneHist;
  const bool warp_hist = EPI == kEpiLists && P.hist_mode == kHistSmem;
  const uint32_t hist_words = kHist ? P.nbins * 32u : (warp_hist ? P.nbins * kWarpsPerBlock : 0u);
  // dynamic shared memory: substitution table, histogram, staged A symbols
  // (symbol i of the chunk's word w at 32 * i + w)
  uint16_t* sTab = nullptr;
  uint32_t* hist0 = s_dyn;
  if constexpr (TAB) {
    sTab = reinterpret_cast<uint16_t*>(s_dyn);
    hist0 = s_dyn + kTabBytes / sizeof(uint32_t);
    const uint4* src = reinterpret_cast<const uint4*>(P.sim_tab);
    uint4* dst = reinterpret_cast<uint4*>(sTab);
    for (int q = tid; q < (int)(kTabBytes / sizeof(uint4)); q += kBlock) dst[q] = __ldg(src + q);
  }
  uint32_t* wh = hist0 + (warp_hist ? (size_t)warp * P.nbins : 0);
  uint32_t* sA = hist0 + hist_words + (size_t)warp * P.stage_syms;
  for (uint32_t q = (uint32_t)tid; q < hist_words; q += kBlock) hist0[q] = 0u;
  __syncthreads();
  Terms& T = s_terms[warp];
  AlignTask& Q = s_tasks[warp];
  uint32_t inserts = 0;
  uint64_t hpairs = 0;

  for (;;) {
    unsigned long long t = 0;
    if (lane == 0) t = atomicAdd(P.counter, 1ull);
    t = __shfl_sync(0xffffffffu, t, 0);
    if (t >= P.ntasks) break;
    const Seg* S = P.segs + find_seg(P.segs, P.nsegs, t);
    const uint32_t d = S->dict;
    const uint32_t* src = reinterpret_cast<const uint32_t*>(EPI == kEpiOtherLists && P.terms ? P.terms + d : P.local + d);
    __syncwarp();
    for (int q = lane; q < (int)(sizeof(Terms) / 4); q += 32) reinterpret_cast<uint32_t*>(&T)[q] = src[q];
    if (lane == 0) {
      Q.g = task_geom(*S, t, P.TA);
      Q.la = S->la;
      Q.lb = (int)S->lb;
      Q.mx = Q.lb;
      Q.a_base = S->aenc_base + (Q.g.a0 - S->a_beg) * (uint32_t)Q.la;
      Q.b_base = S->b_base + ((Q.g.b0 - S->b_beg) / 2u) * (uint32_t)(ceil4(Q.lb) / 4);
      Q.check = Q.g.tri && Q.g.a1 > Q.g.b0;
    }
    __syncwarp();
    if ((EPI == kEpiLists || kHist) && P.hist_mode != kHistNone && !hist_covers(P, T, Q)) {
      if (lane == 0) atomicOr(P.err, kErrHistRange);
      continue;
    }
    dp_dispatch<LO, HI, EPI, TAB>(Q.lb, P, T, Q, wh, sA, sTab, s_queue[warp], inserts);
    if (hist_words) {
      hpairs += (uint64_t)(Q.g.a1 - Q.g.a0) * (uint32_t)kWarpB;
      if (hpairs >= kHistFlushPairs) {
        hist_flush(P, wh, lane);
        hpairs = 0;
      }
    }
  }
  if (hist_words) {
    __syncthreads();
    if (warp_hist || warp == 0) hist_flush(P, wh, lane);
  }
  if (P.stats) {
    for (int o = 16; o > 0; o >>= 1) inserts += __shfl_xor_sync(0xffffffffu, inserts, o);
    if (lane == 0 && inserts) atomicAdd(P.stats, (unsigned long long)inserts);
  }
}

}  // namespace nw
