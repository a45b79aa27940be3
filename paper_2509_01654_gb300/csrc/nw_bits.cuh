// nw_bits.cuh -- the bit-parallel alignment kernel (sm_103a): for match /
// mismatch scorings whose shifted recurrence has few steps (below), 64 cells
// of Algorithm 1's matrix advance per group of logic instructions.
//
// The rows, and why they hold, are in nw_bitrow.cuh.
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
// warps share them and take P.sub A words (kBitSub, fewer in small tasks) at a
// time each.  A row costs one broadcast read of the A symbol's code and one
// conflict-free 8-byte read.
//
// Score.  G = g * (sum of the word's h) = g * (sum of the planes' bit counts);
// for m >= 3 the planes are first recoded to binary digits, so that a word
// takes two or three bit counts.
//
// What bounds it: the logic pipe.  A row of (1, -1, -1), steps (3, 1), is 14
// logic operations and 3 additions per 32 columns, 34 instructions a lane for up
// to 48 cells where the DPX cell takes 3 for 2.  600k words, top-10 and histogram:
// 1,129 ms on the DPX kernel, 390 here, of which the logic operations at the
// measured LOP3 rate are 272 (the additions have a second pipe: 100 lanes a clock
// against 64), lists that move about 25 and the histogram's shared additions 13 to
// 20; the rest is issue slots and stalls (at 100k words the logic pipe is 70.5 %
// active, issue 65.8 %).
#pragma once

#include "nw_bitrow.cuh"
#include "nw_dp.cuh"

namespace nw {

// The A words of one task against the lane's K words (b = b0 + 32 w + lane).
template <int MM, int XX, int EPI, int K>
__device__ __forceinline__ void bit_task(const AlignParams& P, const Terms& T, const AlignTask& Q,
                                         const unsigned char* masks, uint32_t* wh, uint16_t* sA, uint32_t* queue,
                                         uint32_t& inserts) {
  constexpr int PITCH = bit_pitch(K);
  constexpr bool kSplit = PITCH == 8 || PITCH == 16 || PITCH == 32;
  constexpr bool kLists = EPI != kEpiMatrix;
  constexpr bool kHist = EPI == kEpiListsLaneHist;
  constexpr int KP = (K + 1) / 2;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const TaskGeom g = Q.g;
  const int pconst = T.gap * (Q.la + Q.lb);  // score = G + pconst
  const bool check = Q.check;
  const int la = Q.la;

  // columns of the lane's words: all of them, and all but each word's last
  B64 FM{0u, 0u}, NL{0u, 0u};
  {
    const uint64_t f = (1ull << Q.lb) - 1ull;
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
  const bool full = __all_sync(0xffffffffu, vmask == (1u << K) - 1u) && !check;

  // list bounds in G, packed for the prefilter (see neg_bound16): the lane's
  // B words, and A word c0 + lane of the words staged last
  uint32_t nB2[KP];
  uint32_t my_nA2 = 0u;
  auto load_bounds_B = [&]() {
#pragma unroll
    for (int i = 0; i < KP; ++i) {
      int t[2] = {INT_MAX, INT_MAX};
#pragma unroll
      for (int h = 0; h < 2; ++h)
        if (T.B.slots && ((vmask >> (2 * i + h)) & 1u))
          t[h] = g_bound(P, T, __ldcg(T.B.thr + g.b0 + 32u * (2 * i + h) + lane), Q.mx, pconst);
      nB2[i] = neg_bound2(t[0], t[1]);
    }
  };
  auto load_bound_A = [&](uint32_t c0, uint32_t nA) {
    const int t = T.A.slots && (uint32_t)lane < nA ? g_bound(P, T, __ldcg(T.A.thr + c0 + lane), Q.mx, pconst) : INT_MAX;
    my_nA2 = neg_bound2(t, t);
  };
  if constexpr (kLists) load_bounds_B();
  uint32_t waiting = 0u;  // queued candidates (warp-uniform)
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
    // their codes (two zero entries beyond for the reads ahead)
    __syncwarp();
    {
      const uint32_t total = nA * (uint32_t)la;
      const uint32_t* src = T.a_sym + Q.a_base + (size_t)(c0 - g.a0) * (uint32_t)la;
      const uint32_t shift = T.shift;
      for (uint32_t i = lane; i < total + 2u; i += 32u)
        sA[i] = i < total ? (uint16_t)((__ldg(src + i) & 0xffffu) >> shift) : (uint16_t)0;
    }
    const uint32_t my_orig = (EPI == kEpiMatrix && (uint32_t)lane < nA) ? __ldg(T.A.perm + c0 + lane) : 0u;
    if constexpr (kLists) load_bound_A(c0, nA);
    __syncwarp();

    const unsigned char* mrow = masks + lane * 8;
    const uint16_t* sp = sA;
    uint2 mv = *reinterpret_cast<const uint2*>(mrow + sp[0] * kMaskRow);
    uint32_t o1 = sp[1];
    auto next_mask = [&]() {  // the row's mask; the next one's read is issued
      const B64 M{mv.x, mv.y};
      mv = *reinterpret_cast<const uint2*>(mrow + o1 * kMaskRow);
      o1 = sp[2];
      ++sp;
      return M;
    };
    for (uint32_t w0 = 0; w0 < nA; ++w0) {
      const uint32_t a = c0 + w0;
      B64 H[bit_planes(MM, XX)];
      if (la > 0) {
        bit_first<MM, XX, kSplit>(H, next_mask(), NL);
        // (unrolled by 1, 2, 4: 388, 394, 398 ms at 600k words; eight bodies
        // share the instruction cache)
#pragma unroll 1
        for (int r = 1; r < la; ++r) bit_next<MM, XX, kSplit>(H, next_mask(), NL);
      } else {
#pragma unroll
        for (int x = 0; x < bit_planes(MM, XX); ++x) H[x] = {0u, 0u};
      }
      B64 D[bit_digits(MM)];
      bit_digit_planes<MM, XX>(H, D);
      int gv[K];
      bit_scores<MM, K>(D, FM, coef, gv);

      if constexpr (EPI == kEpiMatrix) {
        const uint32_t oa = __shfl_sync(0xffffffffu, my_orig, (int)w0);
#pragma unroll
        for (int w = 0; w < K; ++w) {
          if (!((vmask >> w) & 1u) || (check && a >= g.b0 + 32u * w + lane)) continue;
          const uint64_t i = oa < ob[w] ? oa : ob[w], j = oa < ob[w] ? ob[w] : oa;
          const uint64_t off = upper_offset(i, j, P.n);
          if (off >= P.mat_lo && off < P.mat_hi) P.mat[off] = (int8_t)(gv[w] + pconst);
        }
      } else {
        if constexpr (kHist) {
          // lane columns: a warp's additions never collide
          if (full) {
#pragma unroll
            for (int w = 0; w < K; ++w) atomicAdd(hcol + 32 * gv[w], 1u);
          } else {
#pragma unroll
            for (int w = 0; w < K; ++w)
              if (((vmask >> w) & 1u) && (!check || a < g.b0 + 32u * w + lane)) atomicAdd(hcol + 32 * gv[w], 1u);
          }
        } else if (EPI == kEpiLists && P.hist_mode != kHistNone) {
#pragma unroll
          for (int w = 0; w < K; ++w)
            if (((vmask >> w) & 1u) && (!check || a < g.b0 + 32u * w + lane))
              hist_add(P, wh, gv[w] + pconst - P.hist_lo);
        }
        // prefilter: non-zero when some word's G reaches its own list's bound,
        // or the largest G reaches the A word's
        uint32_t res[KP];
#pragma unroll
        for (int i = 0; i < KP; ++i)
          res[i] = (uint32_t)gv[2 * i] + (2 * i + 1 < K ? (uint32_t)gv[2 * i + 1 < K ? 2 * i + 1 : 0] * 65536u : 0u);
        const uint32_t nA2 = __shfl_sync(0xffffffffu, my_nA2, (int)w0);
        uint32_t top = res[0], any = __viaddmax_s16x2_relu(res[0], nB2[0], 0u);
#pragma unroll
        for (int i = 1; i < KP; ++i) {
          top = __vmaxs2(top, res[i]);
          any = __viaddmax_s16x2(res[i], nB2[i], any);
        }
        any = __viaddmax_s16x2(top, nA2, any);
        if (__any_sync(0xffffffffu, any != 0u)) {
          uint32_t cand = 0u;  // bit w: word w is a candidate
#pragma unroll
          for (int w = 0; w < K; ++w) {
            // the packed test again, one half at a time on plain integers
            const uint32_t n2 = __vmaxs2(nB2[w >> 1], nA2);
            const int nb = (w & 1) ? (int)n2 >> 16 : (int)(int16_t)n2;
            const bool in = gv[w] + nb > 0 && (!check || a < g.b0 + 32u * w + lane);
            cand |= (in ? 1u : 0u) << w;
          }
          cand &= vmask;
          bool filed = false;
          while (__any_sync(0xffffffffu, cand != 0u)) {
            const int w = __ffs(cand) - 1;  // (-1: nothing left, the entry is not used)
            uint32_t G = res[0];
#pragma unroll
            for (int i = 1; i < KP; ++i) G = (w >> 1) == i ? res[i] : G;
            G = (w & 1) ? G >> 16 : G & 0xffffu;
            filed |= queue_candidate<kFileAhead<EPI>>(P, T, Q, queue, waiting, inserts, cand != 0u,
                                     (G << 16) | ((a - g.a0) << 8) | (32u * (uint32_t)w + (uint32_t)lane));
            cand &= cand - 1u;
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

// Blocks per SM the kernel is compiled for: 5 leave the row loop and the
// epilogue ~100 registers a thread.  600k words: 4 blocks 407 ms, 5 blocks
// 394, 6 blocks 408, 8 blocks 414 (the row loop unrolled twice).
constexpr int kBitMinBlocks = 5;

template <int MM, int XX, int EPI>
__global__ void __launch_bounds__(kBitBlock, kBitMinBlocks) nw_bit_kernel(const __grid_constant__ AlignParams P) {
  extern __shared__ __align__(16) unsigned char s_bits[];
  __shared__ unsigned long long s_task[2];
  __shared__ uint32_t s_seg[2];
  __shared__ uint32_t s_queue[kBitWarps][kQueueEntries];
  // the task's terms and geometry live in shared memory: most of them are
  // read on the rare paths only, and registers are what bounds the block count
  __shared__ Terms T;
  __shared__ AlignTask Q;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  // dynamic shared memory: match masks, histogram (lane columns shared by the
  // block, or one array per warp), staged A symbols
  constexpr bool kHist = EPI == kEpiListsLaneHist;
  const bool warp_hist = EPI == kEpiLists && P.hist_mode == kHistSmem;
  const uint32_t hist_words = kHist ? P.nbins * 32u : (warp_hist ? P.nbins * kBitWarps : 0u);
  unsigned char* masks = s_bits;
  uint32_t* hist0 = reinterpret_cast<uint32_t*>(s_bits + P.mask_bytes);
  uint32_t* wh = hist0 + (warp_hist ? (size_t)warp * P.nbins : 0);
  uint16_t* sA = reinterpret_cast<uint16_t*>(hist0 + hist_words) + (size_t)warp * P.stage_syms;
  for (uint32_t q = (uint32_t)tid; q < hist_words; q += kBitBlock) hist0[q] = 0u;
  uint64_t hpairs = 0;
  uint32_t inserts = 0;
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
      const uint32_t* src = reinterpret_cast<const uint32_t*>(EPI == kEpiOtherLists && P.terms ? P.terms + d : P.local + d);
      if (tid < (int)(sizeof(Terms) / 4)) reinterpret_cast<uint32_t*>(&T)[tid] = src[tid];
    }
    if (tid == kBitBlock - 1) {
      const int K = bit_words_per_lane((int)S->lb);
      Q.g = task_geom(*S, t, P.TA, 32u * (uint32_t)K);
      Q.K = K;
      Q.la = S->la;
      Q.lb = (int)S->lb;
      Q.mx = Q.la > Q.lb ? Q.la : Q.lb;
      Q.a_base = S->aenc_base + (Q.g.a0 - S->a_beg) * (uint32_t)Q.la;
      Q.b_base = S->b_base + (Q.g.b0 - S->b_beg) * (uint32_t)Q.lb;
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
            atomicOr(reinterpret_cast<uint32_t*>(masks + c * kMaskRow) + lane * 2 + (bit >> 5), 1u << (bit & 31));
          }
        }
      }
    }
    if ((EPI == kEpiLists || kHist) && P.hist_mode != kHistNone && !hist_covers(P, T, Q)) {
      if (tid == 0) atomicOr(P.err, kErrHistRange);
      continue;  // block-uniform
    }
    __syncthreads();
    switch (K) {
      case 8: bit_task<MM, XX, EPI, 8>(P, T, Q, masks, wh, sA, s_queue[warp], inserts); break;
      case 7: bit_task<MM, XX, EPI, 7>(P, T, Q, masks, wh, sA, s_queue[warp], inserts); break;
      case 6: bit_task<MM, XX, EPI, 6>(P, T, Q, masks, wh, sA, s_queue[warp], inserts); break;
      case 5: bit_task<MM, XX, EPI, 5>(P, T, Q, masks, wh, sA, s_queue[warp], inserts); break;
      case 4: bit_task<MM, XX, EPI, 4>(P, T, Q, masks, wh, sA, s_queue[warp], inserts); break;
      case 3: bit_task<MM, XX, EPI, 3>(P, T, Q, masks, wh, sA, s_queue[warp], inserts); break;
      case 2: bit_task<MM, XX, EPI, 2>(P, T, Q, masks, wh, sA, s_queue[warp], inserts); break;
      default: bit_task<MM, XX, EPI, 1>(P, T, Q, masks, wh, sA, s_queue[warp], inserts); break;
    }
    if (hist_words) {
      hpairs += (uint64_t)(Q.g.a1 - Q.g.a0) * (32u * (uint32_t)K);  // (more than the warp's share)
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
