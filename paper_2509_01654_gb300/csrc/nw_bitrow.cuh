// nw_bitrow.cuh -- one row of Algorithm 1's matrix in bit planes, shared by the
// bit-parallel kernels: all pairs and queries (nw_bits.cuh), explicit pairs and
// proposal candidates (nw_bitpairs.cuh).
//
// Recurrence.  With G[i][j] = H[i][j] - p*(i + j) (see nw_dp.cuh)
//     G[i][j] = max(G[i-1][j-1] + s, G[i-1][j], G[i][j-1]),  G[i][0] = G[0][j] = 0,
// s = s'_m on equal symbols and s'_x+ = max(s'_x, 0) otherwise.  Dividing by
// g = gcd(s'_m, s'_x+) leaves steps (m, x).  The horizontal and vertical
// differences h = G[i][j] - G[i][j-1] and v = G[i][j] - G[i-1][j] lie in
// 0 .. m, and one cell maps the difference h' above it and the difference v'
// to its left to
//     c = max(s, h', v'),   v = c - h',   h = c - v'
// (G[i-1][j-1] taken from the cell's three terms).  This is the bit-vector
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
#pragma once

#include <stdint.h>

#include "nw_internal.cuh"

namespace nw {

// The bit planes of 64 columns, or of 32.
struct B64 {
  uint32_t lo, hi;
};
struct B32 {
  uint32_t lo;
};
__device__ __forceinline__ B32 operator&(B32 a, B32 b) { return {a.lo & b.lo}; }
__device__ __forceinline__ B32 operator|(B32 a, B32 b) { return {a.lo | b.lo}; }
__device__ __forceinline__ B32 operator^(B32 a, B32 b) { return {a.lo ^ b.lo}; }
__device__ __forceinline__ B32 operator~(B32 a) { return {~a.lo}; }
__device__ __forceinline__ B64 operator&(B64 a, B64 b) { return {a.lo & b.lo, a.hi & b.hi}; }
__device__ __forceinline__ B64 operator|(B64 a, B64 b) { return {a.lo | b.lo, a.hi | b.hi}; }
__device__ __forceinline__ B64 operator^(B64 a, B64 b) { return {a.lo ^ b.lo, a.hi ^ b.hi}; }
__device__ __forceinline__ B64 operator~(B64 a) { return {~a.lo, ~a.hi}; }

// a + b: with Split (no word straddles bit 32) the halves are independent
template <bool Split>
__device__ __forceinline__ B32 add_cols(B32 a, B32 b) {
  return {a.lo + b.lo};
}
template <bool Split>
__device__ __forceinline__ B64 add_cols(B64 a, B64 b) {
  if constexpr (Split) {
    return {a.lo + b.lo, a.hi + b.hi};
  } else {
    const uint64_t s = (((uint64_t)a.hi << 32) | a.lo) + (((uint64_t)b.hi << 32) | b.lo);
    return {(uint32_t)s, (uint32_t)(s >> 32)};
  }
}

// One row: H[1..m] (index a - 1) of row i - 1 becomes row i.
template <int MM, int XX, bool Split, class W>
__device__ __forceinline__ void bit_row(W (&H)[MM], const W M, const W NL) {
  W U[MM + 1];  // U[a], a = 1..m (v' >= a)
  const W z = ~H[0] & NL;
  // (M | U[m]) and (M | H[m]) stand in for M: where v' = m the cell is a
  // match's anyway (v' - h' = m - h'), which saves the last term of each sum
#pragma unroll
  for (int a = MM; a >= 1; --a) {
    if (a > XX) {
      W g;
      if (a == MM) {
        g = M & z;
      } else {
        W t = M;  // M & ~H[m-a+1], joined by U[m] (b = m - a) under the same mask
        t = (t | U[MM]) & ~H[MM - a];
#pragma unroll
        for (int b = 1; b < MM - a; ++b) t = t | (~H[b] & U[a + b]);
        g = t & NL;
        // g may hold bits with H[1] = 0 and set: they are run starts too
      }
      const W P = g | z;
      const W s = add_cols<Split>(P, g);
      U[a] = P ^ g ^ s;
    } else {
      W t = a == MM ? (M & ~H[0]) : ((M | U[MM]) & ~H[MM - a]);
#pragma unroll
      for (int b = XX - a + 1 > 1 ? XX - a + 1 : 1; b < MM - a; ++b) t = t | (~H[b] & U[a + b]);
      t = (t | ~H[XX - a]) & NL;
      U[a] = add_cols<Split>(t, t);
    }
  }
  W N[MM];
  const W q = M | H[MM - 1];
#pragma unroll
  for (int a = 1; a <= MM; ++a) {
    W t = q & ~U[MM - a + 1];
    const int b0 = a <= XX ? XX - a + 1 : 0;
#pragma unroll
    for (int b = b0; b < MM - a; ++b) t = t | (~U[b + 1] & H[a + b - 1]);
    if (a <= XX) t = t | ~U[XX - a + 1];
    N[a - 1] = t;
  }
#pragma unroll
  for (int a = 0; a < MM; ++a) H[a] = N[a];
}

// Planes a row's state takes: thermometer planes, except for the steps (3, 1)
// of the paper's scoring, which keep h as two binary digits (below).
__host__ __device__ constexpr int bit_planes(int m, int x) { return m == 3 && x == 1 ? 2 : m; }

// One row of the steps (3, 1) on the binary digits H[0] + 2 H[1] of h.  The
// cell's c = max(s, h', v') is 1, 2 or 3: c >= 2 is C2 = M | h' >= 2 | v' >= 2,
// and c is odd unless it is 2.  v' = 3 and v' >= 2 come from the two carry
// chains above; the parities of v and h follow from c = v + h' = h + v' alone,
// without a plane for v >= 1: 14 logic operations and three additions, against
// 16 on thermometer planes.
template <bool Split, class W>
__device__ __forceinline__ void bit_row31(W (&H)[2], const W M, const W NL) {
  const W h0 = H[0], h1 = H[1];
  const W z = ~h1 & ~h0 & NL;                    // h' = 0
  const W g3 = M & z;
  const W U3 = add_cols<Split>(z, g3) ^ (z & ~M);   // v' = 3
  const W r = M | U3;
  const W g2 = r & ~h1 & NL;                     // c = 3 and h' <= 1
  const W U2 = add_cols<Split>(g2 | z, g2) ^ (z & ~g2);  // v' >= 2
  const W C2 = M | h1 | U2;
  const W odd = r | ((h1 & h0) | ~C2);           // c = 1 or 3
  const W v0 = (odd ^ h0) & NL;                  // v odd
  const W u0 = add_cols<Split>(v0, v0);             // v' odd
  H[0] = odd ^ u0;
  H[1] = C2 ^ U2 ^ (~odd & u0);
}
// The first row (h' = 0): v is 3 from a match on and 1 before it, so c is odd,
// v' is odd past a word's first column, and h = c - v'.
template <bool Split, class W>
__device__ __forceinline__ void bit_row31_first(W (&H)[2], const W M, const W NL) {
  const W g3 = M & NL;
  const W U3 = add_cols<Split>(NL, g3) ^ (NL & ~M);
  H[0] = ~add_cols<Split>(NL, NL);
  H[1] = M & ~U3;
}

// One row of the steps (2, 1), the general row with its terms written out: 9
// logic operations and two additions.  (As an instance of bit_row the compiler
// spilled 700 to 880 bytes a thread in every alignment kernel of this class: top-10
// lists and histogram of 20,000 words of 24 symbols, 128 codes, 8.5 ms, of 40
// symbols, 256 codes, 46.8 ms, slower than the DPX kernel's 28.2; written out 3.5
// and 12.5 ms.)
template <bool Split, class W>
__device__ __forceinline__ void bit_row21(W (&H)[2], const W M, const W NL) {
  const W h1 = H[0], h2 = H[1];
  const W z = ~h1 & NL;
  const W g = M & z;
  const W U2 = add_cols<Split>(z, g) ^ (z & ~g);  // v' = 2
  const W v1 = (((M | U2) & ~h2) | ~h1) & NL;     // v >= 1
  const W U1 = add_cols<Split>(v1, v1);
  const W q = M | h2;
  H[0] = (q & ~U2) | ~U1;
  H[1] = q & ~U1;
}

// The state recoded to binary digits: h = sum over d of 2^d * D[d].
__host__ __device__ constexpr int bit_digits(int m) { return m == 1 ? 1 : (m <= 3 ? 2 : 3); }
template <int MM, int XX, class W>
__device__ __forceinline__ void bit_digit_planes(const W (&H)[bit_planes(MM, XX)], W (&D)[bit_digits(MM)]) {
  if constexpr (MM == 3 && XX == 1) {
    D[0] = H[0];
    D[1] = H[1];
  } else if constexpr (MM == 1) {
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

// any later row, and row 1 from nothing
template <int MM, int XX, bool Split, class W>
__device__ __forceinline__ void bit_next(W (&H)[bit_planes(MM, XX)], const W M, const W NL) {
  if constexpr (MM == 3 && XX == 1) bit_row31<Split>(H, M, NL);
  else if constexpr (MM == 2) bit_row21<Split>(H, M, NL);
  else bit_row<MM, XX, Split>(H, M, NL);
}
template <int MM, int XX, bool Split, class W>
__device__ __forceinline__ void bit_first(W (&H)[bit_planes(MM, XX)], const W M, const W NL) {
  if constexpr (MM == 3 && XX == 1) {
    bit_row31_first<Split>(H, M, NL);
  } else {
#pragma unroll
    for (int a = 0; a < MM; ++a) H[a] = W{};  // folds most of the row away
    bit_next<MM, XX, Split>(H, M, NL);
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

// G of words 0..K-1 at a pitch of PITCH columns (real units: coef = g)
template <int MM, int K, int W = 0, int PITCH = bit_pitch(K)>
__device__ __forceinline__ void bit_scores(const B64 (&D)[bit_digits(MM)], B64 FM, int coef, int (&g)[K]) {
  if constexpr (W < K) {
    int v = 0;
#pragma unroll
    for (int d = 0; d < bit_digits(MM); ++d) v += field_count<W, PITCH>(D[d], FM) * (coef << d);
    g[W] = v;
    bit_scores<MM, K, W + 1, PITCH>(D, FM, coef, g);
  }
}

// the words' lengths from their field masks
template <int K, int W, int PITCH>
__device__ __forceinline__ void field_lengths(B64 FM, int (&len)[K]) {
  if constexpr (W < K) {
    len[W] = field_count<W, PITCH>(FM, FM);
    field_lengths<K, W + 1, PITCH>(FM, len);
  }
}

}  // namespace nw
