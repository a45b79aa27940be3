// Maps a range of lengths, and reduced steps (m, x), to their alignment kernels
// across the instantiation units.
#include "nw_launch.h"

namespace nw {
const void* dp_kernel_range_0(int epi, bool tab);
const void* dp_kernel_range_1(int epi, bool tab);
const void* dp_kernel_range_2(int epi, bool tab);
const void* dp_kernel_range_3(int epi, bool tab);

const void* dp_kernel(int range, int epi, bool tab) {
  switch (range) {
    case 0: return dp_kernel_range_0(epi, tab);
    case 1: return dp_kernel_range_1(epi, tab);
    case 2: return dp_kernel_range_2(epi, tab);
    case 3: return dp_kernel_range_3(epi, tab);
    default: return nullptr;
  }
}

#define NW_BIT_ALL(F) F(1, 0) F(2, 1) F(3, 1) F(3, 2) F(4, 1) F(4, 3) F(5, 1) F(5, 2) F(5, 3) F(5, 4)
#define NW_BIT_DECL(m, x)                      \
  const void* bit_kernel_##m##_##x(int epi);   \
  const void* bit_pairs_##m##_##x(bool wide);  \
  const void* bit_rescore_##m##_##x();
NW_BIT_ALL(NW_BIT_DECL)

const void* bit_kernel(int m, int x, int epi) {
#define NW_BIT_CASE(a, b) \
  if (m == a && x == b) return bit_kernel_##a##_##b(epi);
  NW_BIT_ALL(NW_BIT_CASE)
#undef NW_BIT_CASE
  return nullptr;
}
const void* bit_pairs(int m, int x, bool wide) {
#define NW_BIT_CASE(a, b) \
  if (m == a && x == b) return bit_pairs_##a##_##b(wide);
  NW_BIT_ALL(NW_BIT_CASE)
#undef NW_BIT_CASE
  return nullptr;
}
const void* bit_rescore(int m, int x) {
#define NW_BIT_CASE(a, b) \
  if (m == a && x == b) return bit_rescore_##a##_##b();
  NW_BIT_ALL(NW_BIT_CASE)
#undef NW_BIT_CASE
  return nullptr;
}
}  // namespace nw
