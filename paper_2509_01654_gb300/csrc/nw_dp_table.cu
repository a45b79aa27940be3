// Maps a length LB, and reduced steps (m, x), to their alignment kernels across
// the instantiation units.
#include "nw_launch.h"

namespace nw {
const void* dp_kernel_range_0(int LB, int epi, bool tab);
const void* dp_kernel_range_11(int LB, int epi, bool tab);
const void* dp_kernel_range_21(int LB, int epi, bool tab);
const void* dp_kernel_range_31(int LB, int epi, bool tab);

const void* dp_kernel(int LB, int epi, bool tab) {
  if (LB < 0 || LB > kMaxLen) return nullptr;
  if (LB <= 10) return dp_kernel_range_0(LB, epi, tab);
  if (LB <= 20) return dp_kernel_range_11(LB, epi, tab);
  if (LB <= 30) return dp_kernel_range_21(LB, epi, tab);
  return dp_kernel_range_31(LB, epi, tab);
}

#define NW_BIT_ALL(F) F(1, 0) F(2, 1) F(3, 1) F(3, 2) F(4, 1) F(4, 3) F(5, 1) F(5, 2) F(5, 3) F(5, 4)
#define NW_BIT_DECL(m, x) const void* bit_kernel_##m##_##x(int epi);
NW_BIT_ALL(NW_BIT_DECL)

const void* bit_kernel(int m, int x, int epi) {
#define NW_BIT_CASE(a, b) \
  if (m == a && x == b) return bit_kernel_##a##_##b(epi);
  NW_BIT_ALL(NW_BIT_CASE)
  return nullptr;
}
}  // namespace nw
