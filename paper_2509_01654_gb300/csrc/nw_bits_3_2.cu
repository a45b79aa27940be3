// Bit-parallel alignment kernels for the reduced steps match 3, mismatch 2.
#define NW_BIT_M 3
#define NW_BIT_X 2
#include "nw_bits_inst.inc"
