// Bit-parallel alignment kernels for the reduced steps match 3, mismatch 1.
#define NW_BIT_M 3
#define NW_BIT_X 1
#include "nw_bits_inst.inc"
