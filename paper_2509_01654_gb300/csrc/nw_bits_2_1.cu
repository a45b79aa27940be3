// Bit-parallel alignment kernels for the reduced steps match 2, mismatch 1.
#define NW_BIT_M 2
#define NW_BIT_X 1
#include "nw_bits_inst.inc"
