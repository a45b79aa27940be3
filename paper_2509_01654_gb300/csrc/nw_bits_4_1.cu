// Bit-parallel alignment kernels for the reduced steps match 4, mismatch 1.
#define NW_BIT_M 4
#define NW_BIT_X 1
#include "nw_bits_inst.inc"
