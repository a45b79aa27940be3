// Bit-parallel alignment kernels for the reduced steps match 4, mismatch 3.
#define NW_BIT_M 4
#define NW_BIT_X 3
#include "nw_bits_inst.inc"
