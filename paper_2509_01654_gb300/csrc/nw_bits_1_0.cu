// Bit-parallel alignment kernels for the reduced steps match 1, mismatch 0.
#define NW_BIT_M 1
#define NW_BIT_X 0
#include "nw_bits_inst.inc"
