// Bit-parallel alignment kernels for the reduced steps match 5, mismatch 4.
#define NW_BIT_M 5
#define NW_BIT_X 4
#include "nw_bits_inst.inc"
