// DPX alignment kernels for the longer word lengths 11 to 20.
#define NW_DP_RANGE 1
#include "nw_dp_inst.inc"
