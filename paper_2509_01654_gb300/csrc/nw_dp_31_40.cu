// DPX alignment kernels for the longer word lengths 31 to 40.
#define NW_DP_RANGE 3
#include "nw_dp_inst.inc"
