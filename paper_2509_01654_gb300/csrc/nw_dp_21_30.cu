// DPX alignment kernels for the longer word lengths 21 to 30.
#define NW_DP_RANGE 2
#include "nw_dp_inst.inc"
