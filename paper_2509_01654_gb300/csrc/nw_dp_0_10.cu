// DPX alignment kernels for the longer word lengths 0 to 10.
#define NW_DP_RANGE 0
#include "nw_dp_inst.inc"
