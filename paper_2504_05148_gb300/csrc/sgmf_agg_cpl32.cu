// sgmf_agg_cpl32.cu -- aggregation kernels with 32 disparity cells per lane (Dp = 256).
#include "sgmf_sweep.cuh"

SGMF_AGG_INSTANTIATE(32)
