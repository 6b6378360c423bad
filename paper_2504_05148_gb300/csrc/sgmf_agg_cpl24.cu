// sgmf_agg_cpl24.cu -- aggregation kernels with 24 disparity cells per lane (Dp = 192).
#include "sgmf_sweep.cuh"

SGMF_AGG_INSTANTIATE(24)
