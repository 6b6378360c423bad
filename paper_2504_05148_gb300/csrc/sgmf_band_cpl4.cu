// sgmf_band_cpl4.cu -- banded aggregation kernels with 4 band cells per lane (bands of 64).
#include "sgmf_band_sweep.cuh"

SGMF_BAND_INSTANTIATE(4)
