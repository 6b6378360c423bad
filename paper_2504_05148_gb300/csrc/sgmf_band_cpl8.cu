// sgmf_band_cpl8.cu -- banded aggregation kernels with 8 band cells per lane (bands of 128).
#include "sgmf_band_sweep.cuh"

SGMF_BAND_INSTANTIATE(8)
