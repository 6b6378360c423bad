// sgmf_aggregate.cu -- picks the aggregation kernels for a context's lane
// width and path-cost width: the full-range kernels (sgmf_lines.cuh,
// sgmf_rows.cuh, sgmf_sweep.cuh: 8-lane groups, Dp = 8 CPL) and the banded
// ones (sgmf_band_agg.cuh, sgmf_band_sweep.cuh: 16-lane groups, Dp = 16 CPL).
// Each lane width is instantiated in its own translation unit.
#include <cstdint>

#include "sgmf_internal.cuh"

namespace sgmf {

#define SGMF_AGG_DECLARE                                                                    \
  template <int CPL, bool S8>                                                              \
  cudaError_t launch_lines_t(const KParams &k, const Buffers &b, int nf, cudaStream_t s);  \
  template <int CPL, bool S8>                                                              \
  cudaError_t launch_rows_t(const KParams &k, const Buffers &b, int nf, cudaStream_t s);   \
  template <int CPL>                                                                       \
  cudaError_t launch_sweep_t(const KParams &k, const Buffers &b, int nf, cudaStream_t s);  \
  template <int CPL>                                                                       \
  int sweep_plan_t(const KParams &k, int nb, int *slots);

SGMF_AGG_DECLARE
namespace oct {
SGMF_AGG_DECLARE
template <int CPL>
cudaError_t launch_wta_t(const KParams &k, const Buffers &b, int nf, int16_t *out, cudaStream_t s);
}
#undef SGMF_AGG_DECLARE

// FN<CPL, S8> of the context's lane width
#define SGMF_DISPATCH(FN, ...)                                       \
  switch ((k.band ? 100 : 0) + k.DPL * 2 + (spill8 ? 1 : 0)) {       \
    case 4: return oct::FN<8, false>(__VA_ARGS__);                   \
    case 5: return oct::FN<8, true>(__VA_ARGS__);                    \
    case 8: return oct::FN<16, false>(__VA_ARGS__);                  \
    case 9: return oct::FN<16, true>(__VA_ARGS__);                   \
    case 12: return oct::FN<24, false>(__VA_ARGS__);                 \
    case 13: return oct::FN<24, true>(__VA_ARGS__);                  \
    case 16: return oct::FN<32, false>(__VA_ARGS__);                 \
    case 17: return oct::FN<32, true>(__VA_ARGS__);                  \
    case 104: return FN<4, false>(__VA_ARGS__);                      \
    case 105: return FN<4, true>(__VA_ARGS__);                       \
    case 108: return FN<8, false>(__VA_ARGS__);                      \
    case 109: return FN<8, true>(__VA_ARGS__);                       \
    default: return cudaErrorInvalidValue;                           \
  }
// FN<CPL>
#define SGMF_DISPATCH_W(FN, ERR, ...)                                \
  switch ((k.band ? 100 : 0) + k.DPL) {                              \
    case 2: return oct::FN<8>(__VA_ARGS__);                          \
    case 4: return oct::FN<16>(__VA_ARGS__);                         \
    case 6: return oct::FN<24>(__VA_ARGS__);                         \
    case 8: return oct::FN<32>(__VA_ARGS__);                         \
    case 102: return FN<4>(__VA_ARGS__);                             \
    case 104: return FN<8>(__VA_ARGS__);                             \
    default: return ERR;                                             \
  }

cudaError_t launch_agg_lines(const KParams &k, const Buffers &b, int nf, bool spill8, cudaStream_t s) {
  SGMF_DISPATCH(launch_lines_t, k, b, nf, s)
}

cudaError_t launch_agg_rows(const KParams &k, const Buffers &b, int nf, bool spill8, cudaStream_t s) {
  SGMF_DISPATCH(launch_rows_t, k, b, nf, s)
}

cudaError_t launch_agg_sweep(const KParams &k, const Buffers &b, int nf, cudaStream_t s) {
  SGMF_DISPATCH_W(launch_sweep_t, cudaErrorInvalidValue, k, b, nf, s)
}

cudaError_t launch_agg_wta(const KParams &k, const Buffers &b, int nf, int16_t *out, cudaStream_t s) {
  switch (k.band ? 0 : k.DPL) {
    case 2: return oct::launch_wta_t<8>(k, b, nf, out, s);
    case 4: return oct::launch_wta_t<16>(k, b, nf, out, s);
    case 6: return oct::launch_wta_t<24>(k, b, nf, out, s);
    case 8: return oct::launch_wta_t<32>(k, b, nf, out, s);
    default: return cudaErrorInvalidValue;
  }
}

int agg_sweep_plan(const KParams &k, int nb, int *slots) { SGMF_DISPATCH_W(sweep_plan_t, 0, k, nb, slots) }

}  // namespace sgmf
