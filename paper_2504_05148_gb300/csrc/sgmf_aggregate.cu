// sgmf_aggregate.cu -- picks the aggregation kernels (sgmf_lines.cuh,
// sgmf_wta.cuh, sgmf_rows.cuh, sgmf_sweep.cuh) for a context's lane width
// (Dp = 8 CPL cells a vector) and path-cost width.  Each lane width is
// instantiated in its own translation unit (sgmf_agg_cpl*.cu).
#include <cstdint>

#include "sgmf_internal.cuh"

namespace sgmf {
namespace oct {
template <int CPL, bool S8>
cudaError_t launch_lines_t(const KParams &k, const Buffers &b, int nf, cudaStream_t s);
template <int CPL, bool S8>
cudaError_t launch_rows_t(const KParams &k, const Buffers &b, int nf, cudaStream_t s);
template <int CPL, bool S8>
cudaError_t launch_wta_t(const KParams &k, const Buffers &b, int nf, int16_t *out, cudaStream_t s);
template <int CPL>
cudaError_t launch_sweep_t(const KParams &k, const Buffers &b, int nf, cudaStream_t s);
template <int CPL>
int sweep_plan_t(const KParams &k, int nb, int *slots);
}  // namespace oct

// FN<CPL, S8> of the context's lane width, Dp = 32 * DPL = 8 * CPL
#define SGMF_DISPATCH(FN, ...)                       \
  switch (k.DPL * 2 + (bytes ? 1 : 0)) {             \
    case 4: return oct::FN<8, false>(__VA_ARGS__);   \
    case 5: return oct::FN<8, true>(__VA_ARGS__);    \
    case 8: return oct::FN<16, false>(__VA_ARGS__);  \
    case 9: return oct::FN<16, true>(__VA_ARGS__);   \
    case 12: return oct::FN<24, false>(__VA_ARGS__); \
    case 13: return oct::FN<24, true>(__VA_ARGS__);  \
    case 16: return oct::FN<32, false>(__VA_ARGS__); \
    case 17: return oct::FN<32, true>(__VA_ARGS__);  \
    default: return cudaErrorInvalidValue;           \
  }
// FN<CPL>
#define SGMF_DISPATCH_W(FN, ERR, ...)                \
  switch (k.DPL) {                                   \
    case 2: return oct::FN<8>(__VA_ARGS__);          \
    case 4: return oct::FN<16>(__VA_ARGS__);         \
    case 6: return oct::FN<24>(__VA_ARGS__);         \
    case 8: return oct::FN<32>(__VA_ARGS__);         \
    default: return ERR;                             \
  }

cudaError_t launch_agg_lines(const KParams &k, const Buffers &b, int nf, bool bytes, cudaStream_t s) {
  SGMF_DISPATCH(launch_lines_t, k, b, nf, s)
}

cudaError_t launch_agg_rows(const KParams &k, const Buffers &b, int nf, bool bytes, cudaStream_t s) {
  SGMF_DISPATCH(launch_rows_t, k, b, nf, s)
}

cudaError_t launch_agg_wta(const KParams &k, const Buffers &b, int nf, bool bytes, int16_t *out, cudaStream_t s) {
  SGMF_DISPATCH(launch_wta_t, k, b, nf, out, s)
}

cudaError_t launch_agg_sweep(const KParams &k, const Buffers &b, int nf, cudaStream_t s) {
  SGMF_DISPATCH_W(launch_sweep_t, cudaErrorInvalidValue, k, b, nf, s)
}

int agg_sweep_plan(const KParams &k, int nb, int *slots) { SGMF_DISPATCH_W(sweep_plan_t, 0, k, nb, slots) }

}  // namespace sgmf
