// sgmf_check.cuh -- the pieces of the three-view stereo-LiDAR consistency
// check, Eq. 6 (Sec. IV-C), for the kernels that run it.
//
// D^{c*}_p = d*_p when
//   the stereo term holds: q_m = (x - d*, y) is in the image and
//   |d*_p - d'(q_m)| <= lr, or
//   the LiDAR term holds: some valid raw d-bar_q, q in the (2rc+1)^2 window
//   K_p (clipped), has |d*_p - d-bar_q| <= tc -- i.e. the window's presence
//   masks have a bit in [d* - tc, d* + tc];
// otherwise -1.  The raw map d-bar is used, never d-hat.  `consistency`
// selects the Table V variants.  With the sub-pixel fit on, a kept pixel
// carries its sub-pixel disparity (1/16 px) instead of d*; the test itself
// is always on the integer d*.
#pragma once
#include <cstdint>

#include "sgmf_internal.cuh"

namespace sgmf {

// whether the LiDAR term decides the pixel
__device__ __forceinline__ bool check_needs_lidar(const KParams &k, bool stereo_ok) {
  return k.consistency == 2 || (k.consistency == 0 && !stereo_ok);
}

__device__ __forceinline__ bool check_passes(const KParams &k, bool stereo_ok, bool lidar_ok) {
  switch (k.consistency) {
    case 1: return stereo_ok;
    case 2: return lidar_ok;
    case 3: return true;
    default: return stereo_ok || lidar_ok;
  }
}

// The LiDAR term of pixel (x, y) with winner ds.  boxC holds the row ORs of
// the presence masks (|x' - x| <= rc); the 2 rc + 1 rows of the window are ORed
// here, for the small fraction of the pixels that need them.
__device__ __forceinline__ bool check_lidar_term(const KParams &k, const Buffers &b, int x, int y, int ds) {
  const int lo = max(ds - k.tc, 0), hi = min(ds + k.tc, k.D - 1);
  const size_t plane = (size_t)k.W * k.H;
  const int y0 = max(y - k.rc, 0), y1 = min(y + k.rc, k.H - 1);
  bool ok = false;
  for (int w = lo >> 5; w <= (hi >> 5) && !ok; ++w) {
    const int a = max(lo - 32 * w, 0), e = min(hi - 32 * w, 31);   // bit range [a, e] of word w
    const uint32_t upto = e == 31 ? 0xffffffffu : ((1u << (e + 1)) - 1u);
    const uint32_t rng = upto & ~((1u << a) - 1u);
    const uint32_t *col = b.boxC + w * plane + x;
    // the window's rows, eight loads in flight at a time
    for (int yy = y0; yy <= y1 && !ok; yy += 8) {
      uint32_t acc = 0u;
#pragma unroll
      for (int j = 0; j < 8; ++j)
        if (yy + j <= y1) acc |= col[(size_t)(yy + j) * k.W];
      ok = (acc & rng) != 0u;
    }
  }
  return ok;
}

// pixel p's output: d* (or its sub-pixel value) where the check passed
__device__ __forceinline__ void check_store(const KParams &k, const Buffers &b, int16_t *out, size_t p, int ds,
                                            bool ok) {
  const int16_t v = k.subpixel ? b.dsub[p] : (int16_t)ds;
  out[p] = ok ? v : (int16_t)-1;
}

}  // namespace sgmf
