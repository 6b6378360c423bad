// sgmf_check.cu -- three-view stereo-LiDAR consistency check, Eq. 6 (Sec. IV-C).
#include <cstdint>

#include "sgmf_check.cuh"

namespace sgmf {

__global__ void __launch_bounds__(256) k_consistency(KParams k, Buffers b0, int16_t *__restrict__ out) {
  const int x = blockIdx.x * 32 + (threadIdx.x & 31);
  const int y = blockIdx.y * 8 + (threadIdx.x >> 5);
  if (x >= k.W || y >= k.H) return;
  const Buffers b = frame_view(k, b0, blockIdx.z);
  if (gated_off(b.gate, k.gate_run)) return;
  out += (size_t)blockIdx.z * frame_px(k);
  const size_t p = (size_t)y * k.W + x;
  const int ds = b.dstar[p];
  bool stereo_ok = false, lidar_ok = false;
  if (k.consistency != 2 && k.consistency != 3) {
    const int xm = x - ds;
    // (d' is always valid for the plain method; the banded mode marks a right
    // pixel whose diagonal meets no band with -1, and the term then fails)
    const int dp = xm >= 0 ? (int)b.dprime[(size_t)y * k.W + xm] : -1;
    stereo_ok = dp >= 0 && abs(ds - dp) <= k.lr;
  }
  if (check_needs_lidar(k, stereo_ok)) lidar_ok = check_lidar_term(k, b, x, y, ds);
  check_store(k, b, out, p, ds, check_passes(k, stereo_ok, lidar_ok));
}

cudaError_t launch_consistency(const KParams &k, const Buffers &b, int nf, int16_t *out, cudaStream_t s) {
  dim3 grid((k.W + 31) / 32, (k.H + 7) / 8, nf);
  k_consistency<<<grid, 256, 0, s>>>(k, b, out);
  return cudaGetLastError();
}

}  // namespace sgmf
