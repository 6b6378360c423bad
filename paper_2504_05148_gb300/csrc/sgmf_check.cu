// sgmf_check.cu -- three-view stereo-LiDAR consistency check, Eq. 6 (Sec. IV-C).
#include <cstdint>

#include "sgmf_check.cuh"

namespace sgmf {

// Tiles of 32 columns by 8 kRows rows.  First every pixel's stereo term; the
// pixels that the LiDAR term decides (a minority, scattered over the warps) go
// on a list in shared memory, which the block's threads then take densely, so
// that no warp walks a window's rows for a few of its lanes.  What bounds it is
// the latency of the window's loads.  12 frames of 640 x 480, D = 64: 65 -> 33 us
// against a thread that does both terms of its pixel.
constexpr int kRows = 4;

__global__ void __launch_bounds__(256) k_consistency(KParams k, Buffers b0, int16_t *__restrict__ out) {
  __shared__ uint32_t list[256 * kRows];   // ds << 16 | row in the tile << 8 | column in the tile
  __shared__ int n_list;
  const Buffers b = frame_view(k, b0, blockIdx.z);
  if (gated_off(b.gate, k.gate_run)) return;
  out += (size_t)blockIdx.z * frame_px(k);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int xb = blockIdx.x * 32, yb = blockIdx.y * (8 * kRows), x = xb + lane;
  if (threadIdx.x == 0) n_list = 0;
  __syncthreads();
  int ds[kRows];
#pragma unroll
  for (int j = 0; j < kRows; ++j) {
    const int y = yb + warp + 8 * j;
    ds[j] = x < k.W && y < k.H ? (int)b.dstar[(size_t)y * k.W + x] : 0;
  }
  // (d' is always valid for the plain method; the banded mode marks a right
  // pixel whose diagonal meets no band with -1, and the term then fails)
  int dp[kRows];
#pragma unroll
  for (int j = 0; j < kRows; ++j) {
    const int y = yb + warp + 8 * j, xm = x - ds[j];
    dp[j] = x < k.W && y < k.H && xm >= 0 && k.consistency != 2 && k.consistency != 3
                ? (int)b.dprime[(size_t)y * k.W + xm] : -1;
  }
#pragma unroll
  for (int j = 0; j < kRows; ++j) {
    const int y = yb + warp + 8 * j;
    const bool in = x < k.W && y < k.H;
    const bool stereo_ok = dp[j] >= 0 && abs(ds[j] - dp[j]) <= k.lr;
    const bool later = in && check_needs_lidar(k, stereo_ok);
    const uint32_t m = __ballot_sync(0xffffffffu, later);
    int base = 0;
    if (lane == 0 && m) base = atomicAdd(&n_list, __popc(m));
    base = __shfl_sync(0xffffffffu, base, 0);
    if (later)
      list[base + __popc(m & ((1u << lane) - 1u))] = (uint32_t)ds[j] << 16 | (uint32_t)(warp + 8 * j) << 8 | lane;
    else if (in)
      check_store(k, b, out, (size_t)y * k.W + x, ds[j], check_passes(k, stereo_ok, false));
  }
  __syncthreads();
  const int n = n_list;
  for (int i = threadIdx.x; i < n; i += 256) {
    const uint32_t e = list[i];
    const int d = (int)e >> 16, py = yb + (int)(e >> 8 & 255u), px = xb + (int)(e & 255u);
    check_store(k, b, out, (size_t)py * k.W + px, d, check_lidar_term(k, b, px, py, d));
  }
}

cudaError_t launch_consistency(const KParams &k, const Buffers &b, int nf, int16_t *out, cudaStream_t s) {
  dim3 grid((k.W + 31) / 32, (k.H + 8 * kRows - 1) / (8 * kRows), nf);
  k_consistency<<<grid, 256, 0, s>>>(k, b, out);
  return cudaGetLastError();
}

}  // namespace sgmf
