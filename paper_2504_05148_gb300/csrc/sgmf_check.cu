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

// A thread per pixel that takes both terms, in tiles of 32 columns by 8 rows:
// where the list has nothing to gather or the call too few tiles of it
__global__ void __launch_bounds__(256) k_consistency_px(KParams k, Buffers b0, int16_t *__restrict__ out) {
  const int x = blockIdx.x * 32 + (threadIdx.x & 31), y = blockIdx.y * 8 + (threadIdx.x >> 5);
  if (x >= k.W || y >= k.H) return;
  const Buffers b = frame_view(k, b0, blockIdx.z);
  if (gated_off(b.gate, k.gate_run)) return;
  out += (size_t)blockIdx.z * frame_px(k);
  const size_t p = (size_t)y * k.W + x;
  const int ds = b.dstar[p], xm = x - ds;
  const int dp = xm >= 0 && k.consistency != 2 && k.consistency != 3 ? (int)b.dprime[(size_t)y * k.W + xm] : -1;
  const bool stereo_ok = dp >= 0 && abs(ds - dp) <= k.lr;
  const bool lidar_ok = check_needs_lidar(k, stereo_ok) && check_lidar_term(k, b, x, y, ds);
  check_store(k, b, out, p, ds, check_passes(k, stereo_ok, lidar_ok));
}

// The list costs a call its atomics, a barrier and a fourth of the CTAs: about 2
// us where a window of few rows leaves nothing to win them back (one frame of 640 x
// 480, r_c = 0 16.5 us a call by pixels, 18.7 with the list; r_c = 4 18.6, 20.7;
// r_c = 8 19.4, 19.6; r_c = 80 41.3, 35.8; 8 frames of 320 x 240, 4 tiles a SM, r_c = 0
// the kernel 10.2, 12.3, r_c = 6 16.4, 14.3), and where the LiDAR term alone
// decides, every pixel is on it: one frame of 640 x 480, r_c = 20 20.7 us by pixels,
// 24.8 with the list, 8 frames of 320 x 240 32.7, 28.6 for their shape.
static bool by_pixel(const KParams &k, long tiles) {
  const bool every = k.consistency == 2;           // every pixel is on the list
  if (every && k.rc == 0) return true;
  if (!every && (k.consistency != 0 || k.rc > 4)) return false;
  int sms = 0;
  return sm_count(&sms) == cudaSuccess && tiles < (k.rc <= 4 ? 5L : 4L) * sms;
}

cudaError_t launch_consistency(const KParams &k, const Buffers &b, int nf, int16_t *out, cudaStream_t s) {
  const dim3 grid((k.W + 31) / 32, (k.H + 8 * kRows - 1) / (8 * kRows), nf);
  if (by_pixel(k, (long)grid.x * grid.y * grid.z))
    k_consistency_px<<<dim3(grid.x, (k.H + 7) / 8, nf), 256, 0, s>>>(k, b, out);
  else
    k_consistency<<<grid, 256, 0, s>>>(k, b, out);
  return cudaGetLastError();
}

}  // namespace sgmf
