// sgmf_wta.cuh -- path sum S, winner d* (Eq. 3), the right view's d' and the
// three-view check (Eq. 6) from the line walks' byte vectors.
//
// Where every direction's path costs lie in memory as byte vectors (line
// kernels, costs that fit a byte), nothing is left to walk: a CTA takes one
// image row, each of its 8-lane groups a segment of it, so that a call of few
// frames fills the GPU.  The kernel is bound by reading the vectors (8 bytes a
// cell with eight paths), which its lanes copy ahead into their places of a
// shared-memory ring (cp.async).  Measured on 1242 x 375, D = 128: 113 us for
// one frame, 605 us for 8 (6.3 TB/s), check included, where the row walk that
// formed S on the way and the check kernel took 371 and 985 us.
//
// d' is a systolic running min inside a segment: the best key S << 8 | d of
// right pixel x' = x - d moves one disparity slot per step; the slot that
// leaves, and at the segment's end the slots left, are min-merged into the
// row's d' keys in shared memory.  Then the row's check: every pixel's stereo
// term from those keys, and the LiDAR term, gathered over the row, for the
// pixels it decides.
#pragma once

#include "sgmf_check.cuh"
#include "sgmf_lanes.cuh"

namespace sgmf {
namespace oct {

struct WtaArgs {
  KParams k;
  Buffers b;                    // frame 0's maps (d*, d', d-sub, row ORs, gate)
  const uint8_t *vec[4];        // frame 0's vector pairs: two byte vectors, 2 Dp bytes per pixel
  size_t vec_frame[4];          // bytes from one frame to the next
  uint16_t *dbg_sum;            // frame 0's S (u16 vectors), or null
  int16_t *out;
};

// NP: vector pairs
template <int CPL, int NP>
struct WtaCfg {
  static constexpr int Dp = kGL * CPL, kVec = 32 * CPL, kSlot = 2 * NP * kVec;
  static constexpr int R = CPL == 8 ? 8 : (CPL == 16 ? 4 : 2);   // slots: one step each, about 16 KB a warp
  static constexpr int kMaxWarps = 8;
  static int warps(int W) { return max(1, min(kMaxWarps, (W + 319) / 320)); }   // segments of about 80 pixels
  // the rings, the row's d' keys (u32), d* and the list of undecided pixels (u16)
  static int smem(int W) { return warps(W) * R * kSlot + (W + 3) / 4 * 4 * 8; }
};

template <int CPL, int NP>
__global__ void __launch_bounds__(256) k_wta(const __grid_constant__ WtaArgs a) {
  using CF = WtaCfg<CPL, NP>;
  constexpr int NW = CPL / 2, Dp = CF::Dp, R = CF::R;
  extern __shared__ __align__(128) uint8_t smem[];
  __shared__ int n_list;
  const int f = blockIdx.y, y = blockIdx.x;
  if (gated_off(a.b.gate ? a.b.gate + f : nullptr, a.k.gate_run)) return;
  const int W = a.k.W, D = a.k.D;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, grp = lane / kGL, lig = lane % kGL;
  const int nwarp = blockDim.x >> 5, Wr = (W + 3) / 4 * 4;
  uint32_t *merge = reinterpret_cast<uint32_t *>(smem + nwarp * R * CF::kSlot);   // [Wr] key of each right pixel
  uint16_t *ds_s = reinterpret_cast<uint16_t *>(merge + Wr);                      // [Wr] d*
  uint16_t *list = ds_s + Wr;                                                     // [Wr]
  const Buffers b = frame_view(a.k, a.b, f);
  const size_t row = (size_t)y * W;
  for (int i = threadIdx.x; i < W; i += blockDim.x) merge[i] = 0xffffffffu;
  if (threadIdx.x == 0) n_list = 0;
  __syncthreads();
  {
    // the group's segment [x0, x1): equal lengths, the last ones may be short or empty
    const int seg = (W + kGW * nwarp - 1) / (kGW * nwarp), gi = warp * kGW + grp;
    const int x0 = min(gi * seg, W), x1 = min(x0 + seg, W);
    uint8_t *ring = smem + warp * R * CF::kSlot;
    const uint32_t ring_s = smem_u32(ring);
    const uint8_t *pv[NP];
#pragma unroll
    for (int j = 0; j < NP; ++j)
      pv[j] = a.vec[j] + f * a.vec_frame[j] + (row + min(x0, W - 1)) * 2 * Dp + lig * Vec8<CPL>::kLane;
    auto copy = [&](uint32_t slot, bool move) {
#pragma unroll
      for (int j = 0; j < NP; ++j) {
        copy8<CPL>(slot + 2 * j * CF::kVec, lane, pv[j]);
        copy8<CPL>(slot + (2 * j + 1) * CF::kVec, lane, pv[j] + Dp);
        if (move) pv[j] += 2 * Dp;
      }
    };
    // a group past its segment's end copies the segment's last pixel again
    for (int t = 0; t < R; ++t) {
      copy(ring_s + t * CF::kSlot, x0 + t + 1 < x1);
      cp_commit();
    }
    uint32_t kb[NW];
#pragma unroll
    for (int i = 0; i < NW; ++i) {
      const int d0 = lig * CPL + i, d1 = d0 + NW;
      kb[i] = (uint32_t)(d0 & 0xff) | ((uint32_t)(d1 & 0xff) << 8) | (d0 >= D ? 0xff0000u : 0u) |
              (d1 >= D ? 0xff000000u : 0u);
    }
    const int end_lane = (D - 1) / CPL, end_cell = (D - 1) % CPL;
    uint8_t *dbg = (f == 0 && a.dbg_sum != nullptr)
                       ? reinterpret_cast<uint8_t *>(a.dbg_sum) + row * Dp * 2 + lig * Vec16<CPL>::kLane
                       : nullptr;
    uint32_t acc[CPL];
#pragma unroll
    for (int j = 0; j < CPL; ++j) acc[j] = 0xffffffffu;
    const uint32_t z0[CPL / 4] = {};
    int base = 0;
    for (int t = 0; t < seg; ++t) {
      const int x = x0 + t;
      const bool act = x < x1;
      cp_wait<R - 1>();
      uint32_t Sm[NW];
#pragma unroll
      for (int w = 0; w < NW; ++w) Sm[w] = 0u;
#pragma unroll
      for (int j = 0; j < NP; ++j) {
        uint32_t T[NW], U[NW];
        slot8<CPL>(ring + base + 2 * j * CF::kVec, lane, z0, T);
        slot8<CPL>(ring + base + (2 * j + 1) * CF::kVec, lane, z0, U);
#pragma unroll
        for (int i = 0; i < NW; ++i) Sm[i] = j == 0 ? T[i] + U[i] : Sm[i] + T[i] + U[i];
      }
      copy(ring_s + base, x + R + 1 < x1);
      cp_commit();
      base = base + CF::kSlot == R * CF::kSlot ? 0 : base + CF::kSlot;
      if (dbg != nullptr && act) store_u16<CPL>(dbg + (size_t)x * Dp * 2, Sm);
      // keys S << 8 | d; padding keys have 0xff in the top byte
      uint32_t key[CPL];
#pragma unroll
      for (int i = 0; i < NW; ++i) {
        key[i] = prmt(Sm[i], kb[i], 0x6104);
        key[i + NW] = prmt(Sm[i], kb[i], 0x7325);
      }
      uint32_t best[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        best[j] = key[j];
#pragma unroll
        for (int i = j + 4; i < CPL; i += 4) best[j] = min(best[j], key[i]);
      }
      const uint32_t win = group_min_u32(min(min(best[0], best[1]), min(best[2], best[3])));
      const int ds = (int)(win & 0xffu);
      if (lig == 0 && act) {
        ds_s[x] = (uint16_t)ds;
        b.dstar[row + x] = (int16_t)ds;
      }
      if (a.k.subpixel) {
        // parabola through S(d*-1), S(d*), S(d*+1); the lanes holding the two
        // neighbours contribute them, every other lane the neutral 0xffffffff
        uint32_t sm = 0xffffffffu, sp = 0xffffffffu;
#pragma unroll
        for (int j = 0; j < CPL; ++j) {
          const int d = lig * CPL + j;
          sm = d + 1 == ds ? key[j] >> 8 : sm;
          sp = d == ds + 1 ? key[j] >> 8 : sp;
        }
        sm = group_min_u32(sm);
        sp = group_min_u32(sp);
        if (lig == 0 && act) b.dsub[row + x] = (int16_t)subpixel_disp(ds, D, sm, win >> 8, sp);
      }
      // right view: the keys move up a slot, then S(x, d) is folded in
      const uint32_t below = __shfl_up_sync(kAll, acc[CPL - 1], 1, kGL);
#pragma unroll
      for (int j = CPL - 1; j > 0; --j) acc[j] = min(acc[j - 1], key[j]);
      acc[0] = min(lig == 0 ? 0xffffffffu : below, key[0]);
      if (act && t + 1 < x1 - x0) {
        const int xr = x - (D - 1);              // slot D - 1 leaves
        if (lig == end_lane && xr >= 0) {
          uint32_t v = acc[CPL - 1];
          if (end_cell != CPL - 1) {
#pragma unroll
            for (int j = 0; j < CPL - 1; ++j)
              if (j == end_cell) v = acc[j];
          }
          atomicMin(&merge[xr], v);
        }
      } else if (act) {
        // the segment's last pixel: every slot leaves
#pragma unroll
        for (int j = 0; j < CPL; ++j) {
          const int d = lig * CPL + j;
          if (d < D && x >= d) atomicMin(&merge[x - d], acc[j]);
        }
      }
    }
    cp_wait<0>();
  }
  __syncthreads();
  // the row's d' and the stereo term; the pixels left to the LiDAR term are listed
  for (int x = threadIdx.x; x < W; x += blockDim.x) {
    const int ds = ds_s[x], xm = x - ds;
    b.dprime[row + x] = (int16_t)(merge[x] & 0xffu);
    const bool stereo = xm >= 0 && abs(ds - (int)(merge[xm] & 0xffu)) <= a.k.lr;
    if (check_needs_lidar(a.k, stereo))
      list[atomicAdd(&n_list, 1)] = (uint16_t)x;
    else
      check_store(a.k, b, a.out + f * frame_px(a.k), row + x, ds, check_passes(a.k, stereo, false));
  }
  __syncthreads();
  for (int i = threadIdx.x; i < n_list; i += blockDim.x) {
    const int x = list[i], ds = ds_s[x];
    check_store(a.k, b, a.out + f * frame_px(a.k), row + x, ds, check_lidar_term(a.k, b, x, y, ds));
  }
}

template <int CPL, int NP>
static cudaError_t launch_wta_v(const WtaArgs &a, int nf, cudaStream_t s) {
  using CF = WtaCfg<CPL, NP>;
  static bool done[64] = {};
  const int most = CF::kMaxWarps * CF::R * CF::kSlot + kMaxDim * 8;
  cudaError_t e = smem_optin(k_wta<CPL, NP>, most, done);
  if (e != cudaSuccess) return e;
  k_wta<CPL, NP><<<dim3(a.k.H, nf), 32 * CF::warps(a.k.W), CF::smem(a.k.W), s>>>(a);
  return cudaGetLastError();
}

template <int CPL>
cudaError_t launch_wta_t(const KParams &k, const Buffers &b, int nf, int16_t *out, cudaStream_t s) {
  WtaArgs a = {};
  a.k = k;
  a.b = b;
  a.dbg_sum = b.dbg_sum;
  a.out = out;
  const int nfam = k.num_paths == 8 ? 3 : 1;
  for (int i = 0; i <= nfam; ++i) {
    uint8_t *v[2];
    size_t frame[2];
    family_vectors(k, b, true, i == nfam ? 3 : i, v, frame);
    a.vec[i] = v[0];
    a.vec_frame[i] = frame[0];
  }
  return nfam == 3 ? launch_wta_v<CPL, 4>(a, nf, s) : launch_wta_v<CPL, 2>(a, nf, s);
}

}  // namespace oct
}  // namespace sgmf
