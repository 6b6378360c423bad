// sgmf_wta.cuh -- path sum S, winner d* (Eq. 3), the right view's d' and the
// three-view check (Eq. 6) from vectors of path costs in memory.
//
// Behind the line walks every direction's path costs lie in memory and nothing
// is left to walk: a CTA takes one image row, each of its 8-lane groups a
// segment of it, so that a call of few frames fills the GPU.  The kernel is
// bound by reading the vectors (8 bytes a cell with eight directions' byte
// vectors), which its lanes copy ahead into their places of a shared-memory
// ring (cp.async).  Measured on 1242 x 375, D = 128: 113 us for one frame,
// 605 us for 8 (6.3 TB/s), check included, where the row walk that formed S on
// the way and the check kernel took 371 and 985 us.
//
// d' is a systolic running min inside a segment: the best key S << 8 | d of
// right pixel x' = x - d moves one disparity slot per step; the slot that
// leaves, and at the segment's end the slots left, are min-merged into the
// row's d' keys in shared memory.  On the bands the slots are band positions
// (slot s: right pixel x - lo - s) and all leave where the band start changes;
// segments are whole band tiles, so that this is every eighth step for the four
// groups of a warp together.  Then the row's check: every pixel's stereo term
// from those keys, and the LiDAR term, gathered over the row, for the pixels it
// decides.
#pragma once

#include "sgmf_check.cuh"
#include "sgmf_lanes.cuh"

namespace sgmf {
namespace oct {

constexpr int kMaxWtaVec = 7;

struct WtaArgs {
  KParams k;
  Buffers b;                    // frame 0's maps (d*, d', d-sub, row ORs, gate)
  const uint8_t *vec[kMaxWtaVec];   // frame 0's vectors, 2 Dp bytes per pixel
  size_t vec_frame[kMaxWtaVec];     // bytes from one frame to the next
  const uint8_t *cost;          // HALF: frame 0's cost volume
  StepConsts sc;                // HALF
  uint16_t *dbg_sum;            // frame 0's S (u16 vectors), or null
  int16_t *out;
};

// NP: pairs of byte vectors side by side; NS: u16 vectors (after the pairs);
// HALF: the cost bytes too (after the vectors)
template <int CPL, int NP, int NS, bool HALF>
struct WtaCfg {
  static constexpr int Dp = kGL * CPL, k8 = 32 * CPL, NV = NP + NS, kSlot = (2 * NV + (HALF ? 1 : 0)) * k8;
  // slots: one step each, about 16 KB a warp (at least 2; HALF, which computes
  // more per step and needs the warps: about 12 KB)
  static constexpr int R = HALF ? (kSlot * 4 <= 12288 ? 4 : (kSlot * 3 <= 16384 ? 3 : 2))
                                : (kSlot * 8 <= 16384 ? 8 : (kSlot * 4 <= 16384 ? 4 : 2));
  // at most 8 warps a CTA, and what the shared memory of the widest row leaves
  static constexpr int kFit = (226 * 1024 - kMaxDim * 8) / (R * kSlot), kMaxWarps = kFit < 8 ? kFit : 8;
  static_assert(kMaxWarps >= 1, "a warp's ring fits beside the widest row");
  // segments of about 80 pixels; HALF: two CTAs a SM at least
  static int warps(int W) {
    int n = max(1, min(kMaxWarps, (W + 319) / 320));
    if (HALF) n = max(1, min(n, (112 * 1024 - W * 8) / (R * kSlot)));
    return n;
  }
  // the rings, the row's d' keys (u32), d* and the list of undecided pixels (u16)
  static int smem(int W) { return warps(W) * R * kSlot + (W + 3) / 4 * 4 * 8; }
};

// HALF: the walks left the vectors of odd rows (rows family: of odd columns)
// out.  A direction's vector there is one step of Eq. 2 from its predecessor,
// which lies in an even row (column) and was stored.  At D = 128 the kernel then
// executes 565 instructions per 512 cells instead of 173 and is ALU-bound (78 %
// of the pipe): 8 frames of 1242 x 375 605 -> 760 us, the walks 1185 -> 857.
template <int CPL, int NP, int NS, bool BANDED, bool HALF>
__global__ void __launch_bounds__(256) k_wta(const __grid_constant__ WtaArgs a) {
  using CF = WtaCfg<CPL, NP, NS, HALF>;
  static_assert(!HALF || (NS == 0 && !BANDED), "HALF: byte vectors of the full range");
  constexpr int NW = CPL / 2, Dp = CF::Dp, R = CF::R, NV = CF::NV;
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
    int seg = (W + kGW * nwarp - 1) / (kGW * nwarp);
    if constexpr (BANDED) seg = (seg + kBandTile - 1) / kBandTile * kBandTile;
    if constexpr (HALF) seg = (seg + 1) / 2 * 2;     // segments start at even columns
    const int gi = warp * kGW + grp;
    const int x0 = min(gi * seg, W), x1 = min(x0 + seg, W);
    uint8_t *ring = smem + warp * R * CF::kSlot;
    const uint32_t ring_s = smem_u32(ring);
    const uint8_t *pv[NV];
    [[maybe_unused]] const uint8_t *pc = nullptr;
    [[maybe_unused]] const bool odd_row = HALF && (y & 1);
#pragma unroll
    for (int j = 0; j < NV; ++j)
      pv[j] = a.vec[j] + f * a.vec_frame[j] + (row + (HALF ? 0 : min(x0, W - 1))) * 2 * Dp +
              lig * (j < NP ? Vec8<CPL>::kLane : Vec16<CPL>::kLane);
    if constexpr (HALF) pc = a.cost + f * frame_cells(a.k) + row * Dp + lig * Vec8<CPL>::kLane;
    // step t's copies into a slot.  A group past its segment's end copies the
    // segment's last pixel again (HALF: goes on, to the row's last)
    auto copy = [&](uint32_t slot, int t) {
      if constexpr (HALF) {
        const int x = min(x0 + t, W - 1);
        copy8<CPL>(slot + 2 * NP * CF::k8, lane, pc + (size_t)x * Dp);
        // the rows' vectors of an even column, or right -> left the next column's
        if (!(t & 1)) copy8<CPL>(slot, lane, pv[0] + (size_t)x * (2 * Dp));
        copy8<CPL>(slot + CF::k8, lane, pv[0] + (size_t)(t & 1 ? min(x + 1, W - 1) : x) * (2 * Dp) + Dp);
        // where the predecessors lie: the row above (the down directions) and
        // below (the up ones; clamped at the last row, the vector is then not used)
        const int xm = max(x - 1, 0), xp = min(x + 1, W - 1);
        const ptrdiff_t up_row = odd_row ? -(ptrdiff_t)W : 0, down_row = odd_row && y + 1 < a.k.H ? W : up_row;
#pragma unroll
        for (int j = 1; j < NP; ++j) {
          const int xd = !odd_row || j == 1 ? x : (j == 2 ? xm : xp), xu = !odd_row || j == 1 ? x : (j == 2 ? xp : xm);
          copy8<CPL>(slot + 2 * j * CF::k8, lane, pv[j] + (up_row + xd) * (2 * Dp));
          copy8<CPL>(slot + (2 * j + 1) * CF::k8, lane, pv[j] + (down_row + xu) * (2 * Dp) + Dp);
        }
      } else {
#pragma unroll
        for (int j = 0; j < NV; ++j) {
          const uint32_t d = slot + 2 * j * CF::k8;
          if (j < NP) {
            copy8<CPL>(d, lane, pv[j]);
            copy8<CPL>(d + CF::k8, lane, pv[j] + Dp);
          } else {
            copy16<CPL>(d, lane, pv[j]);
          }
          if (x0 + t + 1 < x1) pv[j] += 2 * Dp;
        }
      }
    };
    for (int t = 0; t < R; ++t) {
      copy(ring_s + t * CF::kSlot, t);
      cp_commit();
    }
    [[maybe_unused]] uint32_t z[CPL / 4] = {};
    [[maybe_unused]] Raw8<CPL> right = {};       // HALF: the left -> right vector of the even column before
    [[maybe_unused]] const Edges none = no_neighbours(lig);
    if constexpr (HALF) pad_bytes<CPL>(D, lig, z);
    uint32_t kb[NW];                             // the keys' low bytes (d) and the padding's high ones
    [[maybe_unused]] const int16_t *lo_row = nullptr;
    [[maybe_unused]] int lo = 0;                 // the band start of the tile
    if constexpr (BANDED) {
      lo_row = b.band_lo + (y >> kBandTileLog) * a.k.tw;
    } else {
#pragma unroll
      for (int i = 0; i < NW; ++i) {
        const int d0 = lig * CPL + i, d1 = d0 + NW;
        kb[i] = (uint32_t)(d0 & 0xff) | ((uint32_t)(d1 & 0xff) << 8) | (d0 >= D ? 0xff0000u : 0u) |
                (d1 >= D ? 0xff000000u : 0u);
      }
    }
    const int end_lane = BANDED ? kGL - 1 : (D - 1) / CPL, end_cell = BANDED ? CPL - 1 : (D - 1) % CPL;
    uint8_t *dbg = (f == 0 && a.dbg_sum != nullptr)
                       ? reinterpret_cast<uint8_t *>(a.dbg_sum) + row * Dp * 2 + lig * Vec16<CPL>::kLane
                       : nullptr;
    uint32_t acc[CPL];
#pragma unroll
    for (int j = 0; j < CPL; ++j) acc[j] = 0xffffffffu;
    const uint32_t z0[CPL / 4] = {};
    // every slot of the accumulator to the row's keys; x: the pixel they were last updated at
    auto flush = [&](int x) {
#pragma unroll
      for (int j = 0; j < CPL; ++j) {
        const int xr = x - lo - (lig * CPL + j);
        if ((BANDED ? acc[j] != 0xffffffffu : lig * CPL + j < D) && xr >= 0) atomicMin(&merge[xr], acc[j]);
      }
    };
    int base = 0;
    for (int t = 0; t < seg; ++t) {
      const int x = x0 + t;
      const bool act = x < x1;
      if constexpr (BANDED) {
        if (t % kBandTile == 0) {
          const int now = lo_row[min(x, W - 1) >> kBandTileLog];
          if (t == 0 || now != lo) {
            if (t > 0 && act) flush(x - 1);      // (a group past its end was flushed there)
#pragma unroll
            for (int j = 0; j < CPL; ++j) acc[j] = 0xffffffffu;
            lo = now;
            const uint32_t b0 = (uint32_t)(lo + lig * CPL);
#pragma unroll
            for (int i = 0; i < NW; ++i) kb[i] = (b0 + i) | ((b0 + i + NW) << 8);
          }
          __syncwarp();
        }
      }
      uint32_t Sm[NW];
      if constexpr (HALF) {
        cp_wait<R - 1>();
        const uint8_t *v = ring + base;
        uint32_t C[NW], A[NW], B[NW];
        slot8<CPL>(v + 2 * NP * CF::k8, lane, z, C);
        // A and B: two predecessors' vectors -> their directions' vectors here
        auto step2 = [&]() {
          uint32_t ma, mb;
          group_min2<NW>(A, B, ma, mb);
          step<NW>(A, C, ma, a.sc, none);
          step<NW>(B, C, mb, a.sc, none);
        };
        if (!(t & 1)) {
          slot_raw8<CPL>(v, lane, right);
          expand8<CPL>(right, z0, A);
          slot8<CPL>(v + CF::k8, lane, z0, B);
        } else {
          Raw8<CPL> left;
          slot_raw8<CPL>(v + CF::k8, lane, left);
          if (x + 1 >= W) left = {};             // the path right -> left starts here
          expand8<CPL>(right, z, A);
          expand8<CPL>(left, z, B);
          step2();
        }
#pragma unroll
        for (int w = 0; w < NW; ++w) Sm[w] = A[w] + B[w];
        if (!odd_row) {
#pragma unroll
          for (int j = 1; j < NP; ++j) {
            slot8<CPL>(v + 2 * j * CF::k8, lane, z0, A);
            slot8<CPL>(v + (2 * j + 1) * CF::k8, lane, z0, B);
#pragma unroll
            for (int w = 0; w < NW; ++w) Sm[w] += A[w] + B[w];
          }
        } else {
          const bool last = y + 1 >= a.k.H;
#pragma unroll
          for (int j = 1; j < NP; ++j) {
            Raw8<CPL> dn, up;
            slot_raw8<CPL>(v + 2 * j * CF::k8, lane, dn);
            slot_raw8<CPL>(v + (2 * j + 1) * CF::k8, lane, up);
            // paths that start here: the predecessor lies outside the image
            if (j == 2 ? x == 0 : (j == 3 && x == W - 1)) dn = {};
            if (last || (j == 2 ? x == W - 1 : (j == 3 && x == 0))) up = {};
            expand8<CPL>(dn, z, A);
            expand8<CPL>(up, z, B);
            step2();
#pragma unroll
            for (int w = 0; w < NW; ++w) Sm[w] += A[w] + B[w];
          }
        }
      } else {
        cp_wait<R - 1>();
#pragma unroll
        for (int j = 0; j < NV; ++j) {
          const uint8_t *v = ring + base + 2 * j * CF::k8;
          uint32_t T[NW];
          if (j < NP) {
            uint32_t U[NW];
            slot8<CPL>(v, lane, z0, T);
            slot8<CPL>(v + CF::k8, lane, z0, U);
#pragma unroll
            for (int i = 0; i < NW; ++i) Sm[i] = j == 0 ? T[i] + U[i] : Sm[i] + T[i] + U[i];
          } else {
            slot16<CPL>(v, lane, T);
#pragma unroll
            for (int i = 0; i < NW; ++i) Sm[i] = j == 0 ? T[i] : Sm[i] + T[i];
          }
        }
      }
      copy(ring_s + base, t + R);
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
      if (!BANDED && a.k.subpixel) {
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
        const int xr = x - lo - (BANDED ? Dp - 1 : D - 1);   // the last slot leaves
        if (lig == end_lane && xr >= 0) {
          uint32_t v = acc[CPL - 1];
          if (!BANDED && end_cell != CPL - 1) {
#pragma unroll
            for (int j = 0; j < CPL - 1; ++j)
              if (j == end_cell) v = acc[j];
          }
          atomicMin(&merge[xr], v);
        }
      } else if (act) {
        flush(x);                                // the segment's last pixel: every slot leaves
      }
    }
    cp_wait<0>();
  }
  __syncthreads();
  // the row's d' and the stereo term; the pixels left to the LiDAR term are listed
  for (int x = threadIdx.x; x < W; x += blockDim.x) {
    const int ds = ds_s[x], xm = x - ds;
    // (on the bands a right pixel whose diagonal meets no band has none: -1,
    // and the stereo term fails)
    b.dprime[row + x] = BANDED && merge[x] == 0xffffffffu ? (int16_t)-1 : (int16_t)(merge[x] & 0xffu);
    bool stereo = false;
    if (xm >= 0) {
      const uint32_t m = merge[xm];
      stereo = (!BANDED || m != 0xffffffffu) && abs(ds - (int)(m & 0xffu)) <= a.k.lr;
    }
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

template <int CPL, int NP, int NS, bool BANDED, bool HALF = false>
static cudaError_t launch_wta_v(const WtaArgs &a, int nf, cudaStream_t s) {
  using CF = WtaCfg<CPL, NP, NS, HALF>;
  static bool done[64] = {};
  const int most = CF::kMaxWarps * CF::R * CF::kSlot + kMaxDim * 8;
  cudaError_t e = smem_optin(k_wta<CPL, NP, NS, BANDED, HALF>, most, done);
  if (e != cudaSuccess) return e;
  k_wta<CPL, NP, NS, BANDED, HALF><<<dim3(a.k.H, nf), 32 * CF::warps(a.k.W), CF::smem(a.k.W), s>>>(a);
  return cudaGetLastError();
}

template <int CPL, bool S8, bool BANDED>
static cudaError_t launch_wta_b(const KParams &k, const Buffers &b, int nf, int16_t *out, cudaStream_t s) {
  WtaArgs a = {};
  a.k = k;
  a.b = b;
  a.cost = b.cost;
  a.sc = step_consts(k);
  a.dbg_sum = b.dbg_sum;
  a.out = out;
  int n = 0;
  auto add = [&](const uint8_t *v, size_t frame) {
    a.vec[n] = v;
    a.vec_frame[n++] = frame;
  };
  const int nfam = k.num_paths == 8 ? 3 : 1;
  uint8_t *v[2];
  size_t frame[2];
  family_vectors(k, b, S8, 3, v, frame);
  add(v[0], frame[0]);                           // the rows: a pair of byte vectors, or their u16 sum
  if constexpr (S8 && !BANDED)
    if (k.rows_lines) {                          // the other directions: the sweep's two u16 sums
      for (int i = 0; i < 2; ++i) add(reinterpret_cast<const uint8_t *>(b.part[i]), 2 * frame_cells(k));
      return launch_wta_v<CPL, 1, 2, BANDED>(a, nf, s);
    }
  for (int i = 0; i < nfam; ++i) {
    family_vectors(k, b, S8, i, v, frame);
    add(v[0], frame[0]);
    if (!S8) add(v[1], frame[1]);
  }
  if constexpr (S8 && !BANDED && (CPL == 16 || CPL == 24))
    if (k.half)
      return nfam == 3 ? launch_wta_v<CPL, 4, 0, BANDED, true>(a, nf, s) : launch_wta_v<CPL, 2, 0, BANDED, true>(a, nf, s);
  if constexpr (S8)
    return nfam == 3 ? launch_wta_v<CPL, 4, 0, BANDED>(a, nf, s) : launch_wta_v<CPL, 2, 0, BANDED>(a, nf, s);
  else
    return nfam == 3 ? launch_wta_v<CPL, 0, 7, BANDED>(a, nf, s) : launch_wta_v<CPL, 0, 3, BANDED>(a, nf, s);
}

template <int CPL, bool S8>
cudaError_t launch_wta_t(const KParams &k, const Buffers &b, int nf, int16_t *out, cudaStream_t s) {
  if constexpr (CPL <= 16)
    if (k.band) return launch_wta_b<CPL, S8, true>(k, b, nf, out, s);
  return launch_wta_b<CPL, S8, false>(k, b, nf, out, s);
}

}  // namespace oct
}  // namespace sgmf
