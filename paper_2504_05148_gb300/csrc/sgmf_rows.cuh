// sgmf_rows.cuh -- behind the sweep: the two horizontal directions of Eq. 2, the path sum S, the
// winner d* (Eq. 3) and the right view's d' (Sec. IV-C).
//
// A CTA takes four image rows: its first warp walks them left -> right
// (r = (1,0)), its second right -> left, one row per 8-lane group, so that
// each warp's code knows its direction.  Each warp spills its path costs for
// the half of the row it reaches first; on the other half it reads the other
// warp's spill, adds the vertical and diagonal vectors into S = sum_r L_r, and
// takes d* and d' there.  The two meet once, at a block barrier between the
// halves.
//
// d' is a systolic running min: the best key S << 8 | d of right pixel
// x' = x - d moves one disparity slot per step, so after D steps it has seen
// S(x' + d, d) for every d.  Right pixels whose diagonal crosses the middle
// get keys from both warps, merged in shared memory at the end.
//
// Inputs stream through a ring of shared-memory slots, one step each, filled
// by 8- and 16-byte asynchronous copies (cp.async): a lane copies the pieces it
// will read itself, so a slot needs no barrier, only the lane's own group
// count.  (One bulk copy per row and vector, five to eight a row and chunk of
// four steps, cost the issuing warp 0.3 us a chunk: the copies of a warp's
// lanes issue one after the other.)
#pragma once

#include "sgmf_lanes.cuh"

namespace sgmf {
namespace oct {

constexpr int kSums = 2;        // u16 vectors (the sweep's sums) read per pixel beside cost and spill

struct RowArgs {
  KParams k;
  const uint8_t *cost;
  const uint8_t *vec[kSums];  // frame 0's vertical / diagonal vectors, 2 Dp bytes per pixel
  size_t vec_frame[kSums];    // bytes from one frame to the next
  uint8_t *spill;               // frame 0's row spill region
  size_t spill_frame;
  int16_t *dstar, *dprime;
  int16_t *dsub;                // sub-pixel output (1/16 px), or null when the fit is off
  uint16_t *dbg_sum;            // frame 0's S (u16 vectors), or null
  StepConsts sc;
  const int *gate;              // per-frame gate words of the launch's frames, or null
};

// A slot holds, for the 32 lanes of a warp, the pieces of one step: cost bytes,
// spill, the sums.
template <int CPL, bool S8>
struct RowCfg {
  static constexpr int Dp = kGL * CPL, SB = S8 ? 1 : 2;
  static constexpr int k8 = 32 * CPL, k16 = 2 * k8;              // bytes of a byte / u16 vector of the four rows
  static constexpr int oSpill = k8, oVec = oSpill + (S8 ? k8 : k16), kSlot = oVec + kSums * k16;
  // slots: up to 8 steps (at least 2) in about 32 KB a warp
  static constexpr int R = 8 * kSlot <= 32768 ? 8 : (4 * kSlot <= 32768 ? 4 : 2);
  static constexpr int U = R < 4 ? R : 4;                        // steps unrolled
  static constexpr int kMerge = kGW * Dp * 4;                    // merge words of the four rows
  static constexpr int kSmem = 2 * R * kSlot + kMerge;
};

// what a lane carries along its row
template <int CPL>
struct RowWalk {
  uint32_t L[CPL / 2];
  uint32_t mm;
  uint32_t acc[CPL];            // right-view keys; slot d holds right pixel x - d
};

// the lane's constants of the walk
template <int CPL>
struct RowLane {
  int W, D, xm, lane, lig;
  bool act;                     // the group's row is inside the image
  size_t row;                   // its first pixel
  uint32_t z[CPL / 4], kb[CPL / 2];
  Edges edges;
  int end_lane, end_cell;       // where disparity D - 1 lies
  StepConsts sc;
  uint8_t *spill;               // the lane's first chunk of the row's spill
  uint8_t *dbg;                 // and of its S, or null
  int16_t *dstar, *dprime, *dsub;
  const uint8_t *cost, *vec[kSums];   // the lane's first chunk of the row's pixel 0
  uint32_t *merge;              // the row's merge words; word i: right pixel xm - D + 1 + i
};

template <int CPL, bool S8, bool FWD, bool SECOND>
__device__ __forceinline__ void row_step(RowWalk<CPL> &w, const RowLane<CPL> &g, const uint8_t *slot, int x) {
  using CF = RowCfg<CPL, S8>;
  constexpr int NW = CPL / 2, Dp = CF::Dp;
  const uint32_t z0[CPL / 4] = {};
  uint32_t C[NW];
  slot8<CPL>(slot, g.lane, g.z, C);
  step<NW>(w.L, C, w.mm, g.sc, g.edges);
  w.mm = group_min<NW>(w.L);
  if constexpr (!SECOND) {
    if (g.act) VecW<CPL, S8>::put(g.spill + (size_t)x * Dp * CF::SB, w.L);
  } else {
    uint32_t Sm[NW];
    if constexpr (S8)
      slot8<CPL>(slot + CF::oSpill, g.lane, z0, Sm);
    else
      slot16<CPL>(slot + CF::oSpill, g.lane, Sm);
#pragma unroll
    for (int i = 0; i < NW; ++i) Sm[i] += w.L[i];
#pragma unroll
    for (int j = 0; j < kSums; ++j) {
      const uint8_t *v = slot + CF::oVec + j * CF::k16;
      uint32_t T[NW];
      slot16<CPL>(v, g.lane, T);
#pragma unroll
      for (int i = 0; i < NW; ++i) Sm[i] += T[i];
    }
    if (g.dbg != nullptr && g.act) store_u16<CPL>(g.dbg + (size_t)x * Dp * 2, Sm);
    // keys S << 8 | d; padding keys have 0xff in the top byte
    uint32_t key[CPL];
#pragma unroll
    for (int i = 0; i < NW; ++i) {
      key[i] = prmt(Sm[i], g.kb[i], 0x6104);
      key[i + NW] = prmt(Sm[i], g.kb[i], 0x7325);
    }
    uint32_t best = key[0];
#pragma unroll
    for (int j = 1; j < CPL; ++j) best = min(best, key[j]);
    best = group_min_u32(best);
    if (g.lig == 0 && g.act) g.dstar[x] = (int16_t)(best & 0xffu);
    if (g.dsub != nullptr) {
      // parabola through S(d*-1), S(d*), S(d*+1); the lanes holding the two
      // neighbours contribute them, every other lane the neutral 0xffffffff
      const int ds = (int)(best & 0xffu);
      uint32_t sm = 0xffffffffu, sp = 0xffffffffu;
#pragma unroll
      for (int j = 0; j < CPL; ++j) {
        const int d = g.lig * CPL + j;
        sm = d + 1 == ds ? key[j] >> 8 : sm;
        sp = d == ds + 1 ? key[j] >> 8 : sp;
      }
      sm = group_min_u32(sm);
      sp = group_min_u32(sp);
      if (g.lig == 0 && g.act) g.dsub[x] = (int16_t)subpixel_disp(ds, g.D, sm, best >> 8, sp);
    }
    // right view: walking right the keys move up a slot per step, walking left
    // down a slot; then S(x, d) is folded in
    if constexpr (FWD) {
      uint32_t in = __shfl_up_sync(kAll, w.acc[CPL - 1], 1, kGL);
      if (g.lig == 0) in = 0xffffffffu;
#pragma unroll
      for (int j = CPL - 1; j > 0; --j) w.acc[j] = min(w.acc[j - 1], key[j]);
      w.acc[0] = min(in, key[0]);
      const int xr = x - (g.D - 1);              // slot D - 1 is complete on this half
      if (g.lig == g.end_lane && xr >= 0 && g.act) {
        uint32_t v = w.acc[CPL - 1];
        if (g.end_cell != CPL - 1) {
#pragma unroll
          for (int j = 0; j < CPL - 1; ++j)
            if (j == g.end_cell) v = w.acc[j];
        }
        if (xr >= g.xm)
          g.dprime[xr] = (int16_t)(v & 0xffu);
        else
          atomicMin(&g.merge[xr - (g.xm - g.D + 1)], v);
      }
    } else {
      uint32_t in = __shfl_down_sync(kAll, w.acc[0], 1, kGL);
      if (g.lig == kGL - 1) in = 0xffffffffu;
#pragma unroll
      for (int j = 0; j < CPL - 1; ++j) w.acc[j] = min(w.acc[j + 1], key[j]);
      w.acc[CPL - 1] = min(in, key[CPL - 1]);
      if (g.lig == 0 && g.act) {                 // slot 0: right pixel x
        if (x + g.D - 1 < g.xm)
          g.dprime[x] = (int16_t)(w.acc[0] & 0xffu);
        else
          atomicMin(&g.merge[x - (g.xm - g.D + 1)], w.acc[0]);
      }
    }
  }
}

// One half of a warp's walk over n pixels from x0 on: SECOND the pixels the
// other warp reached first.
template <int CPL, bool S8, bool FWD, bool SECOND>
__device__ __forceinline__ void row_half(RowWalk<CPL> &w, const RowLane<CPL> &g, uint8_t *ring, int x0, int n) {
  using CF = RowCfg<CPL, S8>;
  constexpr int R = CF::R, U = CF::U, Dp = CF::Dp, kMove = FWD ? 1 : -1;
  const uint32_t ring_s = smem_u32(ring);
  // sources of the next step to copy
  const uint8_t *pc = g.cost + (ptrdiff_t)x0 * Dp, *ps = g.spill + (ptrdiff_t)x0 * Dp * CF::SB;
  const uint8_t *pv[kSums];
#pragma unroll
  for (int j = 0; j < kSums; ++j) pv[j] = g.vec[j] + (ptrdiff_t)x0 * 2 * Dp;
  auto copy = [&](uint32_t slot) {
    copy8<CPL>(slot, g.lane, pc);
    pc += kMove * Dp;
    if constexpr (SECOND) {
      if constexpr (S8)
        copy8<CPL>(slot + CF::oSpill, g.lane, ps);
      else
        copy16<CPL>(slot + CF::oSpill, g.lane, ps);
      ps += kMove * Dp * CF::SB;
#pragma unroll
      for (int j = 0; j < kSums; ++j) {
        copy16<CPL>(slot + CF::oVec + j * CF::k16, g.lane, pv[j]);
        pv[j] += kMove * 2 * Dp;
      }
    }
  };
  for (int t = 0; t < R; ++t) {
    if (t < n) copy(ring_s + t * CF::kSlot);
    cp_commit();
  }
  int base = 0;                                  // the slot of step t
  for (int t = 0; t < n; t += U) {
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (t + u >= n) break;
      cp_wait<R - 1>();
      row_step<CPL, S8, FWD, SECOND>(w, g, ring + base + u * CF::kSlot, x0 + kMove * (t + u));
      if (t + u + R < n) copy(ring_s + base + u * CF::kSlot);
      cp_commit();
    }
    base = base + U * CF::kSlot == R * CF::kSlot ? 0 : base + U * CF::kSlot;
  }
  cp_wait<0>();
}

// One warp's walk of its four rows.
template <int CPL, bool S8, bool FWD>
__device__ __forceinline__ void row_walk(const RowLane<CPL> &g, uint8_t *ring) {
  RowWalk<CPL> w;
#pragma unroll
  for (int i = 0; i < CPL / 2; ++i) w.L[i] = 0u;   // the first step starts a path
  w.mm = 0u;
#pragma unroll
  for (int j = 0; j < CPL; ++j) w.acc[j] = 0xffffffffu;
  row_half<CPL, S8, FWD, false>(w, g, ring, FWD ? 0 : g.W - 1, FWD ? g.xm : g.W - g.xm);
  __syncthreads();                               // both first halves are stored
  row_half<CPL, S8, FWD, true>(w, g, ring, FWD ? g.xm : g.xm - 1, FWD ? g.W - g.xm : g.xm);
  if (FWD && g.act) {
    // right pixels x' = W-1-d whose diagonal leaves the image: the slots left
#pragma unroll
    for (int j = 0; j < CPL; ++j) {
      const int d = g.lig * CPL + j, xr = g.W - 1 - d;
      if (d < g.D - 1 && xr >= 0) {
        if (xr >= g.xm)
          g.dprime[xr] = (int16_t)(w.acc[j] & 0xffu);
        else
          atomicMin(&g.merge[xr - (g.xm - g.D + 1)], w.acc[j]);
      }
    }
  }
}

template <int CPL, bool S8>
__global__ void __launch_bounds__(64) k_rows(const __grid_constant__ RowArgs a) {
  using CF = RowCfg<CPL, S8>;
  constexpr int Dp = CF::Dp, NW = CPL / 2;
  extern __shared__ __align__(128) uint8_t smem[];
  const int f = blockIdx.y;
  if (gated_off(a.gate ? a.gate + f : nullptr, a.k.gate_run)) return;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, grp = lane / kGL, lig = lane % kGL;
  const int W = a.k.W, D = a.k.D, y0 = blockIdx.x * kGW, y = min(y0 + grp, a.k.H - 1);
  uint32_t *merge = reinterpret_cast<uint32_t *>(smem + 2 * CF::R * CF::kSlot);
  const size_t fpx = frame_px(a.k), fcells = frame_cells(a.k);
  RowLane<CPL> g;
  g.W = W;
  g.D = D;
  g.xm = W / 2;
  g.lane = lane;
  g.lig = lig;
  g.act = y0 + grp < a.k.H;
  g.row = (size_t)y * W;
  pad_bytes<CPL>(D, lig, g.z);
#pragma unroll
  for (int i = 0; i < NW; ++i) {
    const int d0 = lig * CPL + i, d1 = d0 + NW;
    g.kb[i] = (uint32_t)(d0 & 0xff) | ((uint32_t)(d1 & 0xff) << 8) | (d0 >= D ? 0xff0000u : 0u) |
              (d1 >= D ? 0xff000000u : 0u);
  }
  g.edges = no_neighbours(lig);
  g.end_lane = (D - 1) / CPL;
  g.end_cell = (D - 1) % CPL;
  g.sc = a.sc;
  g.cost = a.cost + f * fcells + g.row * Dp + lig * Vec8<CPL>::kLane;
  g.spill = a.spill + f * a.spill_frame + g.row * Dp * CF::SB + lig * VecW<CPL, S8>::kLane;
#pragma unroll
  for (int j = 0; j < kSums; ++j)
    g.vec[j] = a.vec[j] + f * a.vec_frame[j] + g.row * 2 * Dp + lig * Vec16<CPL>::kLane;
  g.dbg = (f == 0 && a.dbg_sum != nullptr)
              ? reinterpret_cast<uint8_t *>(a.dbg_sum) + g.row * Dp * 2 + lig * Vec16<CPL>::kLane
              : nullptr;
  g.dstar = a.dstar + f * fpx + g.row;
  g.dprime = a.dprime + f * fpx + g.row;
  g.dsub = a.dsub != nullptr ? a.dsub + f * fpx + g.row : nullptr;
  g.merge = merge + grp * Dp;
  for (int i = threadIdx.x; i < kGW * Dp; i += blockDim.x) merge[i] = 0xffffffffu;
  __syncthreads();
  if (warp == 0)
    row_walk<CPL, S8, true>(g, smem);
  else
    row_walk<CPL, S8, false>(g, smem + CF::R * CF::kSlot);
  __syncthreads();
  // right pixels whose diagonal crosses the middle: both warps contributed
  for (int r = warp; r < kGW && y0 + r < a.k.H; r += 2)
    for (int i = lane; i < D - 1; i += 32) {
      const int xr = g.xm - D + 1 + i;
      if (xr >= 0 && xr < g.xm)
        a.dprime[f * fpx + (size_t)(y0 + r) * W + xr] = (int16_t)(merge[r * Dp + i] & 0xffu);
    }
}

template <int CPL, bool S8>
static cudaError_t launch_rows_v(const RowArgs &a, int nf, cudaStream_t s) {
  using CF = RowCfg<CPL, S8>;
  static bool done[64] = {};
  cudaError_t e = smem_optin(k_rows<CPL, S8>, CF::kSmem, done);
  if (e != cudaSuccess) return e;
  k_rows<CPL, S8><<<dim3((a.k.H + kGW - 1) / kGW, nf), 64, CF::kSmem, s>>>(a);
  return cudaGetLastError();
}

template <int CPL, bool S8>
cudaError_t launch_rows_t(const KParams &k, const Buffers &b, int nf, cudaStream_t s) {
  RowArgs a = {};
  const size_t cells = frame_cells(k);
  a.k = k;
  a.cost = b.cost;
  a.spill = static_cast<uint8_t *>(b.spill) + 6 * cells;   // the fourth spill region
  a.spill_frame = 8 * cells;
  a.dstar = b.dstar;
  a.dprime = b.dprime;
  a.dsub = k.subpixel ? b.dsub : nullptr;
  a.dbg_sum = b.dbg_sum;
  a.sc = step_consts(k);
  a.gate = b.gate;
  for (int i = 0; i < kSums; ++i) {
    a.vec[i] = reinterpret_cast<const uint8_t *>(b.part[i]);
    a.vec_frame[i] = 2 * cells;
  }
  return launch_rows_v<CPL, S8>(a, nf, s);
}

}  // namespace oct
}  // namespace sgmf
