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

constexpr int kMaxWtaVec = 8;   // two directions of four families

// a vector kept from one step to the next, as it was stored
template <int CPL, bool S8>
struct Prev {
  Raw8<CPL> r;
  __device__ __forceinline__ void load(const uint8_t *slot, int lane) { slot_raw8<CPL>(slot, lane, r); }
  __device__ __forceinline__ void words(const uint32_t (&z)[CPL / 4], uint32_t (&w)[CPL / 2]) const {
    expand8<CPL>(r, z, w);
  }
};
template <int CPL>
struct Prev<CPL, false> {
  uint32_t w[CPL / 2];
  __device__ __forceinline__ void load(const uint8_t *slot, int lane) { slot16<CPL>(slot, lane, w); }
  __device__ __forceinline__ void words(const uint32_t (&)[CPL / 4], uint32_t (&o)[CPL / 2]) const {
    copy_words<CPL / 2>(o, w);
  }
};

struct WtaArgs {
  KParams k;
  Buffers b;                    // frame 0's maps (d*, d', d-sub, row ORs, gate)
  const uint8_t *vec[kMaxWtaVec];   // frame 0's vectors, 2 Dp bytes per pixel
  size_t vec_frame[kMaxWtaVec];     // bytes from one frame to the next
  const uint8_t *cost;          // half-stored vectors: frame 0's cost volume
  StepConsts sc;                // half-stored vectors
  uint16_t *dbg_sum;            // frame 0's S (u16 vectors), or null
  int16_t *out;
};

// What a slot of the ring holds for one step: the two directions' vectors of
// the rows and of NF families, NS u16 sums, and the cost bytes where the rows'
// vectors are half stored (RH).  S8: vectors of bytes, else u16.
template <int CPL, bool S8, int NF, int NS, bool RH>
struct WtaCfg {
  static constexpr int Dp = kGL * CPL, k8 = 32 * CPL, kV = S8 ? k8 : 2 * k8, NP = NF + 1;
  static constexpr int oSum = 2 * NP * kV, oCost = oSum + NS * 2 * k8, kSlot = oCost + (RH ? k8 : 0);
  // slots: one step each, about 16 KB a warp (at least 2; RH, which computes
  // more per step and needs the warps: about 12 KB)
  static constexpr int R = RH ? (kSlot * 4 <= 12288 ? 4 : (kSlot * 3 <= 16384 ? 3 : 2))
                              : (kSlot * 8 <= 16384 ? 8 : (kSlot * 4 <= 16384 ? 4 : 2));
  // on the bands RH re-indexes vectors: a group's scratch (band_shift)
  static constexpr int kShift = kGW * kGL * CPL * 2;
  static constexpr int warp_bytes(bool banded) { return R * kSlot + (RH && banded ? kShift : 0); }
  static constexpr int kRoom = 226 * 1024;         // dynamic shared memory of a SM's CTAs
  static_assert(R * kSlot + kShift + kMaxDim * 8 <= kRoom, "a warp's ring fits beside the widest row");
  // at most 8 warps, segments of about 80 pixels.  RH: no more warps than two
  // CTAs a SM have room for (at 32 cells a lane about 200 registers: 2 warps a
  // scheduler), unless one alone holds more than those two (wide rows, whose d'
  // keys take the room, and large slots)
  static int warps(int W, bool banded) {
    auto fit = [&](int ctas) { return (kRoom / ctas - W * 8) / warp_bytes(banded); };
    const int n = max(1, min(min(8, fit(1)), (W + 319) / 320));
    const int two = RH ? max(1, min(min(n, CPL == 32 ? 4 : 8), fit(2))) : n;
    return n > 2 * two ? n : two;
  }
  // the rings, the row's d' keys (u32), d* and the list of undecided pixels (u16)
  static int smem(int W, bool banded) { return warps(W, banded) * warp_bytes(banded) + (W + 3) / 4 * 4 * 8; }
};

// Half-stored vectors.  RH, of the rows: the walks left those of odd columns
// out; FH, of the families: those of odd rows.  A direction's vector there is
// one step of Eq. 2 from its predecessor, which lies in an even column (row)
// and was stored; on the bands it is re-indexed first where it lies in another
// tile.  Bytes come with neither or with both.  At D = 128 the kernel with byte
// vectors then executes 593 instructions per 512 cells instead of 351 and is
// ALU-bound (79 % of the pipe): 8 frames of 1242 x 375 605 -> 760 us, the walks
// 1185 -> 857.  u16
// vectors come with RH at least: the rows' two directions then fit the region
// that one sum of both took, whose second walk had to wait for the first and read
// and write all of it (p2 = 300, 1242 x 375, D = 128: one frame 578 -> 439 us a call,
// 32 frames 12302 -> 9018; 1280 x 720 x 16, D = 192 21359 -> 16599).
template <int CPL, bool S8, int NF, int NS, bool BANDED, bool RH, bool FH>
__global__ void __launch_bounds__(256) k_wta(const __grid_constant__ WtaArgs a) {
  using CF = WtaCfg<CPL, S8, NF, NS, RH>;
  static_assert(RH || !FH, "half-stored families come with half-stored rows");
  static_assert(!BANDED || NS == 0, "no sweep on the bands");
  constexpr int NW = CPL / 2, Dp = CF::Dp, R = CF::R, NP = CF::NP, kV = CF::kV;
  extern __shared__ __align__(128) uint8_t smem[];
  __shared__ int n_list;
  const int f = blockIdx.y, y = blockIdx.x;
  if (gated_off(a.b.gate ? a.b.gate + f : nullptr, a.k.gate_run)) return;
  const int W = a.k.W, D = a.k.D;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, grp = lane / kGL, lig = lane % kGL;
  const int nwarp = blockDim.x >> 5, Wr = (W + 3) / 4 * 4;
  uint32_t *merge = reinterpret_cast<uint32_t *>(smem + nwarp * CF::warp_bytes(BANDED));   // [Wr] key of each right pixel
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
    if constexpr (RH) seg = (seg + 1) / 2 * 2;       // segments start at even columns
    const int gi = warp * kGW + grp;
    const int x0 = min(gi * seg, W), x1 = min(x0 + seg, W);
    uint8_t *ring = smem + warp * CF::warp_bytes(BANDED);
    const uint32_t ring_s = smem_u32(ring);
    // a vector's pieces into a slot, and out of it
    auto copy_v = [&](uint32_t slot, const uint8_t *src) {
      if constexpr (S8)
        copy8<CPL>(slot, lane, src);
      else
        copy16<CPL>(slot, lane, src);
    };
    // sources: the rows (0) and families (1 ..), down (left -> right) and up vectors (bytes: a
    // pixel's side by side); then the sums
    const uint8_t *pv[NP][S8 ? 1 : 2];
    [[maybe_unused]] const uint8_t *pq[NS > 0 ? NS : 1];
    [[maybe_unused]] const uint8_t *pc = nullptr;
    [[maybe_unused]] const bool odd_row = FH && (y & 1);
    const int xc = RH ? 0 : min(x0, W - 1);          // the pixel the sources start at
#pragma unroll
    for (int j = 0; j < NP; ++j)
#pragma unroll
      for (int i = 0; i < (S8 ? 1 : 2); ++i)
        pv[j][i] = a.vec[2 * j + i] + f * a.vec_frame[2 * j + i] + (row + xc) * 2 * Dp + lig * VecW<CPL, S8>::kLane;
    auto src = [&](int j, int i) { return S8 ? pv[j][0] + i * Dp : pv[j][S8 ? 0 : i]; };
#pragma unroll
    for (int j = 0; j < NS; ++j)
      pq[j] = a.vec[2 * NP + j] + f * a.vec_frame[2 * NP + j] + (row + xc) * 2 * Dp + lig * Vec16<CPL>::kLane;
    if constexpr (RH) pc = a.cost + f * frame_cells(a.k) + row * Dp + lig * Vec8<CPL>::kLane;
    // step t's copies into a slot.  A group past its segment's end copies the
    // segment's last pixel again (RH: goes on, to the row's last)
    auto copy = [&](uint32_t slot, int t) {
      if constexpr (RH) {
        const int x = min(x0 + t, W - 1);
        copy8<CPL>(slot + CF::oCost, lane, pc + (size_t)x * Dp);
        // the rows' vectors of an even column, or right -> left the next column's;
        // u16: that of even column x lies in pixel x - 1's place (0's in 0's)
        if (!(t & 1)) copy_v(slot, src(0, 0) + (size_t)x * (2 * Dp));
        const int xl = S8 ? (t & 1 ? min(x + 1, W - 1) : x) : (t & 1 ? x : max(x - 1, 0));
        copy_v(slot + kV, src(0, 1) + (size_t)xl * (2 * Dp));
        // where the predecessors lie: the row above (the down directions) and
        // below (the up ones; clamped at the last row, the vector is then not used)
        [[maybe_unused]] const int xm = max(x - 1, 0), xp = min(x + 1, W - 1);
        [[maybe_unused]] const ptrdiff_t up_row = odd_row ? -(ptrdiff_t)W : 0,
                                         down_row = odd_row && y + 1 < a.k.H ? W : up_row;
#pragma unroll
        for (int j = 1; j < NP; ++j) {
          const int xd = !odd_row || j == 1 ? x : (j == 2 ? xm : xp), xu = !odd_row || j == 1 ? x : (j == 2 ? xp : xm);
          copy_v(slot + 2 * j * kV, src(j, 0) + (up_row + xd) * (2 * Dp));
          copy_v(slot + (2 * j + 1) * kV, src(j, 1) + (down_row + xu) * (2 * Dp));
        }
#pragma unroll
        for (int j = 0; j < NS; ++j) copy16<CPL>(slot + CF::oSum + j * 2 * CF::k8, lane, pq[j] + (size_t)x * (2 * Dp));
      } else {
        const bool go = x0 + t + 1 < x1;
#pragma unroll
        for (int j = 0; j < NP; ++j) {
          copy_v(slot + 2 * j * kV, src(j, 0));
          copy_v(slot + (2 * j + 1) * kV, src(j, 1));
#pragma unroll
          for (int i = 0; i < (S8 ? 1 : 2); ++i)
            if (go) pv[j][i] += 2 * Dp;
        }
#pragma unroll
        for (int j = 0; j < NS; ++j) {
          copy16<CPL>(slot + CF::oSum + j * 2 * CF::k8, lane, pq[j]);
          if (go) pq[j] += 2 * Dp;
        }
      }
    };
    for (int t = 0; t < R; ++t) {
      copy(ring_s + t * CF::kSlot, t);
      cp_commit();
    }
    [[maybe_unused]] uint32_t z[CPL / 4] = {};
    [[maybe_unused]] Prev<CPL, S8> right = {};   // RH: the left -> right vector of the even column before
    [[maybe_unused]] const Edges none = no_neighbours(lig);
    if constexpr (RH && !BANDED) pad_bytes<CPL>(D, lig, z);
    uint32_t kb[NW];                             // the keys' low bytes (d) and the padding's high ones
    [[maybe_unused]] const int16_t *lo_row = nullptr;
    [[maybe_unused]] int lo = 0;                 // the band start of the tile
    // RH on the bands: those of the tiles left and right and of the three below (row y + 1's)
    [[maybe_unused]] int lo_l = 0, lo_r = 0, below_l = 0, below_m = 0, below_r = 0;
    [[maybe_unused]] uint32_t *shift = reinterpret_cast<uint32_t *>(ring + R * CF::kSlot) + grp * (kGL * NW);
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
          if constexpr (RH) {
            const int tx = min(x, W - 1) >> kBandTileLog, tl = max(tx - 1, 0), tr = min(tx + 1, a.k.tw - 1);
            const int16_t *lo_next = b.band_lo + (min(y + 1, a.k.H - 1) >> kBandTileLog) * a.k.tw;
            lo_l = lo_row[tl], lo_r = lo_row[tr];
            below_l = lo_next[tl], below_m = lo_next[tx], below_r = lo_next[tr];
          }
          __syncwarp();
        }
      }
      uint32_t Sm[NW];
      cp_wait<R - 1>();
      const uint8_t *v = ring + base;
      // the slot's vector i as words
      auto get = [&](int i, uint32_t (&w)[NW]) {
        if constexpr (S8)
          slot8<CPL>(v + i * kV, lane, z0, w);
        else
          slot16<CPL>(v + i * kV, lane, w);
      };
      auto add2 = [&](const uint32_t (&A)[NW], const uint32_t (&B)[NW]) {
#pragma unroll
        for (int w = 0; w < NW; ++w) Sm[w] += A[w] + B[w];
      };
      if constexpr (RH) {
        uint32_t C[NW], A[NW], B[NW];
        slot8<CPL>(v + CF::oCost, lane, z, C);
        // predecessor i's vector (padding cells above every path cost); zeros where
        // the path starts here
        auto pred = [&](int i, bool start, uint32_t (&w)[NW]) {
          Prev<CPL, S8> p;
          p.load(v + i * kV, lane);
          if (start) p = {};
          p.words(z, w);
        };
        // A and B: two predecessors' vectors -> their directions' vectors here.
        // from_a, from_b: the band starts there
        auto step2 = [&]([[maybe_unused]] int from_a, [[maybe_unused]] int from_b, [[maybe_unused]] bool start_a,
                         [[maybe_unused]] bool start_b) {
          uint32_t ma, mb;
          [[maybe_unused]] Edges ea = none, eb = none;
          group_min2<NW>(A, B, ma, mb);
          if constexpr (BANDED) {
            // (the starts differ only where the step crosses into another tile)
            auto reindex = [&](uint32_t (&w)[NW], int from, bool start, Edges &e) {
              if (!__any_sync(kAll, from != lo)) return;
              e = band_shift<NW>(w, lo - from, shift, lig);
              const uint32_t keep = start ? 0u : 0xffffffffu;
#pragma unroll
              for (int i = 0; i < NW; ++i) w[i] &= keep;
            };
            reindex(A, from_a, start_a, ea);
            reindex(B, from_b, start_b, eb);
          }
          step<NW, BANDED>(A, C, ma, a.sc, ea, lig);
          step<NW, BANDED>(B, C, mb, a.sc, eb, lig);
        };
        if (!(t & 1)) {
          right.load(v, lane);
          if constexpr (!S8) {                   // (the path starts at column 0: its vector is the cost)
            if (x == 0) copy_words<NW>(right.w, C);
          }
          right.words(z0, A);
          get(1, B);
        } else {
          right.words(z, A);
          const bool start = x + 1 >= W;         // (the path right -> left)
          pred(1, start, B);
          step2(lo, t % kBandTile == kBandTile - 1 ? lo_r : lo, false, start);
        }
#pragma unroll
        for (int w = 0; w < NW; ++w) Sm[w] = A[w] + B[w];
        if (!odd_row) {
#pragma unroll
          for (int j = 1; j < NP; ++j) {
            get(2 * j, A);
            get(2 * j + 1, B);
            add2(A, B);
          }
        } else {
          const bool last = y + 1 >= a.k.H;
          // on the bands: the tile column of x - 1 (-1: the one to the left) and x + 1
          const bool first_x = t % kBandTile == 0, last_x = t % kBandTile == kBandTile - 1;
#pragma unroll
          for (int j = 1; j < NP; ++j) {
            // paths that start here: the predecessor lies outside the image
            const bool start_a = j == 2 ? x == 0 : (j == 3 && x == W - 1);
            const bool start_b = last || (j == 2 ? x == W - 1 : (j == 3 && x == 0));
            pred(2 * j, start_a, A);
            pred(2 * j + 1, start_b, B);
            const int up_l = first_x ? lo_l : lo, up_r = last_x ? lo_r : lo;
            const int dn_l = first_x ? below_l : below_m, dn_r = last_x ? below_r : below_m;
            step2(j == 1 ? lo : (j == 2 ? up_l : up_r), j == 1 ? below_m : (j == 2 ? dn_r : dn_l), start_a, start_b);
            add2(A, B);
          }
        }
      } else {
#pragma unroll
        for (int j = 0; j < NP; ++j) {
          const uint8_t *vj = ring + base + 2 * j * CF::k8;
          uint32_t T[NW], U[NW];
          slot8<CPL>(vj, lane, z0, T);
          slot8<CPL>(vj + CF::k8, lane, z0, U);
#pragma unroll
          for (int i = 0; i < NW; ++i) Sm[i] = j == 0 ? T[i] + U[i] : Sm[i] + T[i] + U[i];
        }
      }
#pragma unroll
      for (int j = 0; j < NS; ++j) {
        uint32_t T[NW];
        slot16<CPL>(v + CF::oSum + j * 2 * CF::k8, lane, T);
#pragma unroll
        for (int i = 0; i < NW; ++i) Sm[i] += T[i];
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

template <int CPL, bool S8, int NF, int NS, bool BANDED, bool RH, bool FH = true>
static cudaError_t launch_wta_v(const WtaArgs &a, int nf, cudaStream_t s) {
  using CF = WtaCfg<CPL, S8, NF, NS, RH>;
  static bool done[64] = {};
  cudaError_t e = smem_optin(k_wta<CPL, S8, NF, NS, BANDED, RH, FH>, CF::kRoom, done);
  if (e != cudaSuccess) return e;
  k_wta<CPL, S8, NF, NS, BANDED, RH, FH>
      <<<dim3(a.k.H, nf), 32 * CF::warps(a.k.W, BANDED), CF::smem(a.k.W, BANDED), s>>>(a);
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
  const bool eight = k.num_paths == 8;
  // the rows, then the other families or, behind the sweep, its two u16 sums
  for (int i = 0; i < (k.rows_lines ? 1 : (eight ? 4 : 2)); ++i) {
    uint8_t *v[2];
    size_t frame[2];
    family_vectors(k, b, S8, (i + 3) % 4, v, frame);
    for (int j = 0; j < 2; ++j) add(v[j], frame[j]);
  }
  if constexpr (!BANDED)
    if (k.rows_lines) {
      for (int i = 0; i < 2; ++i) add(reinterpret_cast<const uint8_t *>(b.part[i]), 2 * frame_cells(k));
      return launch_wta_v<CPL, S8, 0, 2, BANDED, !S8, false>(a, nf, s);
    }
  if constexpr (!S8 || (!BANDED && (CPL == 16 || CPL == 24)))
    if (k.half)
      return eight ? launch_wta_v<CPL, S8, 3, 0, BANDED, true>(a, nf, s) : launch_wta_v<CPL, S8, 1, 0, BANDED, true>(a, nf, s);
  return eight ? launch_wta_v<CPL, S8, 3, 0, BANDED, !S8, false>(a, nf, s)
               : launch_wta_v<CPL, S8, 1, 0, BANDED, !S8, false>(a, nf, s);
}

template <int CPL, bool S8>
cudaError_t launch_wta_t(const KParams &k, const Buffers &b, int nf, int16_t *out, cudaStream_t s) {
  if constexpr (CPL <= 16)
    if (k.band) return launch_wta_b<CPL, S8, true>(k, b, nf, out, s);
  return launch_wta_b<CPL, S8, false>(k, b, nf, out, s);
}

}  // namespace oct
}  // namespace sgmf
