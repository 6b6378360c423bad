// sgmf_lines.cuh -- the directions of Eq. 2 (Sec. III) as line walks.
//
// Each direction runs along a family of lines:
//   family 0 (vertical)      line k = column k            down: r=(0,1)   up: r=(0,-1)
//   family 1 (diagonal)      line k: x = (k + y) mod W    down: r=(1,1)   up: r=(-1,-1)
//   family 2 (anti-diagonal) line k: x = (k - y) mod W    down: r=(-1,1)  up: r=(1,-1)
//   family 3 (rows)          line k = row k               right: r=(1,0)  left: r=(-1,0)
// With the modulo every diagonal line has exactly H pixels, and a path
// (re)starts where the line wraps, i.e. where p - r leaves the image.
//
// An 8-lane group walks one line in one direction, a warp four neighbouring
// lines.  The two directions of a family are independent walks (grid.y), and
// so are the families: their launches overlap (programmatic launch), so that a
// call of few frames has eight directions' lines in flight.  A walk is bound
// by its own chain (a step's minimum, three shuffles, feeds the next step)
// when few warps are resident, and by memory otherwise: it reads the cost
// volume once and writes one vector per pixel.  A lane copies its own cost
// bytes kLineAhead steps ahead into its place of a shared-memory ring
// (cp.async): no barrier, and enough in flight for one warp a scheduler.
// Measured on 1242 x 375, D = 128: the six vertical and diagonal directions of
// one frame 442 us when each family walked down then up in a launch of its own,
// all eight directions now 181 us; 8 frames 1358 us for six, 1205 us for eight
// (6.3 TB/s: the DRAM bound).  8 steps ahead: 195 us for one frame, 16: 181.
#pragma once

#include <algorithm>

#include "sgmf_lanes.cuh"

namespace sgmf {
namespace oct {

struct LineArgs {
  KParams k;
  const uint8_t *cost;
  uint8_t *dst[2];        // frame 0's vectors of the down / up walk, pixel stride 2 Dp bytes
  size_t dst_frame[2];    // bytes from one frame to the next
  StepConsts sc;
  const int *gate;        // per-frame gate words of the launch's frames, or null
  const int16_t *lo;      // banded mode: band starts per tile, [frame][th][tw]
};

// A position on a line: its pixel index p, column x, and whether the path
// restarts there.  Wrapping at x = xw the line goes on, a new path, at xs.
template <int FAM>
struct LinePos {
  int p, x, y;                   // (y: banded mode)
  bool start;
  __device__ __forceinline__ void next(int dp, int dx, int dy, int xw, int xs, int W) {
    p += dp;
    y += dy;
    if constexpr (FAM == 3) x += dx;
    if constexpr (FAM == 1 || FAM == 2) {
      x += dx;
      start = x == xw;
      p = start ? p - dx * W : p;
      x = start ? xs : x;
    }
  }
};

constexpr int kLineAhead = 16;   // steps copied ahead (a multiple of the four unrolled)

// HALF: store only the vectors of even rows (rows family: even columns); the
// winner kernel takes the others' step itself.  With u16 vectors the two
// directions of the rows then share a region: that of left -> right in its
// pixel's place, that of right -> left in the place of the pixel before, column
// 0's in its own (the other one there is the cost itself).
// BANDED: on the bands (no padding cells).
template <int CPL, bool S8, int FAM, bool BANDED, bool HALF>
__global__ void __launch_bounds__(256) k_lines(const __grid_constant__ LineArgs a) {
  constexpr int NW = CPL / 2, Dp = kGL * CPL, A = kLineAhead, U = 4, kSlot = 32 * CPL;
  extern __shared__ __align__(128) uint8_t smem[];
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const int f = blockIdx.z;
  const int W = a.k.W, H = a.k.H;
  const int lines = FAM == 3 ? H : W, n = FAM == 3 ? W : H;   // lines, steps of each
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, grp = lane / kGL, lig = lane % kGL;
  const int line0 = (blockIdx.x * (blockDim.x >> 5) + warp) * kGW;
  if (gated_off(a.gate ? a.gate + f : nullptr, a.k.gate_run) || line0 >= lines) {   // warp-uniform
    asm volatile("griddepcontrol.wait;" ::: "memory");
    return;
  }
  const bool up = blockIdx.y != 0;
  const int line = min(line0 + grp, lines - 1);  // a group past the last line repeats it and stores nothing
  const bool act = line0 + grp < lines;
  const uint8_t *cost = a.cost + f * frame_cells(a.k) + lig * Vec8<CPL>::kLane;
  uint8_t *dst = a.dst[up] + f * a.dst_frame[up] + lig * VecW<CPL, S8>::kLane;
  uint8_t *ring = smem + warp * (A * kSlot);
  const uint32_t ring_s = smem_u32(ring);
  uint32_t z[CPL / 4] = {};
  if constexpr (!BANDED) pad_bytes<CPL>(a.k.D, lig, z);
  const Edges none = no_neighbours(lig);
  const StepConsts sc = a.sc;
  // the first pixel and the move per step
  const int dx = FAM == 0 ? 0 : (FAM == 3 ? (up ? -1 : 1) : ((FAM == 1) != up ? 1 : -1));
  const int dy = FAM == 3 ? 0 : (up ? -1 : 1);
  const int xw = dx > 0 ? W : -1, xs = dx > 0 ? 0 : W - 1;
  LinePos<FAM> in;
  in.start = false;                              // (the first step starts from a zero vector anyway)
  int dp;
  if constexpr (FAM == 3) {
    in.x = up ? W - 1 : 0;
    in.y = line;
    in.p = line * W + in.x;
    dp = dx;
  } else {
    in.x = line;
    if (FAM != 0 && up) {
      const int x = (FAM == 1 ? line + (H - 1) : line - (H - 1)) % W;
      in.x = x < 0 ? x + W : x;
    }
    in.y = up ? H - 1 : 0;
    in.p = in.y * W + in.x;
    dp = (up ? -W : W) + dx;
  }
  LinePos<FAM> at = in;                          // in: next step to copy; at: next step to take
  auto copy = [&](uint32_t slot) {
    copy8<CPL>(slot, lane, cost + (size_t)(unsigned)in.p * Dp);
    in.next(dp, dx, dy, xw, xs, W);
  };
#pragma unroll 1
  for (int t = 0; t < A; ++t) {
    if (t < n) copy(ring_s + t * kSlot);
    cp_commit();
  }
  uint32_t L[NW];
#pragma unroll
  for (int w = 0; w < NW; ++w) L[w] = 0u;
  uint32_t mm = 0u;
  // banded: the tile and band start of the step before, the group's shift scratch
  [[maybe_unused]] const int16_t *lo = nullptr;
  [[maybe_unused]] int tile = 0, cur = 0;
  [[maybe_unused]] uint32_t *buf = nullptr;
  if constexpr (BANDED) {
    lo = a.lo + (size_t)f * a.k.th * a.k.tw;
    tile = (at.y >> kBandTileLog) * a.k.tw + (at.x >> kBandTileLog);
    cur = lo[tile];
    buf = reinterpret_cast<uint32_t *>(smem + (blockDim.x >> 5) * (A * kSlot)) + (warp * kGW + grp) * (kGL * NW);
  }
  // the next step's cost bytes are read while this step's minimum is formed
  Raw8<CPL> nxt;
  cp_wait<A - 1>();
  slot_raw8<CPL>(ring, lane, nxt);
  // a step on the bytes read before; slot: the next step's.  The copy into
  // the slot of the step itself follows (its bytes are in registers)
  auto take = [&](const uint8_t *slot) {
    uint32_t C[NW];
    expand8<CPL>(nxt, z, C);
    cp_wait<A - 2>();
    slot_raw8<CPL>(slot, lane, nxt);
    Edges e = none;
    if constexpr (BANDED) {
      const int tl = (at.y >> kBandTileLog) * a.k.tw + (at.x >> kBandTileLog);
      if (__any_sync(kAll, tl != tile)) {
        const int now = lo[tl], delta = now - cur;
        tile = tl;
        cur = now;
        if (__any_sync(kAll, delta != 0)) e = band_shift<NW>(L, delta, buf, lig);
      }
    }
    if constexpr (FAM == 1 || FAM == 2) {
      if (__any_sync(kAll, at.start)) {
        const uint32_t keep = at.start ? 0u : 0xffffffffu;
#pragma unroll
        for (int w = 0; w < NW; ++w) L[w] &= keep;
        mm &= keep;
      }
    }
    step<NW, BANDED>(L, C, mm, sc, e, lig);
    mm = group_min<NW>(L);
    uint8_t *o = dst + (size_t)(unsigned)at.p * (2 * Dp);
    if constexpr (HALF && FAM == 3 && !S8) {
      if (act && !(at.x & 1) && (up || at.x != 0)) VecW<CPL, S8>::put(up && at.x != 0 ? o - 2 * Dp : o, L);
    } else if (act && !(HALF && ((FAM == 3 ? at.x : at.y) & 1))) {
      VecW<CPL, S8>::put(o, L);
    }
    at.next(dp, dx, dy, xw, xs, W);
  };
  int t = 0, base = 0;                           // base: the slot of step t
  for (; t + A + U <= n; t += U) {               // U steps and the U copied into their slots all exist
    const int after = base + U * kSlot == A * kSlot ? 0 : base + U * kSlot;
#pragma unroll
    for (int u = 0; u < U; ++u) {
      take(ring + (u + 1 < U ? base + (u + 1) * kSlot : after));
      copy(ring_s + base + u * kSlot);
      cp_commit();
    }
    base = after;
  }
#pragma unroll 1
  for (; t < n; ++t) {
    const int after = base + kSlot == A * kSlot ? 0 : base + kSlot;
    take(ring + after);                          // (past the last step: bytes never used)
    if (t + A < n) copy(ring_s + base);
    cp_commit();
    base = after;
  }
  cp_wait<0>();
  // complete only after the launches this one overlaps: what follows in the
  // stream then finds every family's vectors
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

template <int CPL, bool S8, int FAM, bool BANDED, bool HALF>
static cudaError_t launch_family(const LineArgs &a, int nf, bool overlap, cudaStream_t s) {
  constexpr int kWarp = kLineAhead * 32 * CPL + (BANDED ? kGW * kGL * CPL * 2 : 0);
  constexpr int kMaxWarps = 8;
  static_assert(kMaxWarps * kWarp <= 224 * 1024, "the rings fit");
  const int warps = std::min(a.k.line_warps, kMaxWarps), per_cta = kGW * warps, lines = FAM == 3 ? a.k.H : a.k.W;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((lines + per_cta - 1) / per_cta, 2, nf);
  cfg.blockDim = dim3(32 * warps);
  cfg.dynamicSmemBytes = warps * kWarp;
  // u16 at 8 cells a lane: one split of the L1 for every family.  An SM changes its
  // split only when it is empty, and these families, left to the driver, asked for
  // different ones: a family waited on every SM for those it overlaps (D = 64, four
  // paths: the walks of 64 x 8192 2754 us, 692 so; of 12 frames of 160 x 90 69, 27).
  // The others agree, and lose by a larger share of shared memory where they read
  // through the L1: bands of 64 5 %, 24 cells a lane 10 %
  static bool done[64] = {};
  const cudaError_t e = once_per_device(done, [](int) {
    auto kern = k_lines<CPL, S8, FAM, BANDED, HALF>;
    const cudaError_t r = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxWarps * kWarp);
    if (r != cudaSuccess || S8 || BANDED || CPL > 8) return r;
    return cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
  });
  if (e != cudaSuccess) return e;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = overlap ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, k_lines<CPL, S8, FAM, BANDED, HALF>, a);
}

// Where a family's down and up vectors of a pixel lie.  S8: side by side,
// [down Dp bytes][up Dp bytes], in the family's buffer (rows: in the fourth
// spill region); u16: the up vectors in the family's buffer, the down vectors
// in the family's spill region, the rows' of both in the fourth (k_lines, HALF).
inline void family_vectors(const KParams &k, const Buffers &b, bool s8, int fam, uint8_t *(&v)[2], size_t (&frame)[2]) {
  const size_t cells = frame_cells(k);
  uint8_t *region = static_cast<uint8_t *>(b.spill) + fam * 2 * cells;
  uint8_t *part = fam < 3 ? reinterpret_cast<uint8_t *>(b.part[fam]) : nullptr;
  if (s8) {
    v[0] = fam < 3 ? part : region;
    v[1] = v[0] + k.Dp;
    frame[0] = frame[1] = (fam < 3 ? 2 : 8) * cells;
  } else {
    v[0] = region;
    v[1] = fam < 3 ? part : region;
    frame[0] = 8 * cells;
    frame[1] = (fam < 3 ? 2 : 8) * cells;
  }
}

template <int CPL, bool S8, bool BANDED>
static cudaError_t launch_walks(const KParams &k, const Buffers &b, int nf, cudaStream_t s) {
  LineArgs a = {};
  a.k = k;
  if (BANDED) a.k.D = k.Dp;                      // cells are band positions
  a.cost = b.cost;
  a.sc = step_consts(k);
  a.gate = b.gate;
  a.lo = b.band_lo;
  // the first launch waits for the cost volume as usual; the others may start
  // beside it (they touch nothing it writes).  The rows, the longest walks, go first
  bool overlap = false;
  cudaError_t e = cudaSuccess;
  auto family = [&](auto fam) {
    constexpr int F = decltype(fam)::value;
    if (e != cudaSuccess) return;
    family_vectors(k, b, S8, F, a.dst, a.dst_frame);
    if constexpr (!S8 && F == 3)
      e = launch_family<CPL, S8, F, BANDED, true>(a, nf, overlap, s);
    else if constexpr (!S8 || (!BANDED && (CPL == 16 || CPL == 24)))
      e = k.half ? launch_family<CPL, S8, F, BANDED, true>(a, nf, overlap, s)
                 : launch_family<CPL, S8, F, BANDED, false>(a, nf, overlap, s);
    else
      e = launch_family<CPL, S8, F, BANDED, false>(a, nf, overlap, s);
    overlap = true;
  };
  family(std::integral_constant<int, 3>{});
  if (k.rows_lines) return e;                       // the other directions are the sweep's
  family(std::integral_constant<int, 0>{});
  if (k.num_paths == 8) {
    family(std::integral_constant<int, 1>{});
    family(std::integral_constant<int, 2>{});
  }
  return e;
}

template <int CPL, bool S8>
cudaError_t launch_lines_t(const KParams &k, const Buffers &b, int nf, cudaStream_t s) {
  if constexpr (CPL <= 16)
    if (k.band) return launch_walks<CPL, S8, true>(k, b, nf, s);
  return launch_walks<CPL, S8, false>(k, b, nf, s);
}

}  // namespace oct
}  // namespace sgmf
