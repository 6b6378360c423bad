// sgmf_lanes.cuh -- the lane layout and the recursion step (Eq. 2) of the
// aggregation kernels, over the full range and on the bands.
//
// A group of 8 lanes holds the Dp disparities of one path-cost vector; lane j
// holds cells [j CPL, (j + 1) CPL), CPL = Dp / 8, as NW = CPL / 2 u16x2 words.
// Word w pairs the cells w (low half) and w + NW (high half), so the d - 1 and
// d + 1 neighbours of a word are the words w - 1 and w + 1 themselves: only
// the first and the last word need a byte permute and a shuffle, where words
// of adjacent cells need a permute per word.  One step of Eq. 2 on a word:
//   t     = viaddmin(vimin3(L(d-1), L(d+1), m + P2 - P1), P1, L(d))
//         = min{ L(d), L(d-1)+P1, L(d+1)+P1, m+P2 }
//   L'(d) = t + C(d) - m                      (one 32-bit add: t >= m per half)
// with m = min_k L(k), a per-lane u16x2 min and three shuffles.  A warp steps
// four vectors at once; a step's fixed work (two neighbour shuffles, the
// minimum's four, a few words of bookkeeping) serves 4 Dp cells.  The 16-lane
// groups of adjacent-cell words that this replaced spent two full-warp
// reductions and Dp / 16 + 1 permutes per 2 Dp cells: at D = 128 a sweep over
// six directions took 592 instructions per 512 cells, now 395 (1242 x 375, one
// wave of frames: 786 -> 602 us).  A step of a line walk at D = 128, with its cost
// bytes and its share of the stores, is 83 instructions for four vectors; where
// few warps share a SM it takes about 146 ns (1242 steps in 181 us).
//
// A path start is the same step applied to an all-zero previous vector (with
// m = 0 it yields L = C).  Disparities d >= D are padding: their cost is
// raised by kInf so they never reach the min.
//
// Memory order of a vector.  Bytes: a lane's CPL bytes are the words' (low,
// high) cells in turn, so one permute turns two words into four bytes and one
// per word back.  u16: the words as they are.  A lane's bytes are one or more
// chunks of one vector access (16 bytes, 8 where CPL is no multiple of 16);
// for CPL = 32 (bytes) and CPL = 16, 32 (u16) the chunks of the 8 lanes are
// interleaved, chunk 0 of every lane first, so that a group's access covers
// 128 consecutive bytes of shared or global memory.
#pragma once
#include <cstdint>

#include "sgmf_internal.cuh"

namespace sgmf {
namespace oct {

constexpr unsigned kAll = 0xffffffffu;
constexpr int kGL = 8;          // lanes per group
constexpr int kGW = 32 / kGL;   // groups (vectors) per warp

// bytes of one chunk, chunks per lane, and the byte offset of lane lig's first
// chunk and of the next one, for the u8 and the u16 form of a vector
template <int CPL>
struct Vec8 {
  static constexpr int CH = CPL % 16 == 0 ? 16 : 8, N = CPL / CH;
  static constexpr int kLane = CPL == 32 ? 16 : CPL, kNext = CPL == 32 ? 128 : CH;
};
template <int CPL>
struct Vec16 {
  static constexpr int N = CPL / 8;
  static constexpr bool kInter = CPL == 16 || CPL == 32;
  static constexpr int kLane = kInter ? 16 : 2 * CPL, kNext = kInter ? 128 : 16;
};

// the u8 chunks at p (the lane's first chunk) as raw 32-bit words
template <int CPL>
struct Raw8 {
  uint32_t v[CPL / 4];
};

template <int CPL>
__device__ __forceinline__ void load_raw8(const uint8_t *p, Raw8<CPL> &r) {
  using V = Vec8<CPL>;
#pragma unroll
  for (int q = 0; q < V::N; ++q) {
    if constexpr (V::CH == 16) {
      const uint4 t = *reinterpret_cast<const uint4 *>(p + q * V::kNext);
      r.v[4 * q] = t.x, r.v[4 * q + 1] = t.y, r.v[4 * q + 2] = t.z, r.v[4 * q + 3] = t.w;
    } else {
      const uint2 t = *reinterpret_cast<const uint2 *>(p + q * V::kNext);
      r.v[2 * q] = t.x, r.v[2 * q + 1] = t.y;
    }
  }
}

// raw bytes -> words; z holds the pad bytes (0x40 for cells d >= D), which
// become the high bytes
template <int CPL>
__device__ __forceinline__ void expand8(const Raw8<CPL> &r, const uint32_t (&z)[CPL / 4], uint32_t (&w)[CPL / 2]) {
#pragma unroll
  for (int j = 0; j < CPL / 4; ++j) {
    w[2 * j] = prmt(r.v[j], z[j], 0x5140);
    w[2 * j + 1] = prmt(r.v[j], z[j], 0x7362);
  }
}

template <int CPL>
__device__ __forceinline__ void load_u8(const uint8_t *p, const uint32_t (&z)[CPL / 4], uint32_t (&w)[CPL / 2]) {
  Raw8<CPL> r;
  load_raw8<CPL>(p, r);
  expand8<CPL>(r, z, w);
}

// words -> bytes (every real value is <= 255 when used)
template <int CPL>
__device__ __forceinline__ void store_u8(uint8_t *p, const uint32_t (&w)[CPL / 2]) {
  using V = Vec8<CPL>;
  uint32_t v[CPL / 4];
#pragma unroll
  for (int j = 0; j < CPL / 4; ++j) v[j] = prmt(w[2 * j], w[2 * j + 1], 0x6420);
#pragma unroll
  for (int q = 0; q < V::N; ++q) {
    if constexpr (V::CH == 16)
      *reinterpret_cast<uint4 *>(p + q * V::kNext) = make_uint4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
    else
      *reinterpret_cast<uint2 *>(p + q * V::kNext) = make_uint2(v[2 * q], v[2 * q + 1]);
  }
}

template <int CPL>
__device__ __forceinline__ void store_u16(uint8_t *p, const uint32_t (&w)[CPL / 2]) {
  using V = Vec16<CPL>;
#pragma unroll
  for (int q = 0; q < V::N; ++q)
    *reinterpret_cast<uint4 *>(p + q * V::kNext) = make_uint4(w[4 * q], w[4 * q + 1], w[4 * q + 2], w[4 * q + 3]);
}

// a vector in the width its path costs need: bytes (S8) or u16
template <int CPL, bool S8>
struct VecW {
  static constexpr int kLane = S8 ? Vec8<CPL>::kLane : Vec16<CPL>::kLane;
  static __device__ __forceinline__ void put(uint8_t *p, const uint32_t (&w)[CPL / 2]) {
    if constexpr (S8)
      store_u8<CPL>(p, w);
    else
      store_u16<CPL>(p, w);
  }
};

// asynchronous copies of a lane's own pieces into shared memory
template <int B>
__device__ __forceinline__ void cp_async(uint32_t dst, const uint8_t *src) {
  if constexpr (B == 16)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// a lane's pieces of a byte / u16 vector: global (lane's first chunk) -> slot,
// and slot -> registers.  slot: the vector's place in the slot, before the lane offset
template <int CPL>
__device__ __forceinline__ void copy8(uint32_t slot, int lane, const uint8_t *src) {
  using V = Vec8<CPL>;
#pragma unroll
  for (int q = 0; q < V::N; ++q) cp_async<V::CH>(slot + (q * 32 + lane) * V::CH, src + q * V::kNext);
}
template <int CPL>
__device__ __forceinline__ void copy16(uint32_t slot, int lane, const uint8_t *src) {
  using V = Vec16<CPL>;
#pragma unroll
  for (int q = 0; q < V::N; ++q) cp_async<16>(slot + (q * 32 + lane) * 16, src + q * V::kNext);
}
template <int CPL>
__device__ __forceinline__ void slot_raw8(const uint8_t *slot, int lane, Raw8<CPL> &r) {
  using V = Vec8<CPL>;
#pragma unroll
  for (int q = 0; q < V::N; ++q) {
    if constexpr (V::CH == 16) {
      const uint4 t = reinterpret_cast<const uint4 *>(slot)[q * 32 + lane];
      r.v[4 * q] = t.x, r.v[4 * q + 1] = t.y, r.v[4 * q + 2] = t.z, r.v[4 * q + 3] = t.w;
    } else {
      const uint2 t = reinterpret_cast<const uint2 *>(slot)[q * 32 + lane];
      r.v[2 * q] = t.x, r.v[2 * q + 1] = t.y;
    }
  }
}
template <int CPL>
__device__ __forceinline__ void slot8(const uint8_t *slot, int lane, const uint32_t (&z)[CPL / 4],
                                      uint32_t (&w)[CPL / 2]) {
  Raw8<CPL> r;
  slot_raw8<CPL>(slot, lane, r);
  expand8<CPL>(r, z, w);
}
template <int CPL>
__device__ __forceinline__ void slot16(const uint8_t *slot, int lane, uint32_t (&w)[CPL / 2]) {
#pragma unroll
  for (int q = 0; q < Vec16<CPL>::N; ++q) {
    const uint4 t = reinterpret_cast<const uint4 *>(slot)[q * 32 + lane];
    w[4 * q] = t.x, w[4 * q + 1] = t.y, w[4 * q + 2] = t.z, w[4 * q + 3] = t.w;
  }
}

// pad bytes of the lane's cells d >= D, in the order of the lane's bytes
template <int CPL>
__device__ __forceinline__ void pad_bytes(int D, int lig, uint32_t (&z)[CPL / 4]) {
#pragma unroll
  for (int i = 0; i < CPL / 4; ++i) {
    uint32_t v = 0;
#pragma unroll
    for (int b = 0; b < 4; ++b)
      if (lig * CPL + 2 * i + (b >> 1) + (b & 1) * (CPL / 2) >= D) v |= (kInf >> 8) << (8 * b);
    z[i] = v;
  }
}


template <int NW>
__device__ __forceinline__ void copy_words(uint32_t (&dst)[NW], const uint32_t (&src)[NW]) {
#pragma unroll
  for (int w = 0; w < NW; ++w) dst[w] = src[w];
}

struct StepConsts {
  uint32_t p1x2;   // P1 in both halves
  uint32_t dpx2;   // (P2 - P1) in both halves
  uint32_t one;    // 1, as a value the compiler cannot see
};
inline StepConsts step_consts(const KParams &k) {
  return {(uint32_t)k.p1 * 0x10001u, (uint32_t)(k.p2 - k.p1) * 0x10001u, 1u};
}
__device__ __forceinline__ uint32_t mad_u32(uint32_t a, uint32_t b, uint32_t c) {
  uint32_t d;
  asm("mad.lo.u32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
  return d;
}

// The group's outer neighbours, as bits ORed into the first / last lane's words:
// 0xffff in the missing neighbour's half (L(-1), L(Dp) only enter a min).  On the
// bands the neighbour's half is cleared first (step) and may hold the previous
// pixel's cell just outside the current band (band_shift).
struct Edges {
  uint32_t lo, hi;
};
__device__ __forceinline__ Edges no_neighbours(int lig) {
  return {lig == 0 ? 0xffffu : 0u, lig == kGL - 1 ? 0xffff0000u : 0u};
}

// One step of Eq. 2 for the lane's words.  mm = min_k L(p - r, k) in both halves.
// MAD: the last addition as a multiply-add (t * 1 + ..), which leaves the ALU
// pipe, the bound of most callers, for the FMA pipe: 2 to 4 % of the walks and
// the winner kernel at up to 8 words a lane; above, and in the sweep at 8, the
// register it costs loses more.
template <int NW, bool BANDED = false, bool MAD = NW <= 8>
__device__ __forceinline__ void step(uint32_t (&L)[NW], const uint32_t (&C)[NW], uint32_t mm, const StepConsts &sc,
                                     Edges e, int lig = 0) {
  const uint32_t below = __shfl_up_sync(kAll, L[NW - 1], 1, kGL);
  const uint32_t above = __shfl_down_sync(kAll, L[0], 1, kGL);
  // below the first word: (cell CPL - 1 of the lane below, own cell NW - 1);
  // above the last: (own cell NW, cell 0 of the lane above)
  uint32_t left = prmt(below, L[NW - 1], 0x5432), last = prmt(L[0], above, 0x5432);
  if constexpr (BANDED) {
    left &= lig == 0 ? 0xffff0000u : 0xffffffffu;
    last &= lig == kGL - 1 ? 0xffffu : 0xffffffffu;
  }
  left |= e.lo;
  last |= e.hi;
  const uint32_t cap = mm + sc.dpx2;           // m + P2 - P1 per half
  const uint32_t negmm = 0u - mm;
#pragma unroll
  for (int i = 0; i < NW; ++i) {
    const uint32_t right = i == NW - 1 ? last : L[i + 1];
    const uint32_t t = __viaddmin_u16x2(__vimin3_u16x2(left, right, cap), sc.p1x2, L[i]);
    left = L[i];
    L[i] = MAD ? mad_u32(t, sc.one, C[i] + negmm) : t + C[i] + negmm;
  }
}

// min of the lane's words, per half
template <int NW>
__device__ __forceinline__ uint32_t lane_min(const uint32_t (&L)[NW]) {
  if constexpr (NW == 4) {
    return __vminu2(__vimin3_u16x2(L[0], L[1], L[2]), L[3]);
  } else if constexpr (NW == 8) {
    return __vimin3_u16x2(__vimin3_u16x2(L[0], L[1], L[2]), __vimin3_u16x2(L[3], L[4], L[5]), __vminu2(L[6], L[7]));
  } else {
    uint32_t v = L[0];
#pragma unroll
    for (int i = 1; i + 1 < NW; i += 2) v = __vimin3_u16x2(v, L[i], L[i + 1]);
    return NW % 2 == 0 ? __vminu2(v, L[NW - 1]) : v;
  }
}

// min over the group's disparities, in both halves
template <int NW>
__device__ __forceinline__ uint32_t group_min(const uint32_t (&L)[NW]) {
  uint32_t v = lane_min<NW>(L);
  v = __vminu2(v, prmt(v, v, 0x1032));
  // two rounds of shuffles instead of three: they are the step's longest chain
  const uint32_t a = __shfl_xor_sync(kAll, v, 1), b = __shfl_xor_sync(kAll, v, 2), c = __shfl_xor_sync(kAll, v, 3);
  v = __vminu2(__vimin3_u16x2(v, a, b), c);
  return __vminu2(v, __shfl_xor_sync(kAll, v, 4));
}

// the minima of two vectors, each in both halves: one pass of shuffles for both
template <int NW>
__device__ __forceinline__ void group_min2(const uint32_t (&A)[NW], const uint32_t (&B)[NW], uint32_t &ma,
                                           uint32_t &mb) {
  const uint32_t va = lane_min<NW>(A), vb = lane_min<NW>(B);
  uint32_t v = __vminu2(prmt(va, vb, 0x5410), prmt(va, vb, 0x7632));
  const uint32_t a = __shfl_xor_sync(kAll, v, 1), b = __shfl_xor_sync(kAll, v, 2), c = __shfl_xor_sync(kAll, v, 3);
  v = __vminu2(__vimin3_u16x2(v, a, b), c);
  v = __vminu2(v, __shfl_xor_sync(kAll, v, 4));
  ma = prmt(v, v, 0x1010);
  mb = prmt(v, v, 0x3232);
}

// min of a u32 over the group
__device__ __forceinline__ uint32_t group_min_u32(uint32_t v) {
#pragma unroll
  for (int s = 1; s < kGL; s *= 2) v = min(v, __shfl_xor_sync(kAll, v, s));
  return v;
}

// ---- disparity bands (banded mode, not in the paper) -----------------------------
// In banded mode cell j of pixel p stands for disparity lo_p + j, with lo_p
// constant on 8 x 8 pixel tiles.  Where the band start changes by delta along a
// path, the previous pixel's path costs are re-indexed: cell j takes old cell
// j + delta, and the cells that have no old counterpart become absent (kInf,
// above every real path cost, so they only ever lose a min).  m of the previous
// pixel stays the min over its own band.  The recursion on the bands is the
// exact dynamic program of Eq. 1 with each pixel's labels restricted to its
// band, so the previous pixel's cell just below the new band (old cell
// delta - 1, for delta > 0) or just above it (old cell B + delta, for
// delta < 0) is still the d-1 / d+1 neighbour of the new band's end cell: the
// shift hands it to the next step as the end lane's edge.
//
// Runs on all 32 lanes: a group with delta = 0 rewrites its cells in place.
// buf: the group's shared scratch, 8 NW words.
template <int NW>
__device__ __forceinline__ Edges band_shift(uint32_t (&L)[NW], int delta, uint32_t *buf, int lig) {
  constexpr int CPL = 2 * NW, B = kGL * CPL;
#pragma unroll
  for (int i = 0; i < NW; ++i) buf[lig * NW + i] = L[i];
  __syncwarp();
  const uint16_t *cells = reinterpret_cast<const uint16_t *>(buf);
  auto old = [&](int c, uint32_t absent) -> uint32_t {   // old cell c
    const int r = c % CPL;
    return (unsigned)c < (unsigned)B ? (uint32_t)cells[2 * (c / CPL * NW + r % NW) + r / NW] : absent;
  };
#pragma unroll
  for (int i = 0; i < NW; ++i) {
    const int c = lig * CPL + i + delta;
    L[i] = old(c, kInf) | old(c + NW, kInf) << 16;
  }
  const uint32_t v = old(lig == 0 ? delta - 1 : B + delta, 0xffffu);
  __syncwarp();
  return {lig == 0 ? v : 0u, lig == kGL - 1 ? v << 16 : 0u};
}

// Sub-pixel disparity in 1/16 px: the vertex of the parabola through sm =
// S(d*-1), s0 = S(d*), sp = S(d*+1); 16 d* at the ends of the range.  d* is the
// smallest argmin: den = sm - 2 s0 + sp > 0 and 16 (sm - sp) > -16 den, so the
// biased numerator is positive: offset = floor((16 (sm - sp) + den) / (2 den)) =
// that quotient - 8.
__device__ __forceinline__ int subpixel_disp(int ds, int D, uint32_t sm, uint32_t s0, uint32_t sp) {
  int v = 16 * ds;
  if (ds > 0 && ds < D - 1) {
    const uint32_t den = sm + sp - 2u * s0;
    v += (int)((16u * sm + 17u * den - 16u * sp) / (2u * den)) - 8;
  }
  return v;
}

// opt in once per device to the kernel's dynamic shared memory
template <typename Kern>
static cudaError_t smem_optin(Kern kern, int bytes, bool (&done)[64]) {
  return once_per_device(done, [&](int) {
    return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  });
}

}  // namespace oct
}  // namespace sgmf
