// sgmf_sweep.cuh -- row-synchronous aggregation of the six vertical and
// diagonal directions of Eq. 2 (Sec. III, 8 paths).
//
// The line kernels walk each line of a family separately and read the cost
// volume once per direction.  Here one thread-block cluster sweeps a whole
// frame row by row: the down sweep carries r = (0,1), (1,1), (-1,1) together,
// the up sweep r = (0,-1), (1,-1), (-1,-1), so a sweep reads every cost row
// once for three directions and writes one u16 sum of the three path costs
// per cell (the row kernel adds the two sums and its own two directions).
//
// A row of the frame is split into strips, one per CTA of the cluster, and a
// strip into runs of P pixels, one per 8-lane group.  A group keeps the
// three path-cost vectors of its P pixels in registers.  From one row to the
// next the vertical direction stays on its pixel, the "from-left" diagonal
// (predecessor x - 1) moves one pixel right and the "from-right" diagonal
// (predecessor x + 1) one pixel left, so the only state that crosses a group
// boundary per row is one vector each way.  Those go through shared-memory
// slots, double-buffered by row parity.  Inside a CTA a split row barrier (an
// mbarrier with one arrival per warp) orders them: a group computes the two
// vectors it sends, waits for the previous row's barrier, reads what entered
// it, stores what it sends, arrives, and only then does the rest of the row,
// so the barrier's latency hides behind almost a full row of work.  The
// strip's end groups exchange with the neighbouring CTAs by st.async, whose
// bytes complete on the receiving CTA's message barrier; a pair of groups
// sends its row-t vectors only after receiving the other's row t-1 vectors,
// which is what makes two slots per direction enough.  No thread waits at
// cluster scope inside the row loop.
//
// Cost rows arrive by bulk copies (one per row and CTA: the strip's pixels
// are contiguous) into a ring of R stages, R - 2 rows ahead.  Every mbarrier
// wait is bounded (the error word records a timeout); the two cluster
// barriers, at the start and the end, are executed by every thread.
//
// What bounds it is the ALU pipe (u16x2 minima and adds at half rate).
#pragma once

#include "sgmf_lines.cuh"
#include "sgmf_rows.cuh"
#include "sgmf_wta.cuh"

namespace sgmf {
namespace oct {

struct SweepArgs {
  KParams k;
  const uint8_t *cost;
  uint8_t *sum[2];        // down / up sweep sums, u16 vectors [F][H][W][Dp]
  int *err;
  StepConsts sc;
  int strip;              // pixels per CTA (= 4 * warps * P)
  const int *gate;        // per-frame gate words of the launch's frames, or null
};

template <int CPL>
struct SweepCfg {
  static constexpr int Dp = kGL * CPL, NW = CPL / 2;
  // pixels per group: 3 P NW words of path costs a lane, at most 96.  (Two CTAs
  // a SM of 6 warps and 168 registers, ring of 3 rows: 32 frames of 1242 x 375,
  // D = 128 3.30 against 3.00 ms; more warps do not help, the ALU pipe is full)
  static constexpr int P = CPL <= 16 ? 4 : 2;
  static constexpr int kMaxWarps = CPL <= 16 ? 8 : 10;
  static constexpr int kMaxCluster = 16;         // CTAs per cluster (above 8: non-portable)
  static constexpr int kMaxRow = CPL <= 16 ? 2048 : 1280;   // pixels of a row the sweep takes
  static constexpr int R = 4;                    // ring stages (rows)
  static constexpr int kBars = (R + 6) / 2 * 2;  // R + 5 mbarriers, padded: the slots start on 16 bytes
  static_assert(kBars >= R + 5 && kBars % 2 == 0, "room for the barriers, and aligned slots");
  static constexpr int kSlot = (NW + 1) * kGL;   // words of one exchanged vector: NW words + m, per lane
  // at least kExclusive bytes: one CTA per SM, so that the clusters the
  // device holds at once are the SMs the sweep occupies
  static constexpr int kExclusive = 120 * 1024;
  // the sums leave by bulk copies where the buffers fit beside the ring: per
  // warp two staging buffers (by row parity) of its 4 P pixels' u16 sums
  static constexpr bool kBulkSums = CPL <= 16;
  static constexpr int kSumBuf = kGW * P * Dp * 2;   // bytes of one buffer
  static constexpr int smem_bytes(int warps) {
    return max(kExclusive, R * (kGW * warps * P) * Dp + kBars * 8 + 2 * 2 * (kGW * warps) * kSlot * 4 +
                               (kBulkSums ? warps * 2 * kSumBuf + 128 : 0));
  }
};

// ---- cluster primitives (inline PTX) -----------------------------------------------
// The .aligned forms need the whole warp at the same instruction: each call
// first reconverges the warp.
__device__ __forceinline__ void cluster_arrive() {
  __syncwarp();
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}

__device__ __forceinline__ void cluster_wait() {
  __syncwarp();
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// address of the same shared-memory location in CTA `rank` of the cluster
__device__ __forceinline__ uint32_t cluster_map(uint32_t saddr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(saddr), "r"(rank));
  return r;
}

// asynchronous 16- and 4-byte stores into (another CTA's) shared memory whose
// completion counts the bytes on the mbarrier at mbar (same CTA as addr)
__device__ __forceinline__ void st_async4(uint32_t addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d,
                                          uint32_t mbar) {
  asm volatile(
      "st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(addr),
      "r"(a), "r"(b), "r"(c), "r"(d), "r"(mbar)
      : "memory");
}
__device__ __forceinline__ void st_async(uint32_t addr, uint32_t v, uint32_t mbar) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];" ::"r"(addr), "r"(v),
               "r"(mbar)
               : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t *bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

template <int CPL>
__global__ void __launch_bounds__(32 * SweepCfg<CPL>::kMaxWarps, 1) k_sweep(const __grid_constant__ SweepArgs a) {
  using CF = SweepCfg<CPL>;
  constexpr int P = CF::P, NW = CF::NW, Dp = CF::Dp, R = CF::R, SL = CF::kSlot;
  constexpr uint32_t kMsgBytes = SL * 4;            // one exchanged vector: 8 lanes x (NW + 1) words
  extern __shared__ __align__(128) uint8_t smem[];
  const int W = a.k.W, H = a.k.H, strip = a.strip;
  const int rank = blockIdx.x, ncta = gridDim.x;   // the cluster spans grid.x
  const bool up = blockIdx.y != 0;
  const int f = blockIdx.z;
  // a skipped frame: every CTA of the cluster (one frame) returns before any copy or barrier
  if (gated_off(a.gate ? a.gate + f : nullptr, a.k.gate_run)) return;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, grp = lane / kGL, lig = lane % kGL;
  const int nwarp = blockDim.x >> 5, ng = kGW * nwarp, gi = warp * kGW + grp;
  const int x_cta = rank * strip;
  const int npx = min(strip, W - x_cta);           // >= 1: the cluster has ceil(W / strip) CTAs
  const int xg = x_cta + gi * P;                   // the group's first pixel
  uint8_t *ring = smem;
  // mbarriers: R ring stages, the row barrier of the CTA, and the four
  // message barriers [dir][parity] of the vectors that arrive from the
  // neighbouring CTAs (dir 0: into group 0 from the left, dir 1: into the
  // last group from the right)
  uint64_t *bars = reinterpret_cast<uint64_t *>(smem + R * strip * Dp);
  uint64_t *rowbar = bars + R;
  uint64_t *rx = bars + R + 1;
  // exchange slots [dir][parity][group]: four words a lane at a time
  // ([word / 4][lane][word % 4]), then the lanes' minima
  uint32_t *slots = reinterpret_cast<uint32_t *>(bars + CF::kBars);
  const uint8_t *cost = a.cost + f * frame_cells(a.k);
  // this frame's sums, 2 Dp bytes per pixel
  uint8_t *sum_f = a.sum[up ? 1 : 0] + f * frame_cells(a.k) * 2;

  if (threadIdx.x == 0) {
    for (int s = 0; s < R; ++s) mbar_init(&bars[s], 1);
    mbar_init(rowbar, (uint32_t)nwarp);             // one arrival per warp and row
    for (int i = 0; i < 4; ++i) mbar_init(&rx[i], 1);   // the receiver's expect_tx arrival
    mbar_fence_init();
  }
  __syncthreads();
  int issued = 0;                                  // thread 0: rows whose copy was issued
  auto issue = [&](int t) {
    const int y = up ? H - 1 - t : t;
    mbar_expect_tx(&bars[t % R], (uint32_t)(npx * Dp));
    bulk_g2s(ring + (size_t)(t % R) * strip * Dp, cost + ((size_t)y * W + x_cta) * Dp, (uint32_t)(npx * Dp),
             &bars[t % R]);
    issued = t + 1;
  };
  if (threadIdx.x == 0) {
    issue(0);
    if (H > 1) issue(1);
  }
  // every CTA of the cluster runs, its barriers initialised, before the first remote store
  cluster_arrive();
  cluster_wait();

  uint32_t z[CPL / 4];
  pad_bytes<CPL>(a.k.D, lig, z);
  const Edges none = no_neighbours(lig);
  const StepConsts sc = a.sc;
  // path-cost vectors of the group's pixels and their minima: vertical,
  // from-left diagonal (predecessor x - 1), from-right diagonal (x + 1)
  uint32_t V[P][NW], DL[P][NW], DR[P][NW];
  uint32_t mV[P], mL[P], mR[P];
#pragma unroll
  for (int i = 0; i < P; ++i) {
#pragma unroll
    for (int w = 0; w < NW; ++w) V[i][w] = DL[i][w] = DR[i][w] = 0u;
    mV[i] = mL[i] = mR[i] = 0u;
  }
  // where this group's two outgoing vectors go: the neighbouring groups'
  // slots, in this CTA (plain stores) or, for the strip's end groups, in the
  // neighbouring CTA (st.async, completing on that CTA's message barrier)
  auto slot = [&](int dir, int par, int g) { return slots + ((dir * 2 + par) * ng + g) * SL; };
  const bool remote_r = gi == ng - 1, remote_l = gi == 0;
  const bool send_r = !remote_r || rank + 1 < ncta, send_l = !remote_l || rank > 0;
  const uint32_t rk_r = remote_r && send_r ? rank + 1 : rank, rk_l = remote_l && send_l ? rank - 1 : rank;
  const int g_r = remote_r ? 0 : gi + 1, g_l = remote_l ? ng - 1 : gi - 1;
  // vectors that arrive from another CTA: group 0 from the left, the last group from the right
  const bool recv_l = gi == 0 && rank > 0, recv_r = gi == ng - 1 && rank + 1 < ncta;
  auto put = [&](int dir, int par, bool remote, int g, uint32_t rk, const uint32_t(&v)[NW], uint32_t m) {
    uint32_t *d = slot(dir, par, g);
    if (remote) {
      const uint32_t base = cluster_map(smem_u32(d), rk), mb = cluster_map(smem_u32(&rx[dir * 2 + par]), rk);
#pragma unroll
      for (int q = 0; q < NW / 4; ++q)
        st_async4(base + q * 128 + lig * 16, v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3], mb);
      st_async(base + NW * 32 + lig * 4, m, mb);
    } else {
#pragma unroll
      for (int q = 0; q < NW / 4; ++q)
        reinterpret_cast<uint4 *>(d)[q * 8 + lig] = make_uint4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
      d[NW * 8 + lig] = m;
    }
  };
  auto get = [&](int dir, int par, uint32_t(&v)[NW], uint32_t &m) {
    const uint32_t *d = slot(dir, par, gi);
#pragma unroll
    for (int q = 0; q < NW / 4; ++q) {
      const uint4 t = reinterpret_cast<const uint4 *>(d)[q * 8 + lig];
      v[4 * q] = t.x, v[4 * q + 1] = t.y, v[4 * q + 2] = t.z, v[4 * q + 3] = t.w;
    }
    m = d[NW * 8 + lig];
  };
  // path starts at the image border: pixel 0's left predecessor is x = -1
  // at the strip of x = 0; a pixel's right predecessor x + 1 = W does not exist
  const uint32_t keep_in_l = xg == 0 ? 0u : 0xffffffffu;
  // warps whose groups touch neither border need none of the masks below
  const bool plain = __all_sync(kAll, xg > 0 && xg + P < W);
  // one Eq. 2 step from predecessor (pr, mp) on costs Cc: the new vector.  Its
  // min follows, two vectors at a time (one pass of shuffles for both: 32 frames
  // of 1242 x 375, D = 128 3.08 -> 3.00 ms)
  auto move = [&](uint32_t(&o)[NW], const uint32_t(&pr)[NW], uint32_t mp, const uint32_t(&Cc)[NW]) {
    copy_words<NW>(o, pr);
    step<NW, false, (NW < 8)>(o, Cc, mp, sc, none);
  };
  bool ok = true;
  auto bounded = [&](uint64_t *bar, uint32_t parity) {
    if (!mbar_wait_bounded(bar, parity, kWaitLimit)) {
      set_error(a.err, kErrTimeout);
      ok = false;
    }
  };
  // the warp's sum staging buffers (kBulkSums), after the slots, 128-byte aligned
  uint8_t *wsum = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(slots + 2 * 2 * ng * SL) + 127) &
                                              ~uintptr_t(127)) +
                  (size_t)warp * 2 * CF::kSumBuf;
  const int xw = x_cta + warp * kGW * P;                 // the warp's first pixel
  const int nvw = max(0, min(kGW * P, W - xw));          // its pixels inside the image

  for (int t = 0; t < H; ++t) {
    bounded(&bars[t % R], (uint32_t)(t / R) & 1u);
    const uint8_t *st = ring + (size_t)(t % R) * strip * Dp + gi * P * Dp + lig * Vec8<CPL>::kLane;
    const int y = up ? H - 1 - t : t;
    uint32_t C0[NW], CP[NW];
    load_u8<CPL>(st, z, C0);
    load_u8<CPL>(st + (P - 1) * Dp, z, CP);
    // the two vectors this group sends: from-left of its last pixel (from
    // its own pixel P-2), from-right of its first pixel (from its pixel 1)
    uint32_t eL[NW], eR[NW], meL, meR;
    {
      uint32_t pr[NW], mpr = mR[1];
      copy_words<NW>(pr, DR[1]);
      if (!plain) {
        const uint32_t kr = xg + 1 < W ? 0xffffffffu : 0u;   // pixel 0's right predecessor inside
#pragma unroll
        for (int w = 0; w < NW; ++w) pr[w] &= kr;
        mpr &= kr;
      }
      move(eL, DL[P - 2], mL[P - 2], CP);
      move(eR, pr, mpr, C0);
      group_min2<NW>(eL, eR, meL, meR);
    }
    // the vectors entering this group from the previous row
    uint32_t inL[NW], inR[NW], minL = 0u, minR = 0u;
#pragma unroll
    for (int w = 0; w < NW; ++w) inL[w] = inR[w] = 0u;
    if (t > 0) {
      const int par = (t - 1) & 1;
      // every warp of the CTA has stored row t - 1's vectors (and finished row t - 2)
      bounded(rowbar, (uint32_t)(t - 1) & 1u);
      if (recv_l || recv_r) {
        uint64_t *mb = &rx[(recv_l ? 0 : 1) * 2 + par];
        if (lig == 0) mbar_expect_tx(mb, kMsgBytes);
        bounded(mb, (uint32_t)((t - 1) >> 1) & 1u);
      }
      get(0, par, inL, minL);
      get(1, par, inR, minR);
    }
    // the ring stage of row t - 2 is free: every warp finished that row before its row t - 1 arrival
    // (row t - 1 may still be read), so rows up to t - 2 + R may be on their way
    if (threadIdx.x == 0 && issued < H && issued <= t - 2 + R) issue(issued);
    if (t + 1 < H) {
      // row t's outgoing vectors (the last row's have no reader)
      const int par = t & 1;
      if (send_r) put(0, par, remote_r, g_r, rk_r, eL, meL);
      if (send_l) put(1, par, remote_l, g_l, rk_l, eR, meR);
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(rowbar);
    // the rest of the row
    if (!plain) {
      const uint32_t kl = keep_in_l, kr = xg + P < W ? 0xffffffffu : 0u;
#pragma unroll
      for (int w = 0; w < NW; ++w) {
        inL[w] &= kl;
        inR[w] &= kr;
      }
      minL &= kl;
      minR &= kr;
    }
    uint32_t carry[NW], mcarry = mL[0];
    copy_words<NW>(carry, DL[0]);
    move(DL[0], inL, minL, C0);
#pragma unroll
    for (int i = 0; i < P; ++i) {
      uint32_t C[NW];
      if (i == 0)
        copy_words<NW>(C, C0);
      else if (i == P - 1)
        copy_words<NW>(C, CP);
      else
        load_u8<CPL>(st + i * Dp, z, C);
      move(V[i], V[i], mV[i], C);
      if (i >= 1 && i <= P - 2) {
        uint32_t nxt[NW];
        const uint32_t mnxt = mL[i];
        copy_words<NW>(nxt, DL[i]);
        move(DL[i], carry, mcarry, C);
        group_min2<NW>(V[i], DL[i], mV[i], mL[i]);
        copy_words<NW>(carry, nxt);
        mcarry = mnxt;
        uint32_t pr[NW], mpr = mR[i + 1];
        copy_words<NW>(pr, DR[i + 1]);
        if (!plain) {
          const uint32_t ki = xg + i + 1 < W ? 0xffffffffu : 0u;
#pragma unroll
          for (int w = 0; w < NW; ++w) pr[w] &= ki;
          mpr &= ki;
        }
        move(DR[i], pr, mpr, C);
        if (i % 2 == 0) group_min2<NW>(DR[i - 1], DR[i], mR[i - 1], mR[i]);   // (i = 1 waits for i = 2)
      } else if (i == 0) {
        group_min2<NW>(V[0], DL[0], mV[0], mL[0]);
        copy_words<NW>(DR[0], eR);
        mR[0] = meR;
      } else {
        copy_words<NW>(DL[P - 1], eL);
        mL[P - 1] = meL;
        move(DR[P - 1], inR, minR, C);
        group_min2<NW>(V[P - 1], DR[P - 1], mV[P - 1], mR[P - 1]);
      }
      uint32_t sum[NW];
#pragma unroll
      for (int w = 0; w < NW; ++w) sum[w] = V[i][w] + DL[i][w] + DR[i][w];
      [[maybe_unused]] const int x = xg + i;
      if constexpr (CF::kBulkSums)   // into the row's staging buffer (pixels outside the image are not copied out)
        store_u16<CPL>(wsum + (t & 1) * CF::kSumBuf + (grp * P + i) * Dp * 2 + lig * Vec16<CPL>::kLane, sum);
      else if (ok && x < W)
        store_u16<CPL>(sum_f + ((size_t)y * W + x) * Dp * 2 + lig * Vec16<CPL>::kLane, sum);
    }
    if constexpr (CF::kBulkSums) {
      // the row's sums of the warp's pixels: one bulk copy from the staging
      // buffer; the buffer of row t - 1 has been read before row t + 1 reuses it
      fence_proxy_async_shared();
      __syncwarp();
      if (lane == 0) {
        if (ok && nvw > 0)
          bulk_s2g(sum_f + ((size_t)y * W + xw) * Dp * 2, wsum + (t & 1) * CF::kSumBuf, (uint32_t)(nvw * Dp * 2));
        bulk_commit();
        bulk_wait_read_all_but_one();
      }
      __syncwarp();
    }
  }
  if constexpr (CF::kBulkSums) {
    if (lane == 0) bulk_wait_all();
  }
  // every message was waited for by its receiver; the cluster barrier keeps
  // every CTA (and its shared memory) alive until all are done
  cluster_arrive();
  cluster_wait();
  if (threadIdx.x == 0 && !ok) {
    for (int h = max(0, issued - R); h < issued; ++h)
      mbar_wait_bounded(&bars[h % R], (uint32_t)(h / R) & 1u, kWaitLimit);
  }
}

// Warps per CTA when a row of W pixels is split over `ctas` CTAs, or 0 when
// that split is not allowed (a CTA above kMaxWarps, or an empty last CTA).
template <int CPL>
inline int sweep_warps(int W, int ctas) {
  using CF = SweepCfg<CPL>;
  if (ctas < 1 || ctas > CF::kMaxCluster) return 0;
  const int warps = (W + ctas * kGW * CF::P - 1) / (ctas * kGW * CF::P);
  if (warps > CF::kMaxWarps || (ctas - 1) * kGW * warps * CF::P >= W) return 0;
  return warps;
}

template <int CPL>
static cudaLaunchConfig_t sweep_config(int nf, int ctas, int warps, cudaStream_t s, cudaLaunchAttribute *attr) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(ctas, 2, nf);
  cfg.blockDim = dim3(32 * warps);
  cfg.dynamicSmemBytes = SweepCfg<CPL>::smem_bytes(warps);
  cfg.stream = s;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = ctas;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cfg;
}

// kernel attributes (once per device): the dynamic shared memory and cluster
// sizes above the portable 8
template <int CPL>
static cudaError_t sweep_attributes() {
  static bool done[64] = {};
  return once_per_device(done, [](int) {
    cudaError_t e = cudaFuncSetAttribute(k_sweep<CPL>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         SweepCfg<CPL>::smem_bytes(SweepCfg<CPL>::kMaxWarps));
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(k_sweep<CPL>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    return e;
  });
}

// The cluster size (CTAs per cluster) for the sweep of a context that runs
// up to nb frames per call, or 0 when it cannot run (8 paths, rows of at most
// kMaxRow pixels).  A call is 2 nb cluster jobs of H rows each; with n clusters resident at once it takes ceil(2 nb / n) waves, and a row takes
// time in proportion to the pixels of one CTA (one CTA per SM).  Among the
// sizes from the smallest that holds a row up to twice that (at most 16) the
// one with the fewest waves x pixels per CTA (ties: the smaller cluster).
template <int CPL>
int sweep_plan_t(const KParams &k, int nb, int *slots) {
  using CF = SweepCfg<CPL>;
  if (k.num_paths != 8) return 0;
  const int lo = (k.W + kGW * CF::kMaxWarps * CF::P - 1) / (kGW * CF::kMaxWarps * CF::P);
  if (k.W > CF::kMaxRow || lo > CF::kMaxCluster || sweep_attributes<CPL>() != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  int best = 0, best_n = 0;
  long best_cost = 0;
  for (int cs = lo; cs <= min(CF::kMaxCluster, 2 * lo); ++cs) {
    const int warps = sweep_warps<CPL>(k.W, cs);
    if (warps == 0) continue;
    cudaLaunchAttribute attr[1];
    cudaLaunchConfig_t cfg = sweep_config<CPL>(1, cs, warps, nullptr, attr);
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, k_sweep<CPL>, &cfg) != cudaSuccess) {
      cudaGetLastError();
      continue;
    }
    if (n < 1) continue;
    const long cost = (long)((2 * nb + n - 1) / n) * (kGW * warps * CF::P);
    if (best == 0 || cost < best_cost) {
      best_cost = cost;
      best = cs;
      best_n = n;
    }
  }
  if (slots != nullptr) *slots = best_n;
  return best;
}

template <int CPL>
cudaError_t launch_sweep_t(const KParams &k, const Buffers &b, int nf, cudaStream_t s) {
  using CF = SweepCfg<CPL>;
  const int ctas = k.sweep_cs, warps = sweep_warps<CPL>(k.W, ctas);
  if (warps == 0) return cudaErrorInvalidValue;
  cudaError_t e = sweep_attributes<CPL>();
  if (e != cudaSuccess) return e;
  SweepArgs a;
  a.k = k;
  a.cost = b.cost;
  a.sum[0] = reinterpret_cast<uint8_t *>(b.part[0]);
  a.sum[1] = reinterpret_cast<uint8_t *>(b.part[1]);
  a.err = b.err;
  a.gate = b.gate;
  a.sc = step_consts(k);
  a.strip = kGW * warps * CF::P;
  cudaLaunchAttribute attr[1];
  cudaLaunchConfig_t cfg = sweep_config<CPL>(nf, ctas, warps, s, attr);
  return cudaLaunchKernelEx(&cfg, k_sweep<CPL>, a);
}

}  // namespace oct
}  // namespace sgmf

// explicit instantiations of one lane width (CPL cells per lane)
#define SGMF_AGG_INSTANTIATE(CPL)                                                                              \
  namespace sgmf {                                                                                             \
  namespace oct {                                                                                              \
  template cudaError_t launch_lines_t<CPL, false>(const KParams &, const Buffers &, int, cudaStream_t);        \
  template cudaError_t launch_lines_t<CPL, true>(const KParams &, const Buffers &, int, cudaStream_t);         \
  template cudaError_t launch_rows_t<CPL, false>(const KParams &, const Buffers &, int, cudaStream_t);         \
  template cudaError_t launch_rows_t<CPL, true>(const KParams &, const Buffers &, int, cudaStream_t);          \
  template cudaError_t launch_wta_t<CPL, false>(const KParams &, const Buffers &, int, int16_t *, cudaStream_t); \
  template cudaError_t launch_wta_t<CPL, true>(const KParams &, const Buffers &, int, int16_t *, cudaStream_t); \
  template cudaError_t launch_sweep_t<CPL>(const KParams &, const Buffers &, int, cudaStream_t);               \
  template int sweep_plan_t<CPL>(const KParams &, int, int *);                                                 \
  }                                                                                                            \
  }
