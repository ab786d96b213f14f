// W4A16 MSD linear layer with few tokens (per weight matrix): decode layers and mixture-of-experts blocks.
//
// Operands are swapped against the many-row kernels of gemm_w4a16.cu: a band of up to 128 weight rows is the MMA A operand, the
// stacked components [Q1; Q2] (NB = 2 ceil8(tokens) rows) are B, and the two passes land in different columns of one accumulator,
// so a weight tile passes the tensor core once and an MMA costs what its tokens are worth.
//
// Bound: HBM for experts (32 of 2048 x 7168, 512 tokens: 53 us, 4.8 TB/s), the chain of two kernels for single layers (16 tokens, 4096 x 14336
// and back: 11.2 and 12.6 us for 31 MB each).  With tiles of 128 token rows, padded and once per component, a 256 x 256 weight stage
// took 0.65 us of tensor time where HBM needs 0.8 for all SMs: 68 and 32 us for the two.  With about 64 tokens and more the components,
// brought once per band, outweigh the weights and those tiles are the shorter way again.
#include <cuda_bf16.h>

#include <cmath>
#include <mutex>

#include "host_common.h"
#include "sm100.cuh"

namespace msd {

constexpr int kDecThreads = 384;                  // weight producer, MMA issuer, four epilogue warps, four scale warps, component and scale producers
constexpr int kDecBoxes = 4;                      // heights of component boxes in a grouped launch
constexpr int kDecBlockK = 256;                   // elements per K block (128 packed bytes, one swizzle row)
constexpr int kDecMaxStages = 16;
constexpr int kDecMaxSets = 4;
constexpr int kDecStoreBytes = 2 * 16 * 128 * 4;  // epilogue staging: two buffers of [16 tokens][128 rows] FP32
constexpr int kDecSmem = 227 * 1024 - 2048;
// Least shared memory of a CTA that waits for others (K split over a cluster).  Every CTA takes all of its SM's tensor memory, and the wait
// for that has no limit: of two such CTAs on one SM the second would wait for the first to end, the first at a cluster barrier
// for the peers of the second or for the second itself.  With more than half of an SM's 228 KB each (1 KB of it the system's) there is
// only one of them, and none beside a CTA of the other kernels whose CTAs wait for one another, which take 160 KB and more.
constexpr int kDecClusterSmem = 116 * 1024;
static_assert(2 * (kDecClusterSmem + 1024) > 228 * 1024, "two CTAs of a cluster would fit one SM");
constexpr int kDecTmemCols = 512;

struct W4DecodeParams {
  int M, NB, N;                 // tokens (ungrouped), most stacked component rows of a group, weight rows of a matrix
  int h, bands, items;          // weight rows per band, bands per matrix, bands of all groups
  int kblocks, kw, ksteps;      // 256-element K blocks, of which a stage holds kw; stages that cover K
  int S, kper;                  // CTAs per band (a cluster) and stages each takes
  int nstages, stage_bytes, x_off, sf_off;      // pipeline, and where a stage's components and scales lie
  int nsfx;                     // 128-row scale blocks of the stacked components (1 or 2)
  int t3;                       // the kw boxes of a stage travel as one 3-D box (K % 256 == 0)
  int early;                    // stages whose weights are asked for before the decomposition has ended
  int nacc, sf_col, set_cols;   // accumulators; first scale column, columns of a set of them
  int nsets;                    // sets of scale columns: stages whose scales are in tensor memory (2 or 4)
  int epi_off;
  int sf_kgroups, row_blocks;   // blocked weight scales: 128-element K groups per row, 128-row blocks per matrix
  const uint8_t* sfw;
  const uint8_t* sfx;
  int sfw_ready;                // sfw was laid out before this call
  void* y;
  int ytype;
  unsigned* status;
};
// Component boxes: in a grouped launch of a quarter, half, three quarters and all of NB rows, of which a group loads the smallest that
// holds its own (32 experts of 2048 x 7168, 6 to 35 tokens each: 51.1 us with one, 49.5 with four).
template <bool kGrouped> struct W4DecodeXMaps { CUtensorMap m[kGrouped ? kDecBoxes : 1]; };
__host__ __device__ inline int w4d_box_rows(int NB, int i) { return (NB * (i + 1) / kDecBoxes + 15) / 16 * 16; }

// Stores `wt` tokens of a band, given as [16][128] values in shared memory, to y rows y_row0 ...; 128 threads, 16-byte vectors.
template <typename OutT>
__device__ __forceinline__ void w4d_store_rows(const OutT* stage, OutT* y, int N, int n0, int rows, int64_t y_row0, int wt, int et) {
  constexpr int kVec = 16 / static_cast<int>(sizeof(OutT)), kSegs = 128 / kVec;
  const int nf = (et % kSegs) * kVec;
  if (nf >= rows) return;                          // (rows is a multiple of 8)
  for (int j = et / kSegs; j < wt; j += 128 / kSegs)
    *reinterpret_cast<uint4*>(y + (y_row0 + j) * N + n0 + nf) = *reinterpret_cast<const uint4*>(stage + j * 128 + nf);
}
template <bool kBf16>
__device__ __forceinline__ void w4d_stage_value(uint8_t* buf, int j, int r, float v) {
  if constexpr (kBf16) reinterpret_cast<__nv_bfloat16*>(buf)[j * 128 + r] = __float2bfloat16_rn(v);
  else reinterpret_cast<float*>(buf)[j * 128 + r] = v;
}

template <bool kGrouped>
__global__ void __launch_bounds__(kDecThreads, 1)
gemm_w4a16_decode_kernel(const __grid_constant__ CUtensorMap tmap_w, const __grid_constant__ W4DecodeXMaps<kGrouped> tmap_x, const W4DecodeParams p,
                         const __grid_constant__ typename W4GroupArg<kGrouped>::type grp) {
  extern __shared__ uint8_t smem_dyn[];
  __shared__ __align__(8) uint64_t full_bar[kDecMaxStages], empty_bar[kDecMaxStages], tfull_bar[2], tempty_bar[2];
  __shared__ __align__(8) uint64_t sf_ready[kDecMaxSets], sf_free[kDecMaxSets];
  __shared__ uint32_t tmem_base_slot;
  __shared__ int abort_flag;

  const int warp = __shfl_sync(0xffffffffu, static_cast<int>(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
  if (p.nstages < 1 || p.kw < 1 || p.kper < 1) return;                  // malformed plan: touch nothing
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_dyn) + 1023) & ~static_cast<uintptr_t>(1023));
  const int S = kGrouped ? 1 : p.S;
  const int rank = S > 1 ? static_cast<int>(cluster_ctarank()) : 0;
  const int item0 = S > 1 ? static_cast<int>(cluster_id()) : static_cast<int>(blockIdx.x);
  const int item_step = S > 1 ? p.items : static_cast<int>(gridDim.x);     // (a cluster has one item)
  const int ks0 = rank * p.kper, ks1 = min(ks0 + p.kper, p.ksteps);

  // Stacked component rows of an item's group: two components of ceil8(tokens) rows, and the rows of the box that brings them.
  struct Rows { int Mp, NB, box, box_rows; };
  auto rows_of = [&](int item) {
    Rows r = {p.NB >> 1, p.NB, 0, p.NB};
    if constexpr (kGrouped) {
      const int g = item / p.bands;
      r.Mp = (grp.off[g + 1] - grp.off[g] + 7) & ~7;
      r.NB = 2 * r.Mp;
      r.box = 0;
      while ((r.box_rows = w4d_box_rows(p.NB, r.box)) < r.NB) ++r.box;
    }
    return r;
  };
  // Where an item's operands lie; ks counts stages.
  struct Pos { int item, ks, w_row, x_row, rb, need2, sfx_off; Rows rows; };
  auto enter = [&](Pos& q) {
    int g = 0, band = q.item, e = 0;
    if constexpr (kGrouped) { g = q.item / p.bands; band = q.item - g * p.bands; e = grp.expert[g]; }
    q.ks = ks0;
    const int row0 = band * p.h;
    q.w_row = e * p.N + row0;
    q.x_row = g * p.NB;
    q.rb = row0 >> 7;
    q.need2 = (row0 & 127) + p.h > 128 && q.rb + 1 < p.row_blocks;
    q.rb += e * p.row_blocks;
    q.sfx_off = g * p.nsfx;
    q.rows = rows_of(q.item);
  };
  auto advance = [&](Pos& q) {
    if (++q.ks < ks1) return;
    q.item += item_step;
    if (q.item < p.items) enter(q);
  };
  auto valid_blocks = [&](int ks) { return min(p.kw, p.kblocks - ks * p.kw); };
  uint64_t pol_w = 0, pol_x = 0;
  // Three producer warps (a copy costs its thread 50 to 100 ns, and a freed stage waits for all of its copies to be issued one after the
  // other): 0 the weights, 10 the components, 11 the scale blocks, lanes 0 and 1 the weights' and 2 and 3 the components'.
  // 32 experts of 2048 x 7168, 16 tokens each: 53.7 us, 61.1 with one warp issuing them all.
  auto load_w = [&](const Pos& q, int stage) {
    const int v = valid_blocks(q.ks);
    if (lane == 0)
      mbar_arrive_expect_tx(&full_bar[stage], static_cast<uint32_t>((p.t3 ? p.kw : v) * (p.h + q.rows.box_rows) * 128 + v * 1024 * (1 + q.need2 + p.nsfx)));
    __syncwarp();
    uint8_t* dst = smem + stage * p.stage_bytes;
    if (p.t3) {
      if (lane == 0) tma_load_3d_hint(dst, &tmap_w, 0, q.w_row, q.ks * p.kw, &full_bar[stage], pol_w);
    } else if (lane < v) {
      tma_load_2d_hint(dst + lane * p.h * 128, &tmap_w, (q.ks * p.kw + lane) * 128, q.w_row, &full_bar[stage], pol_w);
    }
  };
  // (the bytes of these two may be counted before warp 0's arrival announces them: the phase cannot end without it)
  auto load_x = [&](const Pos& q, int stage) {
    uint8_t* dst = smem + stage * p.stage_bytes + p.x_off;
    if (p.t3) {
      if (lane == 0) tma_load_3d_hint(dst, &tmap_x.m[q.rows.box], 0, q.x_row, q.ks * p.kw, &full_bar[stage], pol_x);
    } else if (lane < valid_blocks(q.ks)) {
      tma_load_2d_hint(dst + lane * q.rows.box_rows * 128, &tmap_x.m[q.rows.box], (q.ks * p.kw + lane) * 128, q.x_row, &full_bar[stage], pol_x);
    }
  };
  auto load_sf = [&](const Pos& q, int stage, bool w, bool x) {
    const bool mine = lane < 2 ? w && lane <= q.need2 : x && lane < 2 + p.nsfx;
    if (mine) {
      const uint8_t* base = lane < 2 ? p.sfw : p.sfx;
      const int block = lane < 2 ? q.rb + lane : q.sfx_off + lane - 2;
      bulk_load(smem + stage * p.stage_bytes + p.sf_off + lane * p.kw * 1024, base + (static_cast<size_t>(block) * p.sf_kgroups + 2 * q.ks * p.kw) * 512,
                valid_blocks(q.ks) * 1024, &full_bar[stage]);
    }
  };

  Pos q = {}, first = {};
  int pre = 0;
  const bool producer = warp == 0 || warp == 10 || warp == 11;
  if (warp == 0) {
    if (lane < p.nstages) { mbar_init(&full_bar[lane], 1); mbar_init(&empty_bar[lane], 1); }
    if (lane >= 16 && lane < 18) { mbar_init(&tfull_bar[lane - 16], 1); mbar_init(&tempty_bar[lane - 16], 4); }
    if (lane >= 20 && lane < 20 + kDecMaxSets) { mbar_init(&sf_ready[lane - 20], 4); mbar_init(&sf_free[lane - 20], 1); }
    if (lane == 18) abort_flag = 0;
    mbar_init_fence();
    __syncwarp();
    pol_w = policy_evict_first();
  } else if (warp == 2 && lane < (kGrouped ? kDecBoxes : 1)) {
    tma_prefetch_desc(&tmap_x.m[lane]);
  }
  if (producer) {
    pol_x = policy_evict_last();
    q.item = item0;
    enter(q);
    first = q;
    // the first stages' weights are asked for before the rest of the CTA's set-up
    if (warp == 0)
      for (; pre < p.early && q.item < p.items; ++pre) { load_w(q, pre); advance(q); }
  }
  if (warp == 1) tmem_alloc(&tmem_base_slot, kDecTmemCols);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = tmem_base_slot;
  volatile int* abort = &abort_flag;

  if (producer) {
    if (warp == 11 && p.sfw_ready)
      for (; pre < p.early && q.item < p.items; ++pre) { load_sf(q, pre, true, false); advance(q); }
    // what the kernel launched just before writes: the components, their scales and weight scales that did not come prepared
    pdl_wait_primary();
    if (warp == 11) {
      q = first;
      for (int i = 0; i < pre; ++i) { load_sf(q, i, false, true); advance(q); }
    }
    int stage = pre == p.nstages ? 0 : pre;
    uint32_t phase = pre == p.nstages ? 1 : 0;
    bool ok = true;
    while (q.item < p.items) {
      ok = wait_bounded_warp(&empty_bar[stage], phase ^ 1, abort, p.status);
      if (!ok) break;
      if (warp == 0) load_w(q, stage);
      else if (warp == 10) load_x(q, stage);
      else load_sf(q, stage, true, true);
      advance(q);
      if (++stage == p.nstages) { stage = 0; phase ^= 1; }
    }
    if (!ok) {                     // copies in flight get a bounded time to land before the CTA goes away
      const long long t0 = clock64();
      while (clock64() - t0 < 2000000LL) {}
    }
  } else if (warp == 1) {
    int stage = 0, it = 0, set = 0;
    uint32_t phase = 0, set_phase = 0;
    bool ok = true;
    const uint64_t op_desc = smem_desc(0, 16, 1024, kSwizzle128B);
    const int w_blk = p.h * 8, x_off = p.x_off >> 4;       // in 16-byte units, as descriptors count
    for (int item = item0; item < p.items && ok; item += item_step, ++it) {
      const Rows rows = rows_of(item);
      const uint32_t idesc_lo = idesc_block_scaled(/*E2M1*/ 1, 1, 128, rows.NB, 0, 0), idesc_hi = idesc_block_scaled(1, 1, 128, rows.NB, 2, 2);
      const int x_blk = rows.box_rows * 8;
      const int acc = p.nacc == 2 ? (it & 1) : 0;
      const uint32_t tphase = p.nacc == 2 ? ((it >> 1) & 1) : (it & 1);
      const uint32_t d_tmem = tmem_base + acc * p.NB;
      ok = wait_bounded_warp(&tempty_bar[acc], tphase ^ 1, abort, p.status);
      if (!ok) break;
      tc_fence_after();
      for (int ks = ks0; ks < ks1; ++ks) {
        ok = wait_bounded_warp(&full_bar[stage], phase, abort, p.status) && wait_bounded_warp(&sf_ready[set], set_phase, abort, p.status);
        if (!ok) break;
        tc_fence_after();
        // (the MMA reads 128 rows from where a band's box starts; what it finds past the band ends up in rows that are not stored)
        uint64_t wd = op_desc + static_cast<uint64_t>(smem_u32(smem + stage * p.stage_bytes) >> 4), xd = wd + x_off;
        uint32_t sfw_t = tmem_base + p.sf_col + set * p.set_cols, sfx_t = sfw_t + 8 * p.kw;
        const int v = valid_blocks(ks);
        for (int c = 0; c < v; ++c) {
#pragma unroll
          for (int kk = 0; kk < 4; ++kk)           // 64 elements (32 bytes) per MMA
            mma_mxf4_warp(d_tmem, wd + 2 * kk, xd + 2 * kk, (kk & 1) ? idesc_hi : idesc_lo, sfw_t + 4 * (kk >> 1), sfx_t + 4 * p.nsfx * (kk >> 1),
                          (ks > ks0 || c > 0 || kk > 0) ? 1u : 0u);
          wd += w_blk; xd += x_blk;
          sfw_t += 8; sfx_t += 8 * p.nsfx;
        }
        tc_commit_warp(&sf_free[set]);
        tc_commit_warp(&empty_bar[stage]);
        if (++set == p.nsets) { set = 0; set_phase ^= 1; }
        if (++stage == p.nstages) { stage = 0; phase ^= 1; }
      }
      if (!ok) break;
      tc_commit_warp(&tfull_bar[acc]);
    }
  } else if (warp >= 6) {      // (warps 10 and 11 went the producers' way above)
    // Scale warps.  TMEM lane l of every quadrant holds, in column j of a K group, the four scales of row l + 32 j.  A band starts
    // at any multiple of 8 rows, a 512-byte block at a multiple of 128: rows are looked up one by one (row r of the band is row
    // (row0 % 128) + r of the one or two blocks loaded).
    const int quad = warp & 3;
    int stage = 0, set = 0;
    uint32_t phase = 0, set_phase = 0;
    bool ok = true;
    for (int item = item0; item < p.items && ok; item += item_step) {
      int band = item;
      if constexpr (kGrouped) band = item % p.bands;
      int w_at[4];                    // byte offsets of this lane's four rows in the weight scales of a K group
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int r = ((band * p.h) & 127) + lane + 32 * j;
        w_at[j] = (r >> 7) * p.kw * 1024 + (r & 31) * 16 + ((r >> 5) & 3) * 4;
      }
      for (int ks = ks0; ks < ks1; ++ks) {
        // (a set's first use waits for the phase before the first, which counts as complete)
        ok = wait_bounded(&full_bar[stage], phase, abort, p.status) && wait_bounded(&sf_free[set], set_phase ^ 1, abort, p.status);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        tc_fence_after();
        const uint8_t* sf = smem + stage * p.stage_bytes + p.sf_off;
        const uint32_t col = tmem_base + (static_cast<uint32_t>(quad * 32) << 16) + p.sf_col + set * p.set_cols;
        const int v = valid_blocks(ks);
        for (int c = 0; c < v; ++c) {
          uint32_t s[8];
#pragma unroll
          for (int g = 0; g < 2; ++g)
#pragma unroll
            for (int j = 0; j < 4; ++j) s[4 * g + j] = *reinterpret_cast<const uint32_t*>(sf + (2 * c + g) * 512 + w_at[j]);
          tmem_st8(col + 8 * c, s);
          const uint4* x0 = reinterpret_cast<const uint4*>(sf + (2 * p.kw + c) * 1024) + lane;
          const uint4 a0 = x0[0], a1 = x0[32];
          if (p.nsfx == 1) {
            const uint32_t t[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
            tmem_st8(col + 8 * p.kw + 8 * c, t);
          } else {
            const uint4 b0 = x0[p.kw * 64], b1 = x0[p.kw * 64 + 32];
            const uint32_t t[16] = {a0.x, a0.y, a0.z, a0.w, b0.x, b0.y, b0.z, b0.w, a1.x, a1.y, a1.z, a1.w, b1.x, b1.y, b1.z, b1.w};
            tmem_st16(col + 8 * p.kw + 16 * c, t);
          }
        }
        tmem_st_wait();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&sf_ready[set]);
        if (++set == p.nsets) { set = 0; set_phase ^= 1; }
        if (++stage == p.nstages) { stage = 0; phase ^= 1; }
      }
    }
  }

  const int quad = warp & 3, r = quad * 32 + lane, et = static_cast<int>(threadIdx.x) - 64;
  const bool epi = warp >= 2 && warp < 6;
  const uint32_t t_lane = tmem_base + (static_cast<uint32_t>(quad * 32) << 16);
  if (S == 1) {
    if (epi) {
      int it = 0, buf = 0;
      bool ok = true;
      for (int item = item0; item < p.items && ok; item += item_step, ++it) {
        int band = item, tokens = p.M;
        int64_t y_row0 = 0;
        if constexpr (kGrouped) {
          const int g = item / p.bands;
          band = item - g * p.bands;
          y_row0 = grp.off[g];
          tokens = grp.off[g + 1] - grp.off[g];
        }
        const int acc = p.nacc == 2 ? (it & 1) : 0;
        const uint32_t tphase = p.nacc == 2 ? ((it >> 1) & 1) : (it & 1);
        ok = named_bar_and(1, 128, wait_bounded(&tfull_bar[acc], tphase, abort, p.status));
        if (!ok) break;
        tc_fence_after();
        const int n0 = band * p.h, rows = min(p.h, p.N - n0), Mp = (tokens + 7) & ~7;
        const uint32_t t_row = t_lane + acc * p.NB;
        for (int c0 = 0; c0 < tokens; c0 += 16, buf ^= 1) {
          uint32_t a[16], b[16];
          tmem_ld16(t_row + c0, a);
          tmem_ld16(t_row + Mp + c0, b);      // (a last chunk of 8 tokens reads columns beyond its own, never used)
          tmem_ld_wait();
          if (c0 + 16 >= tokens) {
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&tempty_bar[acc]);
          }
          uint8_t* sb = smem + p.epi_off + buf * (kDecStoreBytes / 2);
          const int wt = min(16, tokens - c0);
          if (p.ytype == MSD_OUT_BF16) {
#pragma unroll
            for (int j = 0; j < 16; ++j) w4d_stage_value<true>(sb, j, r, __uint_as_float(a[j]) + __uint_as_float(b[j]));
            named_bar_sync(1, 128);
            w4d_store_rows(reinterpret_cast<const __nv_bfloat16*>(sb), static_cast<__nv_bfloat16*>(p.y), p.N, n0, rows, y_row0 + c0, wt, et);
          } else {
#pragma unroll
            for (int j = 0; j < 16; ++j) w4d_stage_value<false>(sb, j, r, __uint_as_float(a[j]) + __uint_as_float(b[j]));
            named_bar_sync(1, 128);
            w4d_store_rows(reinterpret_cast<const float*>(sb), static_cast<float*>(p.y), p.N, n0, rows, y_row0 + c0, wt, et);
          }
        }
      }
    }
  } else {
    // K split inside the cluster.  Tokens in groups of four: rank f finishes the groups [f G / S, (f + 1) G / S).  Slot s of a CTA's
    // drained pipeline holds what rank s sent, [group][128 weight rows][4 tokens]: a warp's stores and loads are contiguous.
    const int G = (p.M + 3) >> 2, slot = ((G + S - 1) / S) * 2048;
    bool ok = true;
    if (epi) {
      ok = named_bar_and(1, 128, wait_bounded(&tfull_bar[0], 0, abort, p.status));
      tc_fence_after();
    }
    __syncwarp();
    cluster_arrive_all();                      // every CTA's pipeline is drained
    cluster_wait_all();
    if (epi && ok) {
      int f = 0;
      for (int g0 = 0; g0 < G; g0 += 4) {
        uint32_t a[16], b[16];
        __syncwarp();
        tmem_ld16(t_lane + 4 * g0, a);
        tmem_ld16(t_lane + (p.NB >> 1) + 4 * g0, b);
        tmem_ld_wait();
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int g = g0 + i;
          if (g >= G) break;
          while (g >= (f + 1) * G / S) ++f;
          if (r < p.h) {
            uint32_t v[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) v[j] = __float_as_uint(__uint_as_float(a[4 * i + j]) + __uint_as_float(b[4 * i + j]));
            st_cluster_v4(mapa_shared(smem_u32(smem) + static_cast<uint32_t>(rank * slot + (g - f * G / S) * 2048 + r * 16), f), v[0], v[1], v[2], v[3]);
          }
        }
      }
    }
    __syncwarp();
    cluster_arrive_all();                      // everything has been delivered
    cluster_wait_all();
    if (epi && ok) {
      const int g_begin = rank * G / S, g_end = (rank + 1) * G / S;
      const int n0 = item0 * p.h, rows = min(p.h, p.N - n0);
      int buf = 0;
      for (int g0 = g_begin; g0 < g_end; g0 += 4, buf ^= 1) {
        uint8_t* sb = smem + p.epi_off + buf * (kDecStoreBytes / 2);
        const int ng = min(4, g_end - g0);
        for (int i = 0; i < ng; ++i) {
          float4 acc = *reinterpret_cast<const float4*>(smem + (g0 + i - g_begin) * 2048 + r * 16);
          for (int s = 1; s < S; ++s) {
            const float4 v = *reinterpret_cast<const float4*>(smem + s * slot + (g0 + i - g_begin) * 2048 + r * 16);
            acc.x += v.x; acc.y += v.y; acc.z += v.z; acc.w += v.w;
          }
          const float o[4] = {acc.x, acc.y, acc.z, acc.w};
          if (p.ytype == MSD_OUT_BF16) {
#pragma unroll
            for (int j = 0; j < 4; ++j) w4d_stage_value<true>(sb, 4 * i + j, r, o[j]);
          } else {
#pragma unroll
            for (int j = 0; j < 4; ++j) w4d_stage_value<false>(sb, 4 * i + j, r, o[j]);
          }
        }
        named_bar_sync(1, 128);
        const int wt = min(4 * ng, p.M - 4 * g0);
        if (p.ytype == MSD_OUT_BF16) w4d_store_rows(reinterpret_cast<const __nv_bfloat16*>(sb), static_cast<__nv_bfloat16*>(p.y), p.N, n0, rows, 4 * g0, wt, et);
        else w4d_store_rows(reinterpret_cast<const float*>(sb), static_cast<float*>(p.y), p.N, n0, rows, 4 * g0, wt, et);
      }
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, kDecTmemCols);
  }
}

static bool w4_decode_attr() {
  static DeviceOnce once;
  return once([] {
    return cudaFuncSetAttribute(gemm_w4a16_decode_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kDecSmem) == cudaSuccess &&
           cudaFuncSetAttribute(gemm_w4a16_decode_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kDecSmem) == cudaSuccess;
  });
}

// How many clusters of S CTAs of the kernel the device holds at once, one CTA per SM as in every launch with clusters (0 on error).
static int w4_decode_clusters(int S) {
  static std::mutex mu;
  static int cache[64][9] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64 || S < 1 || S > 8 || !w4_decode_attr()) return 0;
  std::lock_guard<std::mutex> lock(mu);
  if (cache[dev][S]) return cache[dev][S];
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>(S) * 64);
  cfg.blockDim = dim3(kDecThreads);
  cfg.dynamicSmemBytes = kDecSmem;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = static_cast<unsigned>(S);
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, gemm_w4a16_decode_kernel<false>, &cfg) != cudaSuccess) { cudaGetLastError(); return 0; }
  return cache[dev][S] = n;
}

// What a choice of band height, stage width and K split comes to (groups 0: an ungrouped call).  False: it does not fit.
static bool w4_decode_layout(W4DecodeShape* d, int tokens, int groups, int64_t N, int64_t K, int h, int kw, int S) {
  d->h = h; d->kw = kw; d->S = S;
  d->Mp = (tokens + 7) / 8 * 8;
  d->NB = 2 * d->Mp;
  d->nsfx = d->NB > 128 ? 2 : 1;
  d->kblocks = static_cast<int>((K + kDecBlockK - 1) / kDecBlockK);
  if (h < 8 || h > 128 || h % 8 != 0 || kw < 1 || kw > 4 || kw > d->kblocks || S < 1 || S > (groups > 0 ? 1 : 8)) return false;
  d->ksteps = (d->kblocks + kw - 1) / kw;
  d->kper = (d->ksteps + S - 1) / S;
  d->bands = static_cast<int>((N + h - 1) / h);
  d->items = d->bands * (groups > 0 ? groups : 1);
  d->grid = S > 1 ? d->items * S : (d->items < sm_count() ? d->items : sm_count());
  d->x_off = kw * h * 128;
  d->sf_off = d->x_off + kw * d->NB * 128;
  d->stage_bytes = d->sf_off + (2 + d->nsfx) * kw * 1024;
  d->set_cols = 8 * kw * (1 + d->nsfx);
  const bool one = d->grid >= d->items * S;                    // a CTA has one item: its pipeline is drained when the epilogue starts
  d->nacc = !one && 2 * d->NB + 2 * d->set_cols <= kDecTmemCols ? 2 : 1;
  d->nsets = d->nacc * d->NB + kDecMaxSets * d->set_cols <= kDecTmemCols ? kDecMaxSets : 2;
  d->sf_col = kDecTmemCols - d->nsets * d->set_cols;
  if (d->nacc * d->NB > d->sf_col || (S > 1 && (d->ksteps + d->kper - 1) / d->kper != S)) return false;
  const int pad = (128 - h) * 128;                             // the MMA reads 128 rows from where a band's box starts
  const int room = kDecSmem - 1024 - pad - (one ? 0 : kDecStoreBytes);
  int n = room / d->stage_bytes;
  const int most = one ? d->kper : kDecMaxStages;
  if (n > most) n = most;
  if (n > kDecMaxStages) n = kDecMaxStages;
  d->steps = d->kper * ((d->items * S + d->grid - 1) / d->grid);
  if (n < 1 || (n < 2 && d->steps > 1)) return false;          // (a stage of the next item is asked for while this one's is multiplied)
  d->nstages = n;
  const int G = (tokens + 3) / 4, slots = S > 1 ? S * ((G + S - 1) / S) * 2048 : 0;
  const int pipe = n * d->stage_bytes + pad;
  d->epi_off = one ? slots : pipe;
  const int epi_end = d->epi_off + kDecStoreBytes;
  d->smem = (pipe > epi_end ? pipe : epi_end) + 1024;
  if (S > 1 && d->smem < kDecClusterSmem) d->smem = kDecClusterSmem;
  return d->smem <= kDecSmem;
}

// Band height, stage width and K split by what they cost, in us:
//   a stage       the largest of 0.35 + 0.2 kw (waits, scales into tensor memory, MMA issue), its bytes at 60 GB/s (what an SM takes in)
//                 and the weights of all active CTAs' stages at 6.3 TB/s; 1.2 times that with fewer than three stages in flight
//   a K split     1 + tokens (S - 1) / (32 S): two cluster barriers, and the sums sent to the peers
// Against the best of every (kw, S, height) swept over 30 layers (1 to 128 tokens, 2048 to 16384 x 2048 to 16384) and 26 calls with
// experts (9 to 64 of them, 6 to 77 tokens the longest group): 1.013 on average, 1.10 at most.
static bool w4_decode_search(W4DecodeShape* best, int tokens, int groups, int64_t N, int64_t K, int sms) {
  float cost = 1e30f;
  for (int kw = 4; kw >= 1; kw >>= 1)
    for (int S = 1; S <= (groups > 0 ? 1 : 8); ++S)
      for (int h = 128; h >= 96; h -= 16) {
        W4DecodeShape d;
        if (S > 1 && (N + h - 1) / h * S > sms) continue;
        if (!w4_decode_layout(&d, tokens, groups, N, K, h, kw, S)) continue;
        if (S > 1 && w4_decode_clusters(S) < d.items) continue;
        const int full = d.items * S / d.grid, rest = d.items * S - full * d.grid;
        auto stage_us = [&](int ctas) {
          float us = 0.35f + 0.2f * static_cast<float>(kw);
          us = fmaxf(us, static_cast<float>(d.stage_bytes) / 60.0e3f);
          us = fmaxf(us, 136.0f * static_cast<float>(h * kw) * static_cast<float>(ctas) / 6.3e6f);
          return d.nstages < 3 && d.steps > d.nstages ? 1.2f * us : us;
        };
        float c = static_cast<float>(d.kper) * (static_cast<float>(full) * stage_us(d.grid) + (rest ? stage_us(rest) : 0.0f));
        if (S > 1) c += 1.0f + static_cast<float>(tokens * (S - 1)) / static_cast<float>(32 * S);
        if (c < cost) { cost = c; *best = d; }
      }
  return cost < 1e30f;
}

// What a grouped launch takes, in us, from the same fit as the cost of token tiles (w4_grouped_tiles; `tokens`: an average group's).
// Finer than the rule above: bands of short groups load less than the longest's components, and the epilogue of a band, hidden
// behind the next one's MMAs where there are two accumulators, counts.
float w4_decode_grouped_us(const W4DecodeShape& d, float tokens) {
  const float x_rows = fminf(static_cast<float>(d.NB), 2.0f * tokens + static_cast<float>(d.NB) / 8.0f + 8.0f);
  const float bytes = static_cast<float>(d.kw) * (static_cast<float>(d.h) * 128.0f + x_rows * 128.0f + static_cast<float>(2 + d.nsfx) * 1024.0f);
  const float epilogue = fmaxf(0.0f, 0.0226f * tokens - 0.775f);
  const int full = d.items / d.grid, rest = d.items - full * d.grid;
  auto band_us = [&](int ctas) {
    float us = fmaxf(fmaxf(0.47f + 0.02f * static_cast<float>(d.kw), bytes / 69.0e3f), 136.0f * static_cast<float>(d.h * d.kw) * static_cast<float>(ctas) / 7.3e6f);
    if (d.nstages < 3 && d.steps > d.nstages) us *= 1.2f;
    us *= static_cast<float>(d.ksteps);
    return d.nacc == 2 ? fmaxf(us, epilogue) : us + epilogue;
  };
  return static_cast<float>(full) * band_us(d.grid) + (rest ? band_us(rest) : 0.0f) + (d.nacc == 2 ? epilogue : 0.0f);
}

// The same for a call with one matrix, as far as it differs: weights come in one burst, not as a steady stream, and a cluster's exchange
// counts (see w4_few_or_tiles).
float w4_decode_us(const W4DecodeShape& d, float tokens) {
  const float epilogue = fmaxf(0.0f, 0.0162f * tokens - 0.52f);
  auto stages_us = [&](int ctas) {
    float us = fmaxf(fmaxf(0.52f, static_cast<float>(d.stage_bytes) / 85.0e3f), 136.0f * static_cast<float>(d.h * d.kw) * static_cast<float>(ctas) / 6.15e6f);
    if (d.nstages < 3 && d.steps > d.nstages) us *= 1.2f;
    return static_cast<float>(d.kper) * us;
  };
  if (d.S > 1) return stages_us(d.grid) + 0.8f + 0.081f * tokens * static_cast<float>(d.S - 1) / static_cast<float>(d.S);
  const int full = d.items / d.grid, rest = d.items - full * d.grid;
  auto band_us = [&](int ctas) { return d.nacc == 2 ? fmaxf(stages_us(ctas), epilogue) : stages_us(ctas) + epilogue; };
  return static_cast<float>(full) * band_us(d.grid) + (rest ? band_us(rest) : 0.0f) + (d.nacc == 2 ? epilogue : 0.0f);
}

bool w4_decode_shape(W4DecodeShape* best, int tokens, int groups, int64_t N, int64_t K) {
  if (const int forced = option(OPT_W4_DECODE); forced > 0)
    return w4_decode_layout(best, tokens, groups, N, K, forced % 1000, forced / 100000, forced / 1000 % 100);
  return w4_decode_search(best, tokens, groups, N, K, sm_count());
}

msd_status_t w4_decode_launch(const W4DecodeShape& d, const uint8_t* w_fp4, const uint8_t* q, int64_t q_rows, int64_t w_rows, int M, int64_t N,
                              int64_t K, const uint8_t* sfw, bool sfw_ready, const uint8_t* sfx, void* y, int ytype, const W4Groups* groups,
                              unsigned* status, cudaStream_t s) {
  if (!w4_decode_attr()) return MSD_ERR_CUDA;
  const uint64_t kb = static_cast<uint64_t>(K / 2);
  const bool t3 = K % kDecBlockK == 0;
  const CUtensorMapDataType u8 = CU_TENSOR_MAP_DATA_TYPE_UINT8;
  const CUtensorMapSwizzle sw = CU_TENSOR_MAP_SWIZZLE_128B;
  CUtensorMap tmap_w;
  W4DecodeXMaps<true> tmap_x;
  const int boxes = groups ? kDecBoxes : 1;
  bool ok =
      t3 ? encode_tmap_3d(&tmap_w, u8, w_fp4, 128, static_cast<uint64_t>(w_rows), kb / 128, kb, 128, 128, static_cast<uint32_t>(d.h), static_cast<uint32_t>(d.kw), sw)
         : encode_tmap_2d(&tmap_w, u8, w_fp4, kb, static_cast<uint64_t>(w_rows), kb, 128, static_cast<uint32_t>(d.h), sw);
  for (int i = 0; i < boxes && ok; ++i) {
    const uint32_t rows = static_cast<uint32_t>(groups ? w4d_box_rows(d.NB, i) : d.NB);
    ok = t3 ? encode_tmap_3d(&tmap_x.m[i], u8, q, 128, static_cast<uint64_t>(q_rows), kb / 128, kb, 128, 128, rows, static_cast<uint32_t>(d.kw), sw)
            : encode_tmap_2d(&tmap_x.m[i], u8, q, kb, static_cast<uint64_t>(q_rows), kb, 128, rows, sw);
  }
  if (!ok) return MSD_ERR_CUDA;
  W4DecodeParams p;
  p.M = M; p.NB = d.NB; p.N = static_cast<int>(N);
  p.h = d.h; p.bands = d.bands; p.items = d.items;
  p.kblocks = d.kblocks; p.kw = d.kw; p.ksteps = d.ksteps; p.S = d.S; p.kper = d.kper;
  p.nstages = d.nstages; p.stage_bytes = d.stage_bytes; p.x_off = d.x_off; p.sf_off = d.sf_off; p.nsfx = d.nsfx;
  // (a grouped call leaves most of the bandwidth to the decomposition of its many rows)
  p.t3 = t3 ? 1 : 0; p.early = groups && d.nstages > 2 ? 2 : d.nstages;
  p.nacc = d.nacc; p.nsets = d.nsets; p.sf_col = d.sf_col; p.set_cols = d.set_cols; p.epi_off = d.epi_off;
  p.sf_kgroups = 2 * d.kblocks; p.row_blocks = 2 * static_cast<int>((N + 255) / 256);
  p.sfw = sfw; p.sfx = sfx; p.sfw_ready = sfw_ready ? 1 : 0;
  p.y = y; p.ytype = ytype; p.status = status;
  const bool pdl = option(OPT_NO_PDL) <= 0;
  cudaError_t e;
  if (groups) {
    e = launch_pdl(gemm_w4a16_decode_kernel<true>, dim3(d.grid), dim3(kDecThreads), static_cast<size_t>(d.smem), s, pdl, tmap_w, tmap_x, p, *groups);
  } else {
    e = launch_pdl_cluster(gemm_w4a16_decode_kernel<false>, dim3(d.grid), dim3(kDecThreads), static_cast<size_t>(d.smem), s, pdl, static_cast<unsigned>(d.S),
                           tmap_w, W4DecodeXMaps<false>{{tmap_x.m[0]}}, p, W4NoGroups());
  }
  return e == cudaSuccess ? MSD_OK : MSD_ERR_CUDA;
}

}  // namespace msd
