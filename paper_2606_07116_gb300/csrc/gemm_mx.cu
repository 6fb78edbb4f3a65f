// GEMM of the MXFP4 variant (offq_mx_linear; paper Sec. 3.4 "Generality on Data
// Formats": the offsets are the zero-points of a micro-scaled format) on the
// block-scaled FP4 tensor path of sm_103a.
//
//   y[t][n] = s_w[n] * ( s_a[t] * acc[t][n] + sum_b o[t][b] * R[b][n] ),
//   acc[t][n] = sum_k e_a[t][k] 2^sh_a e_w[n][k] 2^sh_w
//
// with E2M1 codes e and, per row and 32 channels, a power of two 2^sh. That is
// what tcgen05.mma kind::mxf4 multiplies: packed E2M1 operands from shared
// memory and UE8M0 scales (the shift + 127) from tensor memory, 64 codes per
// instruction, products exact, fp32 accumulation. So nothing is widened:
//  * the tiled code layout (a 32-row block's 16-byte chunks, 512 bytes per
//    chunk) is already the unswizzled K-major operand layout: 8 rows x 16 bytes
//    contiguous. A 3-D TMA box {512 bytes, row blocks, chunks} lands it with a
//    row-group stride of 128 bytes and a chunk stride of 512 x row blocks;
//  * the shift words (the 4 blocks of a row's 128-code k-tile) go through
//    registers: four warps, one per TMEM lane quarter, add 127 to each byte and
//    store one column per 32-row block; every quarter holds a copy, as the MMA
//    expects its scales.
// Two SMs form a pair (cluster of 2, cta_group::2): M = 256 tokens x N = 192
// channels; each SM holds 128 rows of A and 96 of B, and the scales of its own
// A rows and of all 192 B rows. N = 192 leaves room in tensor memory for two
// accumulators (2 x 192 columns) beside 4 stages of scales, so a tile's
// epilogue, with its offset correction, runs under the next tile's MMAs.
// What bounds it: per 128 codes an SM's shared memory takes 14 KB of TMA writes
// and 14 KB of operand reads against 192 cycles of MMA; below a few hundred
// tokens the chain of one tile's stages. Measured (per call, weights past the
// L2; before: the codes widened to E4M3 by table in converter warps, kind::
// f8f6f4): 4096 x 4096 -> 14336 103 us = 4650 TFLOP/s (308), 4096 x 14336 -> 4096
// 102 us (343), 777 x 4096 -> 4096 16.5 us (30.9), 1 x 4096 -> 4096 10.1 us (30.5);
// with 43 offset blocks (4096 x 11008 -> 4096) 125 us (296), where the epilogue's
// correction takes longer than a tile's MMAs. Output bits are those of the
// widened form (both accumulate exact products in fp32).
//
// Warps: 0 TMA producer, 1 MMA issuer (leader CTA) and TMEM allocation, 2-9
// scales (two groups of four, taking turns by stage of 256 codes: the chain of
// one stage's waits and tensor-memory stores is longer than its MMAs), 10-17
// epilogue (two per quarter, 96 columns each). Every wait is bounded; a wait that runs out aborts the CTA, which lets its copies
// and MMAs in flight finish and records OFFQ_ERR_TIMEOUT.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "offq.h"
#include "offq_device.cuh"
#include "offq_host.h"
#include "pair_common.cuh"

namespace {

using namespace offq;

constexpr int XBM = 128;           // rows of A per CTA
constexpr int XBN = 192;           // output channels per pair tile
constexpr int XBNH = XBN / 2;      // rows of B per CTA
constexpr int XBK = 256;           // codes per stage: two 128-code k-tiles (shift words)
constexpr int kXKt = XBK / 128;
constexpr int kXStages = 4;
constexpr int kXChunks = XBK / 32;
constexpr int kXAStage = XBM * XBK / 2, kXBStage = XBNH * XBK / 2;  // 16 KB, 12 KB
constexpr int kXStage = kXAStage + kXBStage;
constexpr int kXABlocks = XBM / 32, kXBBlocks = XBN / 32, kXBHBlocks = XBNH / 32;
constexpr int kXSf0 = 2 * XBN;     // TMEM: two accumulators, then the scale stages
constexpr int kXSfKt = 16;         // per k-tile: 4 columns for A, 6 for B
constexpr int kXSfCols = kXKt * kXSfKt;
constexpr int kXTmemCols = 512;
static_assert(kXSf0 + kXStages * kXSfCols <= kXTmemCols, "TMEM budget");
constexpr int kXSfGroups = 2;      // groups of four scale warps, taking turns by stage
constexpr int kXEpiWarps = 8, kXFirstSf = 2, kXFirstEpi = kXFirstSf + 4 * kXSfGroups;
constexpr int kXThreads = (kXFirstEpi + kXEpiWarps) * 32;
constexpr int kXEpiCols = XBN / 2;  // accumulator columns per epilogue warp
constexpr int kXMaxG = 48;          // offset blocks staged in shared memory
constexpr int kXSfPrefetch = 2;     // stages of shift words in flight per scale warp
constexpr int kXOutPitch = XBN * 2 + 16;

constexpr int kXOffOut = kXStages * kXStage;          // staged 16-bit output rows
constexpr int kXOffW = kXOffOut + XBM * kXOutPitch;   // s_w, s_a, barriers, misc
constexpr int kXOffSa = kXOffW + XBN * 4;
constexpr int kXNumBars = 3 * kXStages + 5;
constexpr int kXOffBars = kXOffSa + XBM * 4;
constexpr int kXOffMisc = kXOffBars + kXNumBars * 8;
constexpr int kXOffR = (kXOffMisc + 64 + 15) / 16 * 16;  // row sums [G][192], then offsets [128][G | 1]
constexpr int kXSmemMax = 227 * 1024;
static_assert(kXOffR + 1024 + kXMaxG * XBN * 4 + XBM * (kXMaxG + 1) * 4 <= kXSmemMax, "shared memory budget");

// Instruction descriptor of kind::mxf4 with E2M1 A and B (code 1 at bits 7-9 and
// 10-11), UE8M0 scales (bit 23), N >> 3 at bit 17, M >> 7 at bit 27, K = 64, and
// the byte of the scale words that holds the first of the MMA's two blocks
// (bits 4-5 for B, 29-30 for A).
constexpr uint32_t idesc_mxf4(int M, int N, uint32_t byte) {
  return (byte << 4) | (1u << 7) | (1u << 10) | (static_cast<uint32_t>(N >> 3) << 17) | (1u << 23) |
         (static_cast<uint32_t>(M >> 7) << 27) | (byte << 29);
}

struct MxGemmParams {
  const uint8_t* a_shifts;
  const uint8_t* w_shifts;
  const float* a_scale;
  const float* a_offset;  // [T][G] or nullptr
  const float* w_scale;
  const float* rowsum;    // [G][N]
  void* out;
  int64_t ldo;
  int* status;
  int T, N, G;
  int nk;                  // 128-code k-tiles
  int ns;                  // stages of two k-tiles
  int m_pairs, n_tiles, raster_m;
  int t_blocks, n_blocks;  // 32-row blocks present in the code buffers
  int staged;              // row sums and offsets go through shared memory
  int vec_r;               // rows of the row sums allow 16-byte reads
  int async_out;           // 16-bit output and N % 8 == 0: rows leave by bulk copy
};

__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* map, uint32_t bar, int c0, int c1, int c2) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], "
      "[%5];" ::"r"(dst),
      "l"(map), "r"(c0), "r"(c1), "r"(c2), "r"(bar)
      : "memory");
}

// Descriptor of an unswizzled K-major operand: core matrices of 8 rows x 16
// bytes, 128 bytes apart along the rows, `chunk` bytes apart along K.
__device__ __forceinline__ uint64_t smem_desc_plain(uint32_t saddr, uint32_t chunk) {
  return static_cast<uint64_t>((saddr & 0x3FFFFu) >> 4) | (static_cast<uint64_t>(chunk >> 4) << 16) |
         (static_cast<uint64_t>(128u >> 4) << 32) | (static_cast<uint64_t>(1u) << 46);
}

__device__ __forceinline__ void mma2_mxf4(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                          uint32_t sfa, uint32_t sfb, uint32_t accumulate) {
  asm volatile(
      "{\n"
      ".reg .pred p;\n"
      "setp.ne.b32 p, %6, 0;\n"
      "tcgen05.mma.cta_group::2.kind::mxf4.block_scale.scale_vec::2X [%0], %1, %2, %3, [%4], [%5], p;\n"
      "}\n" ::"r"(d_tmem),
      "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(sfa), "r"(sfb), "r"(accumulate)
      : "memory");
}

__device__ __forceinline__ void tmem_st_4cols(uint32_t taddr, const uint32_t* r) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1,%2,%3,%4};" ::"r"(taddr), "r"(r[0]), "r"(r[1]),
               "r"(r[2]), "r"(r[3])
               : "memory");
}
__device__ __forceinline__ void tmem_st_2cols(uint32_t taddr, const uint32_t* r) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x2.b32 [%0], {%1,%2};" ::"r"(taddr), "r"(r[0]), "r"(r[1]) : "memory");
}

// Pair tile index -> (m-pair, n-tile), in raster groups of m-pairs (as the pair
// kernel of gemm.cu: a weight tile is read from DRAM about once per group).
__device__ __forceinline__ void mx_tile(const MxGemmParams& p, int tile, int& mp, int& nt) {
  const int per_group = p.raster_m * p.n_tiles;
  const int grp = tile / per_group;
  const int local = tile - grp * per_group;
  const int m_left = p.m_pairs - grp * p.raster_m;
  const int gm = m_left < p.raster_m ? m_left : p.raster_m;
  nt = local / gm;
  mp = grp * p.raster_m + (local - nt * gm);
}

template <int OUT>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kXThreads, 1)
    mx_gemm_kernel(const __grid_constant__ CUtensorMap amap, const __grid_constant__ CUtensorMap wmap,
                   const MxGemmParams p) {
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  uint8_t* smem = smem_raw + (base - raw);

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const uint32_t rank = cluster_rank();
  const int cluster = blockIdx.x >> 1;
  const int clusters = gridDim.x >> 1;
  const int nk = p.nk, ns = p.ns;
  const int num_tiles = p.m_pairs * p.n_tiles;

  const uint32_t bar0 = base + kXOffBars;
  auto full = [&](int s) { return bar0 + 8u * s; };                    // this CTA's copies landed
  auto ready = [&](int s) { return bar0 + 8u * (kXStages + s); };      // leader: both CTAs' operands and scales
  auto empty = [&](int s) { return bar0 + 8u * (2 * kXStages + s); };  // both: stage s consumed
  auto acc_full = [&](int b) { return bar0 + 8u * (3 * kXStages + b); };       // both: accumulator b complete
  auto acc_empty = [&](int b) { return bar0 + 8u * (3 * kXStages + 2 + b); };  // leader: accumulator b drained
  const uint32_t done = bar0 + 8u * (3 * kXStages + 4);                // leader, after an abort: MMAs finished
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + kXOffMisc);
  volatile int* abort = reinterpret_cast<volatile int*>(smem + kXOffMisc + 16);
  volatile int* epi_stop = reinterpret_cast<volatile int*>(smem + kXOffMisc + 32);

  if (threadIdx.x == 0) {
    for (int s = 0; s < kXStages; ++s) {
      mbar_init(full(s), 1);
      mbar_init(ready(s), 8);
      mbar_init(empty(s), 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(acc_full(b), 1);
      mbar_init(acc_empty(b), 2 * kXEpiWarps);
    }
    mbar_init(done, 1);
    *abort = 0;
    *epi_stop = 0;
    mbar_fence_init();
  }
  if (warp == 1) {
    tmem_alloc2(smem_u32(tmem_slot), kXTmemCols);
    tmem_relinquish2();
  }
  tc_fence_before();
  cluster_sync();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  griddep_wait();
  griddep_launch_dependents();
  int loads = 0;  // producer: k-tiles requested

  if (warp == 0) {
    // ---------------- TMA producer ----------------
    if (lane == 0) {
      tma_prefetch_desc(&amap);
      tma_prefetch_desc(&wmap);
      int s = 0, phase = 0;
      bool ok = true;
      for (int tile = cluster; tile < num_tiles && ok; tile += clusters) {
        int mp, nt;
        mx_tile(p, tile, mp, nt);
        const int ab = (mp * 2 + static_cast<int>(rank)) * kXABlocks;
        const int bb = nt * kXBBlocks + static_cast<int>(rank) * kXBHBlocks;
        for (int kt = 0; kt < ns; ++kt) {
          ok = wait_cluster(empty(s), phase ^ 1, abort);
          if (!ok) break;
          mbar_arrive_expect_tx(full(s), kXStage);
          const uint32_t dst = base + s * kXStage;
          tma_load_3d(dst, &amap, full(s), 0, ab, kt * kXChunks);
          tma_load_3d(dst + kXAStage, &wmap, full(s), 0, bb, kt * kXChunks);
          ++loads;
          if (++s == kXStages) {
            s = 0;
            phase ^= 1;
          }
        }
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    // ---------------- MMA issuer (leader CTA) ----------------
    if (rank == 0) {
      const uint64_t a_desc0 = smem_desc_plain(base, kXABlocks * 512);
      const uint64_t b_desc0 = smem_desc_plain(base + kXAStage, kXBHBlocks * 512);
      int s = 0, phase = 0, lt = 0;
      bool ok = true;
      for (int tile = cluster; tile < num_tiles && ok; tile += clusters, ++lt) {
        const int b = lt & 1;
        ok = __all_sync(0xFFFFFFFFu, wait_cluster(acc_empty(b), ((lt >> 1) & 1) ^ 1, abort));
        if (!ok) break;
        tc_fence_after();
        for (int kt = 0; kt < ns; ++kt) {
          ok = __all_sync(0xFFFFFFFFu, wait_cluster(ready(s), phase, abort));
          if (!ok) break;
          tc_fence_after();
          if (elect_one()) {
            const uint64_t so = static_cast<uint32_t>(s * (kXStage >> 4));
            const uint32_t sf = tmem + kXSf0 + s * kXSfCols;
#pragma unroll
            for (int j = 0; j < 2 * kXKt; ++j)  // 64 codes: two chunks, two bytes of the k-tile's scale words
              mma2_mxf4(tmem + b * XBN, a_desc0 + so + j * (2 * kXABlocks * 512 >> 4),
                        b_desc0 + so + j * (2 * kXBHBlocks * 512 >> 4), idesc_mxf4(2 * XBM, XBN, 2 * (j & 1)),
                        sf + (j >> 1) * kXSfKt, sf + (j >> 1) * kXSfKt + 4, (kt | j) != 0 ? 1u : 0u);
            mma2_commit_both(empty(s));
            if (kt == ns - 1) mma2_commit_both(acc_full(b));
          }
          __syncwarp();
          if (++s == kXStages) {
            s = 0;
            phase ^= 1;
          }
        }
      }
    }
  } else if (warp >= kXFirstSf && warp < kXFirstEpi) {
    // ---------------- scales: shift words -> UE8M0 in tensor memory ----------------
    const uint32_t lane_tm = tmem + (static_cast<uint32_t>((warp & 3) * 32) << 16) + kXSf0;
    const uint32_t ready_l = leader_addr(ready(0));
    constexpr int kWords = kXABlocks + kXBBlocks;
    const int turn = (warp - kXFirstSf) >> 2;  // stages u == turn mod kXSfGroups
    uint32_t ring[kXSfPrefetch][kXKt][kWords];
    int ld_tile = cluster, ld_kt = turn;  // next stage to load
    while (ld_kt >= ns) {
      ld_kt -= ns;
      ld_tile += clusters;
    }
    int set_for = -1;
    const uint32_t* src[2] = {nullptr, nullptr};
    int blocks_a = 0, blocks_b = 0;
    auto load = [&](uint32_t (&v)[kXKt][kWords]) {
      if (ld_tile < num_tiles) {
        if (ld_tile != set_for) {
          set_for = ld_tile;
          int mp, nt;
          mx_tile(p, ld_tile, mp, nt);
          const int ab = (mp * 2 + static_cast<int>(rank)) * kXABlocks, bb = nt * kXBBlocks;
          src[0] = reinterpret_cast<const uint32_t*>(p.a_shifts) + static_cast<int64_t>(ab) * nk * 32 + lane;
          src[1] = reinterpret_cast<const uint32_t*>(p.w_shifts) + static_cast<int64_t>(bb) * nk * 32 + lane;
          blocks_a = p.t_blocks - ab;
          blocks_b = p.n_blocks - bb;
        }
#pragma unroll
        for (int h = 0; h < kXKt; ++h) {
          const int kt = ld_kt * kXKt + h;
#pragma unroll
          for (int i = 0; i < kWords; ++i) {
            const bool a = i < kXABlocks;
            const int blk = a ? i : i - kXABlocks;
            v[h][i] = blk < (a ? blocks_a : blocks_b) && kt < nk
                          ? __ldg(src[a ? 0 : 1] + static_cast<uint32_t>((blk * nk + kt) * 32))
                          : 0u;
          }
        }
        ld_kt += kXSfGroups;
        while (ld_kt >= ns) {
          ld_kt -= ns;
          ld_tile += clusters;
        }
      }
    };
#pragma unroll
    for (int i = 0; i < kXSfPrefetch; ++i) load(ring[i]);
    const int my_tiles = cluster < num_tiles ? (num_tiles - cluster + clusters - 1) / clusters : 0;
    const int64_t total = static_cast<int64_t>(my_tiles) * ns;
    int s = turn, phase = 0;
    bool ok = true;
    for (int64_t u0 = turn; u0 < total && ok; u0 += kXSfPrefetch * kXSfGroups) {
#pragma unroll
      for (int i = 0; i < kXSfPrefetch; ++i) {
        if (u0 + i * kXSfGroups >= total) break;
        ok = __all_sync(0xFFFFFFFFu, wait_cluster(empty(s), phase ^ 1, abort));
        if (!ok) break;
        tc_fence_after();
#pragma unroll
        for (int h = 0; h < kXKt; ++h) {
          uint32_t v[kWords];
#pragma unroll
          for (int j = 0; j < kWords; ++j) v[j] = ring[i][h][j] + 0x7F7F7F7Fu;  // 2^sh as UE8M0 (no carry: sh <= 6)
          const uint32_t dst = lane_tm + s * kXSfCols + h * kXSfKt;
          tmem_st_4cols(dst, v);
          tmem_st_4cols(dst + 4, v + 4);
          tmem_st_2cols(dst + 8, v + 8);
        }
        load(ring[i]);
        tmem_st_wait();
        tc_fence_before();
        // This CTA's operands of the stage have landed too: one arrival tells the leader both.
        ok = __all_sync(0xFFFFFFFFu, wait_cluster(full(s), phase, abort));
        if (!ok) break;
        __syncwarp();
        if (lane == 0) arrive_cluster(ready_l + 8u * s);
        s += kXSfGroups;
        if (s >= kXStages) {
          s -= kXStages;
          phase ^= 1;
        }
      }
    }
  } else if (warp >= kXFirstEpi) {
    // ---------------- epilogue ----------------
    const uint64_t out_pol = l2_evict_first();
    const int quarter = warp & 3;
    const int half = (warp - kXFirstEpi) >> 2;
    const int et = threadIdx.x - kXFirstEpi * 32;
    const int G = p.G, gp = G | 1;
    float* Ws = reinterpret_cast<float*>(smem + kXOffW);
    float* Sa = reinterpret_cast<float*>(smem + kXOffSa);
    float* Rs = reinterpret_cast<float*>(smem + kXOffR);
    float* Os = Rs + G * XBN;
    const bool async_out = OUT != OFFQ_F32 && p.async_out != 0;
    const int rl = quarter * 32 + lane;
    const uint32_t orow_s = base + kXOffOut + rl * kXOutPitch + half * kXEpiCols * 2;
    int lt = 0;
    for (int tile = cluster; tile < num_tiles; tile += clusters, ++lt) {
      int mp, nt;
      mx_tile(p, tile, mp, nt);
      const int m0 = (mp * 2 + static_cast<int>(rank)) * XBM;
      const int nt0 = nt * XBN;
      // The tile's constants, while its MMAs run (asynchronous copies: their latencies overlap).
      auto stage = [](float* dst, const float* src, bool exists) {
        if (exists)
          cp_async<4>(smem_u32(dst), src);
        else
          *dst = 0.f;
      };
      for (int i = et; i < XBN; i += kXEpiWarps * 32) stage(Ws + i, p.w_scale + nt0 + i, nt0 + i < p.N);
      for (int i = et; i < XBM; i += kXEpiWarps * 32) stage(Sa + i, p.a_scale + m0 + i, m0 + i < p.T);
      if (p.staged) {
        for (int i = et; i < G * XBN; i += kXEpiWarps * 32) {
          const int b = i / XBN, n = nt0 + i - b * XBN;
          stage(Rs + i, p.rowsum + static_cast<int64_t>(b) * p.N + n, n < p.N);
        }
        const int rows = p.T - m0 < XBM ? p.T - m0 : XBM;  // may be negative
        const float* o0 = p.a_offset + static_cast<int64_t>(m0) * G;
        for (int i = et; i < XBM * G; i += kXEpiWarps * 32) {
          const int r = i / G, b = i - r * G;
          stage(Os + r * gp + b, o0 + i, p.a_offset != nullptr && r < rows);
        }
      }
      asm volatile("cp.async.wait_all;" ::: "memory");
      epi_sync<kXEpiWarps>();
      const bool ok = __all_sync(0xFFFFFFFFu, wait_cluster(acc_full(lt & 1), (lt >> 1) & 1, abort));
      if (!ok && lane == 0) *epi_stop = 1;
      tc_fence_after();
      const int t = m0 + rl;
      const bool row_ok = t < p.T;
      const int n0 = nt0 + half * kXEpiCols;
      const uint32_t acc_tm =
          tmem + (static_cast<uint32_t>(quarter * 32) << 16) + (lt & 1) * XBN + half * kXEpiCols;
      if (ok) {
        if (async_out) bulk_wait_read_all();  // this row's previous copy has read the buffer
        const float sa = Sa[rl];
        constexpr int CW = 16;
        // A warp whose 32 rows lie past the tokens, or columns past the channels, has nothing to write.
        const int cols = m0 + quarter * 32 < p.T ? (p.N - n0 < kXEpiCols ? p.N - n0 : kXEpiCols) : 0;
        for (int c = 0; c < cols; c += CW) {
          uint32_t acc[CW];
          tmem_ld_16cols(acc_tm + c, acc);
          const int jc = half * kXEpiCols + c;  // column within the tile
          const int nb = n0 + c;
          // Offset correction: block 0 multiplied, then FMAs in block order.
          uint64_t y2[CW / 2];
          if (p.staged) {
            // Several blocks' broadcast reads of R are in flight at a time (unrolled): the chain of one block
            // (a row's offset, four reads, FMAs) is ten times its issue time.
            const float* o = Os + rl * gp;
            const float4* r4 = reinterpret_cast<const float4*>(Rs + jc);
            {
              const uint64_t O2 = pack2(o[0], o[0]);
#pragma unroll
              for (int q = 0; q < CW / 4; ++q) {
                const float4 rv = r4[q];
                y2[2 * q] = mul2v(O2, pack2(rv.x, rv.y));
                y2[2 * q + 1] = mul2v(O2, pack2(rv.z, rv.w));
              }
            }
#pragma unroll 3
            for (int b = 1; b < G; ++b) {
              const float ob = o[b];
              const uint64_t O2 = pack2(ob, ob);
#pragma unroll
              for (int q = 0; q < CW / 4; ++q) {
                const float4 rv = r4[b * (XBN / 4) + q];
                y2[2 * q] = fma2v(O2, pack2(rv.x, rv.y), y2[2 * q]);
                y2[2 * q + 1] = fma2v(O2, pack2(rv.z, rv.w), y2[2 * q + 1]);
              }
            }
          } else if (p.vec_r && nb + CW <= p.N && p.a_offset != nullptr) {
            // Too many blocks to stage: R by 16-byte reads, several blocks' in flight (one element at a time was the
            // larger part of such a layer: 2 x 18944 -> 7808 with 148 blocks 875 us, now 357).
            const float* o = p.a_offset + static_cast<int64_t>(row_ok ? t : 0) * G;
            const float4* r4 = reinterpret_cast<const float4*>(p.rowsum + nb);
            const int64_t pitch = p.N / 4;
            {
              const float ob = __ldg(o);
              const uint64_t O2 = pack2(ob, ob);
#pragma unroll
              for (int q = 0; q < CW / 4; ++q) {
                const float4 rv = __ldg(r4 + q);
                y2[2 * q] = mul2v(O2, pack2(rv.x, rv.y));
                y2[2 * q + 1] = mul2v(O2, pack2(rv.z, rv.w));
              }
            }
#pragma unroll 4
            for (int b = 1; b < G; ++b) {
              const float ob = __ldg(o + b);
              const uint64_t O2 = pack2(ob, ob);
#pragma unroll
              for (int q = 0; q < CW / 4; ++q) {
                const float4 rv = __ldg(r4 + b * pitch + q);
                y2[2 * q] = fma2v(O2, pack2(rv.x, rv.y), y2[2 * q]);
                y2[2 * q + 1] = fma2v(O2, pack2(rv.z, rv.w), y2[2 * q + 1]);
              }
            }
          } else {
            float z[CW];
#pragma unroll
            for (int i = 0; i < CW; ++i) z[i] = 0.f;
            if (p.a_offset != nullptr) {
              for (int b = 0; b < G; ++b) {
                const float ob = __ldg(p.a_offset + static_cast<int64_t>(row_ok ? t : 0) * G + b);
                const float* rb = p.rowsum + static_cast<int64_t>(b) * p.N + nb;
#pragma unroll
                for (int i = 0; i < CW; ++i)
                  if (nb + i < p.N) z[i] = b == 0 ? ob * __ldg(rb + i) : fmaf(ob, __ldg(rb + i), z[i]);
              }
            }
#pragma unroll
            for (int i = 0; i < CW / 2; ++i) y2[i] = pack2(z[2 * i], z[2 * i + 1]);
          }
          tmem_ld_wait_for(acc);
          const uint64_t SA2 = pack2(sa, sa);
          float y[CW];
          const float4* w4 = reinterpret_cast<const float4*>(Ws + jc);
#pragma unroll
          for (int q = 0; q < CW / 4; ++q) {
            const float4 wv = w4[q];
            const uint64_t A0 = pack2(__uint_as_float(acc[4 * q]), __uint_as_float(acc[4 * q + 1]));
            const uint64_t A1 = pack2(__uint_as_float(acc[4 * q + 2]), __uint_as_float(acc[4 * q + 3]));
            unpack2(mul2v(pack2(wv.x, wv.y), fma2v(SA2, A0, y2[2 * q])), y[4 * q], y[4 * q + 1]);
            unpack2(mul2v(pack2(wv.z, wv.w), fma2v(SA2, A1, y2[2 * q + 1])), y[4 * q + 2], y[4 * q + 3]);
          }
          if (async_out) {  // rows past the tokens too: they are not copied out
            uint32_t hv[CW / 2];
#pragma unroll
            for (int i = 0; i < CW / 2; ++i) hv[i] = pack_out<OUT>(y[2 * i], y[2 * i + 1]);
            sts128(orow_s + c * 2, hv[0], hv[1], hv[2], hv[3]);
            sts128(orow_s + c * 2 + 16, hv[4], hv[5], hv[6], hv[7]);
          } else if (row_ok) {
            const int nvalid = p.N - nb < CW ? p.N - nb : CW;
            store_out<OUT, CW>(p.out, static_cast<int64_t>(t) * p.ldo + nb, y, nvalid, out_pol);
          }
          __syncwarp();  // the next columns' load needs every lane
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) arrive_cluster(leader_addr(acc_empty(lt & 1)));
        if (async_out && row_ok && n0 < p.N) {
          const int ncols = p.N - n0 < kXEpiCols ? p.N - n0 : kXEpiCols;
          fence_proxy_async_smem();
          bulk_store(static_cast<uint16_t*>(p.out) + static_cast<int64_t>(t) * p.ldo + n0, orow_s,
                     static_cast<uint32_t>(ncols) * 2, out_pol);
          bulk_commit();
        }
      }
      epi_sync<kXEpiWarps>();  // the staged constants are reused for the next tile
      if (*epi_stop) break;
    }
    bulk_wait_all();  // output rows in flight are written before the CTA ends
  }

  // ---------------- teardown ----------------
  __syncthreads();
  if (*abort) {
    if (warp == 0 && lane == 0) {
      // Copies requested but not consumed land before shared memory is released.
      for (int u = loads > kXStages ? loads - kXStages : 0; u < loads; ++u)
        wait_teardown(full(u % kXStages), (u / kXStages) & 1);
    }
    if (warp == 1 && rank == 0) {
      // The MMAs this warp issued are done when a commit after them arrives. Only here, and only at this CTA's barrier:
      // without an abort every accumulator has been waited for, and an arrival that nobody waits for could reach a CTA
      // that has ended.
      if (elect_one()) mma2_commit(done);
      __syncwarp();
      wait_teardown(done, 0);
    }
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync();  // the pair's MMAs read both CTAs' memory: leave together
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc2(tmem, kXTmemCols);
  }
  if (threadIdx.x == 0 && *abort && p.status != nullptr) atomicExch(p.status, kErrTimeout);
}

// Tiled codes of `blocks` 32-row blocks as [chunk][row block][512 bytes].
bool encode_codes(CUtensorMap* map, const uint8_t* codes, int64_t blocks, int64_t kchunks, int box_blocks) {
  const auto enc = tensor_map_encoder();
  if (enc == nullptr) return false;
  const cuuint64_t dims[3] = {128, static_cast<cuuint64_t>(blocks), static_cast<cuuint64_t>(kchunks)};
  const cuuint64_t strides[2] = {static_cast<cuuint64_t>(kchunks) * 512, 512};
  const cuuint32_t box[3] = {128, static_cast<cuuint32_t>(box_blocks), kXChunks};
  const cuuint32_t elem_strides[3] = {1, 1, 1};
  return enc(map, CU_TENSOR_MAP_DATA_TYPE_UINT32, 3, const_cast<uint8_t*>(codes), dims, strides, box, elem_strides,
             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <int OUT>
int launch_mx(const CUtensorMap& amap, const CUtensorMap& wmap, const MxGemmParams& p, cudaStream_t s) {
  if (!smem_optin<mx_gemm_kernel<OUT>>(kXSmemMax)) return OFFQ_ERR_CUDA;
  const int sms = device_sms();
  if (sms < 2) return OFFQ_ERR_CUDA;
  const int64_t tiles = static_cast<int64_t>(p.m_pairs) * p.n_tiles;
  const int clusters = static_cast<int>(tiles < sms / 2 ? tiles : sms / 2);
  const size_t bytes = kXOffR + 1024 + (p.staged ? p.G * XBN * 4 + XBM * (p.G | 1) * 4 : 0);
  return launch_pdl(mx_gemm_kernel<OUT>, dim3(2 * clusters), dim3(kXThreads), bytes, s, amap, wmap, p);
}

}  // namespace

extern "C" int offq_mx_linear(const uint8_t* a_codes, const uint8_t* a_shifts, const float* a_scale,
                              const float* a_offset, int64_t T, int64_t N, int64_t K, int32_t g,
                              const uint8_t* w_codes, const uint8_t* w_shifts, const float* w_scale,
                              const float* w_offsum, void* out, int out_dtype, int64_t ldo, void* stream) {
  const int ob = elem_bytes(out_dtype);
  if (ob == 0 || T < 0 || N < 1 || !is_pow2(g) || g < 32 || g > 8192) return OFFQ_ERR_INVALID_ARG;
  if (K <= 0 || K % g != 0 || K % 128 != 0 || ldo < N) return OFFQ_ERR_INVALID_ARG;
  if (K > kMaxGemmK || T > 0x3FFFFFFF || N > 0x3FFFFFFF) return OFFQ_ERR_UNSUPPORTED;
  if (T == 0) return OFFQ_OK;
  if (a_codes == nullptr || a_shifts == nullptr || a_scale == nullptr || w_codes == nullptr || w_shifts == nullptr ||
      w_scale == nullptr || w_offsum == nullptr || out == nullptr)
    return OFFQ_ERR_INVALID_ARG;
  if (!aligned(a_codes, 16) || !aligned(w_codes, 16) || !aligned(out, 16) || (ldo * ob) % 16 != 0 ||
      !aligned(a_shifts, 4) || !aligned(w_shifts, 4) || !aligned(a_scale, 4) || !aligned(w_scale, 4) ||
      !aligned(w_offsum, 4) || (a_offset != nullptr && !aligned(a_offset, 4)))
    return OFFQ_ERR_MISALIGNED;
  MxGemmParams p{};
  p.a_shifts = a_shifts;
  p.w_shifts = w_shifts;
  p.a_scale = a_scale;
  p.a_offset = a_offset;
  p.w_scale = w_scale;
  p.rowsum = w_offsum;
  p.out = out;
  p.ldo = ldo;
  p.status = device_status_ptr();
  p.T = static_cast<int>(T);
  p.N = static_cast<int>(N);
  p.G = static_cast<int>(K / g);
  p.nk = static_cast<int>(K / 128);
  p.ns = (p.nk + kXKt - 1) / kXKt;
  p.m_pairs = static_cast<int>((T + 2 * XBM - 1) / (2 * XBM));
  p.n_tiles = static_cast<int>((N + XBN - 1) / XBN);
  // Raster groups of m-pairs whose activation codes total at most ~32 MB.
  int64_t rm = (int64_t{32} << 20) / (2 * XBM * (K / 2));
  if (rm < 1) rm = 1;
  p.raster_m = static_cast<int>(rm < p.m_pairs ? rm : p.m_pairs);
  p.t_blocks = static_cast<int>((T + 31) / 32);
  p.n_blocks = static_cast<int>((N + 31) / 32);
  p.staged = p.G <= kXMaxG;
  p.vec_r = aligned(w_offsum, 16) && N % 4 == 0;
  p.async_out = out_dtype != OFFQ_F32 && N % 8 == 0;
  CUtensorMap amap, wmap;
  if (!encode_codes(&amap, a_codes, p.t_blocks, K / 32, kXABlocks) ||
      !encode_codes(&wmap, w_codes, p.n_blocks, K / 32, kXBHBlocks))
    return OFFQ_ERR_CUDA;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  switch (out_dtype) {
    case OFFQ_F32: return launch_mx<OFFQ_F32>(amap, wmap, p, s);
    case OFFQ_BF16: return launch_mx<OFFQ_BF16>(amap, wmap, p, s);
    case OFFQ_F16: return launch_mx<OFFQ_F16>(amap, wmap, p, s);
    default: return OFFQ_ERR_INVALID_ARG;
  }
}
