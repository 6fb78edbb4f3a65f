// W4A4 GEMM of the OffQ path (offq_w4a4_linear) on the 5th-generation tensor
// cores of sm_103a, with the dequant + offset epilogue fused.
//
//   y[t][n] = s_w[n] * ( s_a[t] * (acc'[t][n] - 8 Rt[n]) + sum_b o[t][b] * R[b][n] )
//   acc'[t][n] = sum_k (q_a[t][k] + 8) * q_w[n][k],   Rt[n] = sum_b R[b][n]
//
// acc' is what the tensor cores accumulate: activation codes are stored as
// u = q + 8 (1..15) and weight codes as sign-magnitude q (-7..7). Both widen to
// E4M3 bytes whose values are exact integers times 2^-9: bytes 0x00..0x0F are
// the values 0..15 * 2^-9 (subnormals and the first binade share one step), and
// the sign bit negates. Every product and partial sum is then an integer times
// 2^-18 below 2^24 * 2^-18 for K <= 65536, exact in the fp32 accumulator. The
// "+8" is removed in the epilogue, still exactly: acc' - 8 Rt[n] is the integer
// dot product times 2^-18, with the weight row sum Rt = sum_k q_w[n][k] (the
// block row sums R added up). Only then is it scaled, so an output near zero
// is not the small difference of two large rounded terms.
//
// Design. Widening 4-bit codes to fp8 operands costs shared-memory bandwidth,
// which the tensor core's operand reads share. So:
//  * two SMs form a pair (cluster of 2, tcgen05 cta_group::2) computing a
//    256 x 256 tile; each SM holds 128 rows of A and half (128 rows) of B, and
//    the pair's MMA reads each half of B once for both SMs;
//  * A never touches shared memory: converter warps load its packed codes with
//    coalesced 16-byte loads, widen them in registers and write the E4M3
//    operand straight into tensor memory (tcgen05.st), where the MMA reads it;
//  * B is loaded the same way, widened, and stored once into the 128-byte-
//    swizzled K-major shared-memory layout the MMA reads;
//  * both code matrices use a 32-row tiled layout, so each 16-byte load of a
//    warp covers 512 contiguous bytes and lane i receives row i.
// Per SM and 128-code k-tile this moves 16 KB of shared memory for the MMA's B
// reads and 16 KB of B stores, against 512 cycles of MMA work.
//
// Warp roles per CTA (21 warps):
//   warp 0       TMEM allocation; in the leader CTA, an elected lane issues the MMAs
//   warps 1-8    A converters: two per 32-lane quarter of TMEM, alternating k-tiles
//   warps 9-16   B converters: two per 32-row group, alternating k-tiles
//   warps 17-20  epilogue (one per TMEM quarter, all 256 columns)
// Every wait is bounded; a wait that runs out aborts the CTA and records
// OFFQ_ERR_TIMEOUT in the device status word.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <mutex>

#include "offq.h"
#include "offq_device.cuh"
#include "offq_host.h"
#include "pair_common.cuh"

namespace {

using namespace offq;

constexpr int BM = 128;            // rows of A per CTA (256 per pair)
constexpr int BN = 256;            // output channels per pair tile (128 rows of B per CTA)
constexpr int BNH = BN / 2;        // rows of B held by one CTA
constexpr int BK = 128;            // codes per k-tile
constexpr int kChunksPerKt = BK / 32;  // 16-byte packed chunks per row per k-tile
// Warp roles of one instantiation. kSplitA / kSplitB converter warps serve each
// 32-row group of A / B, taking turns by k-tile; kEpiWarps drain the
// accumulator (one per 32-lane TMEM quarter). 21 warps put 6 on one SM
// sub-partition: 80 registers per thread. (Trading B converters for epilogue
// warps in the several-block kernel left one B warp per group too slow.)
template <bool kOneBlock>
struct Roles {
  // Stages of the operand ring. Several offset blocks take 4, so 128 TMEM columns
  // stay free for half of the precomputed offset correction.
  static constexpr int kStages = kOneBlock ? 6 : 4;
  static constexpr int kSplitA = 2;
  static constexpr int kSplitB = 2;
  static constexpr int kAWarps = 4 * kSplitA, kBWarps = 4 * kSplitB;
  static constexpr int kEpiWarps = 4;  // one per 32-lane TMEM quarter
  static constexpr int kFirstA = 1, kFirstB = kFirstA + kAWarps, kFirstEpi = kFirstB + kBWarps;
  static constexpr int kThreads = (kFirstEpi + kEpiWarps) * 32;
  static_assert(kSplitA <= kStages && kSplitB <= kStages, "a converter's next stage is at most one ring turn ahead");
};
constexpr int kConvWarpsPerCta = 8;  // arrivals per stage and CTA: one per 32-row group of A and of B
// k-tiles of loads in flight per converter thread. With one, a warp's loads
// are issued right after its barrier arrival and have its next turn (two k-tiles
// later) to land, and no load is outstanding when the arrival's release orders
// the warp's earlier memory operations.
constexpr int kPrefetch = 1;
constexpr int kMaxStageG = 48;                       // offset blocks staged in shared memory
constexpr int kAccCols = BN;       // fp32 accumulator columns (TMEM lanes = rows)
constexpr int kACol0 = kAccCols;   // A operand stages live in TMEM after the accumulator
constexpr int kAColsPerStage = BK / 4;  // 4 E4M3 values per 32-bit column
constexpr int kTmemCols = 512;
static_assert(kACol0 + Roles<true>::kStages * kAColsPerStage <= kTmemCols, "TMEM budget");
// Several offset blocks: the correction sum_b o_b R[b][n] of a tile is
// computed while its MMAs run; accumulator columns 0..127 keep theirs in TMEM
// after the A stages, columns 128..255 in shared memory.
constexpr int kCorrCol0 = kACol0 + Roles<false>::kStages * kAColsPerStage;
constexpr int kCorrTmemCols = 128;
static_assert(kCorrCol0 + kCorrTmemCols <= kTmemCols, "TMEM budget with the correction");
constexpr int kBStage = BNH * BK;  // 16 KB of E4M3 per stage
// Output rows staged by the epilogue (16-bit outputs): pitch padded by 16
// bytes, so the 32 rows a warp writes at once fall in distinct bank groups. The
// correction's columns 128..255 lie in the same bytes of their row before.
constexpr int kOutPitch = BN * 2 + 16;
static_assert((BN - kCorrTmemCols) * 4 + 16 == kOutPitch, "a row's correction half and its outputs share the buffer");

// Shared memory of one instantiation: B stages; the tile's epilogue constants
// (row sums R[b][256 columns], channel scales, offsets o[b][128 rows], s_a);
// the staged output rows, which several offset blocks share with half of their
// correction; barriers.
template <bool kOneBlock>
struct Smem {
  static constexpr int kStages = Roles<kOneBlock>::kStages;
  static constexpr int kNumBars = 2 * kStages + 2;
  static constexpr int kMaxG = kOneBlock ? 1 : kMaxStageG;
  static constexpr int kOPitch = kOneBlock ? BM : BM + 4;  // floats per block of staged offsets
  static constexpr int kOffB = 0;
  static constexpr int kOffR = kOffB + kStages * kBStage;
  static constexpr int kOffW = kOffR + kMaxG * BN * 4;
  static constexpr int kOffO = kOffW + BN * 4;
  static constexpr int kOffSa = kOffO + kMaxG * kOPitch * 4;
  static constexpr int kOffRt = kOffSa + BM * 4;    // several blocks: -8 sum_b R[b][n] per column
  static constexpr int kOffOut = kOffRt + BN * 4;   // staged output rows; several blocks: first the correction half
  static constexpr int kOffBars = kOffOut + BM * kOutPitch;
  static constexpr int kOffMisc = kOffBars + kNumBars * 8;
  static constexpr int kBytes = kOffMisc + 64 + 1024;  // + slack to align the base to 1024
  static_assert(kBytes <= 227 * 1024, "shared memory budget");
  static_assert(kOffOut % 16 == 0, "bulk copies need 16-byte aligned rows");
};

constexpr uint32_t kIdesc = idesc_e4m3_f32(2 * BM, BN);  // pair MMA: M = 256, N = 256

struct GemmParams {
  const uint8_t* a_codes;  // tiled [ceil(T/32)*32][K/2]
  const uint8_t* w_codes;  // tiled [ceil(N/32)*32][K/2]
  const float* a_scale;
  const float* a_offset;  // [T][G] or nullptr
  const float* w_scale;
  const float* rowsum;    // [G][N]
  void* out;
  int64_t ldo;
  int32_t* acc_debug;
  int* status;
  int T, N, K, G;
  int m_pairs, n_tiles;    // pair tiles: m_pairs x n_tiles
  int raster_m;            // m-pairs per raster group (see tile_mn)
  int t_blocks, n_blocks;  // 32-row tiles present in the code buffers
  int kchunks;             // K / 32
  int vec_ok;              // rowsum and w_scale rows are 16-byte aligned
  int async_out;           // 16-bit output, N % 8 == 0, no debug output: rows leave by bulk copy
};

// Loads the four 16-byte chunks of k-tile kt of one row of a tiled code matrix
// (zeros where the row block or the chunk does not exist).
// blk: this lane's first byte of the row block (nullptr if the block does not
// exist); the block's chunk c starts 512 * c bytes further.
// pol: the L2 policy of the loads.
__device__ __forceinline__ void load_kt(const uint8_t* blk, int kchunks, int kt, uint4 (&v)[kChunksPerKt],
                                        uint64_t pol) {
#pragma unroll
  for (int j = 0; j < kChunksPerKt; ++j) {
    const int c = kt * kChunksPerKt + j;
    if (blk != nullptr && c < kchunks)
      v[j] = ldg_stream_hint(blk + c * 512, pol);
    else
      v[j] = make_uint4(0u, 0u, 0u, 0u);
  }
}

// Pair tile index -> (m-pair, n-tile). Tiles are taken in groups of raster_m
// m-pairs; within a group the m-pair runs fastest. The clusters running at one
// time then share a few weight tiles across all m-pairs of the group, so each
// weight tile comes from DRAM about once per group while the group's
// activation rows (at most ~32 MB, chosen on the host) stay in L2.
__device__ __forceinline__ void tile_mn(const GemmParams& p, int tile, int& mp, int& nt) {
  const int per_group = p.raster_m * p.n_tiles;
  const int grp = tile / per_group;
  const int local = tile - grp * per_group;
  const int m_left = p.m_pairs - grp * p.raster_m;
  const int gm = m_left < p.raster_m ? m_left : p.raster_m;
  nt = local / gm;
  mp = grp * p.raster_m + (local - nt * gm);
}

__device__ __forceinline__ void tmem_ld_8cols(uint32_t taddr, uint32_t (&r)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr)
               : "memory");
}
// 16 TMEM lanes x 32 columns: lane l of the warp gives, for each 8-column group
// j, row l / 4 columns 2 (l % 4) and + 1 in r[4j], r[4j + 1] and row l / 4 + 8 in
// r[4j + 2], r[4j + 3].
__device__ __forceinline__ void tmem_st_16rows_32cols(uint32_t taddr, const uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.st.sync.aligned.16x256b.x4.b32 [%0], "
      "{%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};" ::"r"(taddr),
      "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]),
      "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
      : "memory");
}
__device__ __forceinline__ void tmem_ld_16rows_32cols(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.16x256b.x4.b32 "
      "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
}
// Where column c of a tile lies so that a lane's 8 columns of 32 (2 m, 2 m + 1 of each 8) are 32 contiguous bytes.
__device__ __forceinline__ int frag_pos(int c) { return (c & ~31) + (c & 6) * 4 + ((c >> 3) & 3) * 2 + (c & 1); }
__device__ __forceinline__ void lds_4x64(const float* p, uint64_t (&v)[4]) {
  const ulonglong2 a = *reinterpret_cast<const ulonglong2*>(p), b = *reinterpret_cast<const ulonglong2*>(p + 4);
  v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y;
}
// Four 8 x 8 matrices of 16-bit values: lane l gives row l / 4, columns 2 (l % 4) and + 1 of matrix j in r[j], and in
// addr the address of row l % 8 of matrix l / 8.
__device__ __forceinline__ void stmatrix4(uint32_t addr, const uint32_t (&r)[4]) {
  asm volatile("stmatrix.sync.aligned.m8n8.x4.shared.b16 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(r[0]), "r"(r[1]),
               "r"(r[2]), "r"(r[3])
               : "memory");
}
__device__ __forceinline__ uint64_t lds64(uint32_t addr) {
  uint64_t v;
  asm volatile("ld.shared.b64 %0, [%1];" : "=l"(v) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ void sts64(uint32_t addr, uint32_t a, uint32_t b) {
  asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(addr), "r"(a), "r"(b) : "memory");
}

// Row block (of 32 rows) of this CTA's A rows / B rows for a pair tile.
__device__ __forceinline__ int a_block(const GemmParams& p, int tile, uint32_t rank, int quarter) {
  int mp, nt;
  tile_mn(p, tile, mp, nt);
  return (mp * 2 * BM + static_cast<int>(rank) * BM + quarter * 32) >> 5;
}

__device__ __forceinline__ int b_block(const GemmParams& p, int tile, uint32_t rank, int wb) {
  int mp, nt;
  tile_mn(p, tile, mp, nt);
  return (nt * BN + static_cast<int>(rank) * BNH + wb * 32) >> 5;
}

// Persistent pair kernel: cluster c processes pair tiles c, c + clusters, ...
// (pair tile index mapped to (m-pair, n-tile) by tile_mn). The k-tile counter g runs
// across tiles so the stage ring never drains between tiles.
// kOneBlock: the offsets span the whole row (G == 1). kWindows: more than
// kMaxStageG offset blocks, staged in windows of that many (2048 tokens x 11904 ->
// 4096 with 93 blocks 139 us; read from global memory at the tile end, 1537). Each
// runs its own instantiation, so the register allocation of the common one-block
// kernel does not carry the G-term epilogue loop, nor that of up to kMaxStageG
// blocks the reload of a window's sums (6912 -> 2560, 27 blocks: 50 us, 56 with it).
// All have 80 registers; with windows two of the three output types spill 4 to 12 bytes.
template <int OUT, bool kOneBlock, bool kWindows>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(Roles<kOneBlock>::kThreads, 1)
    w4a4_gemm_kernel(const GemmParams p) {
  constexpr float kAccScale = 262144.0f;  // operands are integers times 2^-9: the accumulator carries 2^-18
  extern __shared__ uint8_t smem_raw[];
  using SL = Smem<kOneBlock>;
  using RL = Roles<kOneBlock>;
  constexpr int kStages = RL::kStages;
  constexpr int kFirstA = RL::kFirstA, kFirstB = RL::kFirstB, kFirstEpi = RL::kFirstEpi;
  constexpr int kEpiWarps = RL::kEpiWarps;
  constexpr int kOffB = SL::kOffB, kOffR = SL::kOffR, kOffW = SL::kOffW, kOffO = SL::kOffO, kOffSa = SL::kOffSa;
  constexpr int kOffBars = SL::kOffBars, kOffMisc = SL::kOffMisc, kOPitch = SL::kOPitch;
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  uint8_t* smem = smem_raw + (base - raw);

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const uint32_t rank = cluster_rank();
  const int cluster = blockIdx.x >> 1;
  const int clusters = gridDim.x >> 1;
  const int nk = (p.K + BK - 1) / BK;
  const int num_tiles = p.m_pairs * p.n_tiles;

  const uint32_t bar0 = base + kOffBars;
  auto full = [&](int s) { return bar0 + 8u * s; };                // leader: operands of stage s ready
  auto empty = [&](int s) { return bar0 + 8u * (kStages + s); };   // both: stage s consumed
  const uint32_t acc_full = bar0 + 8u * (2 * kStages);             // both: accumulator complete
  const uint32_t acc_empty = bar0 + 8u * (2 * kStages + 1);        // leader: accumulator drained
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + kOffMisc);
  volatile int* abort = reinterpret_cast<volatile int*>(smem + kOffMisc + 16);

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(full(s), 2 * kConvWarpsPerCta);
      mbar_init(empty(s), 1);
    }
    mbar_init(acc_full, 1);
    mbar_init(acc_empty, 2 * kEpiWarps);
    *abort = 0;
    mbar_fence_init();
  }
  if (warp == 0) {
    tmem_alloc2(smem_u32(tmem_slot), kTmemCols);
    tmem_relinquish2();
  }
  tc_fence_before();
  cluster_sync();  // barriers initialised and TMEM allocated in both CTAs
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  // Setup above touches no global memory; from here on, the inputs of the
  // previous kernel in the stream must be complete.
  griddep_wait();
  griddep_launch_dependents();
  int mma_tiles = 0;

  if (warp == 0) {
    // ---------------- MMA issuer (leader CTA) ----------------
    // The whole warp runs the loop; an elected lane issues (elect_one).
    if (rank == 0) {
      const uint64_t desc0 = smem_desc_sw128(base + kOffB);
      int s = 0, phase = 0, lt = 0;  // stage and phase parity of the next k-tile
      for (int tile = cluster; tile < num_tiles; tile += clusters, ++lt) {
        if (!__all_sync(0xFFFFFFFFu, wait_cluster(acc_empty, (lt & 1) ^ 1, abort))) break;
        tc_fence_after();
        bool ok = true;
        for (int kt = 0; kt < nk; ++kt) {
          ok = __all_sync(0xFFFFFFFFu, wait_cluster(full(s), phase, abort));
          if (!ok) break;
          tc_fence_after();
          if (elect_one()) {
            const uint64_t desc = desc0 + static_cast<uint32_t>(s * (kBStage >> 4));
#pragma unroll
            for (int kk = 0; kk < BK / 32; ++kk)
              mma2_ts(tmem, tmem + kACol0 + s * kAColsPerStage + 8 * kk, desc + 2 * kk, kIdesc, (kt | kk) != 0 ? 1u : 0u);
            mma2_commit_both(empty(s));
          }
          __syncwarp();
          if (++s == kStages) {
            s = 0;
            phase ^= 1;
          }
        }
        if (elect_one()) mma2_commit_both(acc_full);
        __syncwarp();
        mma_tiles = lt + 1;
        if (!ok) break;
      }
    }
  } else if (warp < kFirstEpi) {
    // ---------------- converters: packed codes -> E4M3 operands ----------------
    // A warps write 32 TMEM lanes (their quarter); B warps write 32 rows of the
    // shared-memory stage. Each thread keeps kPrefetch k-tiles of loads in
    // flight in a register ring.
    const bool is_a = warp < kFirstB;
    const int quarter = warp & 3;
    const int wb = (warp - kFirstB) & 3;
    const int part = is_a ? (warp - kFirstA) >> 2 : (warp - kFirstB) >> 2;  // k-tiles g == part mod split
    static_assert(RL::kSplitA == RL::kSplitB, "one k-tile stride for both converter kinds");
    constexpr int split = RL::kSplitA;
    const uint32_t full_l = leader_addr(full(0));
    const uint8_t* codes = is_a ? p.a_codes : p.w_codes;
    // The raster keeps a group of m-pairs' activation codes for every n-tile, so
    // they are kept in L2 ahead of the weight tiles streaming past them.
    const uint64_t pol = is_a ? l2_evict_last() : l2_evict_normal();
    const int rb_count = is_a ? p.t_blocks : p.n_blocks;
    // This lane's first byte of the row block a tile needs (nullptr: the block
    // lies past the buffer's rows). Computed once per tile, not per load.
    auto block_ptr = [&](int tile) -> const uint8_t* {
      const int rb = is_a ? a_block(p, tile, rank, quarter) : b_block(p, tile, rank, wb);
      return rb < rb_count ? codes + static_cast<int64_t>(rb) * p.kchunks * 512 + lane * 16 : nullptr;
    };
    uint4 ring[kPrefetch][kChunksPerKt];
    int ld_tile = cluster, ld_kt = 0;  // next k-tile to load
    auto advance1 = [&](int& tile, int& kt) {
      if (++kt == nk) {
        kt = 0;
        tile += clusters;
      }
    };
    auto advance = [&](int& tile, int& kt) {
#pragma unroll
      for (int i = 0; i < split; ++i) advance1(tile, kt);
    };
#pragma unroll
    for (int i = 0; i < split; ++i)
      if (i < part) advance1(ld_tile, ld_kt);
    const int start_tile = ld_tile, start_kt = ld_kt;
#pragma unroll
    for (int i = 0; i < kPrefetch; ++i) {
      if (ld_tile < num_tiles) load_kt(block_ptr(ld_tile), p.kchunks, ld_kt, ring[i], pol);
      advance(ld_tile, ld_kt);
    }
    int tile = start_tile, kt = start_kt;
    int s = part, phase = 0;  // stage and phase parity of this warp's k-tile g (g == part mod split)
    int blk_tile = ld_tile;  // the tile whose row block blk points into
    const uint8_t* blk = ld_tile < num_tiles ? block_ptr(ld_tile) : nullptr;
    bool run = tile < num_tiles;
    while (run) {
#pragma unroll
      for (int slot = 0; slot < kPrefetch; ++slot) {
        if (!run) break;
        // Warp-uniform outcome, so the __syncwarp below is reached by all lanes. After
        // an abort no stage frees up again, so this wait is where a converter stops.
        if (!__all_sync(0xFFFFFFFFu, wait_cluster(empty(s), phase ^ 1, abort))) {
          run = false;
          break;
        }
        if (is_a) {
          tc_fence_after();
          uint32_t f8[32];
#pragma unroll
          for (int j = 0; j < kChunksPerKt; ++j) {
            widen_act(ring[slot][j].x, f8[8 * j + 0], f8[8 * j + 1]);
            widen_act(ring[slot][j].y, f8[8 * j + 2], f8[8 * j + 3]);
            widen_act(ring[slot][j].z, f8[8 * j + 4], f8[8 * j + 5]);
            widen_act(ring[slot][j].w, f8[8 * j + 6], f8[8 * j + 7]);
          }
          tmem_st_32cols(tmem + (static_cast<uint32_t>(quarter * 32) << 16) + kACol0 + s * kAColsPerStage, f8);
          tmem_st_wait();
          tc_fence_before();
        } else {
          const int r = wb * 32 + lane;
          const uint32_t st = base + kOffB + s * kBStage + r * 128;
#pragma unroll
          for (int j = 0; j < kChunksPerKt; ++j) {
            uint32_t a0, a1, a2, a3, b0, b1, b2, b3;
            widen_weight(ring[slot][j].x, a0, a1);
            widen_weight(ring[slot][j].y, a2, a3);
            widen_weight(ring[slot][j].z, b0, b1);
            widen_weight(ring[slot][j].w, b2, b3);
            sts128(st + (((2 * j) ^ (r & 7)) << 4), a0, a1, a2, a3);
            sts128(st + (((2 * j + 1) ^ (r & 7)) << 4), b0, b1, b2, b3);
          }
          fence_proxy_async_smem();
        }
        __syncwarp();
        if (lane == 0) arrive_cluster(full_l + 8u * s);
        // Refill this slot kPrefetch k-tiles ahead.
        if (ld_tile < num_tiles) {
          if (ld_tile != blk_tile) {
            blk_tile = ld_tile;
            blk = block_ptr(ld_tile);
          }
          load_kt(blk, p.kchunks, ld_kt, ring[slot], pol);
        }
        advance(ld_tile, ld_kt);
        advance(tile, kt);
        s += split;
        if (s >= kStages) {
          s -= kStages;
          phase ^= 1;
        }
        run = tile < num_tiles;  // warp-uniform
      }
    }
  } else {
    // ---------------- epilogue ----------------
    const uint64_t out_pol = l2_evict_first();  // outputs: nothing here reads them again
    const int quarter = warp & 3;              // TMEM lanes this warp may read
    const int et = threadIdx.x - kFirstEpi * 32;
    const int G = kOneBlock ? 1 : p.G;
    float* Rs = reinterpret_cast<float*>(smem + kOffR);
    float* Ws = reinterpret_cast<float*>(smem + kOffW);
    float* Os = reinterpret_cast<float*>(smem + kOffO);
    float* Sa = reinterpret_cast<float*>(smem + kOffSa);
    float* Rt = reinterpret_cast<float*>(smem + SL::kOffRt);  // several blocks: -8 sum_b R[b][n]
    const uint32_t acc_empty_l = leader_addr(acc_empty);
    // Loop exit decided only from a flag the epilogue warps write before their
    // own barrier, so all its warps leave together (bar.sync has no timeout).
    volatile int* epi_stop = reinterpret_cast<volatile int*>(smem + kOffMisc + 32);
    if (et == 0) *epi_stop = 0;
    epi_sync<kEpiWarps>();
    int lt = 0;
    for (int tile = cluster; tile < num_tiles; tile += clusters, ++lt) {
      int mp, nt;
      tile_mn(p, tile, mp, nt);
      const int m0 = mp * 2 * BM + static_cast<int>(rank) * BM;
      const int nt0 = nt * BN;
      // Stage this tile's constants while the main loop runs.
      if constexpr (kOneBlock) {
        for (int i = et; i < BN; i += kEpiWarps * 32) {
          const bool in = nt0 + i < p.N;
          Rs[frag_pos(i)] = in ? __ldg(p.rowsum + nt0 + i) : 0.f;
          Ws[frag_pos(i)] = in ? __ldg(p.w_scale + nt0 + i) : 0.f;
        }
        const bool in = m0 + et < p.T;
        Sa[et] = in ? __ldg(p.a_scale + m0 + et) : 0.f;
        Os[et] = in && p.a_offset != nullptr ? __ldg(p.a_offset + m0 + et) : 0.f;
        epi_sync<kEpiWarps>();
      } else {
        // Asynchronous copies, so their latencies overlap: 9.5 k cycles at 43 blocks (22 k as loads into registers).
        // R: thread et takes columns 2 et and 2 et + 1 of every block, placed so that the 8 columns a lane multiplies
        // below are 32 contiguous bytes. More than kMaxStageG blocks come in windows, the correction carried on.
        const int c2 = 2 * et, n2 = nt0 + c2;
        float* rdst = Rs + (c2 & ~31) + (c2 & 7) * 4 + ((c2 >> 3) & 3) * 2;
        Ws[c2] = n2 < p.N ? __ldg(p.w_scale + n2) : 0.f;
        Ws[c2 + 1] = n2 + 1 < p.N ? __ldg(p.w_scale + n2 + 1) : 0.f;
        Sa[et] = m0 + et < p.T ? __ldg(p.a_scale + m0 + et) : 0.f;
        if (p.async_out) bulk_wait_read_all();  // this row's previous output copy has read the buffer
        float rt0 = 0.f, rt1 = 0.f;
        for (int b0 = 0; b0 < (kWindows ? G : 1); b0 += kMaxStageG) {
        const int Gw = kWindows && G - b0 > kMaxStageG ? kMaxStageG : G - b0;  // blocks of this window
        if (kWindows && b0 > 0) epi_sync<kEpiWarps>();  // the previous window has been read
        if (p.vec_ok && n2 < p.N) {
          const float* src = p.rowsum + static_cast<int64_t>(b0) * p.N + n2;
          for (int b = 0; b < Gw; ++b, src += p.N) cp_async<8>(smem_u32(rdst + b * BN), src);
        } else {
          for (int b = 0; b < Gw; ++b) {
            const float* src = p.rowsum + static_cast<int64_t>(b0 + b) * p.N + n2;
            rdst[b * BN] = n2 < p.N ? __ldg(src) : 0.f;
            rdst[b * BN + 1] = n2 + 1 < p.N ? __ldg(src + 1) : 0.f;
          }
        }
        // Offsets, [b][row]: rows q, q + 8, q + 16, q + 24 of a 32-row group side by side.
        {
          const float* o0 = p.a_offset + static_cast<int64_t>(m0) * G + b0;
          const int step_r = kEpiWarps * 32 / Gw, step_b = kEpiWarps * 32 - step_r * Gw;
          int r = et / Gw, b = et - r * Gw;
          while (r < BM) {
            float* dst = Os + b * kOPitch + (r & ~31) + (r & 7) * 4 + ((r >> 3) & 3);
            if (p.a_offset != nullptr && m0 + r < p.T)
              cp_async<4>(smem_u32(dst), o0 + static_cast<int64_t>(r) * G + b);
            else
              *dst = 0.f;
            r += step_r;
            b += step_b;
            if (b >= Gw) {
              b -= Gw;
              ++r;
            }
          }
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
        // Rt[n] = -8 sum_b R[b][n]: integers, exact in fp32. (This thread's own copies.)
#pragma unroll 4
        for (int bb = 0; bb < Gw; ++bb) {
          const float2 v = *reinterpret_cast<const float2*>(rdst + bb * BN);
          rt0 += v.x;
          rt1 += v.y;
        }
        Rt[c2] = rt0 * -8.f;
        Rt[c2 + 1] = rt1 * -8.f;
        epi_sync<kEpiWarps>();
        // While this tile's MMAs run: its offset correction, per element the same chain as at the tile end (block 0
        // multiplied, then FMAs in block order). A lane takes 4 rows x 8 columns at a time, the fragment that a
        // 16-lane x 256-bit TMEM store takes: 3 shared reads of 16 bytes per 32 multiply-adds, where one row and 16
        // columns per lane took 5 per 16. With 43 blocks it still is the longest part of a tile (2048 tokens x 11008 ->
        // 4096 98.6 -> 74.5 us with the staging and the drain): 59 k cycles, about half of them multiply-adds at one
        // warp per sub-partition. Reading a block ahead (81 us: registers) and scalar multiply-adds (80 us) were slower.
        const int q = lane >> 2, m = lane & 3;
        const float* op = Os + quarter * 32 + q * 4;
        const uint32_t corr_tm = tmem + (static_cast<uint32_t>(quarter * 32) << 16) + kCorrCol0;
        const uint32_t corr_s = base + SL::kOffOut + (quarter * 32 + q) * kOutPitch + m * 8;
        for (int sb = 0; sb < BN / 32; ++sb) {
          const float* rp = Rs + sb * 32 + m * 8;
          uint64_t y[4][4];  // [row q + 8 i][column pair 8 j + 2 m]
          const uint32_t tm = corr_tm + sb * 32;
          const uint32_t sm = corr_s + (sb * 32 - kCorrTmemCols) * 4;
          int bb = 0;
          if (!kWindows || b0 == 0) {
            const float4 o = *reinterpret_cast<const float4*>(op);
            const float4 ra = *reinterpret_cast<const float4*>(rp), rb = *reinterpret_cast<const float4*>(rp + 4);
            const uint64_t R[4] = {pack2(ra.x, ra.y), pack2(ra.z, ra.w), pack2(rb.x, rb.y), pack2(rb.z, rb.w)};
            const uint64_t O[4] = {pack2(o.x, o.x), pack2(o.y, o.y), pack2(o.z, o.z), pack2(o.w, o.w)};
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
              for (int j = 0; j < 4; ++j) y[i][j] = mul2v(O[i], R[j]);
            bb = 1;
          } else if (sb * 32 < kCorrTmemCols) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              uint32_t u[16];
              tmem_ld_16rows_32cols(tm + (static_cast<uint32_t>(16 * h) << 16), u);
              tmem_ld_wait_for(u);
#pragma unroll
              for (int j = 0; j < 4; ++j) {
                y[2 * h][j] = pack2(__uint_as_float(u[4 * j]), __uint_as_float(u[4 * j + 1]));
                y[2 * h + 1][j] = pack2(__uint_as_float(u[4 * j + 2]), __uint_as_float(u[4 * j + 3]));
              }
            }
          } else {
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
              for (int j = 0; j < 4; ++j) y[i][j] = lds64(sm + 8 * i * kOutPitch + 32 * j);
          }
#pragma unroll 2
          for (; bb < Gw; ++bb) {
            const float4 o = *reinterpret_cast<const float4*>(op + bb * kOPitch);
            const float4 ra = *reinterpret_cast<const float4*>(rp + bb * BN);
            const float4 rb = *reinterpret_cast<const float4*>(rp + bb * BN + 4);
            const uint64_t R[4] = {pack2(ra.x, ra.y), pack2(ra.z, ra.w), pack2(rb.x, rb.y), pack2(rb.z, rb.w)};
            const uint64_t O[4] = {pack2(o.x, o.x), pack2(o.y, o.y), pack2(o.z, o.z), pack2(o.w, o.w)};
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
              for (int j = 0; j < 4; ++j) y[i][j] = fma2v(O[i], R[j], y[i][j]);
          }
          if (sb * 32 < kCorrTmemCols) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              uint32_t u[16];
#pragma unroll
              for (int j = 0; j < 4; ++j) {
                float v0, v1, v2, v3;
                unpack2(y[2 * h][j], v0, v1);
                unpack2(y[2 * h + 1][j], v2, v3);
                u[4 * j] = __float_as_uint(v0); u[4 * j + 1] = __float_as_uint(v1);
                u[4 * j + 2] = __float_as_uint(v2); u[4 * j + 3] = __float_as_uint(v3);
              }
              tmem_st_16rows_32cols(tm + (static_cast<uint32_t>(16 * h) << 16), u);
            }
          } else {
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
              for (int j = 0; j < 4; ++j) {
                float v0, v1;
                unpack2(y[i][j], v0, v1);
                sts64(sm + 8 * i * kOutPitch + 32 * j, __float_as_uint(v0), __float_as_uint(v1));
              }
          }
        }
        tmem_st_wait();
        }
        __syncwarp();  // a row's correction comes from four lanes
      }
      const bool ok = __all_sync(0xFFFFFFFFu, wait_cluster(acc_full, lt & 1, abort));
      if (!ok && lane == 0) *epi_stop = 1;
      tc_fence_after();
      const int rl = quarter * 32 + lane;
      const int t = m0 + rl;
      const bool row_ok = t < p.T;
      const uint32_t acc_tm = tmem + (static_cast<uint32_t>(quarter * 32) << 16);
      constexpr int CW = 16;  // accumulator columns per TMEM load
      bool released = false;
      // The accumulator has been read: the next tile's MMAs may start.
      auto release = [&] {
        tc_fence_before();
        __syncwarp();
        if (lane == 0) arrive_cluster(acc_empty_l);
        released = true;
      };
      const uint32_t orow_s = base + SL::kOffOut + rl * kOutPitch;
      const bool async_out = OUT != OFFQ_F32 && p.async_out != 0;
      if (!ok) {
        // Aborted: nothing to drain.
      } else if (async_out) {
        // 16-bit rows go to shared memory and leave by one bulk copy per row, so the tile's output write overlaps the
        // next tile's MMAs. No MMA runs during the drain, so its length adds to the tile: the next columns are on
        // their way while these are scaled, and the accumulator is handed back before the last of them and the copies.
        // Rows and columns past the end are computed from zeros and not copied, so no lane branches. 9.2 k cycles
        // before, of a tile's 30 k at K = 4096, now 2.9 k: 8192 tokens x 4096 -> 4096 98 -> 89 us, -> 11008 248 ->
        // 222 us; 14 blocks of 1024 -> 4096 at 2048 tokens (there with strided 32-byte stores) 93 -> 88 us.
        if constexpr (kOneBlock) {
          // 16-lane x 256-bit fragments: a lane holds 4 rows x 8 columns of every 32, so R and s_w are read once per 4
          // rows (one row per lane: 128 reads of 16 bytes each, now 32), and one stmatrix stores 8 rows x 32 columns.
          // With one warp per sub-partition the drain's length is its instruction count: 2048 tokens x 4096 -> 4096
          // 29.5 -> 28.9 us, x 8192 -> 28672 290.5 -> 285.0 (without stmatrix 29.2 and 287.7; scalar FMAs 30.5, 296.9).
          // Packed fp32 pairs; each lane rounds as y = s_w * fma(s_a, acc * 2^18, o R)
          // does, with acc = (acc' - 8 R) 2^-18 formed exactly first (s_a * 2^18 and
          // its product with acc are exact).
          const int q = lane >> 2, m = lane & 3;
          const uint64_t M8 = pack2(-0x1p-15f, -0x1p-15f);  // -8 * 2^-18
          float sa2[4], ob[4];  // rows q + 8 i
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            sa2[i] = Sa[quarter * 32 + q + 8 * i] * kAccScale;
            ob[i] = Os[quarter * 32 + q + 8 * i];
          }
          // This lane's row of the 8 x 8 matrices a stmatrix writes: row lane % 8, columns 8 (lane / 8).
          const uint32_t frow_s = base + SL::kOffOut + (quarter * 32 + (lane & 7)) * kOutPitch + (lane >> 3) * 16;
          bulk_wait_read_all();  // these rows' previous copies have read the buffer
          __syncwarp();
          uint64_t R[4], Wc[4];
          // Rows q + 16 h, q + 16 h + 8 of 32 columns.
          auto emit = [&](int sb, int h, const uint32_t (&acc)[CW]) {
#pragma unroll
            for (int i = 0; i < 2; ++i) {
              const int r = 2 * h + i;
              const uint64_t SA2 = pack2(sa2[r], sa2[r]), OB = pack2(ob[r], ob[r]);
              uint32_t hv[4];
#pragma unroll
              for (int j = 0; j < 4; ++j) {
                uint64_t A = pack2(__uint_as_float(acc[4 * j + 2 * i]), __uint_as_float(acc[4 * j + 2 * i + 1]));
                A = fma2v(R[j], M8, A);
                float y0, y1;
                unpack2(mul2v(Wc[j], fma2v(SA2, A, mul2v(OB, R[j]))), y0, y1);
                hv[j] = pack_out<OUT>(y0, y1);
              }
              stmatrix4(frow_s + 8 * r * kOutPitch + sb * 64, hv);
            }
          };
          uint32_t a0[CW], a1[CW];
          tmem_ld_16rows_32cols(acc_tm, a0);
#pragma unroll
          for (int sb = 0; sb < BN / 32; ++sb) {
            lds_4x64(Rs + sb * 32 + m * 8, R);
            lds_4x64(Ws + sb * 32 + m * 8, Wc);
            tmem_ld_wait_for(a0);
            tmem_ld_16rows_32cols(acc_tm + (16u << 16) + sb * 32, a1);
            emit(sb, 0, a0);
            tmem_ld_wait_for(a1);
            if (sb + 1 < BN / 32)
              tmem_ld_16rows_32cols(acc_tm + (sb + 1) * 32, a0);
            else
              release();
            emit(sb, 1, a1);
          }
          fence_proxy_async_smem();  // a row's outputs come from four lanes and leave by one's bulk copy
          __syncwarp();
        } else {
          // Several blocks: columns 128..255 first, from the highest down, because their outputs overwrite corrections
          // of higher columns of the row; then 0..127, whose corrections are in TMEM.
          const float sa = Sa[rl];
          const uint64_t SA = pack2(sa, sa), K18 = pack2(kAccScale, kAccScale);
          const uint32_t corr_tm = tmem + (static_cast<uint32_t>(quarter * 32) << 16) + kCorrCol0;
          // z = s_w * fma(s_a, acc' 2^18 + Rt, correction) of 4 columns from j; the inner sum is an exact integer.
          auto four = [&](int j, uint32_t x0, uint32_t x1, uint32_t x2, uint32_t x3, uint64_t c0, uint64_t c1,
                          uint32_t& h0, uint32_t& h1) {
            const float4 rt = *reinterpret_cast<const float4*>(Rt + j), wv = *reinterpret_cast<const float4*>(Ws + j);
            const uint64_t A0 = fma2v(pack2(__uint_as_float(x0), __uint_as_float(x1)), K18, pack2(rt.x, rt.y));
            const uint64_t A1 = fma2v(pack2(__uint_as_float(x2), __uint_as_float(x3)), K18, pack2(rt.z, rt.w));
            float y0, y1, y2, y3;
            unpack2(mul2v(pack2(wv.x, wv.y), fma2v(SA, A0, c0)), y0, y1);
            unpack2(mul2v(pack2(wv.z, wv.w), fma2v(SA, A1, c1)), y2, y3);
            h0 = pack_out<OUT>(y0, y1);
            h1 = pack_out<OUT>(y2, y3);
          };
          auto pair2 = [](uint32_t a, uint32_t b) { return pack2(__uint_as_float(a), __uint_as_float(b)); };
          auto emit_s = [&](int c, const uint32_t (&acc)[CW]) {
            uint32_t hv[CW / 2];
#pragma unroll
            for (int q4 = 0; q4 < CW / 4; ++q4) {
              const uint4 v = lds128(orow_s + (c * CW - kCorrTmemCols) * 4 + 16 * q4);
              four(c * CW + 4 * q4, acc[4 * q4], acc[4 * q4 + 1], acc[4 * q4 + 2], acc[4 * q4 + 3], pair2(v.x, v.y),
                   pair2(v.z, v.w), hv[2 * q4], hv[2 * q4 + 1]);
            }
            sts128(orow_s + c * CW * 2, hv[0], hv[1], hv[2], hv[3]);
            sts128(orow_s + c * CW * 2 + 16, hv[4], hv[5], hv[6], hv[7]);
          };
          {
            constexpr int kFirst = kCorrTmemCols / CW, kLast = BN / CW - 1;
            uint32_t a0[CW], a1[CW];
            tmem_ld_16cols(acc_tm + kLast * CW, a0);
#pragma unroll
            for (int c = kLast; c > kFirst; c -= 2) {
              tmem_ld_wait_for(a0);
              tmem_ld_16cols(acc_tm + (c - 1) * CW, a1);
              emit_s(c, a0);
              tmem_ld_wait_for(a1);
              if (c - 2 > kFirst) tmem_ld_16cols(acc_tm + (c - 2) * CW, a0);
              emit_s(c - 1, a1);
            }
          }
          auto emit_t = [&](int j, const uint32_t (&acc)[8], const uint32_t (&cr)[8]) {
            uint32_t hv[4];
#pragma unroll
            for (int q4 = 0; q4 < 2; ++q4)
              four(j + 4 * q4, acc[4 * q4], acc[4 * q4 + 1], acc[4 * q4 + 2], acc[4 * q4 + 3],
                   pair2(cr[4 * q4], cr[4 * q4 + 1]), pair2(cr[4 * q4 + 2], cr[4 * q4 + 3]), hv[2 * q4],
                   hv[2 * q4 + 1]);
            sts128(orow_s + j * 2, hv[0], hv[1], hv[2], hv[3]);
          };
          uint32_t a0[8], c0[8], a1[8], c1[8];
          tmem_ld_8cols(acc_tm, a0);
          tmem_ld_8cols(corr_tm, c0);
#pragma unroll
          for (int j = 0; j < kCorrTmemCols; j += 16) {
            tmem_ld_wait_for(a0, c0);
            tmem_ld_8cols(acc_tm + j + 8, a1);
            tmem_ld_8cols(corr_tm + j + 8, c1);
            emit_t(j, a0, c0);
            tmem_ld_wait_for(a1, c1);
            if (j + 16 < kCorrTmemCols) {
              tmem_ld_8cols(acc_tm + j + 16, a0);
              tmem_ld_8cols(corr_tm + j + 16, c0);
            } else {
              release();
            }
            emit_t(j + 8, a1, c1);
          }
        }
        if (row_ok && nt0 < p.N) {
          const int ncols = p.N - nt0 < BN ? p.N - nt0 : BN;
          fence_proxy_async_smem();  // the row's shared stores, visible to the bulk copy
          bulk_store(static_cast<uint16_t*>(p.out) + static_cast<int64_t>(t) * p.ldo + nt0, orow_s,
                     static_cast<uint32_t>(ncols) * 2, out_pol);
          bulk_commit();
        }
      } else {
        // 32-bit outputs, rows that no bulk copy can write, and calls that want the accumulator: straight from
        // registers.
        const float sa = Sa[rl];
        const float ob = kOneBlock ? Os[rl] : 0.f;
        const uint32_t corr_tm = tmem + (static_cast<uint32_t>(quarter * 32) << 16) + kCorrCol0;
        for (int c = 0; c < BN / CW; ++c) {
          const int jc = c * CW;  // column within the tile
          uint32_t acc[CW], cr[CW];
          tmem_ld_16cols(acc_tm + jc, acc);
          if (!kOneBlock && jc < kCorrTmemCols) tmem_ld_16cols(corr_tm + jc, cr);
          tmem_ld_wait_for(acc);
          if (!kOneBlock && jc < kCorrTmemCols) tmem_ld_wait_for(cr);
          const int nb = nt0 + jc;
          if (nb >= p.N) break;
          if (!kOneBlock && jc >= kCorrTmemCols) {
#pragma unroll
            for (int q4 = 0; q4 < CW / 4; ++q4) {
              const uint4 v = lds128(orow_s + (jc - kCorrTmemCols) * 4 + 16 * q4);
              cr[4 * q4] = v.x; cr[4 * q4 + 1] = v.y; cr[4 * q4 + 2] = v.z; cr[4 * q4 + 3] = v.w;
            }
          }
          const int nvalid = p.N - nb < CW ? p.N - nb : CW;
          float z[CW];
#pragma unroll
          for (int jj = 0; jj < CW; ++jj) {
            const float r8 = kOneBlock ? Rs[frag_pos(jc + jj)] * -8.f : Rt[jc + jj];
            const float corr = kOneBlock ? ob * Rs[frag_pos(jc + jj)] : __uint_as_float(cr[jj]);
            const float accf = fmaf(__uint_as_float(acc[jj]), kAccScale, r8);  // an exact integer
            z[jj] = Ws[kOneBlock ? frag_pos(jc + jj) : jc + jj] * fmaf(sa, accf, corr);
          }
          if (row_ok) store_out<OUT, CW>(p.out, static_cast<int64_t>(t) * p.ldo + nb, z, nvalid, out_pol);
          if (row_ok && p.acc_debug != nullptr) {
            int32_t* d = p.acc_debug + static_cast<int64_t>(t) * p.N + nb;
#pragma unroll
            for (int jj = 0; jj < CW; ++jj)
              if (jj < nvalid) d[jj] = __float2int_rn(__uint_as_float(acc[jj]) * 262144.0f);
          }
          __syncwarp();  // the next columns' load needs every lane
        }
      }
      if (ok && !released) release();
      epi_sync<kEpiWarps>();  // the staged constants are reused for the next tile
      if (*epi_stop) break;
    }
    bulk_wait_all();  // output rows in flight are written before the CTA ends
  }

  // ---------------- teardown ----------------
  if (*abort && warp == 0 && lane == 0 && rank == 0 && mma_tiles > 0) {
    // Let the MMAs already issued finish before tensor memory is released.
    wait_teardown(acc_full, (mma_tiles - 1) & 1);
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync();  // the pair's MMAs read both CTAs' memory: leave together
  if (warp == 0) {
    tc_fence_after();
    tmem_dealloc2(tmem, kTmemCols);
  }
  if (threadIdx.x == 0 && *abort && p.status != nullptr) atomicExch(p.status, kErrTimeout);
}

template <int OUT, bool kOneBlock, bool kWindows>
int launch_gemm(const GemmParams& p, cudaStream_t s) {
  auto kern = w4a4_gemm_kernel<OUT, kOneBlock, kWindows>;
  constexpr int kThreads = Roles<kOneBlock>::kThreads;
  constexpr int kSmemBytes = Smem<kOneBlock>::kBytes;
  if (!smem_optin<w4a4_gemm_kernel<OUT, kOneBlock, kWindows>>(kSmemBytes)) return OFFQ_ERR_CUDA;
  const int sms = device_sms();
  if (sms < 2) return OFFQ_ERR_CUDA;
  const int tiles = p.m_pairs * p.n_tiles;
  const int clusters = tiles < sms / 2 ? tiles : sms / 2;
  return launch_pdl(kern, dim3(2 * clusters), dim3(kThreads), kSmemBytes, s, p);
}

int dispatch_gemm(const GemmParams& p, int out_dtype, cudaStream_t s) {
  const bool windows = p.G > kMaxStageG;
  switch (out_dtype) {
    case OFFQ_F32:
      return p.G == 1 ? launch_gemm<OFFQ_F32, true, false>(p, s)
             : windows ? launch_gemm<OFFQ_F32, false, true>(p, s)
                       : launch_gemm<OFFQ_F32, false, false>(p, s);
    case OFFQ_BF16:
      return p.G == 1 ? launch_gemm<OFFQ_BF16, true, false>(p, s)
             : windows ? launch_gemm<OFFQ_BF16, false, true>(p, s)
                       : launch_gemm<OFFQ_BF16, false, false>(p, s);
    case OFFQ_F16:
      return p.G == 1 ? launch_gemm<OFFQ_F16, true, false>(p, s)
             : windows ? launch_gemm<OFFQ_F16, false, true>(p, s)
                       : launch_gemm<OFFQ_F16, false, false>(p, s);
    default: return OFFQ_ERR_INVALID_ARG;
  }
}

// The shapes, tile counts and raster of one launch (arguments already checked).
GemmParams gemm_params(const uint8_t* a_codes, const float* a_scale, const float* a_offset, int64_t T, int64_t N,
                       int64_t K, int32_t g, const uint8_t* w_codes, const float* w_scale, const float* w_offsum,
                       void* out, int out_dtype, int64_t ldo, int32_t* acc_debug) {
  GemmParams p{};
  p.a_codes = a_codes;
  p.w_codes = w_codes;
  p.a_scale = a_scale;
  p.a_offset = a_offset;
  p.w_scale = w_scale;
  p.rowsum = w_offsum;
  p.out = out;
  p.ldo = ldo;
  p.acc_debug = acc_debug;
  p.status = device_status_ptr();
  p.T = static_cast<int>(T);
  p.N = static_cast<int>(N);
  p.K = static_cast<int>(K);
  p.G = static_cast<int>(K / g);
  p.m_pairs = static_cast<int>((T + 2 * BM - 1) / (2 * BM));
  p.n_tiles = static_cast<int>((N + BN - 1) / BN);
  // Raster groups of m-pairs whose activation codes total at most ~32 MB.
  const int64_t pair_bytes = 2 * BM * (K / 2);
  int64_t rm = (int64_t{32} << 20) / pair_bytes;
  if (rm < 1) rm = 1;
  p.raster_m = static_cast<int>(rm < p.m_pairs ? rm : p.m_pairs);
  p.t_blocks = static_cast<int>((T + 31) / 32);
  p.n_blocks = static_cast<int>((N + 31) / 32);
  p.kchunks = static_cast<int>(K / 32);
  p.vec_ok = aligned(w_offsum, 16) && aligned(w_scale, 16) && (N % 4 == 0);
  p.async_out = out_dtype != OFFQ_F32 && N % 8 == 0 && acc_debug == nullptr;
  return p;
}

// The form a shape takes: the cluster form where its cost rule says so, else by tokens.
int linear_form(int64_t T, int64_t N, int64_t K, int32_t g) {
  if (mid_takes(T, N, K, K / g)) return OFFQ_FORM_MID;
  return T <= few_max_tokens() ? OFFQ_FORM_FEW : OFFQ_FORM_PAIR;
}

// The shape rules of offq_w4a4_linear.
int check_linear_shape(int64_t T, int64_t N, int64_t K, int32_t g) {
  if (T < 0 || N < 1 || !is_pow2(g) || g < 32 || g > 8192) return OFFQ_ERR_INVALID_ARG;
  if (K <= 0 || K % g != 0 || K % 32 != 0) return OFFQ_ERR_INVALID_ARG;
  if (K > kMaxGemmK || T > 0x3FFFFFFF || N > 0x3FFFFFFF) return OFFQ_ERR_UNSUPPORTED;
  return OFFQ_OK;
}

}  // namespace

extern "C" int offq_w4a4_linear_form(int64_t T, int64_t N, int64_t K, int32_t g) {
  const int rc = check_linear_shape(T, N, K, g);
  if (rc != OFFQ_OK) return rc;
  return device_sms() < 1 ? OFFQ_ERR_CUDA : linear_form(T, N, K, g);
}

extern "C" int offq_w4a4_linear(const uint8_t* a_codes, const float* a_scale, const float* a_offset, int64_t T,
                                int64_t N, int64_t K, int32_t g, const uint8_t* w_codes, const float* w_scale,
                                const float* w_offsum, void* out, int out_dtype, int64_t ldo, int32_t* acc_debug,
                                void* stream) {
  const int ob = elem_bytes(out_dtype);
  const int rc = check_linear_shape(T, N, K, g);
  if (ob == 0 || ldo < N || rc == OFFQ_ERR_INVALID_ARG) return OFFQ_ERR_INVALID_ARG;
  if (rc != OFFQ_OK) return rc;
  if (T == 0) return OFFQ_OK;
  if (a_codes == nullptr || a_scale == nullptr || w_codes == nullptr || w_scale == nullptr || w_offsum == nullptr ||
      out == nullptr)
    return OFFQ_ERR_INVALID_ARG;
  if (!aligned(a_codes, 16) || !aligned(w_codes, 16) || !aligned(out, 16) || (ldo * ob) % 16 != 0 ||
      !aligned(a_scale, 4) || !aligned(w_scale, 4) || !aligned(w_offsum, 4) ||
      (a_offset != nullptr && !aligned(a_offset, 4)) || (acc_debug != nullptr && !aligned(acc_debug, 4)))
    return OFFQ_ERR_MISALIGNED;

  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const int form = linear_form(T, N, K, g);
  if (form == OFFQ_FORM_MID)
    return w4a4_linear_mid(a_codes, a_scale, a_offset, T, N, K, g, w_codes, w_scale, w_offsum, out, out_dtype, ldo,
                           acc_debug, s);
  if (form == OFFQ_FORM_FEW)
    return w4a4_linear_few(a_codes, a_scale, a_offset, T, N, K, g, w_codes, w_scale, w_offsum, out, out_dtype, ldo,
                           acc_debug, s);
  const GemmParams p = gemm_params(a_codes, a_scale, a_offset, T, N, K, g, w_codes, w_scale, w_offsum, out, out_dtype,
                                   ldo, acc_debug);
  return dispatch_gemm(p, out_dtype, s);
}
