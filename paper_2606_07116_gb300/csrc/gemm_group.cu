// W4A4 GEMM with per-group activation scales and zero-points
// (offq_w4a4_linear_group): the paper's evaluated activation setting, groups
// of 128 channels quantized asymmetrically (Sec. 3 Eq. 1 with its zero-point,
// Sec. 4 settings), against per-channel symmetric 4-bit weights.
//
//   y[t][n] = s_w[n] * sum_j s[t][j] * (P_j[t][n] - z[t][j] * R[j][n])
//   P_j[t][n] = sum_{k in group j} u[t][k] * q_w[n][k]
//
// u in [0, 15] is the stored code (Eq. 1's x_q), q_w in [-7, 7], and R[j][n]
// the integer row sum of the weight codes over group j. Both codes widen to
// exact E4M3 operands (bytes 0x00..0x0F are 0..15 * 2^-9), so P_j, an integer
// times 2^-18 below 2^24 * 2^-18, is exact in the fp32 accumulator.
//
// One 128-code k-tile is one group, so the per-(token, group) scale cannot sit
// in the operands: the pair MMA (M 256, N 128) writes each group's P_j into one
// of three TMEM partial buffers, and sixteen scaler warps fold it into a running
// fp32 sum held in their registers,
//   d = fma(-z, R, acc)   (exact while |z R| < 2^24),   S = fma(s, d, S),
// (on the accumulator's values * 2^-18, with the factors scaled to match),
// while the MMA fills the other buffers. After a tile's last group the scalers
// multiply by s_w and store y, rounding once to the output type.
//
// What bounds it: issue slots of the SM sub-partitions and the chain of one group.
// Per group a sub-partition has 32 rows x 128 columns to fold (256 cycles of its
// FMA pipe) among about 780 warp instructions (waits, TMEM and shared-memory loads,
// conversions, bookkeeping: 3130 per CTA), and the kernel takes about 1130 cycles
// per group against 296 of MMA (N = 128, A in tensor memory). Hence four
// scaler warps per sub-partition (the latency of one is three times its issue
// time), R read while the partial is waited for, s, z and R in shared memory in
// windows of 16 groups (read from global memory per lane, one row each, they cost
// 32 cache lines per load), and the registers shifted from the converters to the
// scalers. The zero-point sits with the scalers' FMAs: subtracting it in the
// converters costs more issue slots (byte-wise |u - z| and its sign, ~20 operations
// per 8 codes against 3 for the plain nibbles) and still needs the FMA for a group
// that does not straddle zero.
//
// At a few groups the time is the chain around them, so: the windows' copies cover
// only what exists, come from three warps and arrive on their barrier by themselves
// (one warp that zero-filled the rest and waited for its copies: 64 x 512 -> 512
// 6.7 us, now 5.5); a tile's channel scales come with its last window (handed round
// by shuffles, 0.4 us of that); each role reaches its wait for the kernel ahead with
// its registers and addresses ready (0.2 us); outputs leave in whole 64-byte runs.
//
// Measured (per call, weights past the L2; before: eight scaler warps, two
// buffers, z in the operands, s and z by per-lane loads): 2048 x 4096 -> 4096
// 72.4 us (126.8), -> 11008 175.8 us (315.7), 2048 x 11008 -> 4096 185.8 us
// (321.3), 1 x 4096 -> 11008 36.8 us (54.8), 64 x 512 -> 512 5.5 us (6.3), 2048 x
// 512 -> 8192 27.4 us (34.9), 2048 x 256 -> 8192 20.0 us (23.2). Only at one group,
// and at two with few tokens, does the former still lead (64 x 128 -> 128 4.1 us
// against 3.6, 64 x 256 -> 8192 5.7 against 5.3).
//
// TMEM (512 columns per CTA): P0, P1, P2 [0, 384), 4 A stages of 32 columns.
//
// Warp roles per CTA (32 warps of 64 registers, with 60 / 96 bytes of spill stores / loads; 48 after the start for
// warps 0-15, 80 for the scalers):
//   warp 0       TMEM allocation; in the leader CTA, an elected lane issues the MMAs
//   warps 1-3    stage the windows of s, z and R (cp.async)
//   warps 4-11   A converters: two per 32-lane TMEM quarter, taking turns by group
//   warps 12-15  B converters: two per 32-row group (64 rows of B per CTA)
//   warps 16-31  scalers and epilogue, four per TMEM quarter (32 columns each)
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

constexpr int GBM = 128;         // rows of A per CTA (256 per pair)
constexpr int GBN = 128;         // output channels per pair tile
constexpr int GBNH = GBN / 2;    // rows of B held by one CTA
constexpr int GBK = 128;         // codes per k-tile = one activation group
constexpr int kGroup = GBK;
constexpr int kGChunks = GBK / 32;  // 16-byte packed chunks per row per k-tile
constexpr int kGStages = 4;
constexpr int kGBufs = 3;           // partial buffers
constexpr int kGRing = 1;           // k-tiles of loads in flight per converter thread (two do not fit 64 registers)
constexpr int kGTurns = 2;          // converter warps per row group, taking turns
constexpr int kGFirstA = 4, kGFirstB = kGFirstA + 4 * kGTurns;
constexpr int kGFirstSc = kGFirstB + GBNH / 32 * kGTurns;
constexpr int kGScWarps = 16;            // four per TMEM quarter
constexpr int kGScCols = GBN / (kGScWarps / 4);  // columns per scaler warp
constexpr int kGThreads = (kGFirstSc + kGScWarps) * 32;
constexpr int kGArrivals = 4 + GBNH / 32;  // per stage and CTA: one per A quarter and per B row group
constexpr int kGACol0 = kGBufs * GBN;      // A stages
constexpr int kGAColsPerStage = GBK / 4;
constexpr int kGTmemCols = 512;
static_assert(kGACol0 + kGStages * kGAColsPerStage <= kGTmemCols, "TMEM budget");
static_assert(kGTurns <= kGStages, "a converter's next stage is at most one ring turn ahead");
constexpr int kGBStage = GBNH * GBK;  // 8 KB of E4M3 per stage
constexpr uint32_t kGIdesc = idesc_e4m3_f32(2 * GBM, GBN);  // pair MMA: M = 256, N = 128

// Windows of 16 groups, double-buffered: s and z as [128 rows][16 groups], the four
// 16-byte pieces of a row at piece ^ (row / 2 % 4), so that eight rows' reads of one
// piece fall in distinct banks; R as [16 groups][128 columns]; a tile's last window
// with the channel scales.
constexpr int kGWin = 16;
constexpr int kGWinThreads = 96;               // warps 1-3
constexpr int kWinRows = GBM * kGWin * 4;          // 8 KB of s (and of z)
constexpr int kWinR = kGWin * GBN * 4;             // 8 KB of R
constexpr int kWinW = 2 * kWinRows + kWinR;        // a tile's last window: its channel scales, 512 bytes
constexpr int kWinBytes = kWinW + GBN * 4;

constexpr int kGOffWin = kGStages * kGBStage;
constexpr int kGOutBytes = 32 * 64;      // a scaler warp's buffer for its outputs' way out
constexpr int kGOffOut = kGOffWin + 2 * kWinBytes;
constexpr int kGOffBars = kGOffOut + kGScWarps * kGOutBytes;
constexpr int kGNumBars = 2 * kGStages + 2 * kGBufs + 4;
constexpr int kGOffMisc = kGOffBars + kGNumBars * 8;
constexpr int kGUsed = kGOffMisc + 64 + 1024;
// Padded so that one CTA holds an SM: the pair allocates all 512 TMEM columns.
constexpr int kGBytes = kGUsed < 120 * 1024 ? 120 * 1024 : kGUsed;

struct GroupParams {
  const uint8_t* a_codes;  // tiled [ceil(T/32)*32][K/2], unsigned codes
  const uint8_t* w_codes;  // tiled [ceil(N/32)*32][K/2]
  const float* a_scale;    // [T][Gq]
  const float* a_zero;     // [T][Gq]
  const float* w_scale;    // [N]
  const float* gsum;       // [Gq][N]
  void* out;
  int64_t ldo;
  int* status;
  int T, N, K, Gq;
  int m_pairs, n_tiles;
  int t_blocks, n_blocks;
  int kchunks;  // K / 32
  int vec_sz;   // rows of s and z allow 16-byte copies
  int vec_r;    // rows of R allow 16-byte copies
  int vec_w;    // s_w too
};

// Arrives on the mbarrier once all cp.async of this thread so far have landed (the arrival counts against the
// barrier's initial count).
__device__ __forceinline__ void cp_async_arrive(uint32_t bar) {
  asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ float2 lds_f2(uint32_t addr) {
  float2 r;
  asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(r.x), "=f"(r.y) : "r"(addr) : "memory");
  return r;
}

// Byte of group g (of 16) of row r within a window's s or z part.
__device__ __forceinline__ uint32_t win_off(int r, int g) {
  return static_cast<uint32_t>(r * 64 + (((g >> 2) ^ ((r >> 1) & 3)) << 4) + (g & 3) * 4);
}

// Persistent pair kernel over pair tiles (m_pair * n_tiles + n_tile), cluster c
// taking tiles c, c + clusters, ... The global group counter j runs across
// tiles: operand stage j mod 4, partial buffer j mod 3; windows count per tile.
template <int OUT>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kGThreads, 1)
    w4a4_group_gemm_kernel(const GroupParams p) {
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  uint8_t* smem = smem_raw + (base - raw);

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const uint32_t rank = cluster_rank();
  const int cluster = blockIdx.x >> 1;
  const int clusters = gridDim.x >> 1;
  const int nk = p.Gq;
  const int num_tiles = p.m_pairs * p.n_tiles;

  const uint32_t bar0 = base + kGOffBars;
  auto full = [&](int s) { return bar0 + 8u * s; };                  // leader: operands of stage s ready
  auto empty = [&](int s) { return bar0 + 8u * (kGStages + s); };    // both: stage s consumed
  auto pfull = [&](int b) { return bar0 + 8u * (2 * kGStages + b); };            // both: partial b written
  auto pempty = [&](int b) { return bar0 + 8u * (2 * kGStages + kGBufs + b); };  // leader: partial b read
  auto wfull = [&](int w) { return bar0 + 8u * (2 * kGStages + 2 * kGBufs + w); };       // window staged
  auto wempty = [&](int w) { return bar0 + 8u * (2 * kGStages + 2 * kGBufs + 2 + w); };  // window read
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + kGOffMisc);
  volatile int* abort = reinterpret_cast<volatile int*>(smem + kGOffMisc + 16);

  if (threadIdx.x == 0) {
    for (int s = 0; s < kGStages; ++s) {
      mbar_init(full(s), 2 * kGArrivals);
      mbar_init(empty(s), 1);
    }
    for (int b = 0; b < kGBufs; ++b) {
      mbar_init(pfull(b), 1);
      mbar_init(pempty(b), 2 * kGScWarps);
    }
    for (int w = 0; w < 2; ++w) {
      mbar_init(wfull(w), kGWinThreads);
      mbar_init(wempty(w), kGScWarps);
    }
    *abort = 0;
    mbar_fence_init();
  }
  if (warp == 0) {
    tmem_alloc2(smem_u32(tmem_slot), kGTmemCols);
    tmem_relinquish2();
  }
  tc_fence_before();
  cluster_sync();  // barriers initialised and TMEM allocated in both CTAs
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  uint32_t mma_groups = 0;
  auto start_grid = [] {
    griddep_wait();
    griddep_launch_dependents();
  };

  // 16 warps x 48 + 16 warps x 80 = the 32 x 64 registers of the launch.
  if (warp < kGFirstSc) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 48;");
    if (warp == 0) {
      // ---------------- MMA issuer (leader CTA) ----------------
      start_grid();
      // The whole warp runs the loop; an elected lane issues (elect_one).
      if (rank == 0) {
        const uint64_t desc0 = smem_desc_sw128(base);
        int s = 0, phase = 0, b = 0, bphase = 0;
        bool ok = true;
        for (int tile = cluster; tile < num_tiles && ok; tile += clusters) {
          for (int kt = 0; kt < nk; ++kt) {
            ok = __all_sync(0xFFFFFFFFu, wait_cluster(pempty(b), bphase ^ 1, abort) &&
                                             wait_cluster(full(s), phase, abort));
            if (!ok) break;
            tc_fence_after();
            if (elect_one()) {
              const uint64_t desc = desc0 + static_cast<uint32_t>(s * (kGBStage >> 4));
#pragma unroll
              for (int kk = 0; kk < GBK / 32; ++kk)
                mma2_ts(tmem + b * GBN, tmem + kGACol0 + s * kGAColsPerStage + 8 * kk, desc + 2 * kk, kGIdesc,
                        kk != 0 ? 1u : 0u);
              mma2_commit_both(empty(s));
              mma2_commit_both(pfull(b));
            }
            __syncwarp();
            ++mma_groups;
            if (++s == kGStages) {
              s = 0;
              phase ^= 1;
            }
            if (++b == kGBufs) {
              b = 0;
              bphase ^= 1;
            }
          }
        }
      }
    } else if (warp < kGFirstA) {
      // ---------------- windows of s, z and R ----------------
      // Only what exists is copied: rows and columns past the end feed sums that are not stored.
      const int wt = threadIdx.x - 32;  // of the kGWinThreads that stage
      start_grid();
      int w = 0, wphase = 0;
      bool ok = true;
      for (int tile = cluster; tile < num_tiles && ok; tile += clusters) {
        const int m0 = (tile / p.n_tiles) * 2 * GBM + static_cast<int>(rank) * GBM;
        const int n = (tile % p.n_tiles) * GBN + 4 * lane;
        const int rows = p.T - m0 < GBM ? p.T - m0 : GBM;  // may be negative
        for (int k0 = 0; k0 < nk; k0 += kGWin) {
          ok = __all_sync(0xFFFFFFFFu, wait_cluster(wempty(w), wphase ^ 1, abort));
          if (!ok) break;
          const uint32_t wb = base + kGOffWin + w * kWinBytes;
          const int ng = nk - k0 < kGWin ? nk - k0 : kGWin;
          const int pieces = (ng + 3) / 4;  // of four groups per row: 1 to 4, which divide kGWinThreads
          const int g = wt % pieces * 4;
          for (int r = wt / pieces; r < rows; r += kGWinThreads / pieces) {
            const int64_t src = static_cast<int64_t>(m0 + r) * nk + k0 + g;
            const uint32_t dst = wb + win_off(r, g);
            if (p.vec_sz) {  // nk % 4 == 0: pieces are whole
              cp_async<16>(dst, p.a_scale + src);
              cp_async<16>(dst + kWinRows, p.a_zero + src);
            } else {
#pragma unroll
              for (int i = 0; i < 4; ++i) {
                if (g + i < ng) {
                  cp_async<4>(dst + 4 * i, p.a_scale + src + i);
                  cp_async<4>(dst + kWinRows + 4 * i, p.a_zero + src + i);
                }
              }
            }
          }
          for (int i = warp - 1; i < ng; i += kGWinThreads / 32) {
            const float* src = p.gsum + static_cast<int64_t>(k0 + i) * p.N + n;
            const uint32_t dst = wb + 2 * kWinRows + i * GBN * 4 + lane * 16;
            if (p.vec_r) {  // N % 4 == 0: whole pieces
              if (n < p.N) cp_async<16>(dst, src);
            } else {
#pragma unroll
              for (int q = 0; q < 4; ++q)
                if (n + q < p.N) cp_async<4>(dst + 4 * q, src + q);
            }
          }
          if (k0 + kGWin >= nk && warp == 1) {
            const float* src = p.w_scale + n;
            const uint32_t dst = wb + kWinW + lane * 16;
            if (p.vec_w) {
              if (n < p.N) cp_async<16>(dst, src);
            } else {
#pragma unroll
              for (int q = 0; q < 4; ++q)
                if (n + q < p.N) cp_async<4>(dst + 4 * q, src + q);
            }
          }
          // Arrives when this thread's copies have landed: the next window's are issued meanwhile.
          cp_async_arrive(wfull(w));
          w ^= 1;
          if (w == 0) wphase ^= 1;
        }
      }
      asm volatile("cp.async.wait_all;" ::: "memory");  // after an abort too, no copy outlives the CTA
    } else if (warp >= kGFirstA && warp < kGFirstSc) {
      // ---------------- converters: packed codes -> E4M3 operands ----------------
      // Two warps per 32-row group take turns by group, each with kGRing of its
      // k-tiles' loads in flight (a register ring).
      const bool is_a = warp < kGFirstB;
      const int quarter = warp & 3;
      const int wb = is_a ? 0 : (warp - kGFirstB) & 1;
      const int turn = is_a ? (warp - kGFirstA) >> 2 : (warp - kGFirstB) >> 1;
      const uint32_t full_l = leader_addr(full(0));
      const uint8_t* codes = is_a ? p.a_codes : p.w_codes;
      const int rb_count = is_a ? p.t_blocks : p.n_blocks;
      // The next k-tile to load: tile, group, and this lane's address of it (nullptr: the row block lies past the
      // buffer's rows). K is a multiple of 128, so a group's four chunks exist.
      const uint8_t* src = nullptr;
      int ld_tile = cluster, ld_kt = turn;
      auto new_tile = [&]() {
        while (ld_kt >= nk) {
          ld_kt -= nk;
          ld_tile += clusters;
        }
        const int rb = is_a ? ((ld_tile / p.n_tiles) * 2 * GBM + static_cast<int>(rank) * GBM + quarter * 32) >> 5
                            : ((ld_tile % p.n_tiles) * GBN + static_cast<int>(rank) * GBNH + wb * 32) >> 5;
        src = ld_tile < num_tiles && rb < rb_count
                  ? codes + (static_cast<int64_t>(rb) * p.kchunks + ld_kt * kGChunks) * 512 + lane * 16
                  : nullptr;
      };
      auto load_next = [&](uint4 (&v)[kGChunks]) {
#pragma unroll
        for (int j = 0; j < kGChunks; ++j) v[j] = src != nullptr ? ldg_stream(src + j * 512) : make_uint4(0u, 0u, 0u, 0u);
        ld_kt += kGTurns;
        if (ld_kt < nk)
          src = src != nullptr ? src + kGTurns * kGChunks * 512 : nullptr;
        else
          new_tile();
      };
      new_tile();
      start_grid();
      // This warp's groups: every kGTurns-th of all tiles' groups.
      const int my_tiles = cluster < num_tiles ? (num_tiles - cluster + clusters - 1) / clusters : 0;
      int64_t left = (static_cast<int64_t>(my_tiles) * nk - turn + kGTurns - 1) / kGTurns;
      uint4 ring[kGRing][kGChunks];
#pragma unroll
      for (int r = 0; r < kGRing; ++r) load_next(ring[r]);
      int s = turn, phase = 0;
      bool run = true;
      while (run) {
#pragma unroll
        for (int r = 0; r < kGRing; ++r) {
          if (left-- <= 0) {
            run = false;
            break;
          }
          if (!__all_sync(0xFFFFFFFFu, wait_cluster(empty(s), phase ^ 1, abort))) {
            run = false;
            break;
          }
          if (is_a) {
            tc_fence_after();
            const uint32_t dst = tmem + (static_cast<uint32_t>(quarter * 32) << 16) + kGACol0 + s * kGAColsPerStage;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              uint32_t f8[16];
#pragma unroll
              for (int c = 0; c < 2; ++c) {
                const uint4& v = ring[r][2 * h + c];
                widen_act(v.x, f8[8 * c + 0], f8[8 * c + 1]);
                widen_act(v.y, f8[8 * c + 2], f8[8 * c + 3]);
                widen_act(v.z, f8[8 * c + 4], f8[8 * c + 5]);
                widen_act(v.w, f8[8 * c + 6], f8[8 * c + 7]);
              }
              tmem_st_16cols(dst + 16 * h, f8);
            }
            tmem_st_wait();
            tc_fence_before();
          } else {
            const int rr = wb * 32 + lane;
            const uint32_t st = base + s * kGBStage + rr * 128;
#pragma unroll
            for (int c = 0; c < kGChunks; ++c) {
              uint32_t a0, a1, a2, a3, b0, b1, b2, b3;
              widen_weight(ring[r][c].x, a0, a1);
              widen_weight(ring[r][c].y, a2, a3);
              widen_weight(ring[r][c].z, b0, b1);
              widen_weight(ring[r][c].w, b2, b3);
              sts128(st + (((2 * c) ^ (rr & 7)) << 4), a0, a1, a2, a3);
              sts128(st + (((2 * c + 1) ^ (rr & 7)) << 4), b0, b1, b2, b3);
            }
            fence_proxy_async_smem();
          }
          __syncwarp();
          if (lane == 0) arrive_cluster(full_l + 8u * s);
          load_next(ring[r]);  // this ring slot's next k-tile
          s += kGTurns;
          if (s >= kGStages) {
            s -= kGStages;
            phase ^= 1;
          }
        }
      }
    }
  } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 80;");
    // ---------------- scalers and epilogue ----------------
    const int quarter = warp & 3;
    const int c0 = ((warp - kGFirstSc) >> 2) * kGScCols;  // this warp's first column of the tile
    const int rl = quarter * 32 + lane;                   // TMEM lane = row within the CTA
    const uint32_t lane_base = tmem + (static_cast<uint32_t>(quarter * 32) << 16) + c0;
    const uint32_t pempty_l = leader_addr(pempty(0));
    int b = 0, bphase = 0, w = 0, wphase = 0;
    bool ok = true;
    start_grid();
    for (int tile = cluster; tile < num_tiles && ok; tile += clusters) {
      const int m0 = (tile / p.n_tiles) * 2 * GBM + static_cast<int>(rank) * GBM;
      const int t = m0 + rl;
      const int n0 = (tile % p.n_tiles) * GBN + c0;
      const bool warp_on = m0 + quarter * 32 < p.T && n0 < p.N;  // else nothing of this warp's is written
      uint64_t S2[kGScCols / 2];  // running sums of this row's columns c0 .. c0 + kGScCols, packed in pairs
#pragma unroll
      for (int i = 0; i < kGScCols / 2; ++i) S2[i] = 0ull;
      for (int k0 = 0; k0 < nk && ok; k0 += kGWin) {
        ok = __all_sync(0xFFFFFFFFu, wait_cluster(wfull(w), wphase, abort));
        if (!ok) break;
        const uint32_t wb = base + kGOffWin + w * kWinBytes;
        const int ng = nk - k0 < kGWin ? nk - k0 : kGWin;
        for (int g2 = 0; g2 < ng && ok; g2 += 2) {
          const float2 s2 = lds_f2(wb + win_off(rl, g2)), z2 = lds_f2(wb + kWinRows + win_off(rl, g2));
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            if (g2 + i >= ng) break;
            // The accumulator holds P * 2^-18 (each E4M3 operand carries 2^-9): with
            // d' = acc - z 2^-18 R, s 2^18 d' = s (P - z R), all scalings exact.
            const float sg = (i == 0 ? s2.x : s2.y) * 262144.0f;
            const float nz = (i == 0 ? z2.x : z2.y) * -3.814697265625e-06f;
            // R of the first 16 columns is read while the partial is waited for.
            const float4* rrow = reinterpret_cast<const float4*>(smem + kGOffWin + w * kWinBytes + 2 * kWinRows +
                                                                 (g2 + i) * GBN * 4 + c0 * 4);
            float4 r[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) r[q] = rrow[q];
            ok = __all_sync(0xFFFFFFFFu, wait_cluster(pfull(b), bphase, abort));
            if (!ok) break;
            tc_fence_after();
            if (warp_on) {
              const uint64_t SG = pack2(sg, sg);
              const uint64_t NZ = pack2(nz, nz);
#pragma unroll
              for (int c = 0; c < kGScCols / 16; ++c) {
                uint32_t pv[16];
                tmem_ld_16cols(lane_base + b * GBN + c * 16, pv);
                tmem_ld_wait_for(pv);
                if (c == kGScCols / 16 - 1) {
                  // The partial is in registers: its buffer may take another group.
                  tc_fence_before();
                  __syncwarp();
                  if (lane == 0) arrive_cluster(pempty_l + 8u * b);
                }
                uint64_t d[8];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                  d[2 * q] = fma2v(NZ, pack2(r[q].x, r[q].y),
                                   pack2(__uint_as_float(pv[4 * q]), __uint_as_float(pv[4 * q + 1])));
                  d[2 * q + 1] = fma2v(NZ, pack2(r[q].z, r[q].w),
                                       pack2(__uint_as_float(pv[4 * q + 2]), __uint_as_float(pv[4 * q + 3])));
                }
                if (c + 1 < kGScCols / 16) {
#pragma unroll
                  for (int q = 0; q < 4; ++q) r[q] = rrow[4 * (c + 1) + q];
                }
#pragma unroll
                for (int q = 0; q < 8; ++q) S2[c * 8 + q] = fma2v(SG, d[q], S2[c * 8 + q]);
              }
            } else if (lane == 0) {
              arrive_cluster(pempty_l + 8u * b);
            }
            if (++b == kGBufs) {
              b = 0;
              bphase ^= 1;
            }
          }
        }
        if (!ok) break;
        if (k0 + kGWin >= nk) {
          // The tile's last window carries its channel scales.
          const float4* wrow = reinterpret_cast<const float4*>(smem + kGOffWin + w * kWinBytes + kWinW + c0 * 4);
#pragma unroll
          for (int q = 0; q < kGScCols / 4; ++q) {
            const float4 wv = wrow[q];
            S2[2 * q] = mul2v(pack2(wv.x, wv.y), S2[2 * q]);
            S2[2 * q + 1] = mul2v(pack2(wv.z, wv.w), S2[2 * q + 1]);
          }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(wempty(w));
        w ^= 1;
        if (w == 0) wphase ^= 1;
      }
      if (ok && warp_on && n0 + kGScCols <= p.N) {
        // Through the warp's buffer, 64 bytes of a row at a time, so that four lanes store one row's 64 bytes: a lane
        // per row touches 32 lines with each store (2 k cycles a tile: 2048 x 512 -> 8192 32.2 us, now 27.4). Piece q of
        // row r lies at q ^ (r / 2 % 4): no bank conflicts. A ragged edge leaves directly.
        constexpr int kElem = OUT == OFFQ_F32 ? 4 : 2, kPer = 16 / kElem;
        const uint32_t buf = base + kGOffOut + (warp - kGFirstSc) * kGOutBytes;
        const int row0 = m0 + quarter * 32;
#pragma unroll
        for (int c = 0; c < kGScCols; c += 4 * kPer) {
          __syncwarp();  // the buffer has been read
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            uint32_t v[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              float y0, y1;
              if constexpr (OUT == OFFQ_F32) {
                unpack2(S2[(c + 4 * q) / 2 + i / 2], y0, y1);
                v[i] = __float_as_uint((i & 1) == 0 ? y0 : y1);
              } else {
                unpack2(S2[(c + 8 * q) / 2 + i], y0, y1);
                v[i] = pack_out<OUT>(y0, y1);
              }
            }
            sts128(buf + lane * 64 + ((q ^ ((lane >> 1) & 3)) << 4), v[0], v[1], v[2], v[3]);
          }
          __syncwarp();
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const int r = 8 * i + (lane >> 2), q = lane & 3;
            const uint4 v = lds128(buf + r * 64 + ((q ^ ((r >> 1) & 3)) << 4));
            if (row0 + r < p.T)
              *reinterpret_cast<uint4*>(static_cast<uint8_t*>(p.out) +
                                        (static_cast<int64_t>(row0 + r) * p.ldo + n0 + c + q * kPer) * kElem) = v;
          }
        }
      } else if (ok && warp_on) {
#pragma unroll
        for (int c = 0; c < kGScCols; c += 8) {
          float y[8];
#pragma unroll
          for (int i = 0; i < 4; ++i) unpack2(S2[c / 2 + i], y[2 * i], y[2 * i + 1]);
          const int nvalid = p.N - n0 - c < 8 ? p.N - n0 - c : 8;
          if (t < p.T && nvalid > 0) store_out<OUT, 8>(p.out, static_cast<int64_t>(t) * p.ldo + n0 + c, y, nvalid);
        }
      }
    }
  }

  // ---------------- teardown ----------------
  if (*abort && warp == 0 && lane == 0 && rank == 0 && mma_groups > 0) {
    // Let the MMAs already issued finish before tensor memory is released.
    const uint32_t last = mma_groups - 1;
    wait_teardown(pfull(last % kGBufs), (last / kGBufs) & 1u);
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync();
  if (warp == 0) {
    tc_fence_after();
    tmem_dealloc2(tmem, kGTmemCols);
  }
  if (threadIdx.x == 0 && *abort && p.status != nullptr) atomicExch(p.status, kErrTimeout);
}

template <int OUT>
int launch_group_gemm(const GroupParams& p, cudaStream_t s) {
  auto kern = w4a4_group_gemm_kernel<OUT>;
  if (!smem_optin<w4a4_group_gemm_kernel<OUT>>(kGBytes)) return OFFQ_ERR_CUDA;
  const int sms = device_sms();
  if (sms < 2) return OFFQ_ERR_CUDA;
  const int tiles = p.m_pairs * p.n_tiles;
  const int clusters = tiles < sms / 2 ? tiles : sms / 2;
  return launch_pdl(kern, dim3(2 * clusters), dim3(kGThreads), kGBytes, s, p);
}

}  // namespace

extern "C" int offq_w4a4_linear_group(const uint8_t* a_codes, const float* a_scale, const float* a_zero, int64_t T,
                                      int64_t N, int64_t K, int32_t group, const uint8_t* w_codes,
                                      const float* w_scale, const float* w_groupsum, void* out, int out_dtype,
                                      int64_t ldo, void* stream) {
  const int ob = elem_bytes(out_dtype);
  if (ob == 0 || T < 0 || N < 1 || K <= 0 || ldo < N) return OFFQ_ERR_INVALID_ARG;
  if (group != kGroup) return group > 0 ? OFFQ_ERR_UNSUPPORTED : OFFQ_ERR_INVALID_ARG;
  if (K % kGroup != 0) return OFFQ_ERR_INVALID_ARG;
  if (K > kMaxGemmK || T > 0x3FFFFFFF || N > 0x3FFFFFFF) return OFFQ_ERR_UNSUPPORTED;
  if (T == 0) return OFFQ_OK;
  if (a_codes == nullptr || a_scale == nullptr || a_zero == nullptr || w_codes == nullptr || w_scale == nullptr ||
      w_groupsum == nullptr || out == nullptr)
    return OFFQ_ERR_INVALID_ARG;
  if (!aligned(a_codes, 16) || !aligned(w_codes, 16) || !aligned(out, 16) || (ldo * ob) % 16 != 0 ||
      !aligned(a_scale, 4) || !aligned(a_zero, 4) || !aligned(w_scale, 4) || !aligned(w_groupsum, 4))
    return OFFQ_ERR_MISALIGNED;
  GroupParams p{};
  p.a_codes = a_codes;
  p.w_codes = w_codes;
  p.a_scale = a_scale;
  p.a_zero = a_zero;
  p.w_scale = w_scale;
  p.gsum = w_groupsum;
  p.out = out;
  p.ldo = ldo;
  p.status = device_status_ptr();
  p.T = static_cast<int>(T);
  p.N = static_cast<int>(N);
  p.K = static_cast<int>(K);
  p.Gq = static_cast<int>(K / kGroup);
  p.m_pairs = static_cast<int>((T + 2 * GBM - 1) / (2 * GBM));
  p.n_tiles = static_cast<int>((N + GBN - 1) / GBN);
  p.t_blocks = static_cast<int>((T + 31) / 32);
  p.n_blocks = static_cast<int>((N + 31) / 32);
  p.kchunks = static_cast<int>(K / 32);
  p.vec_sz = p.Gq % 4 == 0 && aligned(a_scale, 16) && aligned(a_zero, 16);
  p.vec_r = N % 4 == 0 && aligned(w_groupsum, 16);
  p.vec_w = N % 4 == 0 && aligned(w_scale, 16);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  switch (out_dtype) {
    case OFFQ_F32: return launch_group_gemm<OFFQ_F32>(p, s);
    case OFFQ_BF16: return launch_group_gemm<OFFQ_BF16>(p, s);
    case OFFQ_F16: return launch_group_gemm<OFFQ_F16>(p, s);
    default: return OFFQ_ERR_INVALID_ARG;
  }
}
