// W4A4 GEMM of the OffQ path for batches between decode and prefill: the same
// product and epilogue as w4a4_gemm_kernel (paper Sec. 1, Eq. 5),
//
//   y[t][n] = s_w[n] * ( s_a[t] * (acc'[n][t] - 8 Rt[n]) + sum_b o[t][b] * R[b][n] ),
//   acc'[n][t] = sum_k q_w[n][k] * (q_a[t][k] + 8),   Rt[n] = sum_b R[b][n].
//
// Here the pair kernel's 256 x 256 tiles are too few to fill the chip (16 for
// 4096 channels and up to 256 tokens, on 76 pairs), and each walks all of K.
// And from 17 tokens on, warp-level MMAs over all of a large layer's weights take
// longer than this. So:
//  * a CTA takes 128 output channels (the MMA's M side) x up to 128 tokens (N,
//    a multiple of 16 near an equal share of the tokens) and, in a cluster of
//    S = 1, 2, 4 or 8, an S-th of K; S is the largest that one wave holds. The
//    partial accumulators are integers times 2^-18, so their sum is exact in
//    any order: every CTA sends the columns it does not own into their owner's
//    shared memory, and each owner finishes its own;
//  * converter warps as in the pair kernel: weights are widened in registers
//    into tensor memory, token codes into the 128-byte-swizzled shared-memory
//    operand; four stages of 128 codes;
//  * one output tile per CTA, so the converter warps turn into the epilogue's;
//  * before the wait for the kernel ahead, the CTA asks the L2 for its weight
//    codes (a prefetch; the loads themselves come after the wait).
// Warps: 0 MMA issuer (and TMEM allocation), 1-8 weight converters (two per
// 32-row TMEM quarter, taking turns by k-tile), 9-16 token converters (as many
// per 32-token group as there are, up to three). Every wait is bounded; a wait
// that runs out aborts the CTA, which still passes its cluster's barriers, and
// records OFFQ_ERR_TIMEOUT in the device status word.
//
// What bounds it: a converter warp's chain per k-tile (wait, widen, store, arrive)
// at about 660 cycles per k-tile and CTA; the rest is the chain around it: 2000
// cycles to the first operands, and with S > 1 about 5000 for the exchange.
// Measured (per call, weights past the L2; before: the decode kernel of 128
// channels x all of K per CTA up to 64 tokens, the pair kernel above): 64 x
// 4096 -> 4096 9.0 us (16.7), 201 x 4096 -> 4096 12.4 (18.2), 64 x 11008 -> 4096 with
// 43 offset blocks 14.8 (85.1), 201 x 11008 -> 4096 26.0 (52.3), 128 x 8192 -> 1024
// 12.3 (29.8), 201 x 1920 -> 5376 13.2 (22.7). Two CTAs per SM of half the warps: within
// 10 % either way, worse where S > 1.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "offq.h"
#include "offq_device.cuh"
#include "offq_host.h"
#include "pair_common.cuh"

namespace {

using namespace offq;

constexpr int kMidM = 128;             // output channels per CTA
constexpr int kMidMaxN = 128;          // tokens per CTA
constexpr int kMidBK = 128;            // codes per k-tile
constexpr int kMidStages = 4;
constexpr int kMidConvA = 8, kMidConvB = 8;
constexpr int kMidWarps = 1 + kMidConvA + kMidConvB;
constexpr int kMidThreads = kMidWarps * 32;
constexpr int kMidParts = (kMidConvA + kMidConvB) / 4;  // epilogue warps per TMEM quarter
constexpr int kMidChunk = 16;          // accumulator columns that change hands together
constexpr int kMidChunkBytes = kMidChunk * kMidM * 4;
constexpr int kMidACol0 = kMidMaxN;    // tensor memory: accumulator, then the A stages
constexpr int kMidAColsPerStage = kMidBK / 4;
constexpr int kMidTmemCols = 256;
constexpr int kMidOutBytes = 8 * 32 * 4;  // an epilogue warp's transposition buffer: 8 tokens x 32 channels
static_assert(kMidACol0 + kMidStages * kMidAColsPerStage <= kMidTmemCols, "TMEM budget");
constexpr int kMidPrefetch = 2;   // k-tiles of loads in flight per converter thread
constexpr int kMidDist = 12;     // k-tiles of weight codes asked into the L2 ahead of their loads
constexpr int kMidSmemMax = 200 * 1024;

struct MidParams {
  const uint8_t* a_codes;
  const uint8_t* w_codes;
  const float* a_scale;
  const float* a_offset;   // [T][G] or nullptr
  const float* w_scale;
  const float* rowsum;     // [G][N]
  void* out;
  int64_t ldo;
  int32_t* acc_debug;
  int* status;
  int T, N, G;
  int nt;                  // tokens per tile (MMA N)
  int t_tiles;             // token tiles
  int S;                   // CTAs per cluster, which split K
  int nk;                  // k-tiles
  int kchunks;             // K / 32
  int a_blocks, w_blocks;  // 32-row blocks of the code buffers
  int staged;              // row sums and offsets go through shared memory
  int gp;                  // staged offsets per token, G rounded up to a multiple of 4
  int stages, b_stage;     // operand stages, bytes of one B stage (nt rows of 128 bytes)
  int off_red, off_sa, off_out, off_bars;  // shared memory, after the B stages
  int off_o;               // staged offsets, within the B stages' space
};

// D[tmem] (+)= A[tmem] * B[smem]^T, one CTA, E4M3 operands, fp32 accumulate.
__device__ __forceinline__ void mma_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc,
                                       uint32_t accumulate) {
  asm volatile(
      "{\n"
      ".reg .pred p;\n"
      "setp.ne.b32 p, %4, 0;\n"
      "tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], [%1], %2, %3, p;\n"
      "}\n" ::"r"(d_tmem),
      "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}

__device__ __forceinline__ uint32_t cluster_addr(uint32_t local, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(local), "r"(rank));
  return r;
}
__device__ __forceinline__ void st_cluster_v4(uint32_t addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
  asm volatile("st.shared::cluster.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(a), "r"(b), "r"(c), "r"(d) : "memory");
}
// Byte of columns 4 i .. 4 i + 3 of a row within an exchanged chunk of 16
// columns: 64 bytes per row, its pieces rotated so that eight rows' accesses of
// one piece fall in distinct banks.
__device__ __forceinline__ uint32_t red_off(int row, int i) {
  return static_cast<uint32_t>(row * 64 + (((i + (row >> 1)) & 3) << 4));
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }

__device__ __forceinline__ void tmem_ld_8cols(uint32_t taddr, uint32_t (&r)[8]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];\n"
      "tcgen05.wait::ld.sync.aligned;"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
      : "r"(taddr)
      : "memory");
}

template <int OUT>
__global__ void __launch_bounds__(kMidThreads, 1) w4a4_mid_kernel(const MidParams p) {
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  uint8_t* smem = smem_raw + (base - raw);

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const int S = p.S;
  const int rank = blockIdx.x % S;
  const int unit = blockIdx.x / S;           // token tiles of one channel tile are neighbours
  const int mt = unit / p.t_tiles, tt = unit - mt * p.t_tiles;
  const int n0 = mt * kMidM;                 // first output channel
  const int t0 = tt * p.nt;                  // first token
  const int kt0 = static_cast<int>(static_cast<int64_t>(rank) * p.nk / S);
  const int kt1 = static_cast<int>(static_cast<int64_t>(rank + 1) * p.nk / S);
  const int nch = p.nt / kMidChunk;          // accumulator chunks of the tile
  const int ch0 = rank * nch / S, ch1 = (rank + 1) * nch / S;  // the ones this CTA finishes
  const int max_own = (nch + S - 1) / S;

  const uint32_t bar0 = base + p.off_bars;
  auto full = [&](int s) { return bar0 + 8u * s; };
  auto empty = [&](int s) { return bar0 + 8u * (kMidStages + s); };
  const uint32_t acc_full = bar0 + 8u * (2 * kMidStages);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + p.off_bars + 8 * (2 * kMidStages + 1));
  volatile int* abort = reinterpret_cast<volatile int*>(tmem_slot + 1);

  // L2 prefetch of one k-tile (2 KB, contiguous) of a weight converter's row block.
  auto prefetch_w = [&](int kt) {
    const int rb = (n0 >> 5) + (warp & 3);
    const int c = kt * 4 + (lane >> 2);
    if (lane < 16 && rb < p.w_blocks && kt < kt1 && c < p.kchunks)
      asm volatile("prefetch.global.L2 [%0];" ::"l"(p.w_codes + (static_cast<int64_t>(rb) * p.kchunks + c) * 512 +
                                                   (lane & 3) * 128));
  };

  const int b_groups = (p.nt + 31) / 32;
  if (threadIdx.x == 0) {
    for (int s = 0; s < kMidStages; ++s) {
      mbar_init(full(s), 4 + b_groups);
      mbar_init(empty(s), 1);
    }
    mbar_init(acc_full, 1);
    *abort = 0;
    mbar_fence_init();
  }
  if (warp == 0) {
    tmem_alloc(smem_u32(tmem_slot), kMidTmemCols);
    tmem_relinquish();
  } else if (warp <= 4) {
    // The first k-tiles of this warp's weight row block.
    for (int i = 0; i < kMidDist; ++i) prefetch_w(kt0 + i);
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  if (S > 1) cluster_arrive();  // waited for before the first store into another CTA
  griddep_wait();
  griddep_launch_dependents();
  float* sSa = reinterpret_cast<float*>(smem + p.off_sa);  // scales of this CTA's own tokens
  for (int i = threadIdx.x; i < (ch1 - ch0) * kMidChunk; i += kMidThreads) {
    const int tok = t0 + ch0 * kMidChunk + i;
    if (tok < p.T)
      cp_async<4>(smem_u32(sSa + i), p.a_scale + tok);
    else
      sSa[i] = 0.f;
  }

  if (warp == 0) {
    // ---------------- MMA issuer ----------------
    // The whole warp runs the loop; an elected lane issues (elect_one).
    const uint32_t idesc = idesc_e4m3_f32(kMidM, p.nt);
    const uint64_t desc0 = smem_desc_sw128(base);
    int s = 0, phase = 0;
    for (int kt = kt0; kt < kt1; ++kt) {
      if (!__all_sync(0xFFFFFFFFu, mbar_wait(full(s), phase, abort))) break;
      tc_fence_after();
      if (elect_one()) {
        const uint64_t desc = desc0 + static_cast<uint32_t>(s * p.b_stage >> 4);
#pragma unroll
        for (int kk = 0; kk < kMidBK / 32; ++kk)
          mma_ts(tmem, tmem + kMidACol0 + s * kMidAColsPerStage + 8 * kk, desc + 2 * kk, idesc,
                 (kt != kt0 || kk != 0) ? 1u : 0u);
        mma_commit(empty(s));
      }
      __syncwarp();
      if (++s == p.stages) {
        s = 0;
        phase ^= 1;
      }
    }
    if (elect_one()) mma_commit(acc_full);  // also after an abort: tells the teardown the MMAs are done
    __syncwarp();
  } else {
    // ---------------- converters: packed codes -> E4M3 operands ----------------
    const bool is_a = warp <= kMidConvA;
    const int quarter = warp & 3;
    const int bw = warp - 1 - kMidConvA;
    const int grp = bw % b_groups;                                     // B: 32-token group
    const int turns = is_a ? kMidConvA / 4 : (kMidConvB / b_groups < 3 ? kMidConvB / b_groups : 3);  // at most the stages
    const int turn = is_a ? (warp - 1) >> 2 : bw / b_groups;           // k-tiles kt0 + turn, + turns, ...
    const int rb = is_a ? (n0 >> 5) + quarter : 0;
    const uint8_t* blk = nullptr;
    bool row_ok;
    if (is_a) {
      row_ok = rb < p.w_blocks;
      blk = p.w_codes + static_cast<int64_t>(rb) * p.kchunks * 512 + lane * 16;
    } else {
      const int tok = t0 + grp * 32 + lane;  // a tile's tokens need not start on a 32-row block
      row_ok = (tok >> 5) < p.a_blocks;
      blk = p.a_codes + static_cast<int64_t>(tok >> 5) * p.kchunks * 512 + (tok & 31) * 16;
    }
    auto load = [&](int kt, uint4 (&v)[4]) {
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int c = kt * 4 + j;
        if (row_ok && kt < kt1 && c < p.kchunks)
          v[j] = is_a ? ldg_stream(blk + c * 512) : *reinterpret_cast<const uint4*>(blk + c * 512);
        else
          v[j] = make_uint4(0u, 0u, 0u, 0u);
      }
    };
    uint4 ring[kMidPrefetch][4];
#pragma unroll
    for (int i = 0; i < kMidPrefetch; ++i) load(kt0 + turn + i * turns, ring[i]);
    int s = turn, phase = 0;  // turn < stages
    bool run = turn < turns;
    for (int kb = kt0 + turn; kb < kt1 && run; kb += kMidPrefetch * turns) {
#pragma unroll
      for (int i = 0; i < kMidPrefetch; ++i) {
        const int kt = kb + i * turns;
        if (kt >= kt1) break;
        if (!__all_sync(0xFFFFFFFFu, mbar_wait(empty(s), phase ^ 1, abort))) {
          run = false;
          break;
        }
        if (is_a) {
          tc_fence_after();
          uint32_t f8[32];
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            widen_weight(ring[i][j].x, f8[8 * j + 0], f8[8 * j + 1]);
            widen_weight(ring[i][j].y, f8[8 * j + 2], f8[8 * j + 3]);
            widen_weight(ring[i][j].z, f8[8 * j + 4], f8[8 * j + 5]);
            widen_weight(ring[i][j].w, f8[8 * j + 6], f8[8 * j + 7]);
          }
          tmem_st_32cols(tmem + (static_cast<uint32_t>(quarter * 32) << 16) + kMidACol0 + s * kMidAColsPerStage, f8);
          tmem_st_wait();
          tc_fence_before();
        } else {
          const int r = grp * 32 + lane;
          if (r < p.nt) {  // the last group of a tile may be half
            const uint32_t st = base + s * p.b_stage + r * 128;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              uint32_t a0, a1, a2, a3, b0, b1, b2, b3;
              widen_act(ring[i][j].x, a0, a1);
              widen_act(ring[i][j].y, a2, a3);
              widen_act(ring[i][j].z, b0, b1);
              widen_act(ring[i][j].w, b2, b3);
              sts128(st + (((2 * j) ^ (r & 7)) << 4), a0, a1, a2, a3);
              sts128(st + (((2 * j + 1) ^ (r & 7)) << 4), b0, b1, b2, b3);
            }
          }
          fence_proxy_async_smem();
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(full(s));
        load(kt + kMidPrefetch * turns, ring[i]);
        if (is_a) prefetch_w(kt + kMidDist);
        s += turns;
        if (s >= p.stages) {
          s -= p.stages;
          phase ^= 1;
        }
      }
    }
  }

  // ---------------- partial sums to their owners ----------------
  // The issuer always commits acc_full; its wait is bounded like the others.
  bool ok = __all_sync(0xFFFFFFFFu, mbar_wait(acc_full, 0, abort)) && !*abort;
  tc_fence_after();
  // The MMAs have read their operands: the B stages take the epilogue's constants.
  if (p.staged) {
#pragma unroll 4
    for (int i = threadIdx.x; i < p.G * kMidM; i += kMidThreads) {
      const int n = n0 + (i & (kMidM - 1));
      if (n < p.N)
        cp_async<4>(base + i * 4, p.rowsum + static_cast<int64_t>(i / kMidM) * p.N + n);
      else
        *reinterpret_cast<float*>(smem + i * 4) = 0.f;
    }
    if (p.a_offset != nullptr) {
      const int own_t0 = t0 + ch0 * kMidChunk;
      const int left = p.T - own_t0, own = (ch1 - ch0) * kMidChunk;
      const int cnt = (left < own ? left : own) * p.G;  // may be negative
      for (int i = threadIdx.x; i < cnt; i += kMidThreads) {
        const int r = i / p.G, b = i - r * p.G;
        cp_async<4>(base + p.off_o + (r * p.gp + b) * 4, p.a_offset + static_cast<int64_t>(own_t0) * p.G + i);
      }
    }
  }

  const int quarter = warp & 3, part = (warp - 1) >> 2;  // epilogue roles of the converter warps
  const uint32_t lane_tm = tmem + (static_cast<uint32_t>(quarter * 32) << 16);
  const int row = quarter * 32 + lane;
  if (S > 1) {
    cluster_wait();
    if (warp > 0 && ok) {
      for (int c = part; c < nch; c += kMidParts) {
        int d = 0;
        while ((d + 1) * nch / S <= c) ++d;  // the owner of chunk c
        if (d != rank) {
          uint32_t v[kMidChunk];
          tmem_ld_16cols(lane_tm + c * kMidChunk, v);
          tmem_ld_wait_for(v);
          const int src = rank < d ? rank : rank - 1;
          const uint32_t dst = cluster_addr(base + p.off_red, d) +
                               (src * max_own + c - d * nch / S) * kMidChunkBytes;
#pragma unroll
          for (int i = 0; i < kMidChunk / 4; ++i)
            st_cluster_v4(dst + red_off(row, i), v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
        }
      }
    }
    cluster_arrive();
    cluster_wait();
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();  // the staged constants; and every warp has seen whether the CTA aborted
  ok = ok && !*abort;

  // ---------------- epilogue: lane = channel, 8 tokens at a time ----------------
  if (warp > 0 && ok) {
    const int n = n0 + row;
    const bool n_ok = n < p.N;
    const float* sR = reinterpret_cast<const float*>(smem) + row;
    float rt = 0.f;
    if (p.staged) {
  #pragma unroll 4
      for (int b = 0; b < p.G; ++b) rt += sR[b * kMidM];
    } else if (n_ok) {
      for (int b = 0; b < p.G; ++b) rt += __ldg(p.rowsum + static_cast<int64_t>(b) * p.N + n);
    }
    const float m8r = rt * -0x1p-15f;  // -8 Rt 2^-18: exact
    const float sw = n_ok ? __ldg(p.w_scale + n) : 0.f;
    const bool has_off = p.a_offset != nullptr;
    for (int h = part; h < (ch1 - ch0) * 2; h += kMidParts) {
      const int col = ch0 * kMidChunk + h * 8;  // within the tile
      const int tok0 = t0 + col;
      __syncwarp();  // the load needs every lane; channels past the end took other branches
      uint32_t av[8];
      tmem_ld_8cols(lane_tm + col, av);
      float acc[8], cv[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        acc[i] = __uint_as_float(av[i]);
        cv[i] = 0.f;
      }
      for (int k = 0; k < S - 1; ++k) {
        const uint8_t* r = smem + p.off_red + (k * max_own + (h >> 1)) * kMidChunkBytes;
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          const float4 v = *reinterpret_cast<const float4*>(r + red_off(row, 2 * (h & 1) + i));
          acc[4 * i] += v.x;
          acc[4 * i + 1] += v.y;
          acc[4 * i + 2] += v.z;
          acc[4 * i + 3] += v.w;
        }
      }
      if (has_off && p.staged) {
        const float* o = reinterpret_cast<const float*>(smem + p.off_o) + h * 8 * p.gp;
        for (int b = 0; b < p.gp; b += 4) {
          float rv[4];
#pragma unroll
          for (int j = 0; j < 4; ++j) rv[j] = b + j < p.G ? sR[(b + j) * kMidM] : 0.f;
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const float4 ov = *reinterpret_cast<const float4*>(o + i * p.gp + b);
            cv[i] = b == 0 ? ov.x * rv[0] : fmaf(ov.x, rv[0], cv[i]);
            if (b + 1 < p.G) cv[i] = fmaf(ov.y, rv[1], cv[i]);
            if (b + 2 < p.G) cv[i] = fmaf(ov.z, rv[2], cv[i]);
            if (b + 3 < p.G) cv[i] = fmaf(ov.w, rv[3], cv[i]);
          }
        }
      } else if (has_off && n_ok) {
        for (int b = 0; b < p.G; ++b) {
          const float rv = __ldg(p.rowsum + static_cast<int64_t>(b) * p.N + n);
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const float o = tok0 + i < p.T ? __ldg(p.a_offset + static_cast<int64_t>(tok0 + i) * p.G + b) : 0.f;
            cv[i] = b == 0 ? o * rv : fmaf(o, rv, cv[i]);
          }
        }
      }
      const float4 s0 = *reinterpret_cast<const float4*>(sSa + h * 8), s1 = *reinterpret_cast<const float4*>(sSa + h * 8 + 4);
      const float sa[8] = {s0.x, s0.y, s0.z, s0.w, s1.x, s1.y, s1.z, s1.w};
      const int64_t off = static_cast<int64_t>(tok0) * p.ldo + n;
      const int valid = n_ok ? p.T - tok0 : 0;  // tokens of the eight that exist
      float y[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const float a = (acc[i] + m8r) * 262144.0f;  // exact: the integer dot product
        y[i] = sw * fmaf(sa[i], a, cv[i]);
      }
      const int nb = n0 + quarter * 32;  // the warp's first channel
      if (nb + 32 <= p.N) {
        // Transposed through the warp's buffer, so a lane stores 16 bytes of one token.
        constexpr int kElem = OUT == OFFQ_F32 ? 4 : 2, kPer = 16 / kElem, kLanes = 32 / kPer;  // lanes per token
        uint8_t* buf = smem + p.off_out + (warp - 1) * kMidOutBytes;
        __syncwarp();
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          if constexpr (OUT == OFFQ_F32)
            reinterpret_cast<float*>(buf)[i * 32 + lane] = y[i];
          else if constexpr (OUT == OFFQ_BF16)
            reinterpret_cast<__nv_bfloat16*>(buf)[i * 32 + lane] = __float2bfloat16_rn(y[i]);
          else
            reinterpret_cast<__half*>(buf)[i * 32 + lane] = __float2half_rn(y[i]);
        }
        __syncwarp();
#pragma unroll
        for (int i0 = 0; i0 < 8; i0 += 32 / kLanes) {
          const int i = i0 + lane / kLanes;
          if (tok0 + i < p.T)
            *reinterpret_cast<uint4*>(static_cast<uint8_t*>(p.out) +
                                      ((tok0 + i) * p.ldo + nb) * kElem + (lane % kLanes) * 16) =
                *reinterpret_cast<const uint4*>(buf + i * 32 * kElem + (lane % kLanes) * 16);
        }
      } else {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          if (i < valid) {
            if (OUT == OFFQ_F32) {
              static_cast<float*>(p.out)[off + i * p.ldo] = y[i];
            } else if (OUT == OFFQ_BF16) {
              static_cast<__nv_bfloat16*>(p.out)[off + i * p.ldo] = __float2bfloat16_rn(y[i]);
            } else {
              static_cast<__half*>(p.out)[off + i * p.ldo] = __float2half_rn(y[i]);
            }
          }
        }
      }
      if (p.acc_debug != nullptr) {
#pragma unroll
        for (int i = 0; i < 8; ++i)
          if (i < valid) p.acc_debug[static_cast<int64_t>(tok0 + i) * p.N + n] = __float2int_rn(acc[i] * 262144.0f);
      }
    }
  }

  // ---------------- teardown ----------------
  if (threadIdx.x == 0 && *abort) mbar_wait_teardown(acc_full, 0);  // MMAs in flight finish before TMEM is released
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    tmem_dealloc(tmem, kMidTmemCols);
  }
  if (threadIdx.x == 0 && *abort && p.status != nullptr) atomicExch(p.status, kErrTimeout);
}

// Whether K may be split over S CTAs: at least four k-tiles each, and one wave.
// Clusters of eight do not fill the chip (1024 x 8192 at 201 tokens, 16 of them:
// 22.9 us against 11.3 with clusters of four), so they have to fit in two thirds of it.
bool split_fits(int64_t S, int64_t tiles, int64_t nk, int64_t sms) {
  return nk >= 4 * S && tiles * S <= (S < 8 ? sms : sms * 2 / 3);
}

template <int OUT>
int launch_mid(const MidParams& p, int64_t ctas, size_t bytes, cudaStream_t s) {
  if (!smem_optin<w4a4_mid_kernel<OUT>>(kMidSmemMax)) return OFFQ_ERR_CUDA;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>(ctas));
  cfg.blockDim = dim3(kMidThreads);
  cfg.dynamicSmemBytes = bytes;
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = static_cast<unsigned>(p.S);
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, w4a4_mid_kernel<OUT>, p) == cudaSuccess ? OFFQ_OK : OFFQ_ERR_CUDA;
}

}  // namespace

namespace offq {

// Microseconds a call takes in this form and in its neighbours, fitted to all of
// them measured over N = 512 .. 28672, K = 512 .. 28672 and 4 .. 1100 tokens
// (weights past the L2). Here: waves of CTAs, each of a fixed cost, a cost per
// k-tile and an exchange that grow with its tokens, and one per offset block.
// The pair kernel: waves of 256 x 256 tiles, each bound by its MMAs or by its offset
// correction. The few-token kernel with two token tiles: its warp-level MMAs over
// all weights (with one tile, to 16 tokens, it is the faster one at most sizes and
// at the others within 5 %). The fit is within 20 % of each side, and where two are
// closer than that it matters little which is taken: 400 x 4096 -> 4096 15.2 here
// against 17.4 in pairs; 201 x 4096 -> 11008 29.8 against 18.0; 257 x 11008 -> 4096
// (43 blocks) 37.0 against 40.0, 1100 tokens 84.9 against 74.1; 32 x 8192 -> 16896
// 19.5 against 30.2 few-token, 32 x 4096 -> 4096 8.2 against 6.0.
bool mid_takes(int64_t T, int64_t N, int64_t K, int64_t G) {
  constexpr int64_t kFewTile = 16;
  const int sms = device_sms();
  if (sms < 2 || T <= kFewTile) return false;
  const int64_t nk = (K + kMidBK - 1) / kMidBK;
  const int64_t tiles = (N + kMidM - 1) / kMidM * ((T + kMidMaxN - 1) / kMidMaxN);
  int64_t S = 1;
  while (S < 8 && split_fits(S * 2, tiles, nk, sms)) S *= 2;
  const double k = static_cast<double>(nk), blocks = G > 1 ? static_cast<double>(G) : 0.0;
  const double fill = static_cast<double>(T) / static_cast<double>((T + kMidMaxN - 1) / kMidMaxN * kMidMaxN);
  const double exchange = S > 1 ? 5.6 + 2.0 * fill : 5.0;
  const double mid = static_cast<double>((tiles * S + sms - 1) / sms) *
                     ((0.21 + 0.12 * fill) * k / static_cast<double>(S) + exchange + 0.15 * blocks);
  if (T <= few_max_tokens()) return mid < 2.0 + 2.5e-7 * static_cast<double>(N) * static_cast<double>(K);
  const double waves = static_cast<double>(((N + 255) / 256 * ((T + 255) / 256) + sms / 2 - 1) / (sms / 2));
  const double mma = 0.08 * k + waves * (0.31 * k + 2.0);
  const double corr = G > 1 ? waves * (0.14 * k + 0.45 * blocks + 3.0) : 0.0;
  const double pair = 3.0 + (mma > corr ? mma : corr);
  return mid < pair;
}

// The mid-size form of offq_w4a4_linear (arguments checked by the caller).
int w4a4_linear_mid(const uint8_t* a_codes, const float* a_scale, const float* a_offset, int64_t T, int64_t N,
                    int64_t K, int32_t g, const uint8_t* w_codes, const float* w_scale, const float* w_offsum,
                    void* out, int out_dtype, int64_t ldo, int32_t* acc_debug, cudaStream_t stream) {
  const int sms = device_sms();
  if (sms < 1) return OFFQ_ERR_CUDA;
  MidParams p{};
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
  p.G = static_cast<int>(K / g);
  p.nk = static_cast<int>((K + kMidBK - 1) / kMidBK);
  p.kchunks = static_cast<int>(K / 32);
  p.a_blocks = static_cast<int>((T + 31) / 32);
  p.w_blocks = static_cast<int>((N + 31) / 32);
  p.t_tiles = static_cast<int>((T + kMidMaxN - 1) / kMidMaxN);
  const int per = static_cast<int>((T + p.t_tiles - 1) / p.t_tiles);
  p.nt = (per + 15) / 16 * 16;
  const int64_t tiles = (N + kMidM - 1) / kMidM * p.t_tiles;
  p.b_stage = p.nt * kMidBK;
  const int misc = kMidMaxN * 4 + (kMidConvA + kMidConvB) * kMidOutBytes + 8 * (2 * kMidStages + 1) + 16 + 1024;
  const int nch = p.nt / kMidChunk;
  auto red_bytes = [&](int S) { return (S - 1) * ((nch + S - 1) / S) * kMidChunkBytes; };
  p.S = 1;
  while (p.S < 8 && split_fits(p.S * 2, tiles, p.nk, sms) &&
         (kMidStages - 1) * p.b_stage + red_bytes(p.S * 2) + misc <= kMidSmemMax)
    p.S *= 2;
  const int own = (nch + p.S - 1) / p.S;
  p.gp = (p.G + 3) / 4 * 4;
  const int red = red_bytes(p.S);
  p.stages = kMidStages * p.b_stage + red + misc <= kMidSmemMax ? kMidStages : kMidStages - 1;
  // The epilogue's constants take the B stages' space, and some beyond it where they need it and it is there.
  p.off_o = p.G * kMidM * 4;
  const int64_t consts = static_cast<int64_t>(p.off_o) + own * kMidChunk * p.gp * 4;
  p.staged = consts + red + misc <= kMidSmemMax;
  p.off_red = p.stages * p.b_stage;
  if (p.staged && consts > p.off_red) p.off_red = static_cast<int>((consts + 15) / 16 * 16);
  p.off_sa = p.off_red + red;
  p.off_out = p.off_sa + kMidMaxN * 4;
  p.off_bars = p.off_out + (kMidConvA + kMidConvB) * kMidOutBytes;
  const size_t bytes = static_cast<size_t>(p.off_red) + red + misc;
  const int64_t ctas = tiles * p.S;
  if (ctas > 0x7FFFFFFF) return OFFQ_ERR_UNSUPPORTED;
  switch (out_dtype) {
    case OFFQ_F32: return launch_mid<OFFQ_F32>(p, ctas, bytes, stream);
    case OFFQ_BF16: return launch_mid<OFFQ_BF16>(p, ctas, bytes, stream);
    case OFFQ_F16: return launch_mid<OFFQ_F16>(p, ctas, bytes, stream);
    default: return OFFQ_ERR_INVALID_ARG;
  }
}

}  // namespace offq
