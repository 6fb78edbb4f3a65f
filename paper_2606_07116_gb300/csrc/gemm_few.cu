// W4A4 GEMM of the OffQ path for few tokens (decode): the same product and
// epilogue as w4a4_gemm_kernel (paper Sec. 1: all matrix multiplications in
// uniform 4-bit execution; Eq. 5: the offsets meet the weight block row sums),
//
//   y[t][n] = s_w[n] * ( s_a[t] * (acc'[n][t] - 8 Rt[n]) + sum_b o[t][b] * R[b][n] ),
//   acc'[n][t] = sum_k q_w[n][k] * (q_a[t][k] + 8),   Rt[n] = sum_b R[b][n].
//
// Few tokens (T <= 32; from 17 on only layers small enough that the tcgen05
// form of gemm_mid.cu is slower): warp-level MMA (mma.sync m16n8k16, fp16
// operands, fp32 accumulate).
//
// The weights stream once from HBM and meet at most 32 tokens, so the time is
// that stream plus the chain of latencies from the end of the kernel ahead
// (which makes the activations) to this one's last store. So:
//  * the weight codes go from global memory straight into the registers of the
//    warp that multiplies them. Lane (g, t) of a warp (g = lane / 4, t = lane %
//    4) loads the 16-byte chunk 4 s + t of weight rows g, g + 8, g + 16, g + 24
//    of the CTA's 32-row block (8 rows of a chunk are 128 contiguous bytes).
//    Both operands of an MMA may list K in any common order, so word j of those
//    chunks becomes MMAs 2 j and 2 j + 1 of the step as it lies;
//  * a code becomes an fp16 operand with shifts and masks alone (seven per 8
//    codes), as an integer times a power of two: products are integers times
//    2^-40, exact in the fp32 accumulator (|sum| < 2^24). The fp8 form of
//    mma.sync converts its operands to fp16 on every MMA on this part (500
//    against 1019 MAC per clock and SM), and the tensor cores proper (tcgen05)
//    need the operands in shared or tensor memory first: a pipeline whose fill
//    alone took longer than this whole kernel (14.3 us for 4096 x 4096 at 8
//    tokens, against 3.6 here);
//  * 8 warps split K. Each keeps two k-steps (4 KB) of weight codes in flight.
//    Prefetches of the CTA's weights into L2 are issued before the wait for the
//    kernel ahead (programmatic dependent launch), and up to 4 tokens the first
//    two k-steps' loads and the constants' as well: that kernel makes the
//    activations, not the weights, and the caller keeps to it (offq.h). From 5
//    tokens on nothing but the prefetch of the codes comes before the wait (4096
//    -> 4096 at 5 tokens 4.0 us, with early loads 3.7; prefetching the scales and
//    row sums too was slower at most sizes);
//  * the token codes come through a small cp.async ring per warp (no barrier);
//  * the warps' partial sums (exact in any order) meet in shared memory, and
//    each warp finishes whole tokens, lane = output channel.
// Measured per call, back to back over weight copies past the L2 (before: dp4a
// up to 4 tokens, tcgen05 above): 4096 -> 4096 3.6 / 4.0 / 4.5 / 6.1 us at 1 /
// 8 / 16 / 32 tokens (7.1 / 14.3 / 14.4 / 15.0); 4096 -> 11008 6.8 / 7.3 / 10.5 at
// 1 / 8 / 16 (7.9 / 14.8 / 15.0); 11008 -> 4096 with 43 offset blocks 8.2 / 8.8 /
// 10.3 / 14.2 (22.3 / 38.0 / 38.6 / 53.9). What bounds it: 1.6 us of launch and
// dependency per call, then the latency of two weight loads per warp; above 8
// tokens the mask-and-shift work per token.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "offq.h"
#include "offq_device.cuh"
#include "offq_host.h"
#include "pair_common.cuh"

namespace {

using namespace offq;

constexpr int kFewWarps = 8;
constexpr float kFewUnit = 0x1p40f;       // an accumulator is the integer product times 2^-16 2^-24
constexpr int kFewMaxT = 32;
constexpr int kFewPitch = 36;            // floats per token row of the partial sums (bank-conflict-free)
constexpr int kFewStageG = 64;           // offset blocks staged in shared memory
constexpr int kFewStageO = 2048;         // token offsets staged in shared memory
constexpr int kFewL2Bytes = 128 * 1024;  // most bytes of a CTA's codes prefetched into L2

struct FewParams {
  const uint8_t* a_codes;
  const uint8_t* w_codes;
  const float* a_scale;
  const float* a_offset;   // [T][G] or nullptr
  const float* w_scale;
  const float* rowsum;     // [G][N]
  void* out;
  int64_t ldo;
  int32_t* acc_debug;
  int T, N, G, kchunks;
  int staged;              // rowsum and offsets go through shared memory
};

// Eight weight codes (interleaved sign-magnitude word) as half pairs of channels
// (k, k + 4): a byte with the sign at bit 7 and the magnitude at bits 0-2, as a
// half's high byte over a zero low byte, is the magnitude times 2^-16 (the
// first two binades of a half are one uniform grid).
__device__ __forceinline__ void weight_halves(uint32_t w, uint32_t (&p)[4]) {
  const uint32_t r = __funnelshift_r(w, w, 4);
  p[0] = (w << 8) & 0x87008700u;
  p[1] = (r << 8) & 0x87008700u;
  p[2] = w & 0x87008700u;
  p[3] = r & 0x87008700u;
}

// Eight activation codes as half pairs of the same channels: u * 2^-24 (a
// subnormal half is its bit pattern times 2^-24).
__device__ __forceinline__ void act_halves(uint32_t w, uint32_t (&p)[4]) {
  p[0] = w & 0x000F000Fu;
  p[1] = (w >> 4) & 0x000F000Fu;
  p[2] = (w >> 8) & 0x000F000Fu;
  p[3] = (w >> 12) & 0x000F000Fu;
}

__device__ __forceinline__ void mma_f16_16x8x16(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                                uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

__device__ __forceinline__ uint32_t word_of(const uint4& v, int j) {
  return j == 0 ? v.x : j == 1 ? v.y : j == 2 ? v.z : v.w;
}

__device__ __forceinline__ void few_cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }

// NT: 8-token tiles per CTA (and warp); kFewWarps warps split K. CTAS: CTAs per
// SM the registers are budgeted for. EARLY (of the kernel): reads_early().
template <int NT, int CTAS>
struct Few {
  static constexpr int KS = kFewWarps;
  static constexpr int kTokens = NT * 8;
  static constexpr int kPdW = 2;                                  // k-steps of weight codes in flight per warp (registers)
  static constexpr int kPdA = NT == 1 ? 8 : NT == 2 ? 6 : 4;      // k-steps of token codes in flight per warp (shared memory)
  static constexpr int kChunkPitch = kTokens * 16 + 32;           // four chunks' 8-lane phases in distinct banks
  static constexpr int kRing = kPdA * 4 * kChunkPitch;            // bytes per warp
  static constexpr int kRedFloats = KS * kTokens * kFewPitch;
  // The partial sums reuse the ring: its copies have been read by then.
  static constexpr int kMain = KS * kRing > kRedFloats * 4 ? KS * kRing : kRedFloats * 4;
};

template <int OUT, int NT, int CTAS, bool EARLY>
__global__ void __launch_bounds__(kFewWarps * 32, CTAS) w4a4_few_kernel(const FewParams p) {
  using F = Few<NT, CTAS>;
  constexpr int KS = F::KS;
  extern __shared__ __align__(16) uint8_t few_smem[];
  float* red = reinterpret_cast<float*>(few_smem);             // [KS][kTokens][kFewPitch]
  float* sR = reinterpret_cast<float*>(few_smem + F::kMain);   // [G][32] row sums
  float* sO = sR + (p.staged ? p.G * 32 : 0);                  // [kTokens][G] offsets
  const int ks = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int g = lane >> 2, t = lane & 3;
  const int kc = p.kchunks;
  const int rb = blockIdx.x;
  const int n = rb * 32 + lane;                       // epilogue: this lane's output channel
  const int steps = (kc + 3) / 4;
  const int per = (steps + KS - 1) / KS;
  const int s0 = ks * per;
  const int s1 = s0 + per < steps ? s0 + per : steps;

  // Step s of this lane starts at byte 2048 s of its row block (and at 2048 s of
  // the tokens' block); chunks past K read as zeros.
  const uint8_t* wblk = p.w_codes + static_cast<int64_t>(rb) * kc * 512;
  const uint32_t wend = static_cast<uint32_t>(4 * s1 + t < kc ? 4 * s1 + t : kc) * 512u;
  auto load_w = [&](uint32_t off, uint4 (&v)[4]) {
#pragma unroll
    for (int i = 0; i < 4; ++i) v[i] = off < wend ? ldg_stream(wblk + off + i * 128) : make_uint4(0u, 0u, 0u, 0u);
  };
  uint32_t off = static_cast<uint32_t>(s0) * 2048u + static_cast<uint32_t>(t * 512 + g * 16);
  uint4 wv[F::kPdW][4];
  auto first_w = [&] {
#pragma unroll
    for (int i = 0; i < F::kPdW; ++i) load_w(off + i * 2048u, wv[i]);
  };
  // Each warp asks the L2 for its own share of K, so all warps' first steps come first (one request
  // for the CTA's whole block delivers the last warp's first codes after everyone else's last ones:
  // 4096 -> 4096 at 17 tokens 6.7 us against 6.0, 11008 -> 4096 at 1 token 8.7 against 8.2).
  auto prefetch_w = [&] {
    const int c0 = 4 * s0, c1 = 4 * s1 < kc ? 4 * s1 : kc;
    if (lane == 0 && c0 < c1) {
      const int bytes = (c1 - c0) * 512 < kFewL2Bytes / KS ? (c1 - c0) * 512 : kFewL2Bytes / KS;
      asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(wblk + c0 * 512), "r"(bytes) : "memory");
    }
  };
  // The epilogue's constants: the channel's scale, and the block row sums.
  float sw;
  auto constants = [&] {
    sw = n < p.N ? __ldg(p.w_scale + n) : 0.f;
    if (p.staged) {
      for (int i = threadIdx.x; i < p.G * 32; i += KS * 32) {
        const int nn = rb * 32 + (i & 31);
        if (nn < p.N)
          cp_async<4>(smem_u32(sR + i), p.rowsum + static_cast<int64_t>(i >> 5) * p.N + nn);
        else
          sR[i] = 0.f;
      }
    }
  };
  if constexpr (EARLY) {
    first_w();
    prefetch_w();
    constants();
    griddep_wait();
    griddep_launch_dependents();
  } else {
    prefetch_w();
    griddep_wait();
    first_w();
    griddep_launch_dependents();
  }
  // The warp's token codes: a ring of k-steps, chunk c of step s as kTokens rows
  // of 16 bytes. Lane l copies 16-byte pieces l, l + 32, ... of a step's 4 chunks.
  const uint32_t ring = smem_u32(few_smem) + ks * F::kRing;
  auto copy_a = [&](int s, int slot) {
    if (s < s1) {
#pragma unroll
      for (int i = 0; i < NT; ++i) {
        const int piece = lane + 32 * i, c = piece / F::kTokens, r = piece % F::kTokens;
        const uint32_t dst = ring + (slot * 4 + c) * F::kChunkPitch + r * 16;
        if (4 * s + c < kc)
          cp_async<16>(dst, p.a_codes + static_cast<uint32_t>(4 * s + c) * 512u + r * 16);
        else
          sts128(dst, 0u, 0u, 0u, 0u);
      }
    }
    few_cp_commit();
  };
#pragma unroll
  for (int i = 0; i < F::kPdA - 1; ++i) copy_a(s0 + i, i);
  if constexpr (!EARLY) constants();  // they join the next group of copies
  if (p.staged && p.a_offset != nullptr) {
    const int cnt = p.T * p.G;
    for (int i = threadIdx.x; i < cnt; i += KS * 32)
      cp_async<4>(smem_u32(sO + i), p.a_offset + i);
  }
  // Scales of the tokens this warp finishes: lane i holds token ks + KS i.
  const int my_tok = ks + KS * lane;
  const float sa_l = ks + KS * lane < F::kTokens && my_tok < p.T ? __ldg(p.a_scale + my_tok) : 0.f;

  float acc[2][NT][4];
#pragma unroll
  for (int m = 0; m < 2; ++m)
#pragma unroll
    for (int j = 0; j < NT; ++j)
#pragma unroll
      for (int i = 0; i < 4; ++i) acc[m][j][i] = 0.f;

  int slot = 0, fill = F::kPdA - 1;  // ring slots of this step and of the step copied next
  for (int sb = s0; sb < s1; sb += F::kPdW) {
#pragma unroll
    for (int u = 0; u < F::kPdW; ++u) {
      const int s = sb + u;
      if (s >= s1) break;
      asm volatile("cp.async.wait_group %0;" ::"n"(F::kPdA - 2) : "memory");
      __syncwarp();  // this step's codes are in; every lane has read the slot filled next
      copy_a(s + F::kPdA - 1, fill);
      uint4(&w)[4] = wv[u];
      uint4 a[NT];
#pragma unroll
      for (int q = 0; q < NT; ++q)
        a[q] = lds128(ring + (slot * 4 + t) * F::kChunkPitch + (8 * q + g) * 16);
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        uint32_t wp[4][4];  // rows g, g + 8, g + 16, g + 24: four half pairs each
#pragma unroll
        for (int i = 0; i < 4; ++i) weight_halves(word_of(w[i], j), wp[i]);
#pragma unroll
        for (int q = 0; q < NT; ++q) {
          uint32_t ap[4];
          act_halves(word_of(a[q], j), ap);
#pragma unroll
          for (int m = 0; m < 2; ++m) {
            mma_f16_16x8x16(acc[m][q], wp[2 * m][0], wp[2 * m + 1][0], wp[2 * m][1], wp[2 * m + 1][1], ap[0], ap[1]);
            mma_f16_16x8x16(acc[m][q], wp[2 * m][2], wp[2 * m + 1][2], wp[2 * m][3], wp[2 * m + 1][3], ap[2], ap[3]);
          }
        }
      }
      load_w(off + F::kPdW * 2048u, w);
      off += 2048u;
      slot = slot + 1 == F::kPdA ? 0 : slot + 1;
      fill = fill + 1 == F::kPdA ? 0 : fill + 1;
    }
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();  // every warp is done with its ring, which the partial sums overwrite
  // Partial sums: element (row 16 m + 8 h + g, token 8 q + 2 t + e) is acc[m][q][2 h + e].
  {
    float* r = red + ks * F::kTokens * kFewPitch;
#pragma unroll
    for (int m = 0; m < 2; ++m)
#pragma unroll
      for (int q = 0; q < NT; ++q)
#pragma unroll
        for (int i = 0; i < 4; ++i)
          r[(8 * q + 2 * t + (i & 1)) * kFewPitch + 16 * m + 8 * (i >> 1) + g] = acc[m][q][i];
  }
  __syncthreads();

  // Epilogue: lane = output channel n, tokens ks, ks + KS, ...; the chain of the
  // pair kernel, term for term: corr = sum_b o R (block 0 multiplied, then FMAs
  // in block order), a = acc' - 8 Rt (exact), y = s_w fma(s_a, a, corr).
  constexpr int NI = (F::kTokens + KS - 1) / KS;
  float cv[NI];
#pragma unroll
  for (int i = 0; i < NI; ++i) cv[i] = 0.f;
  float rt = 0.f;
  const bool has_off = p.a_offset != nullptr;
  if (p.staged) {
#pragma unroll 4
    for (int b = 0; b < p.G; ++b) {
      const float rv = sR[b * 32 + lane];
      rt += rv;
      if (has_off) {
#pragma unroll
        for (int i = 0; i < NI; ++i) {
          const float o = sO[(ks + KS * i) * p.G + b];
          cv[i] = b == 0 ? o * rv : fmaf(o, rv, cv[i]);
        }
      }
    }
  } else if (n < p.N) {
    for (int b = 0; b < p.G; ++b) {
      const float rv = __ldg(p.rowsum + static_cast<int64_t>(b) * p.N + n);
      rt += rv;
#pragma unroll
      for (int i = 0; i < NI; ++i) {
        const int tok = ks + KS * i;
        const float o = has_off && tok < p.T ? __ldg(p.a_offset + static_cast<int64_t>(tok) * p.G + b) : 0.f;
        cv[i] = b == 0 ? o * rv : fmaf(o, rv, cv[i]);
      }
    }
  }
#pragma unroll
  for (int i = 0; i < NI; ++i) {
    const int tt = ks + KS * i, tok = tt;
    const float sa = __shfl_sync(0xFFFFFFFFu, sa_l, i);
    if (tt >= F::kTokens || tok >= p.T || n >= p.N) continue;
    float acc_s = 0.f;
#pragma unroll
    for (int k = 0; k < KS; ++k) acc_s += red[(k * F::kTokens + tt) * kFewPitch + lane];
    acc_s *= kFewUnit;
    const float a = acc_s - 8.f * rt;  // exact: the integer dot product
    const float y = sw * fmaf(sa, a, cv[i]);
    const int64_t o = static_cast<int64_t>(tok) * p.ldo + n;
    if (OUT == OFFQ_F32) {
      static_cast<float*>(p.out)[o] = y;
    } else if (OUT == OFFQ_BF16) {
      static_cast<__nv_bfloat16*>(p.out)[o] = __float2bfloat16_rn(y);
    } else {
      static_cast<__half*>(p.out)[o] = __float2half_rn(y);
    }
    if (p.acc_debug != nullptr)
      p.acc_debug[static_cast<int64_t>(tok) * p.N + n] = __float2int_rn(acc_s);
  }
}

// CTAs per SM, up to 8 tokens: with more than two weight blocks per SM the call is the
// stream, and three CTAs (80 registers) keep it fuller (4096 -> 11008: 7.3 us against 8.1 with
// two); up to two blocks per SM, two CTAs (128 registers) have the shorter chain (8192 x 28672:
// 24.5 us against 37.0; 4096 x 4096: 3.6 against 3.8).
template <int OUT, int NT, int CTAS, bool EARLY>
int launch_few(FewParams p, cudaStream_t s) {
  using F = Few<NT, CTAS>;
  p.staged = p.G <= kFewStageG && F::kTokens * p.G <= kFewStageO;
  const size_t bytes = F::kMain + (p.staged ? p.G * 32 + F::kTokens * p.G : 0) * sizeof(float);
  if (!smem_optin<w4a4_few_kernel<OUT, NT, CTAS, EARLY>>(F::kMain + (kFewStageG * 32 + kFewStageO) * 4)) return OFFQ_ERR_CUDA;
  const dim3 grid((p.N + 31) / 32);
  return launch_pdl(w4a4_few_kernel<OUT, NT, CTAS, EARLY>, grid, dim3(kFewWarps * 32), bytes, s, p);
}

template <int OUT>
int dispatch_few(const FewParams& p, bool many_blocks, bool early, cudaStream_t s) {
  if (early) return many_blocks ? launch_few<OUT, 1, 3, true>(p, s) : launch_few<OUT, 1, 2, true>(p, s);
  if (p.T <= 8) return many_blocks ? launch_few<OUT, 1, 3, false>(p, s) : launch_few<OUT, 1, 2, false>(p, s);
  if (p.T <= 16) return launch_few<OUT, 2, 2, false>(p, s);
  return launch_few<OUT, 4, 2, false>(p, s);
}

// Whether the weights may be read before the kernel ahead has finished, which asks of the caller
// that it does not write them and release its dependents early: the calls that offq.h lists, and
// no others.
constexpr int kEarlyTokens = 4;
constexpr int64_t kEarlyActs = 96 * 1024;
bool reads_early(int64_t T, int64_t K) {
  return T <= kEarlyTokens && (T > 2 ? kEarlyTokens : T) * K <= kEarlyActs;
}

}  // namespace

namespace offq {

int few_max_tokens() { return kFewMaxT; }

// The few-token form of offq_w4a4_linear (arguments checked by the caller; 1 <= T <= few_max_tokens()).
int w4a4_linear_few(const uint8_t* a_codes, const float* a_scale, const float* a_offset, int64_t T, int64_t N,
                    int64_t K, int32_t g, const uint8_t* w_codes, const float* w_scale, const float* w_offsum,
                    void* out, int out_dtype, int64_t ldo, int32_t* acc_debug, cudaStream_t stream) {
  const int sms = device_sms();
  if (sms < 1) return OFFQ_ERR_CUDA;
  FewParams p{};
  p.a_codes = a_codes;
  p.w_codes = w_codes;
  p.a_scale = a_scale;
  p.a_offset = a_offset;
  p.w_scale = w_scale;
  p.rowsum = w_offsum;
  p.out = out;
  p.ldo = ldo;
  p.acc_debug = acc_debug;
  p.T = static_cast<int>(T);
  p.N = static_cast<int>(N);
  p.G = static_cast<int>(K / g);
  p.kchunks = static_cast<int>(K / 32);
  const bool early = reads_early(T, K);
  const bool many = (N + 31) / 32 > 2 * sms;
  switch (out_dtype) {
    case OFFQ_F32: return dispatch_few<OFFQ_F32>(p, many, early, stream);
    case OFFQ_BF16: return dispatch_few<OFFQ_BF16>(p, many, early, stream);
    case OFFQ_F16: return dispatch_few<OFFQ_F16>(p, many, early, stream);
    default: return OFFQ_ERR_INVALID_ARG;
  }
}

}  // namespace offq
