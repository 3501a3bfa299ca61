// Intra-block rotation + quantization of a 16-row x 32-column tile of rotated activations by ONE
// warp on the warp-level tensor cores (Algorithm 3 steps 3-4 for one 32-block
// of 16 tokens): y is split into three bfloat16 terms (y = hi + mid + lo up to 2^-24 relative),
// R_intra is bfloat16 already, so every product is exact in fp32 and the fp32-accumulating
// mma.sync m16n8k16 reproduces the fp32 rotation up to the order of additions.  Then Eq. 1 (or the
// NVFP4 / MXINT4 quantizer) on the accumulator fragments: four lanes share a row.
#pragma once
#include <cuda_bf16.h>
#include "nvfp4_quantize.cuh"
#include "mxint4_quantize.cuh"
#include "quantize.cuh"
#include "sm100_ptx.cuh"

namespace torq {

// B fragments of one R_intra block for intra_quantize_frag16.  rb0 / rb1: this lane's ldmatrix row addresses for
// columns 0-15 / 16-31 of rows 0-15 (lane l: row l % 8 of matrix l / 8; matrices (k 0-7, n), (k 8-15, n), (k 0-7, n+8),
// (k 8-15, n+8)); kc_stride: bytes to rows 16-31.
struct IntraFrag { uint32_t b[2][4][2]; };               // [k chunk][n tile][2]
__device__ __forceinline__ void load_intra_frag(uint32_t rb0, uint32_t rb1, uint32_t kc_stride, IntraFrag& f) {
#pragma unroll
  for (int kc = 0; kc < 2; ++kc) {
    ldmatrix_x4_trans(rb0 + kc * kc_stride, f.b[kc][0][0], f.b[kc][0][1], f.b[kc][1][0], f.b[kc][1][1]);
    ldmatrix_x4_trans(rb1 + kc * kc_stride, f.b[kc][2][0], f.b[kc][2][1], f.b[kc][3][0], f.b[kc][3][1]);
  }
}

// Intra rotation and quantization of 16 rows x 32 columns that arrive in the fragment layout (y as
// tmem_ld_16x256b_x4 gives it), so that they never pass through shared memory.  row0: first of the 16 rows;
// scale byte(s) of rows row0 + lane / 4 + 8 rh come back in sb[rh] (0 past the last block for NVFP4; for the other
// formats a block of zeros has byte 0 by itself).
// SHORT_CHAIN: one accumulator per split term, so that only two instructions depend on each other, and the terms added
// smallest first -- for a warp that has one such unit to do and nothing to overlap it with (a single chain of six was
// a third of the unit's time); otherwise one accumulator, which keeps sixteen more registers free.
template <int FMT, bool SHORT_CHAIN = false>
__device__ __forceinline__ void intra_quantize_frag16(const uint32_t (&y)[16], bool has_intra, const IntraFrag& f, int lane,
                                                      int64_t row0, int M, int blk, int nblocks, int d, const NvScale& nvs,
                                                      uint8_t* __restrict__ codes, uint32_t* sb) {
  const int p = lane & 3, r8 = lane >> 2;
  float acc[4][4];
  if (has_intra) {
    uint32_t ah[8], am[8], al[8];                        // A fragments: [k chunk * 4 + (n & 1) * 2 + row half]
#pragma unroll
    for (int n = 0; n < 4; ++n)
#pragma unroll
      for (int rh = 0; rh < 2; ++rh) {
        const int ai = (n >> 1) * 4 + (n & 1) * 2 + rh;
        split3_bf16x2(y[4 * n + 2 * rh], y[4 * n + 2 * rh + 1], ah[ai], am[ai], al[ai]);
      }
#pragma unroll
    for (int n = 0; n < 4; ++n) { acc[n][0] = 0.f; acc[n][1] = 0.f; acc[n][2] = 0.f; acc[n][3] = 0.f; }
    if constexpr (SHORT_CHAIN) {
      float accm[4][4], acch[4][4];
#pragma unroll
      for (int n = 0; n < 4; ++n)
#pragma unroll
        for (int e = 0; e < 4; ++e) { accm[n][e] = 0.f; acch[n][e] = 0.f; }
#pragma unroll
      for (int kc = 0; kc < 2; ++kc)
#pragma unroll
        for (int n = 0; n < 4; ++n) {
          mma_16816_bf16(acc[n], al + 4 * kc, f.b[kc][n]);
          mma_16816_bf16(accm[n], am + 4 * kc, f.b[kc][n]);
          mma_16816_bf16(acch[n], ah + 4 * kc, f.b[kc][n]);
        }
#pragma unroll
      for (int n = 0; n < 4; ++n)
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[n][e] = (acc[n][e] + accm[n][e]) + acch[n][e];
    } else {
#pragma unroll
      for (int kc = 0; kc < 2; ++kc)
#pragma unroll
        for (int n = 0; n < 4; ++n) {
          mma_16816_bf16(acc[n], al + 4 * kc, f.b[kc][n]);
          mma_16816_bf16(acc[n], am + 4 * kc, f.b[kc][n]);
          mma_16816_bf16(acc[n], ah + 4 * kc, f.b[kc][n]);
        }
    }
  } else {
#pragma unroll
    for (int n = 0; n < 4; ++n)
#pragma unroll
      for (int e = 0; e < 4; ++e) acc[n][e] = __uint_as_float(y[4 * n + e]);
  }
#pragma unroll
  for (int rh = 0; rh < 2; ++rh) {
    const float v[8] = {acc[0][2 * rh], acc[0][2 * rh + 1], acc[1][2 * rh], acc[1][2 * rh + 1],
                        acc[2][2 * rh], acc[2][2 * rh + 1], acc[3][2 * rh], acc[3][2 * rh + 1]};
    uint32_t word, sbyte;
    const int64_t row = row0 + r8 + 8 * rh;
    if constexpr (FMT == FMT_MXINT4) {                   // two operand bytes per 8 columns and lane
      uint32_t pr[4];
      mxint4_quantize_row_fragment(v, pr, sbyte);
      if (row < M && blk < nblocks) {
        uint8_t* dst = codes + row * (int64_t)d + (int64_t)blk * 32 + 2 * p;
#pragma unroll
        for (int nt = 0; nt < 4; ++nt) *reinterpret_cast<uint16_t*>(dst + 8 * nt) = (uint16_t)pr[nt];
      }
    } else {
      if constexpr (FMT == FMT_NVFP4) nv_quantize_row_fragment(v, p, nvs, word, sbyte);
      else quantize_row_fragment(v, p, word, sbyte);
      if (row < M && blk < nblocks)
        *reinterpret_cast<uint32_t*>(codes + row * (int64_t)(d / 2) + (int64_t)blk * 16 + 4 * p) = word;
    }
    if constexpr (FMT == FMT_NVFP4) {
      if (blk >= nblocks) sbyte = 0;                     // padding blocks decode to zero
    }
    sb[rh] = sbyte;
  }
}

// Few tokens, ONE FEATURE OF A 32-BLOCK PER LANE, four tokens in registers.
// z[t] = sum_k y[k][t] R[k][lane], fp32, k in index order.  y: shared memory [32 features][4 tokens] fp32, read by broadcast;
// r[i]: R_intra[2 i][lane] (low half) and R_intra[2 i + 1][lane], bf16.
__device__ __forceinline__ void intra_rotate_lane4(uint32_t y_saddr, const uint32_t (&r)[16], float (&z)[4]) {
#pragma unroll
  for (int t = 0; t < 4; ++t) z[t] = 0.f;
#pragma unroll
  for (int k = 0; k < 32; ++k) {
    float4 y;
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(y.x), "=f"(y.y), "=f"(y.z), "=f"(y.w) : "r"(y_saddr + 16u * k));
    const float w = __uint_as_float((k & 1) ? (r[k >> 1] & 0xFFFF0000u) : (r[k >> 1] << 16));
    z[0] = fmaf(y.x, w, z[0]); z[1] = fmaf(y.y, w, z[1]); z[2] = fmaf(y.z, w, z[2]); z[3] = fmaf(y.w, w, z[3]);
  }
}
// Quantizes the 32 features x 4 tokens and stores codes and scale bytes of tokens row0 .. row0 + 3 below M (the scale bytes of the
// others: zero; M = 0: nothing at all).  The arithmetic is that of the row forms above, value by value.
template <int FMT>
__device__ __forceinline__ void quantize_lane4(const float (&z)[4], int lane, int row0, int M, int blk, int d, int kb4, const NvScale& nvs,
                                               uint8_t* __restrict__ codes, uint8_t* __restrict__ scales) {
  float a[4];
  uint32_t sb = 0;                                       // of token row0 + lane % 4 (NVFP4: and this lane's half of the 32 features)
  float f[4];                                            // multiplier of the elements
#pragma unroll
  for (int t = 0; t < 4; ++t) a[t] = fmaxf(0.f, fabsf(z[t]));       // a NaN does not count
  if constexpr (FMT == FMT_NVFP4) {
#pragma unroll
    for (int o = 8; o > 0; o >>= 1)
#pragma unroll
      for (int t = 0; t < 4; ++t) a[t] = fmaxf(a[t], __shfl_xor_sync(0xFFFFFFFFu, a[t], o));
    const int t = lane & 3;                              // one division per lane
    float r;
    nv_block_scale(t == 0 ? a[0] : (t == 1 ? a[1] : (t == 2 ? a[2] : a[3])), nvs, sb, r);
#pragma unroll
    for (int t = 0; t < 4; ++t) f[t] = __shfl_sync(0xFFFFFFFFu, r, (lane & 16) + t);
  } else {
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      uint32_t b;
      block_scale(__uint_as_float(__reduce_max_sync(0xFFFFFFFFu, __float_as_uint(a[t]))), b, f[t]);
      if (lane == t) sb = b;
    }
  }
#pragma unroll
  for (int t = 0; t < 4; ++t) {
    const int row = row0 + t;
    if constexpr (FMT == FMT_MXINT4) {
      const uint32_t w = pack4_e4m3(int4_round(z[t] * f[t]), 0.f, 0.f, 0.f);
      if (row < M) codes[(int64_t)row * d + blk * 32 + lane] = (uint8_t)w;
    } else {
      const float v = __fmul_rn(z[t], f[t]), v1 = __shfl_down_sync(0xFFFFFFFFu, v, 1);
      const uint32_t w = pack8_e2m1(v, v1, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f);
      if (row < M && !(lane & 1)) codes[(int64_t)row * (d / 2) + blk * 16 + (lane >> 1)] = (uint8_t)w;
    }
  }
  if (M > 0 && (lane & 15) < 4 && (FMT == FMT_NVFP4 || lane < 4)) {
    const int row = row0 + (lane & 3);
    const int kb = FMT == FMT_NVFP4 ? 2 * blk + (lane >> 4) : blk;
    scales[scale_offset(row, kb, kb4)] = row < M ? (uint8_t)sb : (uint8_t)0;
  }
}

}  // namespace torq
