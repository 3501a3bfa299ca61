// Block-scaled GEMM for few tokens (M <= 128; Algorithm 3 step 5), where the work is streaming the
// weights from HBM once.  One kernel, no scratch in global memory.
//
// Swapped operands: the tensor-core instruction's 128 rows are 128 output FEATURES (rows of the
// stored weight W' [N, K]) and its N columns are the tokens (16 ... 128, in steps of 16):
//   D[n, m] = sum_k w^[n, k] a^[m, k]
//   A = W tile [128 rows x 128 B of K], scale chunks of W;  B = activation tile [tokens x 128 B],
//   scale chunks of the activations (their single 128-row scale tile).
// A layer has only N / 128 such tiles (40 at N = 5120), so K is split as well: a CLUSTER of S CTAs
// shares one tile, CTA r contracts k range r; the fp32 partial tiles stay on the SMs and are added in rank order (fixed).
// As in the few-token rotation they reach the adding CTA in one of two ways:
//  * PUSH (up to 16 tokens, for K > 2048 up to 32, NVFP4 24): the sums are dealt over all CTAs and warps of the cluster in pieces of 32
//    features x 4 tokens, and every CTA stores its partials of a piece straight from registers into the owner's shared memory (st.async,
//    16 bytes per lane = four tokens of one feature, counted on a barrier of the owning warp), into room of their own.  K = N = 5120, us:
//    pulled 1 token 4.7, 24 tokens 5.6; pushed to one owner per four tokens, into its stages, 4.4 and 16 tokens 4.95; so 4.4, 4.7 and 24
//    tokens 5.25.
//  * pull (more tokens): each CTA writes its partial [token][feature] into its own shared memory, a cluster barrier
//    publishes them, and CTA r adds, for the tokens m = r (mod S), the S partials read with 16-byte ld.shared::cluster.
// With S = 1 (an ordinary launch without clusters) the accumulator goes to Y directly.
//
// Roles per CTA: warp 0 TMA producer, warp 1 MMA issuer (scale chunks shared -> tensor memory, then the
// instructions), warps 2..5 epilogue / reduction.  Shared memory: 4 stages of (16 KiB of W + tokens x
// 128 B + the scale chunks), reused for the partials after the mainloop; at most 113 KiB up to 64 tokens, so
// these CTAs become resident beside those of the few-token rotation that precedes them in the stream and
// fetch their first weight stages while it still runs (the weights are constants of the layer).
#pragma once
#include <cuda_bf16.h>
#include "rotate_fewtok.cuh"
#include "sm100_ptx.cuh"

namespace torq {

template <int FMT = FMT_MXFP4>
struct GemmFewCfg {
  static constexpr int BF = 128;                       // output features per tile = rows of the instruction
  static constexpr int BK = FMT == FMT_MXINT4 ? 128 : 256;   // elements of K per stage (128 bytes per row)
  static constexpr int A_BYTES = BF * 128;             // 16 KiB
  static constexpr int CH = FMT == FMT_NVFP4 ? 4 : (FMT == FMT_MXINT4 ? 1 : 2);   // scale chunks per stage and 128 rows
  static constexpr int SF_BYTES = CH * 512;
  static constexpr int STAGES = 4;
  // (the same for every token count: three stages at 128 tokens would let two CTAs share an SM, clusters of 5
  // instead of 3, which measured 4 - 10 % slower than four stages and one CTA per SM)
  static constexpr int BAR_BYTES = 256;
  static constexpr int THREADS = 192;
  static constexpr int MAX_CLUSTER = 8;
  static constexpr int MAX_TOK = 128;                  // one 128-row scale tile of the activations
  __host__ __device__ static constexpr int stage_bytes(int ntok) {
    return (A_BYTES + ntok * 128 + 2 * SF_BYTES + 1023) / 1024 * 1024;
  }
  // partial sums of the units that one CTA owns, from all CTAs, for any cluster size
  static constexpr int PART_BYTES = 32 * 16;           // of a unit from one CTA: [feature of the quarter][4 tokens]
  static constexpr int MAX_PUSH_TOK = 32;
  __host__ __device__ static constexpr int push_bytes(int M) { return ((M + 3) / 4 * 4 + MAX_CLUSTER - 1) * PART_BYTES; }
  __host__ __device__ static constexpr int pull_smem_bytes(int M) { return STAGES * stage_bytes((M + 15) / 16 * 16) + BAR_BYTES + 1024; }
  // Pushed where the room for what arrives leaves two CTAs per SM (NVFP4: up to 24 tokens); from 17 tokens on for contractions long enough
  // that a cluster of four has work for it (us, pulled / pushed, 32 tokens: N = 4096, K = 2048 3.72 / 4.01, K = 4096 4.47 / 4.49, K =
  // 14336 8.82 / 7.93, layers 4096 x 4096 13.7 / 13.2, 2048 x 4096 9.1 / 9.3; 18 tokens N = K = 5120 5.31 / 4.83).
  __host__ __device__ static constexpr bool push(int M, int K) {
    return M <= 16 || (M <= MAX_PUSH_TOK && K > 2048 && pull_smem_bytes(M) + push_bytes(M) <= 113 * 1024);
  }
  __host__ __device__ static constexpr int smem_bytes(int M, int K) { return pull_smem_bytes(M) + (push(M, K) ? push_bytes(M) : 0); }
  __host__ __device__ static constexpr int ctas_per_sm(int M, int K) { return smem_bytes(M, K) <= 113 * 1024 ? 2 : 1; }
  __host__ __device__ static constexpr int max_smem_bytes() { return pull_smem_bytes(MAX_TOK); }
  static_assert(BF * 4 <= STAGES * 128, "the pulled partial tile lies in the stages after the mainloop");
  __host__ __device__ static constexpr uint32_t tmem_cols(int ntok) {
    return ntok + 8 * CH <= 32 ? 32u : (ntok + 8 * CH <= 64 ? 64u : (ntok + 8 * CH <= 128 ? 128u : 256u));
  }
};

// grid = ceil(N / 128) * S CTAs in clusters of S along x: CTA b works feature tile b / S, k split b % S.
// w_ahead: W tiles beyond the stages that a CTA asks the L2 for.  tmW: Wq [N, K bytes] box [128 x 128]; tmA: Aq [M, K bytes] box [ntok x
// 128]; As / Ws: tiled scales.
// ESETS: sets of four epilogue warps (threads = 64 + 128 ESETS): one set and two CTAs per SM up to 64 tokens (MXINT4: 80, where
// that splits K further); two sets above, where a CTA fills an SM by itself and has some forty tokens to add up and store.
template <int FMT = FMT_MXFP4, int ESETS = 1, bool PUSH = false>
__global__ void __launch_bounds__(64 + 128 * ESETS, ESETS == 1 ? 2 : 1)
gemm_fewtok_kernel(const __grid_constant__ CUtensorMap tmW, const __grid_constant__ CUtensorMap tmA,
                   const uint8_t* __restrict__ As, const uint8_t* __restrict__ Ws, void* __restrict__ Y,
                   int y_is_bf16, int M, int N, int K, int ntok, int S, int w_ahead, float alpha, int* err_word) {
  using C = GemmFewCfg<FMT>;
  constexpr int CH = C::CH;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t* smem_gen = smem_raw + (smem_base - smem_u32(smem_raw));
  const int stage_bytes = C::stage_bytes(ntok);
  const int b_bytes = ntok * 128;
  constexpr int nst = C::STAGES;
  const uint32_t bar_off = nst * stage_bytes;
  const uint32_t bar_base = smem_base + bar_off;
  auto full_bar = [&](int s) { return bar_base + 8u * s; };
  auto empty_bar = [&](int s) { return bar_base + 8u * (C::STAGES + s); };
  const uint32_t accf_bar = bar_base + 8u * (2 * C::STAGES);
  auto recv_bar = [&](int w) { return accf_bar + 8u + 8u * w; };   // PUSH: all partials of the units of epilogue warp w are here
  const uint32_t recv_base = bar_base + C::BAR_BYTES;
  volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(smem_gen + bar_off + 192);
  volatile int* cta_abort = reinterpret_cast<volatile int*>(smem_gen + bar_off + 200);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = blockIdx.x % S, nt = blockIdx.x / S;
  const int k_tiles = (K + C::BK - 1) / C::BK;           // K % 128 == 0: the last stage may be half
  const int kb4 = K / (C::BK / CH);                      // scale chunks per row
  const int kt0 = (int)((long long)k_tiles * rank / S), kt1 = (int)((long long)k_tiles * (rank + 1) / S);
  const uint32_t tmem_cols = C::tmem_cols(ntok);
  // PUSH: unit u = q + 4 c is quarter q of the tile's features and tokens 4 c .. 4 c + 3; CTA u % S owns it, its epilogue warp
  // u / S % 4 adds and stores it
  const int units = 4 * ((M + 3) / 4);

  // The weights and their scales are constants of the layer, never the output of the kernel that runs
  // just before this one: the thread that initialises the barriers sends their loads for the first
  // stages right behind the initialisation (the kernel's time starts with an HBM round trip; tensor-
  // memory allocation and the block-wide barrier come after it instead of before); the activations wait.
  const int pre = (kt1 - kt0) < nst ? (kt1 - kt0) : nst;
  auto stage_tx = [&](int kt) { return (uint32_t)(C::A_BYTES + b_bytes) + 2u * 512u * (uint32_t)min(CH, kb4 - CH * kt); };
  if (threadIdx.x == 0) {
    for (int s = 0; s < nst; ++s) { mbar_init(full_bar(s), 1); mbar_init(empty_bar(s), 1); }
    mbar_init(accf_bar, 1);
    if constexpr (PUSH)
      for (int w = 0; w < 4; ++w) mbar_init(recv_bar(w), 1);
    *cta_abort = 0;
    fence_mbar_init();
    fence_proxy_async_smem();                            // the copy engine sees the initialised barriers
    for (int it = 0; it < pre; ++it) {
      const int kt = kt0 + it;
      const uint32_t st = smem_base + it * stage_bytes;
      mbar_arrive_expect_tx(full_bar(it), stage_tx(kt));
      tma_load_2d(st, &tmW, kt * 128, nt * C::BF, full_bar(it));
      bulk_load_1d(st + C::A_BYTES + b_bytes, Ws + ((size_t)nt * kb4 + CH * kt) * 512,
                   512u * (uint32_t)min(CH, kb4 - CH * kt), full_bar(it));
    }
    tma_prefetch_desc(&tmA);
    if (PUSH && S > 1)
      for (int w = 0; w < 4 && rank + S * w < units; ++w)
        mbar_arrive_expect_tx(recv_bar(w), (uint32_t)((units - rank - S * w + 4 * S - 1) / (4 * S) * S * C::PART_BYTES));
  }
  if (warp == 1) { tmem_alloc(smem_u32(const_cast<uint32_t*>(tmem_slot)), tmem_cols); tmem_relinquish(); }
  tc_fence_before_sync();
  __syncthreads();
  if (PUSH && S > 1) cluster_arrive_relaxed();           // the wait stands before the first access to another CTA
  tc_fence_after_sync();
  const uint32_t tmem_base = *tmem_slot;
  griddep_launch_dependents();
  const int a_pre = PUSH ? pre : 0;                      // activation tiles that the epilogue warps send
  // While the kernel before ends HBM idles: the L2 is asked for W beyond the stages (us, without / with, layers: 128 x 4096 -> 6144 19.05
  // / 18.8, 100 x 4096 -> 12288 21.9 / 21.6, 16 x 8192 -> 8192 29.65 / 29.5).  By a warp that has time for it, in its own branch: in the
  // way of the epilogue warps' dry pass the instructions alone cost up to 3 % (56 x 2048 -> 2048 NVFP4 10.76 / 11.1).
  auto ask = [&]() {
    if (elect_one())
      for (int kt = kt0 + pre; kt < min(kt1, kt0 + pre + w_ahead); ++kt) tma_prefetch_l2_2d(&tmW, kt * 128, nt * C::BF);
    __syncwarp();
  };
  if (PUSH ? warp < 2 : warp != 1) griddep_wait();

  bool acc_ok = false;
  if (warp == 0) {
    // ------------------------------------------------------------------ TMA producer
    bool ok = true;
    for (int kt = kt0 + a_pre, it = a_pre; kt < kt1 && ok; ++kt, ++it) {
      const int s = it % nst;
      if (!mbar_wait_warp(empty_bar(s), ((it / nst) & 1) ^ 1, cta_abort, err_word, SITE_PRODUCER_EMPTY)) {
        ok = false; break;
      }
      const uint32_t st = smem_base + s * stage_bytes;
      const uint32_t sf_bytes = 512u * (uint32_t)min(CH, kb4 - CH * kt);
      if (elect_one()) {
        if (it >= pre) {                                 // the W side of the first stages went out before the wait above
          mbar_arrive_expect_tx(full_bar(s), stage_tx(kt));
          tma_load_2d(st, &tmW, kt * 128, nt * C::BF, full_bar(s));
          bulk_load_1d(st + C::A_BYTES + b_bytes, Ws + ((size_t)nt * kb4 + CH * kt) * 512, sf_bytes, full_bar(s));
        }
        tma_load_2d(st + C::A_BYTES, &tmA, kt * 128, 0, full_bar(s));
        bulk_load_1d(st + C::A_BYTES + b_bytes + C::SF_BYTES, As + (size_t)(CH * kt) * 512, sf_bytes, full_bar(s));
      }
      __syncwarp();
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer
    if constexpr (!PUSH) {
      ask();
      griddep_wait();
    }
    bool ok = true;
    const uint32_t idesc0 = FMT == FMT_NVFP4 ? idesc_nvf4(128, ntok) : idesc_mxf4(128, ntok, 0, 0);
    const uint32_t idesc2 = FMT == FMT_NVFP4 ? idesc_nvf4(128, ntok) : idesc_mxf4(128, ntok, 2, 2);
    const uint32_t sfa_t = tmem_base + ntok, sfb_t = tmem_base + ntok + 4 * CH;     // 4 columns per chunk each
    for (int kt = kt0, it = 0; kt < kt1 && ok; ++kt, ++it) {
      const int s = it % nst;
      if (!mbar_wait_warp(full_bar(s), (it / nst) & 1, cta_abort, err_word, SITE_MMA_FULL)) {
        ok = false; break;
      }
      tc_fence_after_sync();
      const bool two = (kb4 - CH * kt) >= CH;              // K % 256 == 128: the last stage is half
      const uint32_t st = smem_base + s * stage_bytes;
      const uint64_t adesc = make_desc(st, 16, 1024, kSwizzle128);
      const uint64_t bdesc = make_desc(st + C::A_BYTES, 16, 1024, kSwizzle128);
      const uint64_t sfa_d = make_desc(st + C::A_BYTES + b_bytes, 0, 128, 0);
      const uint64_t sfb_d = make_desc(st + C::A_BYTES + b_bytes + C::SF_BYTES, 0, 128, 0);
      if (elect_one()) {
#pragma unroll
        for (int c = 0; c < CH; ++c) {
          if (c < CH / 2 || two) {
            tmem_cp_32x128b_warpx4(sfa_t + 4 * c, sfa_d + 32 * c);
            tmem_cp_32x128b_warpx4(sfb_t + 4 * c, sfb_d + 32 * c);
          }
        }
        if constexpr (FMT == FMT_MXINT4) {                 // a quarter chunk (one scale byte) per instruction
          mma_mxf8(tmem_base, adesc, bdesc, idesc_mxf8(128, ntok, 0), sfa_t, sfb_t, it != 0);
          mma_mxf8(tmem_base, adesc + 2, bdesc + 2, idesc_mxf8(128, ntok, 1), sfa_t, sfb_t, 1);
          mma_mxf8(tmem_base, adesc + 4, bdesc + 4, idesc_mxf8(128, ntok, 2), sfa_t, sfb_t, 1);
          mma_mxf8(tmem_base, adesc + 6, bdesc + 6, idesc_mxf8(128, ntok, 3), sfa_t, sfb_t, 1);
        } else if constexpr (FMT == FMT_NVFP4) {           // one chunk per instruction
#pragma unroll
          for (int j = 0; j < 4; ++j)
            if (j < 2 || two)
              mma_nvf4(tmem_base, adesc + 2 * j, bdesc + 2 * j, idesc0, sfa_t + 4 * j, sfb_t + 4 * j, (it | j) != 0);
        } else {                                           // half a chunk (two scale bytes) per instruction
          mma_mxf4(tmem_base, adesc, bdesc, idesc0, sfa_t, sfb_t, it != 0);
          mma_mxf4(tmem_base, adesc + 2, bdesc + 2, idesc2, sfa_t, sfb_t, 1);
          if (two) {
            mma_mxf4(tmem_base, adesc + 4, bdesc + 4, idesc0, sfa_t + 4, sfb_t + 4, 1);
            mma_mxf4(tmem_base, adesc + 6, bdesc + 6, idesc2, sfa_t + 4, sfb_t + 4, 1);
          }
        }
        tc_commit(empty_bar(s));
      }
      __syncwarp();
    }
    if (ok && elect_one()) tc_commit(accf_bar);
    __syncwarp();
  } else {
    // ------------------------------------------------------------------ epilogue (warps 2..5)
    if constexpr (PUSH) {
      if (warp == 3) ask();
      griddep_wait();
    }
    // The activations of the first stages go out from four warps at once: one warp needs 0.2 us from one stage to the next.
    if (PUSH && warp - 2 < pre && elect_one()) {
      const int it = warp - 2;
      const uint32_t st = smem_base + it * stage_bytes;
      tma_load_2d(st + C::A_BYTES, &tmA, (kt0 + it) * 128, 0, full_bar(it));
      bulk_load_1d(st + C::A_BYTES + b_bytes + C::SF_BYTES, As + (size_t)(CH * (kt0 + it)) * 512,
                   512u * (uint32_t)min(CH, kb4 - CH * (kt0 + it)), full_bar(it));
    }
    __syncwarp();
    // Two passes over the SAME instructions, as in the few-token rotation: pass 0 is a dry run while the
    // mainloop streams (reads this CTA's own shared memory, stores nothing) so that the reduction's code is
    // in the instruction cache when it is needed; pass 1: accumulator -> partials, then the tokens of this CTA.
    const int q = warp & 3;
    const int ew = warp - 2;                             // 0 .. 4 ESETS - 1
    const int feature = q * 32 + lane;                   // of this lane in tensor memory
    const uint32_t tacc = tmem_base + ((uint32_t)(q * 32) << 16);
    if (S == 1) {                                        // nothing to add: accumulator -> Y
      acc_ok = mbar_wait(accf_bar, 0, cta_abort, err_word, SITE_EPI_ACC_FULL);
      acc_ok = __all_sync(0xFFFFFFFFu, acc_ok);
      tc_fence_after_sync();
      const int64_t n = (int64_t)nt * C::BF + feature;
      for (int c0 = 16 * (ew >> 2); acc_ok && c0 < M; c0 += 16 * ESETS) {
        uint32_t v[16];
        tmem_ld_32x32_x16(tacc + c0, v);
        tmem_ld_wait();
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          float y = __uint_as_float(v[j]);
          if constexpr (FMT == FMT_NVFP4) y *= alpha;
          if (c0 + j < M && n < N) {
            if (y_is_bf16) reinterpret_cast<__nv_bfloat16*>(Y)[(int64_t)(c0 + j) * N + n] = __float2bfloat16_rn(y);
            else reinterpret_cast<float*>(Y)[(int64_t)(c0 + j) * N + n] = y;
          }
        }
      }
    } else if constexpr (PUSH) {
      const int w = q;
      // where this warp's partials go: quarter q, tokens 4 c ... (worked out before they are needed: a division takes as long as a store)
      uint32_t dst[C::MAX_PUSH_TOK / 4], dst_bar[C::MAX_PUSH_TOK / 4];
#pragma unroll
      for (int c = 0; c < C::MAX_PUSH_TOK / 4; ++c) {
        const int u = q + 4 * c, ui = u / S, owner = u - ui * S;
        dst[c] = map_to_cta(recv_base + (uint32_t)((ui * S + rank) * C::PART_BYTES + lane * 16), (uint32_t)owner);
        dst_bar[c] = map_to_cta(recv_bar(ui & 3), (uint32_t)owner);
      }
      cluster_wait();
#pragma unroll 1
      for (int pass = rank + S * w < units ? 0 : 1; pass < 2; ++pass) {
        const bool live = pass == 1;
        if (live) {
          acc_ok = mbar_wait(accf_bar, 0, cta_abort, err_word, SITE_EPI_ACC_FULL);
          acc_ok = __all_sync(0xFFFFFFFFu, acc_ok);
          if (!acc_ok) break;
          tc_fence_after_sync();
          uint32_t v[C::MAX_PUSH_TOK];
          tmem_ld_32x32_x16(tacc, *reinterpret_cast<uint32_t(*)[16]>(v));
          if (ntok > 16) tmem_ld_32x32_x16(tacc + 16, *reinterpret_cast<uint32_t(*)[16]>(v + 16));
          tmem_ld_wait();
#pragma unroll
          for (int c = 0; c < C::MAX_PUSH_TOK / 4; ++c)
            if (4 * c < M) st_async_v4(dst[c], v[4 * c], v[4 * c + 1], v[4 * c + 2], v[4 * c + 3], dst_bar[c]);
          if (rank + S * w >= units) break;              // nothing to receive
          const bool ok = mbar_wait_cluster(recv_bar(w), 0, cta_abort, err_word, SITE_EPI_ACC_FULL);
          if (!__all_sync(0xFFFFFFFFu, ok)) break;
        }
#pragma unroll 1
        for (int u = rank + S * w, ui = w; u < units; u += 4 * S, ui += 4) {
          // lane l has feature l of the quarter: one 16-byte load per partial gives its four tokens
          const int m0 = u & ~3;
          const int64_t n = (int64_t)nt * C::BF + (u & 3) * 32 + lane;
          float4 part[C::MAX_CLUSTER];
#pragma unroll
          for (int s = 0; s < C::MAX_CLUSTER; ++s)
            if (s < S)
              asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                           : "=f"(part[s].x), "=f"(part[s].y), "=f"(part[s].z), "=f"(part[s].w)
                           : "r"(recv_base + (uint32_t)((ui * S + s) * C::PART_BYTES + lane * 16)));
          float y[4] = {0.f, 0.f, 0.f, 0.f};             // rank order: the result does not depend on timing
#pragma unroll
          for (int s = 0; s < C::MAX_CLUSTER; ++s)
            if (s < S) { y[0] += part[s].x; y[1] += part[s].y; y[2] += part[s].z; y[3] += part[s].w; }
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            if constexpr (FMT == FMT_NVFP4) y[j] *= alpha;
            if (live && m0 + j < M && n < N) {
              if (y_is_bf16) reinterpret_cast<__nv_bfloat16*>(Y)[(int64_t)(m0 + j) * N + n] = __float2bfloat16_rn(y[j]);
              else reinterpret_cast<float*>(Y)[(int64_t)(m0 + j) * N + n] = y[j];
            }
          }
        }
      }
    } else {
      // A warp takes one token per pass: lane l adds features 4 l .. 4 l + 3 (16-byte loads, 512 contiguous
      // bytes per warp and partial) and stores 8 or 16 bytes of the token's row of Y.  Two tokens per
      // iteration, all their loads issued before the first add: few round trips through the cluster.
      constexpr int NW = 4 * ESETS;
      const int64_t n = (int64_t)nt * C::BF + 4 * lane;
      const uint32_t p_saddr = smem_base;
#pragma unroll 1
      for (int pass = 0; pass < 2; ++pass) {
        const bool live = pass == 1;
        if (live) {
          // ---- epilogue 1: partial tile -> own shared memory
          acc_ok = mbar_wait(accf_bar, 0, cta_abort, err_word, SITE_EPI_ACC_FULL);
          acc_ok = __all_sync(0xFFFFFFFFu, acc_ok);
          if (acc_ok) {
            tc_fence_after_sync();
            float* prow = reinterpret_cast<float*>(smem_gen) + feature;     // partial tile [token][feature]
            for (int c0 = 16 * (ew >> 2); c0 < ntok; c0 += 16 * ESETS) {
              uint32_t v[16];
              tmem_ld_32x32_x16(tacc + c0, v);
              tmem_ld_wait();
#pragma unroll
              for (int j = 0; j < 16; ++j) prow[(c0 + j) * C::BF] = __uint_as_float(v[j]);
            }
          }
          tc_fence_before_sync();
          cluster_sync_all();                              // every CTA's partial tile is visible cluster-wide
        }
        // ---- epilogue 2: add the partials, store Y
        uint32_t p_rank[C::MAX_CLUSTER];
#pragma unroll
        for (int s = 0; s < C::MAX_CLUSTER; ++s)
          p_rank[s] = s < S ? map_to_cta(p_saddr, live ? (uint32_t)s : (uint32_t)rank) : 0u;
        for (int m0 = rank + S * ew; m0 < M; m0 += 2 * NW * S) {
          float4 part[2][C::MAX_CLUSTER];
#pragma unroll
          for (int j = 0; j < 2; ++j) {
            const int m = m0 + NW * S * j;
            if (m < M) {
              const uint32_t off = (uint32_t)((m * C::BF + 4 * lane) * 4);
#pragma unroll
              for (int s = 0; s < C::MAX_CLUSTER; ++s)
                if (s < S)
                  asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
                               : "=f"(part[j][s].x), "=f"(part[j][s].y), "=f"(part[j][s].z), "=f"(part[j][s].w)
                               : "r"(p_rank[s] + off));
            }
          }
#pragma unroll
          for (int j = 0; j < 2; ++j) {
            const int m = m0 + NW * S * j;
            if (m < M) {
              float4 y = make_float4(0.f, 0.f, 0.f, 0.f);  // rank order: the result does not depend on timing
#pragma unroll
              for (int s = 0; s < C::MAX_CLUSTER; ++s)
                if (s < S) { y.x += part[j][s].x; y.y += part[j][s].y; y.z += part[j][s].z; y.w += part[j][s].w; }
              if constexpr (FMT == FMT_NVFP4) { y.x *= alpha; y.y *= alpha; y.z *= alpha; y.w *= alpha; }
              if (live && n < N) {                         // N % 8 == 0: four features are inside or outside together
                if (y_is_bf16) {
                  __nv_bfloat162 h0 = __floats2bfloat162_rn(y.x, y.y), h1 = __floats2bfloat162_rn(y.z, y.w);
                  *reinterpret_cast<uint2*>(reinterpret_cast<__nv_bfloat16*>(Y) + (int64_t)m * N + n) =
                      make_uint2(*reinterpret_cast<uint32_t*>(&h0), *reinterpret_cast<uint32_t*>(&h1));
                } else {
                  *reinterpret_cast<float4*>(reinterpret_cast<float*>(Y) + (int64_t)m * N + n) = y;
                }
              }
            }
          }
        }
      }
    }
    tc_fence_before_sync();
  }
  if (S > 1) {
    if (PUSH) {
      if (warp < 2) cluster_wait();                      // the epilogue warps have waited above
    } else {
      if (warp < 2) { tc_fence_before_sync(); cluster_sync_all(); }        // as the epilogue warps in their pass 1
      cluster_arrive_relaxed();                          // every partial that this warp asked for has come: its sums are out
      cluster_wait();                                    // no CTA of the cluster reads this one's partial tile any more
    }
  }

  // ------------------------------------------------------------------ teardown
  __syncthreads();
  if (PUSH && S > 1 && *cta_abort) cluster_sync_all();   // others may still push to this CTA, see the few-token rotation
  if (warp == 1) {
    tc_fence_after_sync();
    tmem_dealloc(tmem_base, tmem_cols);
  }
}

}  // namespace torq
