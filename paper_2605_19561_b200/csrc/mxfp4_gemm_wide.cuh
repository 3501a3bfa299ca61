// Block-scaled GEMM on CTA pairs in ONE wave (17 tokens and more, the sizes that wide_gemm_width picks): every pair
// works exactly one tile of 256 tokens x `width` output features (a multiple of 64, up to 384), the width chosen so that the tiles just
// fill the pairs.  The pair kernel deals 256-column tiles and pays a whole wave for a remainder, or leaves pairs idle where there are
// few.
//
// As in the pair kernel each CTA stages its own 128 rows of A, its half of the tile's rows of W, its own A scales
// and the whole tile's W scales.  W scales come in chunks of 128 rows (four tensor-memory columns, rows 32 j ... 32 j +
// 31 in column j); the `nchk` chunks that a tile touches are loaded by one box and copied side by side, so that a
// tile which starts 64 rows into its first chunk reads from two columns further on.  A tile wider than 256
// columns is two instructions per K slice that share the A slice, the second always 128 columns.
//
// Nothing overlaps the epilogue here, so it runs on twelve warps and stages its rows in the operand stages, which are
// free by then: accumulator -> registers -> swizzled shared memory -> TMA store of [32 rows x 128 B] boxes.
//
// Roles per CTA: warp 0 TMA producer (one elected thread runs its loop), warp 1 MMA issuer (leader CTA; the whole warp runs the
// loop, an elected lane issues), warps 2..13 epilogue (lane quarter w % 4, three sets).
#pragma once
#include <cuda_bf16.h>
#include "mxfp4_gemm_pair.cuh"
#include "sm100_ptx.cuh"

namespace torq {

template <int FMT = FMT_MXFP4>
struct GemmWideCfg {
  static constexpr int BM = 128;                       // rows per CTA
  static constexpr int BK = GemmPairCfgT<FMT>::BK;     // elements of K per slab (128 bytes per row)
  static constexpr int CH = GemmPairCfgT<FMT>::CH;     // scale chunks per slab and 128 rows
  static constexpr int SF_BOXES = GemmPairCfgT<FMT>::SF_BOXES;
  static constexpr int SF_BOX_WORDS = GemmPairCfgT<FMT>::SF_BOX_WORDS;   // one or two chunks per box
  static constexpr int SF_BOX_BYTES = SF_BOX_WORDS * 4;
  static constexpr int A_BYTES = BM * 128;             // 16 KiB
  static constexpr int MAX_WIDTH = 384;
  static constexpr int AHEAD = 8;                      // slabs of W that the L2 is asked for beyond the stages
  static constexpr int MAX_STAGES = 8;
  static constexpr int ESETS = 3;
  static constexpr int THREADS = 64 + 128 * ESETS;
  static constexpr int OUT_BYTES = 32 * 128;           // one staged box
  static constexpr int SF_COL = MAX_WIDTH;             // A scales, then W scales; accumulator columns below
  __host__ __device__ static constexpr int n0(int width) { return width <= 256 ? width : width - 128; }
  // chunks of W scales a tile can touch: tiles start on multiples of `width`, i.e. 0 or 64 rows into a chunk
  __host__ __device__ static constexpr int chunks(int width) { return (width + (width % 128 ? 64 : 0) + 127) / 128; }
  __host__ __device__ static constexpr int slab_tx(int width) { return A_BYTES + width / 2 * 128 + SF_BOXES * SF_BOX_BYTES * (1 + chunks(width)); }
  __host__ __device__ static constexpr int slab_bytes(int width) { return (slab_tx(width) + 1023) / 1024 * 1024; }
  // K slabs of 128 bytes per stage of the kernel for widths up to `range`
  __host__ __device__ static constexpr int slabs(int range) { return range <= 128 ? 2 : 1; }
  // Two slabs halve the waits and barriers per K, which bound a step of up to 128 columns (us, one slab / two: 200 x 4096, K = 14336
  // 15.9 / 13.2, 300 x 4096, K = 4096 7.3 / 6.7, NVFP4 400 x 4096 8.4 / 7.7, 150 x 5120, K = 5120 7.8 / 6.9, 200 x 6144, K = 4096
  // 7.53 / 7.26), from four slabs on.  With few slabs the first stage is waited for longer (40 x 4096, K = 512 2.90 / 3.02), and so
  // it is with four or five where more than 24 pairs read up to 176 tokens and the last slab is a half one, in NVFP4 with more
  // tokens as well, or the pairs are up to 32 (144 x 4096, K = 1152 4.00 / 4.10, 80 x 2048 3.59 / 3.71, 80 x 4096, K = 1024 3.60 /
  // 3.72, NVFP4 192 x 6144, K = 1152 4.74 / 4.98; beyond the line 112 x 3072, K = 1280 3.77 / 3.70, MXINT4 144 x 6144, K = 640 4.22 /
  // 4.09).
  __host__ __device__ static constexpr bool two_slabs(int64_t M, int64_t K, int64_t pairs) {
    const int64_t k_slabs = (K + BK - 1) / BK;
    if (k_slabs < 4 || k_slabs > 5 || pairs <= 24) return k_slabs >= 4;
    if (K % BK != 0) return M > 176 && FMT != FMT_NVFP4;
    return M > 176 || pairs > 32 || (FMT == FMT_MXINT4 && k_slabs == 5);
  }
  __host__ __device__ static constexpr int range(int width, bool two) { return width > 256 ? 384 : (width > 128 || !two ? 256 : 128); }
  __host__ __device__ static constexpr int stage_bytes(int width, int range) { return slabs(range) * slab_bytes(width); }
  __host__ __device__ static constexpr int stages(int width, int range) {
    return (232448 - 2048) / stage_bytes(width, range) < MAX_STAGES ? (232448 - 2048) / stage_bytes(width, range) : MAX_STAGES;
  }
  __host__ __device__ static constexpr int smem_bytes(int width, int range) { return stages(width, range) * stage_bytes(width, range) + 256 + 1024; }
  static_assert(SF_COL + 4 * CH + 4 * CH * 3 <= 512 && chunks(MAX_WIDTH) <= 3 && chunks(MAX_WIDTH - 64) <= 3, "up to three chunks of W scales");
};

// grid = 2 * rows * cols CTAs in clusters of two: pair p works row tile p % rows (256 tokens), column tile p / rows.
// tmA: [128 x 128 B]; tmB: [n0 / 2 x 128 B]; tmB1: [64 x 128 B] (second instruction); tmSFA / tmSFB: boxes of 1 / nchk
// rows of the scale view; tmY as in the pair kernel.  RANGE: of the width and K (GemmWideCfg).
template <int FMT, int RANGE>
__global__ void __launch_bounds__(GemmWideCfg<FMT>::THREADS, 1)
mxfp4_gemm_wide_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                       const __grid_constant__ CUtensorMap tmB1, const __grid_constant__ CUtensorMap tmSFA,
                       const __grid_constant__ CUtensorMap tmSFB, const __grid_constant__ CUtensorMap tmY, int y_is_bf16,
                       int M, int N, int K, int rows, int width, float alpha, int* err_word) {
  using C = GemmWideCfg<FMT>;
  constexpr int CH = C::CH, SL = C::slabs(RANGE);
  constexpr bool TWO = RANGE > 256;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t* smem_gen = smem_raw + (smem_base - smem_u32(smem_raw));
  const int nst = C::stages(width, RANGE);
  const uint32_t stage_bytes = C::stage_bytes(width, RANGE);
  const uint32_t bar_off = nst * stage_bytes;
  const uint32_t bar_base = smem_base + bar_off;
  auto full_bar = [&](int s) { return bar_base + 8u * s; };
  auto empty_bar = [&](int s) { return bar_base + 8u * (C::MAX_STAGES + s); };
  const uint32_t accf_bar = bar_base + 8u * (2 * C::MAX_STAGES);
  volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(smem_gen + bar_off + 192);
  volatile int* cta_abort = reinterpret_cast<volatile int*>(smem_gen + bar_off + 200);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cluster_ctarank();
  const int pair = blockIdx.x >> 1;
  const int tcol = (pair / rows) * width;
  const int mt = 2 * (pair % rows) + (int)rank;
  const int k_slabs = (K + C::BK - 1) / C::BK, k_tiles = (k_slabs + SL - 1) / SL;   // slabs of K, stages of them (the last may hold one)
  const uint32_t slab_bytes = C::slab_bytes(width);
  const int n0 = C::n0(width), nchk = C::chunks(width);
  const uint32_t b_bytes = (uint32_t)width / 2 * 128;
  const uint32_t sfa_off = C::A_BYTES + b_bytes, sfb_off = sfa_off + C::SF_BOXES * C::SF_BOX_BYTES;

  if (threadIdx.x == 0) {
    for (int s = 0; s < nst; ++s) { mbar_init(full_bar(s), 1); mbar_init(empty_bar(s), 1); }
    mbar_init(accf_bar, 1);
    *cta_abort = 0;
    fence_mbar_init();
  }
  if (warp == 2 && elect_one()) {
    tma_prefetch_desc(&tmB); tma_prefetch_desc(&tmB1); tma_prefetch_desc(&tmSFB);
    tma_prefetch_desc(&tmA); tma_prefetch_desc(&tmSFA); tma_prefetch_desc(&tmY);
  }
  __syncwarp();
  if (warp == 1) { tmem_alloc_pair(smem_u32(const_cast<uint32_t*>(tmem_slot)), 512); tmem_relinquish_pair(); }
  tc_fence_before_sync();
  __syncthreads();
  cluster_sync_after_init();
  tc_fence_after_sync();
  const uint32_t tmem_base = *tmem_slot;
  // The weights and their scales are constants of the layer, never the output of the kernel that runs just before
  // this one: their loads for the first stages go out now, everything else waits for that kernel to complete.
  griddep_launch_dependents();
  const int pre = k_tiles < nst ? k_tiles : nst;

  auto load_a = [&](int s, int kt) {
    const uint32_t bar = map_to_cta(full_bar(s), 0);
    for (int k = kt * SL; k < (kt + 1) * SL && k < k_slabs; ++k) {
      const uint32_t st = smem_base + s * stage_bytes + (k - kt * SL) * slab_bytes;
      tma_load_2d_pair(st, &tmA, k * 128, mt * C::BM, bar);
      // anything outside the buffer arrives as zeros (scale 2^-127 or 0, on operand data that is zero as well)
#pragma unroll
      for (int b = 0; b < C::SF_BOXES; ++b)
        tma_load_2d_pair(st + sfa_off + b * C::SF_BOX_BYTES, &tmSFA, k * CH * 128 + b * C::SF_BOX_WORDS, mt, bar);
    }
  };

  if (warp == 0) {
    // ------------------------------------------------------------------ TMA producer (both CTAs)
    if (elect_one()) {
      const uint32_t leader_full0 = map_to_cta(full_bar(0), 0);
      auto load_w = [&](int s, int kt) {
        const uint32_t bar = leader_full0 + 8u * s;
        const int here = k_slabs - kt * SL < SL ? k_slabs - kt * SL : SL;
        if (rank == 0) mbar_arrive_expect_tx(full_bar(s), 2 * here * C::slab_tx(width));
        for (int i = 0; i < here; ++i) {
          const int k = kt * SL + i;
          const uint32_t st = smem_base + s * stage_bytes + i * slab_bytes;
          tma_load_2d_pair(st + C::A_BYTES, &tmB, k * 128, tcol + (int)rank * (n0 / 2), bar);
          if constexpr (TWO) tma_load_2d_pair(st + C::A_BYTES + n0 / 2 * 128, &tmB1, k * 128, tcol + n0 + (int)rank * 64, bar);
#pragma unroll
          for (int b = 0; b < C::SF_BOXES; ++b)
            tma_load_2d_pair(st + sfb_off + b * nchk * C::SF_BOX_BYTES, &tmSFB, k * CH * 128 + b * C::SF_BOX_WORDS, tcol >> 7, bar);
        }
      };
      for (int i = 0; i < pre; ++i) load_w(i, i);
      griddep_wait();
      int s = 0;                                       // warp 2 sends the A-side loads of the first stages
      uint32_t ph = 0;
      for (int kt = pre; kt < k_tiles; ++kt) {
        if (!mbar_wait_cluster(empty_bar(s), ph, cta_abort, err_word, SITE_PRODUCER_EMPTY)) break;
        load_w(s, kt);
        load_a(s, kt);
        if (++s == nst) { s = 0; ph ^= 1; }
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer (leader only)
    // The whole warp runs the loop and an elected lane issues.  As a loop of one lane, with a loop over the scale chunks inside,
    // issuing took longer than the instructions of a narrow tile: M = 512, N = 4096, K = 14336 23.4 -> 18.8 us, M = 200
    // 19.1 -> 17.0, M = 200, N = 6144, K = 4096 8.45 -> 7.75.
    if (rank == 0) {
      // instruction descriptors of the two widths differ only in the N field ([17,23) = N >> 3)
      const uint32_t less = (uint32_t)((256 - n0) >> 3) << 17;
      constexpr uint32_t less1 = (uint32_t)((256 - 128) >> 3) << 17;
      constexpr uint32_t full_a = FMT == FMT_NVFP4 ? idesc_nvf4(256, 256) : idesc_mxf4(256, 256, 0, 0);
      constexpr uint32_t full_b = FMT == FMT_NVFP4 ? idesc_nvf4(256, 256) : idesc_mxf4(256, 256, 2, 2);
      const uint32_t sfa_t = tmem_base + C::SF_COL, sfb_t = sfa_t + 4 * CH;
      const uint32_t sfb_c = 4u * nchk;                // columns per K chunk
      const uint32_t sfb_m = sfb_t + ((tcol & 127) ? 2u : 0u), sfb_m1 = sfb_m + (uint32_t)n0 / 32;
      const uint32_t acc1 = tmem_base + n0;
      int s = 0;
      uint32_t ph = 0;
      bool ok = true;
      for (int kt = 0; kt < k_tiles; ++kt) {
        ok = mbar_wait_cluster_warp<true>(full_bar(s), ph, cta_abort, err_word, SITE_MMA_FULL);
        if (!ok) break;
        tc_fence_after_sync();
        if (elect_one()) {
#pragma unroll
          for (int i = 0; i < SL; ++i) {
            const int k = kt * SL + i;
            if (SL > 1 && k >= k_slabs) break;
            const bool two = FMT == FMT_MXINT4 || K - k * C::BK > C::BK / 2;       // K % 256 == 128: the last slab is half
            const uint32_t st = smem_base + s * stage_bytes + i * slab_bytes;
            const uint64_t adesc = make_desc(st, 16, 1024, kSwizzle128);
            const uint64_t bdesc = make_desc(st + C::A_BYTES, 16, 1024, kSwizzle128);
            const uint64_t b1desc = make_desc(st + C::A_BYTES + n0 / 2 * 128, 16, 1024, kSwizzle128);
            const uint64_t sfa_d = make_desc(st + sfa_off, 0, 128, 0);
            const uint64_t sfb_d = make_desc(st + sfb_off, 0, 128, 0);
            // scale chunks shared -> tensor memory (descriptor address unit = 16 B)
#pragma unroll
            for (int c = 0; c < CH; ++c) {
              if (CH == 1 || c < CH / 2 || two) {
                tmem_cp_32x128b_warpx4_pair(sfa_t + 4 * c, sfa_d + 32 * c);
#pragma unroll
                for (int t = 0; t < 3; ++t)
                  if (t < nchk)
                    tmem_cp_32x128b_warpx4_pair(sfb_t + c * sfb_c + 4 * t,
                                                sfb_d + ((c >> 1) * nchk + t) * (C::SF_BOX_BYTES / 16) + 32 * (c & 1));
              }
            }
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              if (j < 2 || two) {
                const uint32_t accumulate = (k | j) != 0;
                if constexpr (FMT == FMT_MXINT4) {         // a quarter chunk (one scale byte) per instruction
                  mma_mxf8_pair(tmem_base, adesc + 2 * j, bdesc + 2 * j, idesc_mxf8(256, 256, j) - less, sfa_t, sfb_m, accumulate);
                  if constexpr (TWO)
                    mma_mxf8_pair(acc1, adesc + 2 * j, b1desc + 2 * j, idesc_mxf8(256, 256, j) - less1, sfa_t, sfb_m1, accumulate);
                } else if constexpr (FMT == FMT_NVFP4) {   // one chunk per instruction
                  mma_nvf4_pair(tmem_base, adesc + 2 * j, bdesc + 2 * j, full_a - less, sfa_t + 4 * j, sfb_m + j * sfb_c, accumulate);
                  if constexpr (TWO)
                    mma_nvf4_pair(acc1, adesc + 2 * j, b1desc + 2 * j, full_a - less1, sfa_t + 4 * j, sfb_m1 + j * sfb_c, accumulate);
                } else {                                   // half a chunk (two scale bytes) per instruction
                  const uint32_t id = (j & 1) ? full_b : full_a;
                  mma_mxf4_pair(tmem_base, adesc + 2 * j, bdesc + 2 * j, id - less, sfa_t + 4 * (j >> 1), sfb_m + (j >> 1) * sfb_c, accumulate);
                  if constexpr (TWO)
                    mma_mxf4_pair(acc1, adesc + 2 * j, b1desc + 2 * j, id - less1, sfa_t + 4 * (j >> 1), sfb_m1 + (j >> 1) * sfb_c, accumulate);
                }
              }
            }
          }
          tc_commit_pair(empty_bar(s), 3);
        }
        __syncwarp();
        if (++s == nst) { s = 0; ph ^= 1; }
      }
      if (ok && elect_one()) tc_commit_pair(accf_bar, 3);
    }
    __syncwarp();
  } else {
    // ------------------------------------------------------------------ epilogue (12 warps per CTA)
    const int q = warp & 3;
    const int set = (warp - 2) >> 2;
    // Up to 256 tokens HBM idles until the kernel before has completed: the L2 is asked for the next W (us, without / with, layers: 200 x
    // 4096 -> 6144 21.5 / 21.2, 256 x 5120 -> 5120 27.9 / 27.5, 256 x 4096 -> 14336 25.9 / 25.8; with more row tiles 400 x 4096 -> 4096
    // 25.8 / 26.1).
    const int wrow = tcol + (int)rank * (n0 / 2);      // of W; a last tile narrower than half a tile has none for the second CTA
    if (warp == 3 && rows == 1 && wrow < N && elect_one())
      for (int k = pre * SL; k < min(k_slabs, pre * SL + C::AHEAD); ++k) tma_prefetch_l2_2d(&tmB, k * 128, wrow);
    __syncwarp();
    griddep_wait();                                    // Y may still be read by that kernel
    if (warp == 2) {                                   // from a warp of its own: not behind the W loads of all these stages
      if (elect_one())
        for (int i = 0; i < pre; ++i) load_a(i, i);
      __syncwarp();
    }
    bool ok = mbar_wait_cluster(accf_bar, 0, cta_abort, err_word, SITE_EPI_ACC_FULL);
    ok = __all_sync(0xFFFFFFFFu, ok);
    const int row0 = mt * C::BM + q * 32;
    if (ok && row0 < M) {
      tc_fence_after_sync();
      const uint32_t tacc = tmem_base + ((uint32_t)(q * 32) << 16);
      // two staging buffers per warp in the operand stages (every load has landed and been consumed)
      const uint32_t buf0 = smem_base + (uint32_t)(warp - 2) * 2 * C::OUT_BYTES;
      const uint32_t sw = (uint32_t)(lane & 7);
      auto pack2 = [](uint32_t lo, uint32_t hi) {
        __nv_bfloat162 hh = __floats2bfloat162_rn(__uint_as_float(lo), __uint_as_float(hi));
        return *reinterpret_cast<uint32_t*>(&hh);
      };
      const int unit = y_is_bf16 ? 64 : 32;            // columns of one 128-byte box
      int n = 0;
#pragma unroll 1
      for (int c = set * unit; c < width && tcol + c < N; c += C::ESETS * unit, ++n) {
        const uint32_t buf = buf0 + (n & 1) * C::OUT_BYTES;
        const uint32_t my_row = buf + lane * 128;
        if (lane == 0) bulk_wait_group_read<1>();      // the store before last has read this buffer
        __syncwarp();
#pragma unroll
        for (int half = 0; half < 2; ++half) {
          if (half == 1 && !y_is_bf16) break;
          uint32_t v[32];
          tmem_ld_32x32(tacc + c + 32 * half, v);
          tmem_ld_wait();
          if constexpr (FMT == FMT_NVFP4) {            // product of the two tensor scales
#pragma unroll
            for (int j = 0; j < 32; ++j) v[j] = __float_as_uint(__uint_as_float(v[j]) * alpha);
          }
          auto put16 = [&](int piece, uint32_t a, uint32_t b, uint32_t cc, uint32_t d) {
            asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};"
                         ::"r"(my_row + (((uint32_t)piece ^ sw) << 4)), "r"(a), "r"(b), "r"(cc), "r"(d) : "memory");
          };
          if (y_is_bf16) {
#pragma unroll
            for (int p = 0; p < 4; ++p)
              put16(4 * half + p, pack2(v[8 * p], v[8 * p + 1]), pack2(v[8 * p + 2], v[8 * p + 3]),
                    pack2(v[8 * p + 4], v[8 * p + 5]), pack2(v[8 * p + 6], v[8 * p + 7]));
          } else {
#pragma unroll
            for (int p = 0; p < 8; ++p) put16(p, v[4 * p], v[4 * p + 1], v[4 * p + 2], v[4 * p + 3]);
          }
        }
        fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) {                               // the store clips rows >= M and columns >= N by itself
          tma_store_2d(&tmY, tcol + c, row0, buf);
          bulk_commit_group();
        }
      }
      tc_fence_before_sync();
    }
    if (lane == 0) bulk_wait_group_read<0>();          // shared memory must outlive the stores' reads
  }

  // ------------------------------------------------------------------ teardown
  tc_fence_before_sync();
  __syncthreads();
  if (*cta_abort) {
    for (int i = 0; i < 2000; ++i) __nanosleep(1000);
  }
  cluster_arrive_relaxed();                            // the peer no longer touches this CTA's memory; no data to order
  cluster_wait();
  if (warp == 1) {
    tc_fence_after_sync();
    tmem_dealloc_pair(tmem_base, 512);
  }
}

}  // namespace torq
