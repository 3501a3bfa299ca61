// Rotate + quantize for M > 128 on CTA pairs: the same computation and epilogue as
// rotate_quantize_kernel, but two CTAs (a cluster of 2, one per SM) share one 256 x 256 output
// tile through tcgen05.mma cta_group::2.  Each CTA stages only its own 128 rows of X and its own
// 128 columns of R_inter per K step: 32 KiB per 128 x 256 x 64 of work where the single-CTA kernel
// stages 48, with which it cannot feed the tensor pipe from L2.  Here the loop of loads and
// instructions of a 256 x 256 tile by itself runs at 512 cycles per K step, the instructions' own rate (the
// loads alone take 400, at 22 TB/s): what a long call waits for is the power cap.  Every CTA loads only
// for itself; operand sharing happens inside the MMA, which reads both CTAs' shared memory.
//
// Tiles are dealt round robin from the list MixedTiles describes: 256 x 256 tiles, and where those
// would leave the last wave partly empty, 256 x 192 tiles in its place (N = 192 instructions, 96
// columns of R_inter per CTA, three 32-blocks per epilogue warp instead of four).
//
// Roles per CTA: warp 0 TMA producer (both CTAs), warp 1 MMA issuer (leader CTA only; both
// allocate tensor memory), warps 2..9 epilogue (each CTA drains its own 128 x 256 accumulator).
// Barriers: full[s] lives in the leader and counts the bytes of both CTAs' loads; empty[s] and
// acc_full[a] are local to each CTA and are signalled by the leader's tcgen05.commit to both;
// acc_empty[a] lives in the leader and takes one arrival per epilogue warp of both CTAs (16).
#pragma once
#include <cuda_bf16.h>
#include "l2_requests.cuh"
#include "nvfp4_quantize.cuh"
#include "mxint4_quantize.cuh"
#include "pair_handshake.cuh"
#include "sm100_ptx.cuh"

namespace torq {

struct RotPairCfg {
  static constexpr int BN = 256;                       // tile columns (both CTAs see all of them)
  static constexpr int BM = 128;                       // rows per CTA (256 per pair)
  static constexpr int BK = 64;
  static constexpr int A_BYTES = BM * BK * 2;          // 16 KiB
  static constexpr int B_BOX_BYTES = 64 * BK * 2;      // 64(n) x 64(k) bf16 = 8 KiB
  static constexpr int B_BYTES = (BN / 2 / 64) * B_BOX_BYTES;   // this CTA's 128 columns = 16 KiB
  static constexpr int STAGE_BYTES = A_BYTES + B_BYTES;         // 32 KiB
  static constexpr int STAGES = 6;
  static constexpr int RI_BLOCK_BYTES = 32 * 64;       // bf16, 64-byte swizzle: the last tile
  static constexpr int RI_BYTES = (BN / 32) * 32 * 32 * 4;     // the tile's R_intra blocks: fp32, or bf16
  static constexpr int SMEM_BYTES = STAGES * STAGE_BYTES + RI_BYTES + 256 + 1024;
  static constexpr int NACC = 2;
  static constexpr int TMEM_COLS = 512;
  static constexpr int THREADS = 320;               // producer, MMA issuer, 8 epilogue warps
  static_assert(SMEM_BYTES <= 232448, "shared memory budget");
};

// FMT_NVFP4: the same kernel with the NVFP4 quantizer in the epilogue (two 16-element blocks per
// 32 columns, E4M3 scales, `tensor_scale` the tensor's float32 scale; unused for MXFP4).  R_intra
// is still [d/32, 32, 32]; 16-wide rotations arrive as its block-diagonal form.
// FMT_MXINT4: integer codes written as one E4M3 operand byte per element (`codes` is [M, d] bytes),
// the scale bytes as for MXFP4.
// FMT_F32OUT: no quantizer; `codes` is a float32 [M, d] array that receives Z itself (`scales` unused).
// `x_terms` > 1: X is the sum of that many bfloat16 matrices stored side by side, tmX = [M, x_terms * d]
// (an fp32 matrix split exactly into three bf16 terms); the contraction then runs over all of them
// against the same R_inter, i.e. Z = (X_0 + X_1 + ...) R_inter in one fp32 accumulation.  d % 64 == 0 then.
template <int FMT = FMT_MXFP4>
__global__ void __launch_bounds__(320, 1)
rotate_quantize_pair_kernel(const __grid_constant__ CUtensorMap tmX, const __grid_constant__ CUtensorMap tmR,
                            const __grid_constant__ CUtensorMap tmRn, const __nv_bfloat16* __restrict__ R_intra, uint8_t* __restrict__ codes,
                            uint8_t* __restrict__ scales, int M, int d, float tensor_scale, int x_terms,
                            const MixedTiles tiles, int* err_word) {
  using C = RotPairCfg;
  constexpr int BN = C::BN;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t* smem_gen = smem_raw + (smem_base - smem_u32(smem_raw));
  uint8_t* ri_smem = smem_gen + C::STAGES * C::STAGE_BYTES;
  const uint32_t bar_off = C::STAGES * C::STAGE_BYTES + C::RI_BYTES;
  const uint32_t bar_base = smem_base + bar_off;
  auto full_bar = [&](int s) { return bar_base + 8u * s; };
  auto empty_bar = [&](int s) { return bar_base + 8u * (C::STAGES + s); };
  auto accf_bar = [&](int a) { return bar_base + 8u * (2 * C::STAGES + a); };
  auto acce_bar = [&](int a) { return bar_base + 8u * (2 * C::STAGES + C::NACC + a); };
  const uint32_t alloc_bar = bar_base + 8u * (2 * C::STAGES + 2 * C::NACC);   // in the leader: the other CTA's tensor memory is allocated
  // last tile, per column half: in the leader, both CTAs' split terms of a block; the rotated block
  auto term_bar = [&](int h) { return alloc_bar + 8u + 8u * h; };
  auto rot_bar = [&](int h) { return alloc_bar + 24u + 8u * h; };
  const uint32_t ri_bar = alloc_bar + 40;              // in the leader: the last tile's R_intra is in both CTAs' shared memory
  volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(smem_gen + bar_off + 192);
  volatile int* cta_abort = reinterpret_cast<volatile int*>(smem_gen + bar_off + 200);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cluster_ctarank();             // 0 = leader
  const int pair = blockIdx.x >> 1, npairs = gridDim.x >> 1;
  const int m_tiles = (M + 127) / 128;                 // 128-row tiles that exist
  const int total_tiles = tiles.total;                 // 256-row pair tiles, 256 or 192 columns wide
  const int kr_tiles = (d + C::BK - 1) / C::BK;         // K steps over R_inter; X has x_terms times as many
  const int k_tiles = kr_tiles * x_terms;
  const int nblocks = d / 32;
  const int kb4 = (nblocks + 3) / 4;

  // Set-up.  The producer waits for nothing but the barriers of both CTAs, whose cluster barrier therefore comes before the
  // tensor-memory allocation; the other warps meet behind both on a barrier that the producer only counts itself on.  A CTA whose
  // SM the kernel before leaves last sets the time here: device timestamps, 2048 x 4096, from that kernel's completion to
  // the last pair's first full stage 3.6 us, 2.3 with this set-up and the first X loads from a warp of their own (the layer
  // with N = 6144, where rotation and GEMM have it, 86.1 -> 85.2 us, at the power cap, loops of 0.7 s on each side in turn).
  if (threadIdx.x == 0) {
    for (int s = 0; s < C::STAGES; ++s) { mbar_init(full_bar(s), 1); mbar_init(empty_bar(s), 1); }
    for (int a = 0; a < C::NACC; ++a) { mbar_init(accf_bar(a), 1); mbar_init(acce_bar(a), 16); }
    mbar_init(alloc_bar, 1);
    for (int h = 0; h < 2; ++h) { mbar_init(term_bar(h), 8); mbar_init(rot_bar(h), 1); }
    mbar_init(ri_bar, 2);
    *cta_abort = 0;
    fence_mbar_init();
  }
  if (warp == 2 && elect_one()) { tma_prefetch_desc(&tmX); tma_prefetch_desc(&tmR); tma_prefetch_desc(&tmRn); }
  __syncwarp();
  cluster_arrive_relaxed();
  int mp0, tcol0;                                      // this pair's first tile
  bool narrow0;
  mixed_tile_coords(pair, tiles, mp0, tcol0, narrow0);
  const int pre = k_tiles < C::STAGES ? k_tiles : C::STAGES;
  uint32_t tmem_base = 0;
  if (warp == 0) {
    named_barrier_arrive(2, C::THREADS);
    cluster_wait();                                    // both CTAs' barriers exist before any remote arrive
  } else {
    if (warp == 1) { tmem_alloc_pair(smem_u32(const_cast<uint32_t*>(tmem_slot)), C::TMEM_COLS); tmem_relinquish_pair(); }
    tc_fence_before_sync();
    named_barrier_sync(2, C::THREADS);
    cluster_wait();
    tc_fence_after_sync();
    tmem_base = *tmem_slot;
    if (warp == 1 && rank == 1 && lane == 0) mbar_arrive_cluster(map_to_cta(alloc_bar, 0));   // this CTA's tensor memory is there
  }
  // Set-up above touched no global memory; from here on the previous kernel's results are needed.
  // R_inter is a constant of the layer, never the output of the kernel that runs just before this
  // one: the producer starts the first stages' R_inter loads right away; the X loads and all
  // other global accesses wait until that kernel has completed.
  griddep_launch_dependents();

  if (warp == 0) {
    // ------------------------------------------------------------------ TMA producer (both CTAs)
    // A 192-column tile takes 96 columns of R_inter per CTA: one 64-column box and one 32-column box.
    // Under the 128-byte swizzle a box whose rows are 64 bytes long still lands on a 128-byte pitch, i.e.
    // as the first half of the 64-column layout the instruction's descriptor describes.
    auto load_r = [&](int s, int kr, int my_col, bool narrow) {
      const uint32_t st = smem_base + s * C::STAGE_BYTES;
      const uint32_t leader_full = map_to_cta(full_bar(s), 0);
      if (rank == 0) mbar_arrive_expect_tx(full_bar(s), 2 * (C::STAGE_BYTES - (narrow ? C::B_BOX_BYTES / 2 : 0)));
      tma_load_2d_pair(st + C::A_BYTES, &tmR, my_col, kr * C::BK, leader_full);
      tma_load_2d_pair(st + C::A_BYTES + C::B_BOX_BYTES, narrow ? &tmRn : &tmR, my_col + 64, kr * C::BK, leader_full);
    };
    if (elect_one()) {
      const int my_col = tcol0 + (int)rank * (narrow0 ? kNarrowCols / 2 : BN / 2);
      for (int kt = 0; kt < pre; ++kt) load_r(kt, kt % kr_tiles, my_col, narrow0);
    }
    __syncwarp();
    griddep_wait();
    uint32_t it = pre;                                 // warp 2 sends the X loads of the first stages
    bool ok = true;
    int mp = mp0, tcol = tcol0, kt = pre, kr = pre % kr_tiles;
    bool narrow = narrow0;
    for (int tile = pair; tile < total_tiles && ok; tile += npairs) {
      if (tile != pair) { mixed_tile_coords(tile, tiles, mp, tcol, narrow); kt = 0; kr = 0; }
      const int mt = 2 * mp + (int)rank;
      const int my_col = tcol + (int)rank * (narrow ? kNarrowCols / 2 : BN / 2);
      for (; kt < k_tiles; ++kt, ++it, kr = (kr + 1 == kr_tiles ? 0 : kr + 1)) {
        const int s = it % C::STAGES;
        if (!mbar_wait_cluster_warp(empty_bar(s), ((it / C::STAGES) & 1) ^ 1, cta_abort, err_word,
                               SITE_PRODUCER_EMPTY)) { ok = false; break; }
        if (elect_one()) {
          load_r(s, kr, my_col, narrow);
          tma_load_2d_pair(smem_base + s * C::STAGE_BYTES, &tmX, kt * C::BK, mt * C::BM, map_to_cta(full_bar(s), 0));
        }
        __syncwarp();
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer (leader only)
    if (rank == 0) {
      constexpr uint32_t idesc_wide = idesc_bf16(256, BN, /*A MN-major*/ false, /*B MN-major*/ true);
      constexpr uint32_t idesc_narrow = idesc_bf16(256, kNarrowCols, false, true);
      uint32_t it = 0, tcount = 0;
      bool ok = mbar_wait_cluster_warp<true>(alloc_bar, 0, cta_abort, err_word, SITE_PEER_TMEM);
      for (int tile = pair; tile < total_tiles && ok; tile += npairs, ++tcount) {
        int mp, tcol;
        bool narrow;
        mixed_tile_coords(tile, tiles, mp, tcol, narrow);
        (void)mp; (void)tcol;
        const uint32_t idesc = narrow ? idesc_narrow : idesc_wide;
        const int a = tcount % C::NACC;
        if (!mbar_wait_cluster_warp(acce_bar(a), ((tcount / C::NACC) & 1) ^ 1, cta_abort, err_word,
                               SITE_MMA_ACC_EMPTY)) { ok = false; break; }
        tc_fence_after_sync();
        const uint32_t acc = tmem_base + a * BN;
        for (int kt = 0; kt < k_tiles; ++kt, ++it) {
          const int s = it % C::STAGES;
          if (!mbar_wait_cluster_warp<true>(full_bar(s), (it / C::STAGES) & 1, cta_abort, err_word, SITE_MMA_FULL)) {
            ok = false; break;
          }
          tc_fence_after_sync();
          const uint32_t st = smem_base + s * C::STAGE_BYTES;
          const uint64_t adesc = make_desc(st, 16, 1024, kSwizzle128);
          const uint64_t bdesc = make_desc(st + C::A_BYTES, C::B_BOX_BYTES, 1024, kSwizzle128);
          if (elect_one()) {
#pragma unroll
            for (int j = 0; j < C::BK / 16; ++j)
              mma_bf16_pair(acc, adesc + 2 * j, bdesc + 128 * j, idesc, (kt | j) != 0);
            tc_commit_pair(empty_bar(s), 3);             // stage free in both CTAs
          }
          __syncwarp();
        }
        if (ok && elect_one()) tc_commit_pair(accf_bar(a), 3);   // accumulator ready in both CTAs
        __syncwarp();
        if (FMT != FMT_F32OUT && R_intra != nullptr && ok && tile + npairs >= total_tiles) {
          // Intra-block rotation of the pair's last tile: three split terms x 32 of K per block, terms and result in tensor memory.
          constexpr uint32_t idesc_r = idesc_bf16(256, 32, false, true);
          const int nbb = narrow ? 3 : 4;
          ok = mbar_wait_cluster_warp<true>(ri_bar, 0, cta_abort, err_word, SITE_MMA_FULL);
          for (int i = 0; i < 2 * nbb && ok; ++i) {
            const int h = i & 1, bb = i >> 1;
            if (!mbar_wait_cluster_warp<true>(term_bar(h), bb & 1, cta_abort, err_word, SITE_MMA_FULL)) { ok = false; break; }
            tc_fence_after_sync();
            const uint64_t rdesc = make_desc(smem_u32(ri_smem) + (uint32_t)(h * nbb + bb) * C::RI_BLOCK_BYTES, 2048, 512, kSwizzle64);
            const uint32_t y = acc + (h * nbb + bb) * 32, out = tmem_base + (a ^ 1) * BN + h * 128, lo = out + 32;
            if (elect_one()) {
              mma_bf16_pair_tmem_a(out, lo, rdesc, idesc_r, 0);            // the smallest term first
              mma_bf16_pair_tmem_a(out, lo + 8, rdesc + 64, idesc_r, 1);   // k 16 .. 31: +8 columns of terms, +16 rows of R_intra
              mma_bf16_pair_tmem_a(out, y + 16, rdesc, idesc_r, 1);
              mma_bf16_pair_tmem_a(out, y + 24, rdesc + 64, idesc_r, 1);
              mma_bf16_pair_tmem_a(out, y, rdesc, idesc_r, 1);
              mma_bf16_pair_tmem_a(out, y + 8, rdesc + 64, idesc_r, 1);
              tc_commit_pair(rot_bar(h), 3);
            }
            __syncwarp();
          }
        }
      }
    }
  } else {
    if (warp == 3 && elect_one()) {
      // Until the kernel before has completed HBM idles: the L2 is asked for the first K steps of X, each pair of a row tile for one
      // (us, without / with: layer 1500 x 2048 -> 2048 21.2 / 20.9, 2048 x 4096 -> 6144 81.1 / 80.7).  The step by the tile's column: by
      // the pair's number, the pairs of the second eight row tiles asked for later ones (8192 x 1024 -> 1024 32.9 / 32.6).
      const int kt = x_step_of_tile(tcol0, narrow0);
      const int row = (2 * mp0 + (int)rank) * C::BM;     // the pair's second row tile may not exist
      if (kt < k_tiles && row < M) tma_prefetch_l2_2d(&tmX, kt * C::BK, row);
    }
    __syncwarp();
    griddep_wait();
    if (warp == 2) {
      // The X loads of the first stages: from a warp of its own, so that they go out when the kernel before has completed and
      // not behind the R_inter loads of all these stages (a CTA that finds its SM late is not through with those by then).
      if (elect_one())
        for (int kt = 0; kt < pre; ++kt)
          tma_load_2d_pair(smem_base + kt * C::STAGE_BYTES, &tmX, kt * C::BK, (2 * mp0 + (int)rank) * C::BM, map_to_cta(full_bar(kt), 0));
      __syncwarp();
    }
    // ------------------------------------------------------------------ epilogue (8 warps per CTA)
    // warp w reads lane quarter w % 4 (32 rows) and column half (w - 2) / 4 (four 32-blocks = one
    // 4-byte group of scale bytes; three blocks in a 192-column tile).  Two forms of the intra-block rotation:
    //  * fp32 FMAs, one row per thread, R_intra broadcast from shared memory as fp32.  Bound by
    //    that broadcast (8 bytes per lane and cycle): about 3/4 of a mainloop per tile, which does
    //    not matter while the next tile's mainloop runs beside it on the tensor pipe.
    //  * tcgen05 instructions of both CTAs on three split bf16 terms of y in tensor memory (every product exact, fp32
    //    accumulation), for the CTA's LAST tile, whose epilogue nothing overlaps and beside which half the tensor memory is free.  (As
    //    warp-level MMAs on accumulator fragments that epilogue was bound by those: us, loops of 0.4 s, before / now, rotation
    //    2048 x 4096 59.7 / 58.25, 1900 x 4096 NVFP4 60.0 / 58.6, 8192 x 1024 26.6 / 25.8; shorter loops 58.05 / 56.3, 59.6 / 55.7 and
    //    26.5 / 25.3.)
    const int q = warp & 3;
    const int h = (warp - 2) >> 2;
    const int et = (warp - 2) * 32 + lane;               // 0..255 among the epilogue threads
    const uint32_t ri_saddr = smem_u32(ri_smem);
    uint32_t tcount = 0;
    bool ok = true;
    for (int tile = pair; tile < total_tiles; tile += npairs, ++tcount) {
      int mp, tcol;
      bool narrow;
      mixed_tile_coords(tile, tiles, mp, tcol, narrow);
      const int mt = 2 * mp + (int)rank;
      const int a = tcount % C::NACC;
      const int b0 = tcol >> 5;                          // first 32-block of the tile: even, 2 mod 4 for some narrow tiles
      const int nbb = narrow ? 3 : 4;                    // this warp's blocks: half of the tile's 8 or 6
      const bool last = FMT != FMT_F32OUT && tile + npairs >= total_tiles;
      if (R_intra != nullptr) {
        // Executed by every epilogue thread for every tile, also after a wait has given up.
        named_barrier_sync(1, 256);
        for (int idx = et * 8; ok && idx < (BN / 32) * 1024; idx += 256 * 8) {
          const int lb = idx >> 10, blk = b0 + lb;
          if (last) {                                    // bf16, 16-byte piece c of row i at c ^ ((i >> 1) & 3); rank 1: two pieces on
            const int i = (idx & 1023) >> 5, c = ((idx & 31) >> 3) ^ (2 * (int)rank);
            uint4 v = make_uint4(0u, 0u, 0u, 0u);
            if (blk < nblocks) v = __ldg(reinterpret_cast<const uint4*>(R_intra + (size_t)blk * 1024 + (idx & 1023)));
            *reinterpret_cast<uint4*>(ri_smem + lb * C::RI_BLOCK_BYTES + i * 64 + ((c ^ ((i >> 1) & 3)) << 4)) = v;
          } else {                                       // fp32, dense
            float v[8];
            if (blk < nblocks) load8(R_intra + (size_t)blk * 1024 + (idx & 1023), v);
            else {
#pragma unroll
              for (int i = 0; i < 8; ++i) v[i] = 0.f;
            }
            float* dst = reinterpret_cast<float*>(ri_smem) + idx;
            *reinterpret_cast<float4*>(dst) = make_float4(v[0], v[1], v[2], v[3]);
            *reinterpret_cast<float4*>(dst + 4) = make_float4(v[4], v[5], v[6], v[7]);
          }
        }
        if (last) fence_proxy_async_smem();              // visible to the tensor core's reads
        named_barrier_sync(1, 256);
        if (last && et == 0) mbar_arrive_release_cluster(map_to_cta(ri_bar, 0));
      }
      if (ok) ok = mbar_wait_cluster(accf_bar(a), (tcount / C::NACC) & 1, cta_abort, err_word, SITE_EPI_ACC_FULL);
      ok = __all_sync(0xFFFFFFFFu, ok);
      if (!ok) continue;
      tc_fence_after_sync();
      const uint32_t tacc = tmem_base + ((uint32_t)(q * 32) << 16) + a * BN + h * nbb * 32;
      // Scale bytes: block blk of row r sits in byte blk % 4 of the 4-byte cell of (r, blk / 4).  The four
      // bytes of a wide tile's half are one cell; the three of a narrow tile's half go out one by one.
      const int fb = b0 + h * nbb;
      auto put_scales = [&](uint32_t w, size_t in_tile) {  // byte bb of w = scale of block fb + bb
        if (nbb == 4) {
          if ((fb >> 2) < kb4) *reinterpret_cast<uint32_t*>(scales + ((size_t)mt * kb4 + (fb >> 2)) * 512 + in_tile) = w;
        } else {
          for (int j = 0; j < nbb; ++j) {
            const int blk = fb + j;
            if ((blk >> 2) < kb4) scales[((size_t)mt * kb4 + (blk >> 2)) * 512 + in_tile + (blk & 3)] = (uint8_t)(w >> (8 * j));
          }
        }
      };
      // NVFP4: two bytes per block, cells of two blocks
      auto put_scales16 = [&](uint32_t w01, uint32_t w23, size_t in_tile, int kb4n) {
        if (nbb == 4) {
          if ((fb >> 1) < kb4n) *reinterpret_cast<uint32_t*>(scales + ((size_t)mt * kb4n + (fb >> 1)) * 512 + in_tile) = w01;
          if ((fb >> 1) + 1 < kb4n)
            *reinterpret_cast<uint32_t*>(scales + ((size_t)mt * kb4n + (fb >> 1) + 1) * 512 + in_tile) = w23;
        } else {
          for (int j = 0; j < nbb; ++j) {
            const int blk = fb + j;
            if ((blk >> 1) < kb4n)
              *reinterpret_cast<uint16_t*>(scales + ((size_t)mt * kb4n + (blk >> 1)) * 512 + in_tile + 2 * (blk & 1)) =
                  (uint16_t)((j < 2 ? w01 : w23) >> (16 * (j & 1)));
          }
        }
      };
      {
        // ---- one row per thread
        const int64_t row = (int64_t)mt * C::BM + q * 32 + lane;
        uint32_t sc_word = 0, sc_word2 = 0;              // NVFP4: two groups of four 16-blocks
        NvScale nvs = {};
        if constexpr (FMT == FMT_NVFP4) nvs = nv_scale(tensor_scale);
#pragma unroll 1
        for (int bb = 0; bb < nbb; ++bb) {
          uint32_t yv[32];
          tmem_ld_32x32(tacc + bb * 32, yv);
          tmem_ld_wait();
          if (bb == nbb - 1) {                           // this warp's share is read: tell the leader if it waits for that
            tc_fence_before_sync();
            __syncwarp();
            if (lane == 0 && accumulator_is_waited_for(tile, npairs, C::NACC, total_tiles))
              mbar_arrive_cluster(map_to_cta(acce_bar(a), 0));
          }
          float z[32];
          if (FMT != FMT_F32OUT && last && R_intra != nullptr) {
            // y goes back to tensor memory as hi + mid + lo (bf16, exact): hi and mid over y, lo where the other accumulator's columns of
            // this half were, which these warps have read; the result comes beside it.
            const uint32_t other = tmem_base + ((uint32_t)(q * 32) << 16) + (a ^ 1) * BN + h * 128;
            uint32_t hi[16], mid[16], lo[16];
#pragma unroll
            for (int e = 0; e < 16; ++e) split3_trunc_bf16x2(yv[2 * e], yv[2 * e + 1], hi[e], mid[e], lo[e]);
            tmem_st_32x32_x16(tacc + bb * 32, hi);
            tmem_st_32x32_x16(tacc + bb * 32 + 16, mid);
            tmem_st_32x32_x16(other + 32, lo);
            tmem_st_wait();
            tc_fence_before_sync();
            __syncwarp();
            if (lane == 0) mbar_arrive_cluster(map_to_cta(term_bar(h), 0));
            ok = __all_sync(0xFFFFFFFFu, mbar_wait_cluster(rot_bar(h), bb & 1, cta_abort, err_word, SITE_EPI_ACC_FULL));
            if (!ok) break;
            tc_fence_after_sync();
            tmem_ld_32x32(other, yv);
            tmem_ld_wait();
            tc_fence_before_sync();
#pragma unroll
            for (int j = 0; j < 32; ++j) z[j] = __uint_as_float(yv[j]);
          } else if (R_intra != nullptr) {
            intra_rotate32(yv, ri_saddr + (uint32_t)(h * nbb + bb) * 4096, z);
          } else {
#pragma unroll
            for (int j = 0; j < 32; ++j) z[j] = __uint_as_float(yv[j]);
          }
          const int blk = fb + bb;
          if constexpr (FMT == FMT_F32OUT) {               // the rotated values themselves
            if (row < M && blk < nblocks) {
              float4* dst = reinterpret_cast<float4*>(reinterpret_cast<float*>(codes) + row * (int64_t)d + (int64_t)blk * 32);
#pragma unroll
              for (int j = 0; j < 8; ++j) dst[j] = make_float4(z[4 * j], z[4 * j + 1], z[4 * j + 2], z[4 * j + 3]);
            }
            continue;
          }
          uint4 cw;
          uint32_t sbyte;
          if constexpr (FMT == FMT_MXINT4) {               // one operand byte per element
            uint4 cw2;
            mxint4_quantize_block32(z, cw, cw2, sbyte);
            if (row < M && blk < nblocks) {
              uint4* dst = reinterpret_cast<uint4*>(codes + row * (int64_t)d + (int64_t)blk * 32);
              dst[0] = cw;
              dst[1] = cw2;
            }
          } else {
            if constexpr (FMT == FMT_NVFP4) nv_quantize_2x16(z, nvs, cw, sbyte);
            else quantize_block32(z, cw, sbyte);
            if (row < M && blk < nblocks)
              *reinterpret_cast<uint4*>(codes + row * (int64_t)(d / 2) + (int64_t)blk * 16) = cw;
          }
          if constexpr (FMT == FMT_NVFP4) {
            if (blk >= nblocks) sbyte = 0;               // padding blocks decode to zero
            if (bb < 2) sc_word |= sbyte << (16 * bb);
            else sc_word2 |= sbyte << (16 * (bb - 2));
          } else {
            sc_word |= sbyte << (8 * bb);
          }
        }
        if (!ok) continue;
        if constexpr (FMT == FMT_F32OUT) {
          continue;
        } else if constexpr (FMT == FMT_NVFP4) {
          const int kb4n = (2 * nblocks + 3) / 4;        // 4-byte groups of 16-block scales per row: blocks fb, fb + 1
          if (mt < m_tiles) put_scales16(sc_word, sc_word2, (size_t)lane * 16 + q * 4, kb4n);
        } else {
          if (mt < m_tiles) put_scales(sc_word, (size_t)lane * 16 + q * 4);   // the pair's second row tile may not exist
        }
      }
    }
  }

  // ------------------------------------------------------------------ teardown
  tc_fence_before_sync();
  __syncthreads();
  if (*cta_abort) {
    for (int i = 0; i < 2000; ++i) __nanosleep(1000);
  }
  // The peer no longer touches this CTA's memory after this.  Relaxed: every arrival this CTA sent has been waited for (the
  // last tile of each accumulator sends none), and a release would make each warp wait for its global stores (0.3 - 0.5 us).
  cluster_arrive_relaxed();
  cluster_wait();
  if (warp == 1) {
    tc_fence_after_sync();
    tmem_dealloc_pair(tmem_base, C::TMEM_COLS);
  }
}

}  // namespace torq
