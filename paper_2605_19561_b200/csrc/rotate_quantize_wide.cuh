// Rotate + quantize on CTA pairs in ONE wave: every pair works exactly one tile of 256 tokens x `width` features
// (a multiple of 32, up to 384), the width chosen so that the tiles just fill the pairs.
//
// The pair kernel deals 256-column tiles.  A layer of some hundred tokens has either fewer of those than there are
// pairs, or a few more and pays a second wave for them.  Measured (rotation alone, us, pair kernel / here): 777 x
// 5120 (80 tiles / 4 x 18 of 288) 48.6 / 38.5; 1024 x 5120 48.8 / 40.1; 300 x 4096 (32 / 2 x 32 of 128) 26.0 / 21.2;
// 1000 x 1024 11.7 / 8.4; 1000 x 256 8.0 / 3.9.
//
// A tile wider than 256 columns is two instructions per 16 elements of K that share the X slice, accumulators
// side by side in tensor memory (column c of the tile is accumulator column c).  An instruction of N columns takes the
// larger of N / 2 and 64 + N / 4 cycles, the reading of its slices from shared memory; a second one on the same X
// slice N / 2, but at least 45 however narrow (per 64 of K 256 + 32 columns ran at 692 cycles, 160 + 128 at 576, 256 + 128 at 770),
// so the second one is always 128 columns.  Each CTA of the pair stages its 128 rows of X and half of each instruction's
// columns of R_inter: 64-column boxes of 8 KiB (16 KiB up to 128 columns, where a stage is 128 of K) and, when half of the
// first instruction is no multiple of 64, one narrower box (its rows keep the 128-byte pitch of the swizzle) in a slot of the
// same size.
//
// Bounds: up to 128 columns the latency of the loads and of the hand-overs between the roles (440 cycles per 64 of K at 64
// columns, 460 at 128 with stages of 64, where the instructions take 320 and 384; the same loads alone, from L2, run at 22
// TB/s), above the instructions (500 at 256); then the epilogue, which nothing overlaps.  The intra rotation in it runs as tcgen05
// instructions of both CTAs, y split into three bf16 terms in tensor memory; a lane then holds one row of a block and quantizes it.  As
// warp-level MMAs on the accumulator fragments it was bound by those, about 860 cycles per 32 columns (us, these / here: rotation 777 x
// 5120 44.8 / 42.5, 300 x 2048 8.72 / 8.45, layers 600 x 2048 -> 2048 15.7 / 14.95, loops of 0.5 s 1024 x 4096 -> 4096 44.3 / 43.0).
// Tiles of 32 columns keep that form: a unit of 16 rows for each of eight warps is done before the hand-over to the issuer and back (200
// x 2048 7.68 / 7.88, 256 x 1024 4.48 / 4.64).  Measured no faster: the terms of a set's next block sent before the result of this one is
// waited for (777 x 5120 42.4 / 41.9, but 300 x 2048 8.45 / 8.69: what a short call waits for is this code's instructions), and a warp
// that runs it once ahead (8.45 / 8.58).  Splitting K over the pairs of a larger cluster (partial sums exchanged through distributed
// shared memory) was measured and brought nothing: 300 x 4096 20.9 with two pairs per 256 columns against 21.2.
//
// Roles per CTA: warp 0 TMA producer, warp 1 MMA issuer (leader CTA), warps 2..13 epilogue (lane quarter w % 4, three
// sets of warps).  One elected thread runs the producer's and the issuer's loop.
#pragma once
#include <cuda_bf16.h>
#include "intra_fragment.cuh"
#include "sm100_ptx.cuh"

namespace torq {

struct RotWideCfg {
  static constexpr int BM = 128;                       // rows per CTA
  static constexpr int SLAB = 64;                      // K elements of one 128-byte row of X
  // K per stage: two slabs up to 128 columns, where the waits and the issue of loads per step bound a step and not its math (us, one
  // slab / two: 200 tokens d = 1024 4.87 / 4.48, d = 2048 8.42 / 7.57, 300 tokens d = 4096 18.4 / 17.1; loops of the whole warp
  // instead of one thread 5.51 and 9.10); above, three stages of twice the size lose against six (us, six / three: 600 x 4096 25.6 / 27.8,
  // 300 x 6144 35.5 / 39.3, 400 x 8192 60.3 / 62.8, 160 columns: 1280 x 2048 14.3 / 15.3)
  __host__ __device__ static constexpr int bk(int width) { return width <= 128 ? 2 * SLAB : SLAB; }
  __host__ __device__ static constexpr int a_bytes(int width) { return BM * bk(width) * 2; }       // 32 or 16 KiB
  __host__ __device__ static constexpr int box_bytes(int width) { return 64 * bk(width) * 2; }     // 64 columns of R_inter
  static constexpr int MAX_WIDTH = 384;
  static constexpr int AHEAD = 8;                      // K steps of R_inter that the L2 is asked for beyond the stages
  static constexpr int MAX_STAGES = 6;
  static constexpr int RI_BLOCK_BYTES = 32 * 64;       // R_intra[blk] as bf16 rows of 64 bytes, 16-byte pieces XOR-swizzled
  static constexpr int ESETS = 3;
  static constexpr int THREADS = 64 + 128 * ESETS;
  // Tensor memory behind the accumulator, for the intra rotation of one block per set of warps: the result, 32 columns, and the third split
  // term, 16.  Beside 384 columns there is room for two sets.
  __host__ __device__ static constexpr int sets(int width) { return width + 48 * ESETS <= 512 ? ESETS : 2; }
  __host__ __device__ static constexpr int out_col(int width, int set) { return width + 32 * set; }
  __host__ __device__ static constexpr int lo_col(int width, int set) { return width + 32 * sets(width) + 16 * set; }
  // columns of the first instruction; the second takes the rest
  __host__ __device__ static constexpr int n0(int width) { return width <= 256 ? width : width - 128; }
  __host__ __device__ static constexpr int boxes(int width) { return (n0(width) / 2 + 63) / 64 + (width > 256 ? 1 : 0); }
  __host__ __device__ static constexpr int tail_cols(int width) { return n0(width) / 2 % 64; }         // columns of the narrow box (0: none)
  __host__ __device__ static constexpr int stage_bytes(int width) { return a_bytes(width) + boxes(width) * box_bytes(width); }
  __host__ __device__ static constexpr int stage_tx(int width) { return a_bytes(width) + width / 2 * bk(width) * 2; }   // bytes one CTA loads
  // 192 to 200 KiB of stages whatever the width
  __host__ __device__ static constexpr int stages(int width) { return boxes(width) == 1 ? 4 : (boxes(width) == 2 ? 6 : 5); }
  __host__ __device__ static constexpr int smem_bytes(int width) {
    return stages(width) * stage_bytes(width) + (width / 32) * RI_BLOCK_BYTES + 256 + 1024;
  }
};
static_assert(RotWideCfg::smem_bytes(128) <= 232448 && RotWideCfg::smem_bytes(256) <= 232448 &&
              RotWideCfg::smem_bytes(384) <= 232448, "shared memory budget");
static_assert(RotWideCfg::stages(128) <= RotWideCfg::MAX_STAGES && RotWideCfg::stages(256) <= RotWideCfg::MAX_STAGES &&
              RotWideCfg::stages(384) <= RotWideCfg::MAX_STAGES, "barriers");

// grid = 2 * rows * cols CTAs in clusters of two: pair p works row tile p % rows (256 tokens), column tile p / rows
// (`width` features from column (p / rows) * width on).  tmX: X as (64 of K, token, slab of K), box [64 x 128 x slabs of a
// stage]; tmR: R_inter box [BK of K x 64 columns]; tmRt: box [BK x tail_cols].  d % 128 == 0.  RANGE: 32, 128, 256 or 384, the first
// that is not below the width (two slabs of K per stage, one block; two slabs; one; two instructions per slice).  FMT, `tensor_scale` as
// in the pair kernel.
template <int FMT, int RANGE>
__global__ void __launch_bounds__(RotWideCfg::THREADS, 1)
rotate_quantize_wide_kernel(const __grid_constant__ CUtensorMap tmX, const __grid_constant__ CUtensorMap tmR,
                            const __grid_constant__ CUtensorMap tmRt, const __nv_bfloat16* __restrict__ R_intra,
                            uint8_t* __restrict__ codes, uint8_t* __restrict__ scales, int M, int d,
                            float tensor_scale, int rows, int width, int* err_word) {
  using C = RotWideCfg;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t* smem_gen = smem_raw + (smem_base - smem_u32(smem_raw));
  const int nst = C::stages(width);
  const uint32_t stage_bytes = C::stage_bytes(width);
  const uint32_t ri_off = nst * stage_bytes;
  const uint32_t bar_off = ri_off + (uint32_t)(width / 32) * C::RI_BLOCK_BYTES;
  const uint32_t bar_base = smem_base + bar_off;
  auto full_bar = [&](int s) { return bar_base + 8u * s; };
  auto empty_bar = [&](int s) { return bar_base + 8u * (C::MAX_STAGES + s); };
  const uint32_t accf_bar = bar_base + 8u * (2 * C::MAX_STAGES);
  const uint32_t alloc_bar = accf_bar + 8;             // in the leader: the other CTA's tensor memory is allocated
  auto term_bar = [&](int set) { return accf_bar + 16u + 8u * set; };              // in the leader: both CTAs' split terms of a block
  const uint32_t ri_bar = accf_bar + 16 + 16 * C::ESETS;                           // in the leader: R_intra is in both CTAs' shared memory
  auto rot_bar = [&](int set) { return accf_bar + 16u + 8u * (C::ESETS + set); };  // the rotated block
  volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(smem_gen + bar_off + 192);
  volatile int* cta_abort = reinterpret_cast<volatile int*>(smem_gen + bar_off + 200);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cluster_ctarank();             // 0 = leader
  const int pair = blockIdx.x >> 1;
  const int tcol = (pair / rows) * width;
  const int mt = 2 * (pair % rows) + (int)rank;
  constexpr int BK = C::bk(RANGE), A_BYTES = C::a_bytes(RANGE), BOX_BYTES = C::box_bytes(RANGE);
  constexpr bool TWO = RANGE > 256, kTerms = RANGE > 32;           // kTerms: the intra rotation as tcgen05 instructions
  const int k_tiles = d / BK;
  const int n0 = C::n0(width);
  const int nb = min(width / 32, d / 32 - (tcol >> 5));            // 32-blocks of this tile that exist
  const int sets = C::sets(width);

  // Set-up as in the pair kernels: the producer waits for nothing but the barriers of both CTAs, and the first stages' X loads
  // come from a warp of their own (us, before / after: 200 x 1024 5.25 / 4.87, 200 x 2048 9.35 / 8.42, 300 x 4096 19.2 / 18.5).
  if (threadIdx.x == 0) {
    for (int s = 0; s < nst; ++s) { mbar_init(full_bar(s), 1); mbar_init(empty_bar(s), 1); }
    mbar_init(accf_bar, 1);
    mbar_init(alloc_bar, 1);
    for (int i = 0; i < C::ESETS; ++i) { mbar_init(term_bar(i), 8); mbar_init(rot_bar(i), 1); }
    mbar_init(ri_bar, 2);
    *cta_abort = 0;
    fence_mbar_init();
  }
  if (warp == 2 && elect_one()) { tma_prefetch_desc(&tmX); tma_prefetch_desc(&tmR); tma_prefetch_desc(&tmRt); }
  __syncwarp();
  cluster_arrive_relaxed();
  uint32_t tmem_base = 0;
  if (warp == 0) {
    named_barrier_arrive(2, C::THREADS);
    cluster_wait();                                    // both CTAs' barriers exist before any remote arrive
  } else {
    if (warp == 1) { tmem_alloc_pair(smem_u32(const_cast<uint32_t*>(tmem_slot)), 512); tmem_relinquish_pair(); }
    tc_fence_before_sync();
    named_barrier_sync(2, C::THREADS);
    cluster_wait();
    tc_fence_after_sync();
    tmem_base = *tmem_slot;
    if (warp == 1 && rank == 1 && lane == 0) mbar_arrive_cluster(map_to_cta(alloc_bar, 0));   // this CTA's tensor memory is there
  }
  // R_inter is a constant of the layer, never the output of the kernel that runs just before this one: its
  // loads for the first stages go out now, everything else waits for that kernel to complete.
  griddep_launch_dependents();
  const int pre = k_tiles < nst ? k_tiles : nst;

  if (warp == 0) {
    // ------------------------------------------------------------------ TMA producer (both CTAs)
    if (elect_one()) {
      const int full0 = n0 / 128;                      // whole 64-column boxes of this CTA's half of the first instruction
      const int tail = C::tail_cols(width);
      const int col0 = tcol + (int)rank * (n0 / 2), col1 = tcol + n0 + (int)rank * 64;
      const uint32_t leader_full0 = map_to_cta(full_bar(0), 0);
      auto load_r = [&](int s, int kt) {
        uint32_t dst = smem_base + s * stage_bytes + A_BYTES;
        const uint32_t bar = leader_full0 + 8u * s;
        if (rank == 0) mbar_arrive_expect_tx(full_bar(s), 2 * C::stage_tx(width));
        for (int b = 0; b < full0; ++b, dst += BOX_BYTES) tma_load_2d_pair(dst, &tmR, col0 + 64 * b, kt * BK, bar);
        if (tail) {
          tma_load_2d_pair(dst, &tmRt, col0 + 64 * full0, kt * BK, bar);
          dst += BOX_BYTES;
        }
        if constexpr (TWO) tma_load_2d_pair(dst, &tmR, col1, kt * BK, bar);
      };
      for (int i = 0; i < pre; ++i) load_r(i, i);
      griddep_wait();
      int s = 0;                                       // warp 2 sends the X loads of the first stages
      uint32_t ph = 0;
      for (int kt = pre; kt < k_tiles; ++kt) {
        if (!mbar_wait_cluster(empty_bar(s), ph, cta_abort, err_word, SITE_PRODUCER_EMPTY)) break;
        load_r(s, kt);
        tma_load_3d_pair(smem_base + s * stage_bytes, &tmX, 0, mt * C::BM, kt * (BK / C::SLAB), leader_full0 + 8u * s);
        if (++s == nst) { s = 0; ph ^= 1; }
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer (leader only)
    if (rank == 0 && mbar_wait_cluster_warp<true>(alloc_bar, 0, cta_abort, err_word, SITE_PEER_TMEM) && elect_one()) {
      const uint32_t idesc0 = idesc_bf16(256, n0, /*A MN-major*/ false, /*B MN-major*/ true);
      constexpr uint32_t idesc1 = idesc_bf16(256, 128, false, true);
      int s = 0;
      uint32_t ph = 0;
      bool ok = true;
      for (int kt = 0; kt < k_tiles; ++kt) {
        ok = mbar_wait_cluster<true>(full_bar(s), ph, cta_abort, err_word, SITE_MMA_FULL);
        if (!ok) break;
        tc_fence_after_sync();
        const uint32_t st = smem_base + s * stage_bytes;
        const uint64_t adesc = make_desc(st, 16, 1024, kSwizzle128);
        const uint64_t bdesc = make_desc(st + A_BYTES, BOX_BYTES, 1024, kSwizzle128);
#pragma unroll
        for (int j = 0; j < BK / 16; ++j) {
          const uint64_t aj = adesc + (j >> 2) * (C::BM * C::SLAB * 2 / 16) + 2 * (j & 3);
          mma_bf16_pair(tmem_base, aj, bdesc + 128 * j, idesc0, (kt | j) != 0);
          if constexpr (TWO)                           // the first instruction's half is two boxes then
            mma_bf16_pair(tmem_base + n0, aj, bdesc + 2 * BOX_BYTES / 16 + 128 * j, idesc1, (kt | j) != 0);
        }
        tc_commit_pair(empty_bar(s), 3);            // stage free in both CTAs
        if (++s == nst) { s = 0; ph ^= 1; }
      }
      if (ok) tc_commit_pair(accf_bar, 3);          // accumulator ready in both CTAs
      // Intra-block rotation: block bb by set bb % sets, three split terms x 32 of K, terms and result in tensor memory.
      constexpr uint32_t idesc_r = idesc_bf16(256, 32, false, true);
      if (kTerms && R_intra != nullptr && ok) ok = mbar_wait_cluster<true>(ri_bar, 0, cta_abort, err_word, SITE_MMA_FULL);
      for (int bb = 0, set = 0, r = 0; kTerms && R_intra != nullptr && ok && bb < nb; ++bb) {
        ok = mbar_wait_cluster<true>(term_bar(set), r & 1, cta_abort, err_word, SITE_MMA_FULL);
        if (!ok) break;
        tc_fence_after_sync();
        const uint64_t rdesc = make_desc(smem_base + ri_off + bb * C::RI_BLOCK_BYTES, 2048, 512, kSwizzle64);
        const uint32_t y = tmem_base + bb * 32, lo = tmem_base + C::lo_col(width, set), out = tmem_base + C::out_col(width, set);
        mma_bf16_pair_tmem_a(out, lo, rdesc, idesc_r, 0);            // the smallest term first
        mma_bf16_pair_tmem_a(out, lo + 8, rdesc + 64, idesc_r, 1);   // k 16 .. 31: +8 columns of terms, +16 rows of R_intra
        mma_bf16_pair_tmem_a(out, y + 16, rdesc, idesc_r, 1);
        mma_bf16_pair_tmem_a(out, y + 24, rdesc + 64, idesc_r, 1);
        mma_bf16_pair_tmem_a(out, y, rdesc, idesc_r, 1);
        mma_bf16_pair_tmem_a(out, y + 8, rdesc + 64, idesc_r, 1);
        tc_commit_pair(rot_bar(set), 3);
        if (++set == sets) { set = 0; ++r; }
      }
    }
    __syncwarp();
  } else {
    // ------------------------------------------------------------------ epilogue (12 warps per CTA)
    const int q = warp & 3;
    const int set = (warp - 2) >> 2;
    const int nblocks = d / 32, b0 = tcol >> 5;
    if (warp == 3 && elect_one()) {
      // Until the kernel before has completed HBM idles.  In short calls the L2 is asked for the first K steps of X, one of each row tile
      // per pair that shares it, and, for strips of 64 to 128 columns, for the next R_inter, a strip's steps dealt over its row tiles (us,
      // without / X alone / both, layers: 300 x 2048 -> 2048 14.00 / 13.83 / 13.69, 600 x 2048 15.4 / 15.1 / 14.9, 400 x 4096 -> 4096
      // 25.7 / 25.3 / 25.1, 1500 x 2048 22.0 / 21.6; narrower strips lose by R_inter, 220 x 2048 12.73 / 12.60 / 12.71).  Calls long
      // enough to run at the power cap lose (loops of 0.6 s, 1024 x 4096 44.4 / 44.7 / 45.0, 777 x 5120 60.7 / 60.8).  A box wholly
      // beyond the last token or feature fetches nothing; to leave it out costs more (without / with that guard: 300 x 2048 -> 2048 12.77
      // / 12.81, 1000 x 2048 -> 2048 15.48 / 15.53, 100 x 2048 -> 2048 12.00 / 12.02, three turns each that agree within 0.02).
      if (width * d <= 128 * 4096 && pair / rows < k_tiles) tma_prefetch_l2_3d(&tmX, 0, mt * C::BM, pair / rows * (BK / C::SLAB));
      if (RANGE == 128 && width >= 64)
        for (int kt = pre + pair % rows; kt < min(k_tiles, pre + C::AHEAD); kt += rows)
          for (int c = 0; c < width / 2; c += 64) tma_prefetch_l2_2d(&tmR, tcol + (int)rank * (width / 2) + c, kt * BK);
    }
    __syncwarp();
    if (warp == 2) {
      // X loads of the first stages, from a warp of its own: not behind the R_inter loads of all these stages
      griddep_wait();
      if (elect_one())
        for (int i = 0; i < pre; ++i)
          tma_load_3d_pair(smem_base + i * stage_bytes, &tmX, 0, mt * C::BM, i * (BK / C::SLAB), map_to_cta(full_bar(i), 0));
      __syncwarp();
    }
    if (R_intra != nullptr) {
      // The tile's blocks, rows of 64 bytes under the 64-byte swizzle: 16-byte piece c of row i at c ^ ((i >> 1) & 3).  This CTA's half
      // of the instruction's 32 columns are the first 32 bytes of its rows: rank 1 holds its pieces two on (kTerms).
      for (int idx = (warp - 2) * 32 + lane; idx < nb * 128; idx += 128 * C::ESETS) {
        const int lb = idx >> 7, i = (idx >> 2) & 31, c = (idx & 3) ^ (kTerms ? 2 * (int)rank : 0);
        *reinterpret_cast<uint4*>(smem_gen + ri_off + lb * C::RI_BLOCK_BYTES + i * 64 + ((c ^ ((i >> 1) & 3)) << 4)) =
            __ldg(reinterpret_cast<const uint4*>(R_intra + (size_t)(b0 + lb) * 1024) + (idx & 127));
      }
      if constexpr (kTerms) fence_proxy_async_smem();  // visible to the tensor core's reads
      named_barrier_sync(1, 128 * C::ESETS);
      // kTerms only: without them nobody waits for it, and an arrival that is not waited for could reach a CTA that has exited
      if (kTerms && warp == 2 && lane == 0) mbar_arrive_release_cluster(map_to_cta(ri_bar, 0));
    }
    griddep_wait();                                    // codes and scales may still be read by that kernel
    bool ok = mbar_wait_cluster(accf_bar, 0, cta_abort, err_word, SITE_EPI_ACC_FULL);
    ok = __all_sync(0xFFFFFFFFu, ok);
    tc_fence_after_sync();
    const uint32_t tlane = tmem_base + ((uint32_t)(q * 32) << 16);
    const int64_t row = (int64_t)mt * C::BM + q * 32 + lane;
    const bool live = mt * C::BM + q * 32 < M;         // warp-uniform: else this warp only makes its arrivals
    NvScale nvs = {};
    if constexpr (FMT == FMT_NVFP4) nvs = nv_scale(tensor_scale);
    const int kb4 = FMT == FMT_NVFP4 ? (2 * nblocks + 3) / 4 : (nblocks + 3) / 4;
    if constexpr (!kTerms) {
      // One block: a unit of 16 rows per warp of the first two sets, on accumulator fragments (tmem_ld_16x256b_x4) and warp-level MMAs.
      const int p = lane & 3, r8 = lane >> 2, mh = set;
      if (ok && set < 2 && nb > 0 && mt * C::BM < M) {
        uint32_t y[16];
        tmem_ld_16x256b_x4(tlane + ((uint32_t)(16 * mh) << 16), y);
        tmem_ld_wait();
        // ldmatrix: lane l addresses row l % 8 (+ 8 for odd l / 8) of its matrix, 16-byte piece l / 16 (+ 2)
        const int li = ((lane >> 3) & 1) * 8 + (lane & 7);
        const uint32_t rb = smem_base + ri_off + (uint32_t)li * 64 + (uint32_t)(((lane >> 4) ^ ((li >> 1) & 3)) << 4);
        IntraFrag f;
        if (R_intra != nullptr) load_intra_frag(rb, rb ^ 32u, 16 * 64, f);
        uint32_t sb[2];
        intra_quantize_frag16<FMT>(y, R_intra != nullptr, f, lane, (int64_t)mt * C::BM + q * 32 + 16 * mh, M, b0, nblocks, d, nvs, codes, sb);
        if (p == 0) {                                  // byte b0 % 4 of the 4-byte cell of (row, b0 / 4)
#pragma unroll
          for (int rh = 0; rh < 2; ++rh) {
            const int64_t rr = (int64_t)mt * C::BM + q * 32 + r8 + 16 * mh + 8 * rh;
            if constexpr (FMT == FMT_NVFP4) *reinterpret_cast<uint16_t*>(scales + scale_offset(rr, 2 * b0, kb4)) = (uint16_t)sb[rh];
            else scales[scale_offset(rr, b0, kb4)] = (uint8_t)sb[rh];
          }
        }
      }
    } else {
      const uint32_t term_leader = map_to_cta(term_bar(set), 0);
      // A warp takes 32 rows of a block, one row per lane.  y goes back to tensor memory as hi + mid + lo (bf16, exact): hi and mid over
      // y itself, lo in columns of the set's own, where the result comes as well.
      uint32_t ph = 0;
#pragma unroll 1
      for (int bb = set; ok && set < sets && bb < nb; bb += sets) {
        const int blk = b0 + bb;
        uint32_t y[32];
        if (live) {
          tmem_ld_32x32(tlane + bb * 32, y);
          tmem_ld_wait();
        }
        if (R_intra != nullptr) {
          if (live) {
            uint32_t hi[16], mid[16], lo[16];
#pragma unroll
            for (int e = 0; e < 16; ++e) split3_trunc_bf16x2(y[2 * e], y[2 * e + 1], hi[e], mid[e], lo[e]);
            tmem_st_32x32_x16(tlane + bb * 32, hi);
            tmem_st_32x32_x16(tlane + bb * 32 + 16, mid);
            tmem_st_32x32_x16(tlane + C::lo_col(width, set), lo);
            tmem_st_wait();
          }
          tc_fence_before_sync();
          __syncwarp();
          if (lane == 0) mbar_arrive_cluster(term_leader);
          ok = mbar_wait_cluster(rot_bar(set), ph, cta_abort, err_word, SITE_EPI_ACC_FULL);
          ok = __all_sync(0xFFFFFFFFu, ok);
          if (!ok) break;
          ph ^= 1;
          tc_fence_after_sync();
          if (live) {
            tmem_ld_32x32(tlane + C::out_col(width, set), y);
            tmem_ld_wait();
          }
          tc_fence_before_sync();
        }
        if (live) {
          float z[32];
#pragma unroll
          for (int i = 0; i < 32; ++i) z[i] = __uint_as_float(y[i]);
          uint4 cw, cw2;
          uint32_t sbyte;
          if constexpr (FMT == FMT_MXINT4) mxint4_quantize_block32(z, cw, cw2, sbyte);
          else if constexpr (FMT == FMT_NVFP4) nv_quantize_2x16(z, nvs, cw, sbyte);
          else quantize_block32(z, cw, sbyte);
          if (row < M) {
            if constexpr (FMT == FMT_MXINT4) {           // one operand byte per element
              uint4* dst = reinterpret_cast<uint4*>(codes + row * (int64_t)d + (int64_t)blk * 32);
              dst[0] = cw;
              dst[1] = cw2;
            } else {
              *reinterpret_cast<uint4*>(codes + row * (int64_t)(d / 2) + (int64_t)blk * 16) = cw;
            }
          }
          // rows past the last token of the 128-row scale tile: their sums are zero, and so is their byte
          if constexpr (FMT == FMT_NVFP4) *reinterpret_cast<uint16_t*>(scales + scale_offset(row, 2 * blk, kb4)) = (uint16_t)sbyte;
          else scales[scale_offset(row, blk, kb4)] = (uint8_t)sbyte;
        } else if (mt * C::BM < M) {                     // a quarter without a token
          if constexpr (FMT == FMT_NVFP4) *reinterpret_cast<uint16_t*>(scales + scale_offset(row, 2 * blk, kb4)) = 0;
          else scales[scale_offset(row, blk, kb4)] = 0;
        }
      }
    }
    tc_fence_before_sync();
  }

  // ------------------------------------------------------------------ teardown
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
