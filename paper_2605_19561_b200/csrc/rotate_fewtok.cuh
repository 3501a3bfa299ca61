// Rotate + quantize for few tokens (M <= 256), where the work is streaming R_inter from HBM once
// (Algorithm 3 steps 2-4).  One kernel, no scratch in global memory.
//
// Swapped operands: the tensor-core instruction's 128 rows are 128 output FEATURES (four 32-blocks)
// and its N columns are the tokens (16 ... 256, in steps of 16), so no row of the instruction is padding and the
// accumulator is small:  D[j, m] = sum_i R_inter[i, j] X[m, i].
//   A = R_inter tile [64 (i) x 128 (j)], features contiguous = MN-major, two 64 x 64 boxes (128-B swizzle)
//   B = X tile [tokens x 64 (i)], K-major
// A layer has only d / 128 feature tiles (40 at d = 5120), too few CTAs to pull R_inter at HBM rate,
// so the contraction is also split: a CLUSTER of S CTAs shares one feature tile, CTA r of the cluster
// contracts k range r.  The fp32 partial tiles never leave the SMs: every output has one CTA of the cluster that owns it, adds the S
// partials in rank order (fixed order, so the result does not depend on timing), rotates inside the block and quantizes (Eq. 1).
// The partials reach the owner in one of two ways:
//  * PUSH (up to 32 tokens, with R_intra and clusters of eight up to 56): the pieces of work are small, 32 features x 4
//    tokens, and dealt over all CTAs and warps of the cluster, so that nearly every warp has one and no CTA takes in more than its share
//    (what arrives at one SM comes at about 9 B per cycle).  A CTA stores its partials straight from registers into the owners' shared
//    memory (st.async, 16 bytes per lane = four tokens of one feature, counted on a barrier of the owning warp), into room of their own:
//    nobody has to say first that the stages there are free, and no cluster-wide barrier stands on the path.  The owning warp keeps one
//    feature per lane: the intra rotation is 32 x 4 FMAs per lane on R_intra's column in registers, y read by broadcast.  The other CTAs
//    leave right after their stores, which lets the CTAs of the next kernel in.  Against one owner for a tile (40 KiB to take in at 16
//    tokens, 80 loads per lane to add them, warp-level MMAs), us: rotation of 16 tokens, d = 4096 9.6 -> 8.8, 24 tokens NVFP4 (pulled
//    before) 10.3 -> 9.4.
//  * pull (more tokens): token group g (16 tokens) belongs to CTA g % S.  Every CTA writes its partial [token][feature] into its own shared
//    memory, a cluster barrier publishes them, and the owner reads them with 16-byte ld.shared::cluster and rotates on the warp-level
//    tensor cores (y split into three bf16 terms, fp32 accumulation).  A second barrier, at which a warp arrives
//    as soon as its last such load is back and for which it waits only before it exits, keeps the partials in place
//    (one full barrier at the end: d = 5120, M = 64 14.0 -> 13.7 us, GEMM 6.7 -> 6.1).  CTAs without a unit then leave earlier
//    than the others; where that harms (`together`, see the launch) the second barrier is a full one at the end after all.
//    The epilogue warps of lane quarter q of every CTA own 32-block q of the tile (its R_intra block is fetched into
//    shared memory when the kernel starts, long before it is needed: a first touch of that array from a
//    cold TLB costs microseconds).
// With S = 1 (an ordinary launch without clusters) a warp goes on with its own features.
//
// What the kernel waits for at its start is X (the kernel before writes it): the stages are full of R_inter by then and HBM would idle.  So
// the L2 is asked ahead of that wait for X, and for some R_inter beyond the stages (kAheadTiles): us, layer d = N = 5120, 1 token
// 14.8 -> 14.3, d = 4096, N = 6144, 200 tokens 22.4 -> 21.7.
//
// Roles per CTA: warp 0 TMA producer, warp 1 MMA issuer, warps 2..5 epilogue / reduction.
// Shared memory: 4 stages (5 up to 16 tokens, 3 where more than 32 push) of (16 KiB of R_inter + tokens x 128 B of X); pulled partials
// lie in the same memory after the mainloop, pushed ones behind it.  Up to 64 tokens that is small enough (<= 107 KiB) for two CTAs per
// SM: the grid may exceed the SM count, which keeps more loads in flight; above, one CTA fills an SM, or
// up to 128 tokens two of them with three stages (fewtok_rotation).
#pragma once
#include <cuda_bf16.h>
#include "intra_fragment.cuh"
#include "sm100_ptx.cuh"

namespace torq {

struct RotFewCfg {
  static constexpr int BF = 128;                       // features per tile = rows of the instruction
  static constexpr int BK = 64;
  static constexpr int A_BYTES = BK * BF * 2;          // 16 KiB: two boxes of 64 (k) x 64 (j)
  static constexpr int A_BOX_BYTES = 64 * 64 * 2;
  static constexpr int STAGES = 4, PUSH_STAGES = 5, MAX_STAGES = 5;
  // With three stages two CTAs of 65 to 128 tokens share an SM: for long K ranges, where one CTA per SM leaves SMs without
  // a CTA and too few loads in flight (the rule stands where the kernel is launched).
  static constexpr int SHARED_STAGES = 3, MAX_SHARED_TOK = 128;
  static constexpr int MAX_TOK = 256;                  // N of the instruction: a multiple of 16
  static constexpr int PUSH_TOK = 56;                  // tokens up to which sums are pushed (the rule stands where the kernel is launched)
  static constexpr int PUSH_NTOK = (PUSH_TOK + 15) / 16 * 16;
  static constexpr int PART_BYTES = 32 * 16;           // pushed partial of a unit from one CTA: [feature of the block][4 tokens]
  static constexpr int Y_BYTES = 16 * 33 * 4;          // pull, per epilogue warp: 16 tokens x 32 features, row stride 33
  static constexpr int RI_BYTES = 32 * 80;             // per epilogue warp: R_intra[block] as bf16 rows of 80 bytes
  static constexpr int BAR_BYTES = 256;
  static constexpr int THREADS = 192;
  static constexpr int MAX_CLUSTER = 8;
  __host__ __device__ static constexpr int stage_bytes(int ntok) { return A_BYTES + ntok * BK * 2; }
  // partials of the units that one CTA owns, from all CTAs, for any cluster size; then the y tile of each warp
  __host__ __device__ static constexpr int push_bytes(int ntok) { return (ntok + MAX_CLUSTER - 1) * PART_BYTES + 4 * PART_BYTES; }
  __host__ __device__ static constexpr int smem_bytes(int ntok, int stages, bool push) {
    return stages * stage_bytes(ntok) + BAR_BYTES + (push ? push_bytes(ntok) : 4 * RI_BYTES) + 1024;
  }
  __host__ __device__ static constexpr int ctas_per_sm(int ntok, int stages, bool push) {
    return smem_bytes(ntok, stages, push) <= 113 * 1024 ? 2 : 1;
  }
  __host__ __device__ static constexpr int max_smem_bytes() { return smem_bytes(MAX_TOK, STAGES, false); }
};
// what lies in the stages after the mainloop where partials are pulled: the partial tile (ntok x 512 B) and the y tiles
static_assert(8 * RotFewCfg::Y_BYTES <= 4 * RotFewCfg::A_BYTES && RotFewCfg::BF * 4 <= RotFewCfg::STAGES * RotFewCfg::BK * 2, "reduction buffers");
static_assert(RotFewCfg::ctas_per_sm(16, RotFewCfg::PUSH_STAGES, true) == 2 && RotFewCfg::ctas_per_sm(32, RotFewCfg::STAGES, true) == 2 &&
              RotFewCfg::ctas_per_sm(RotFewCfg::PUSH_NTOK, RotFewCfg::SHARED_STAGES, true) == 2, "two CTAs per SM where sums are pushed");
static_assert(RotFewCfg::ctas_per_sm(RotFewCfg::MAX_SHARED_TOK, RotFewCfg::SHARED_STAGES, false) == 2 &&
              4 * RotFewCfg::Y_BYTES + 80 * RotFewCfg::BF * 4 <= RotFewCfg::SHARED_STAGES * RotFewCfg::stage_bytes(80) &&
              4 * RotFewCfg::Y_BYTES + 128 * RotFewCfg::BF * 4 <= RotFewCfg::SHARED_STAGES * RotFewCfg::stage_bytes(128), "three stages");

// grid = (d / 128 or fewer feature tiles) * S CTAs in clusters of S along x: CTA b works feature tile ft0 + b / S, k split b % S.
// tmX: X [M, d] bf16, box [ntok rows x 64]; tmR: R_inter [d, d] bf16, box [64 x 64].  ntok = M rounded up to
// a multiple of 16.  d % 128 == 0.  `codes` / `scales` / `tensor_scale` as in rotate_quantize_kernel for FMT.
// ESETS: sets of four epilogue warps (threads = 64 + 128 ESETS).  One set where two CTAs share an SM; a CTA that fills an SM
// by itself has several token groups to reduce, rotate and quantize, each a dependent chain of about a microsecond for
// one warp: two sets take them in turn.  NST: stages.  `r_ahead`: R_inter tiles beyond
// the stages that a CTA asks the L2 for.  `together`: the CTAs of a cluster leave together (S > 1 only).
template <int FMT = FMT_MXFP4, int ESETS = 1, bool PUSH = false, int NST = RotFewCfg::STAGES>
__global__ void __launch_bounds__(64 + 128 * ESETS, ESETS == 1 ? 2 : 1)
rotate_fewtok_kernel(const __grid_constant__ CUtensorMap tmX, const __grid_constant__ CUtensorMap tmR,
                     const __nv_bfloat16* __restrict__ R_intra, uint8_t* __restrict__ codes,
                     uint8_t* __restrict__ scales, int M, int d, int ntok, int S, int ft0, int together, int r_ahead,
                     float tensor_scale, int* err_word) {
  using C = RotFewCfg;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t* smem_gen = smem_raw + (smem_base - smem_u32(smem_raw));
  const int stage_bytes = C::stage_bytes(ntok);
  constexpr int nst = NST;
  const uint32_t bar_off = nst * stage_bytes;
  const uint32_t bar_base = smem_base + bar_off;
  auto full_bar = [&](int s) { return bar_base + 8u * s; };
  auto empty_bar = [&](int s) { return bar_base + 8u * (C::MAX_STAGES + s); };
  const uint32_t accf_bar = bar_base + 8u * (2 * C::MAX_STAGES);
  auto recv_bar = [&](int w) { return accf_bar + 8u + 8u * w; };   // PUSH: all partials of the units of epilogue warp w are here
  volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(smem_gen + bar_off + 192);
  volatile int* cta_abort = reinterpret_cast<volatile int*>(smem_gen + bar_off + 200);
  uint8_t* ri_tiles = smem_gen + bar_off + C::BAR_BYTES;    // not part of the stages: filled at kernel start (PUSH: the partials)

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = blockIdx.x % S, ft = ft0 + blockIdx.x / S;
  const int k_tiles = d / C::BK;
  const int kt0 = (int)((long long)k_tiles * rank / S), kt1 = (int)((long long)k_tiles * (rank + 1) / S);
  const uint32_t tmem_cols = ntok <= 32 ? 32u : (ntok <= 64 ? 64u : (ntok <= 128 ? 128u : 256u));
  const int groups = (M + 15) / 16;                      // pull: token groups; group g belongs to CTA g % S
  // PUSH: unit u = q + 4 c is block q of the tile and tokens 4 c .. 4 c + 3.  CTA u % S owns it, epilogue warp u / S % 4 of that
  // CTA works it: the units of warp w are rank + S w, + 4 S, ..., all of the same block.
  const int units = 4 * ((M + 3) / 4);

  // R_inter is a constant of the layer, never the output of the kernel that runs just before this
  // one: the thread that initialises the barriers sends the loads of the first stages' R_inter tiles
  // right behind the initialisation (the kernel's time starts with an HBM round trip; tensor-memory
  // allocation and the block-wide barrier come after it instead of before).  X waits for that kernel.
  const int pre = (kt1 - kt0) < nst ? (kt1 - kt0) : nst;
  if (threadIdx.x == 0) {
    for (int s = 0; s < nst; ++s) { mbar_init(full_bar(s), 1); mbar_init(empty_bar(s), 1); }
    mbar_init(accf_bar, 1);
    if constexpr (PUSH)
      for (int w = 0; w < 4; ++w) mbar_init(recv_bar(w), 1);
    *cta_abort = 0;
    fence_mbar_init();
    fence_proxy_async_smem();                            // the copy engine sees the initialised barriers
    for (int it = 0; it < pre; ++it) {
      const uint32_t st = smem_base + it * stage_bytes;
      mbar_arrive_expect_tx(full_bar(it), (uint32_t)stage_bytes);
      tma_load_2d(st, &tmR, ft * C::BF, (kt0 + it) * C::BK, full_bar(it));
      tma_load_2d(st + C::A_BOX_BYTES, &tmR, ft * C::BF + 64, (kt0 + it) * C::BK, full_bar(it));
    }
    tma_prefetch_desc(&tmX);
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
  uint32_t rr[16];                                       // PUSH: column `lane` of the unit's R_intra block, two rows per word
  if constexpr (PUSH) {
    const int u0 = rank + S * (warp & 3);
#pragma unroll
    for (int k = 0; k < 16; ++k) rr[k] = 0u;
    if (warp >= 2 && R_intra != nullptr && u0 < units) {
      const uint16_t* src = reinterpret_cast<const uint16_t*>(R_intra) + (size_t)(ft * 4 + (u0 & 3)) * 1024 + lane;
#pragma unroll
      for (int k = 0; k < 16; ++k) rr[k] = (uint32_t)__ldg(src + 64 * k) | ((uint32_t)__ldg(src + 64 * k + 32) << 16);
    }
  } else if (warp >= 2 && warp < 6 && R_intra != nullptr && rank < groups) {
    // this warp's R_intra block (a constant of the layer as well), 128 pieces of 16 B: row piece / 4
    uint8_t* r_s = ri_tiles + (warp & 3) * C::RI_BYTES;
    const uint4* src = reinterpret_cast<const uint4*>(R_intra + (size_t)(ft * 4 + (warp & 3)) * 1024);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int piece = lane + 32 * i;
      *reinterpret_cast<uint4*>(r_s + (piece >> 2) * 80 + (piece & 3) * 16) = __ldg(src + piece);
    }
  }
  const int x_pre = !PUSH ? 0 : (pre < 4 ? pre : 4);     // X tiles that the epilogue warps send
  if (warp < 2) griddep_wait();

  bool acc_ok = false;                                   // epilogue warps: the accumulator is complete
  if (warp == 0) {
    // ------------------------------------------------------------------ TMA producer
    bool ok = true;
    for (int kt = kt0 + x_pre, it = x_pre; kt < kt1 && ok; ++kt, ++it) {
      const int s = it % nst;
      if (!mbar_wait_warp(empty_bar(s), ((it / nst) & 1) ^ 1, cta_abort, err_word, SITE_PRODUCER_EMPTY)) {
        ok = false; break;
      }
      const uint32_t st = smem_base + s * stage_bytes;
      if (elect_one()) {
        const bool r_issued = it < pre;                  // R side of this stage went out before the wait above
        if (!r_issued) {
          mbar_arrive_expect_tx(full_bar(s), (uint32_t)stage_bytes);
          tma_load_2d(st, &tmR, ft * C::BF, kt * C::BK, full_bar(s));
          tma_load_2d(st + C::A_BOX_BYTES, &tmR, ft * C::BF + 64, kt * C::BK, full_bar(s));
        }
        tma_load_2d(st + C::A_BYTES, &tmX, kt * C::BK, 0, full_bar(s));
      }
      __syncwarp();
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer
    const uint32_t idesc = idesc_bf16(128, ntok, /*A MN-major*/ true, /*B MN-major*/ false);
    bool ok = true;
    for (int kt = kt0, it = 0; kt < kt1 && ok; ++kt, ++it) {
      const int s = it % nst;
      if (!mbar_wait_warp(full_bar(s), (it / nst) & 1, cta_abort, err_word, SITE_MMA_FULL)) {
        ok = false; break;
      }
      tc_fence_after_sync();
      const uint32_t st = smem_base + s * stage_bytes;
      // A: MN-major.  64 features (128 B) contiguous, k rows 128 B apart, 8-row groups 1024 B apart
      // (stride offset), the next 64 features one box (8 KiB) further (leading offset).
      const uint64_t adesc = make_desc(st, C::A_BOX_BYTES, 1024, kSwizzle128);
      // B: K-major, token rows of 128 B, 8-row groups 1024 B apart.
      const uint64_t bdesc = make_desc(st + C::A_BYTES, 16, 1024, kSwizzle128);
      if (elect_one()) {
#pragma unroll
        for (int j = 0; j < C::BK / 16; ++j)             // K = 16 per instruction: 16 k rows of A = 2 KiB, 32 B of B
          mma_bf16(tmem_base, adesc + 128 * j, bdesc + 2 * j, idesc, (it | j) != 0);
        tc_commit(empty_bar(s));
      }
      __syncwarp();
    }
    if (ok && elect_one()) tc_commit(accf_bar);
    __syncwarp();
  } else {
    // ------------------------------------------------------------------ epilogue (warps 2..5)
    // X is not a constant, but asking the L2 for it changes nothing that a later load sees: one box per CTA until the K range is out.
    // So does asking for R_inter beyond the stages: until X has come the stages stay full and HBM idle.
    if (warp == 2 && elect_one())
      for (int kt = kt0 + ft - ft0; kt < kt1; kt += gridDim.x / S) tma_prefetch_l2_2d(&tmX, kt * C::BK, 0);
    if (warp == 3 && elect_one())
      for (int kt = kt0 + pre; kt < min(kt1, kt0 + pre + r_ahead); ++kt) {
        tma_prefetch_l2_2d(&tmR, ft * C::BF, kt * C::BK);
        tma_prefetch_l2_2d(&tmR, ft * C::BF + 64, kt * C::BK);
      }
    __syncwarp();
    griddep_wait();
    // The X tiles of the first stages go out from four warps at once: one warp needs 0.2 us from one stage to the next.  (PUSH only:
    // elsewhere these warps may still wait for R_intra.  100 tokens, d = 8192: the layer 34.8 / 35.3.)
    if (PUSH && warp - 2 < x_pre && elect_one())
      tma_load_2d(smem_base + (warp - 2) * stage_bytes + C::A_BYTES, &tmX, (kt0 + warp - 2) * C::BK, 0, full_bar(warp - 2));
    __syncwarp();
    // Two passes over the SAME instructions.  Pass 0 is a dry run while the mainloop streams: it reads
    // this CTA's own shared memory (whatever it holds), computes, and stores nothing.  Its only purpose
    // is to have the reduction's code in the instruction cache: executed cold, after the mainloop,
    // that code cost about 2.5 us of instruction fetches -- a fifth of the kernel.  Pass 1 is the
    // real one: accumulator -> partials, then the units of this warp.
    const int q = warp & 3;                              // lane quarter = 32-block of the tile
    const int es = (warp - 2) >> 2;                      // set of epilogue warps
    const int p = lane & 3, r8 = lane >> 2;
    const int nblocks = d / 32;
    const int blk = ft * 4 + q;
    const int kb4 = FMT == FMT_NVFP4 ? (2 * nblocks + 3) / 4 : (nblocks + 3) / 4;
    const uint32_t r_saddr = smem_u32(ri_tiles + q * C::RI_BYTES);
    const uint32_t r_lane = r_saddr + (uint32_t)(((lane >> 3) & 1) * 8 + (lane & 7)) * 80 + (uint32_t)(lane >> 4) * 16;
    const int feature = q * 32 + lane;                   // of this lane in tensor memory
    NvScale nvs = {};
    if constexpr (FMT == FMT_NVFP4) nvs = nv_scale(tensor_scale);
    // rotate inside the block, quantize, store: y in the fragment layout (rows = tokens of group g, columns = features)
    auto finish = [&](const uint32_t (&y)[16], int g, bool live) {
      IntraFrag f;
      if (R_intra != nullptr) load_intra_frag(r_lane, r_lane + 32, 16 * 80, f);
      uint32_t sb[2];
      intra_quantize_frag16<FMT, true>(y, R_intra != nullptr, f, lane, 16 * g, live ? M : 0, blk, nblocks, d, nvs, codes, sb);
      if (p == 0 && live) {
#pragma unroll
        for (int rh = 0; rh < 2; ++rh) {                 // rows of the group past the last token: zero
          const int row = 16 * g + r8 + 8 * rh;
          const uint32_t b = row < M ? sb[rh] : 0u;
          if constexpr (FMT == FMT_NVFP4) *reinterpret_cast<uint16_t*>(scales + scale_offset(row, 2 * blk, kb4)) = (uint16_t)b;
          else scales[scale_offset(row, blk, kb4)] = (uint8_t)b;
        }
      }
    };
    const uint32_t tacc = tmem_base + ((uint32_t)(q * 32) << 16);
    if constexpr (PUSH) {
      const int w = q;                                   // its number among the four: with S = 1 its own features are its units
      const uint32_t recv_base = smem_u32(ri_tiles);
      const uint32_t y_tile = recv_base + (uint32_t)(C::push_bytes(ntok) - 4 * C::PART_BYTES + w * C::PART_BYTES);
      const int ui0 = q / S, owner0 = q - ui0 * S;       // of piece 0 (a division takes as long as a store: not between the stores)
      if (S > 1) cluster_wait();
#pragma unroll 1
      for (int pass = rank + S * w < units ? 0 : 1; pass < 2; ++pass) {
        const bool live = pass == 1;
        if (live) {
          acc_ok = mbar_wait(accf_bar, 0, cta_abort, err_word, SITE_EPI_ACC_FULL);
          acc_ok = __all_sync(0xFFFFFFFFu, acc_ok);
          bool ok = acc_ok;
          if (!ok) break;
          tc_fence_after_sync();
          int ui = ui0, owner = owner0;
#pragma unroll 1
          for (int c0 = 0; c0 < M; c0 += 16) {
            uint32_t v[16];
            tmem_ld_32x32_x16(tacc + c0, v);
            tmem_ld_wait();
#pragma unroll
            for (int c = 0; c < 4; ++c) {
              const uint32_t slot = recv_base + (uint32_t)((ui * S + rank) * C::PART_BYTES + lane * 16);
              if (c0 + 4 * c >= M) break;
              if (S > 1)
                st_async_v4(map_to_cta(slot, (uint32_t)owner), v[4 * c], v[4 * c + 1], v[4 * c + 2], v[4 * c + 3],
                            map_to_cta(recv_bar(ui & 3), (uint32_t)owner));
              else                                       // S = 1: this warp's own units
                asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(slot), "r"(v[4 * c]), "r"(v[4 * c + 1]), "r"(v[4 * c + 2]),
                             "r"(v[4 * c + 3]) : "memory");
              owner += 4;                                // the unit four further on
              while (owner >= S) { owner -= S; ++ui; }
            }
          }
          if (S > 1) {
            if (rank + S * w >= units) break;            // nothing to receive
            ok = __all_sync(0xFFFFFFFFu, mbar_wait_cluster(recv_bar(w), 0, cta_abort, err_word, SITE_EPI_ACC_FULL));
          }
          if (!ok) break;
        }
#pragma unroll 1
        for (int u = rank + S * w, ui = w; u < units; u += 4 * S, ui += 4) {
          const int c = u >> 2, blk_u = ft * 4 + (u & 3);
          float y[4] = {0.f, 0.f, 0.f, 0.f};             // of feature `lane` of the block, four tokens
          float4 part[C::MAX_CLUSTER];
#pragma unroll
          for (int s = 0; s < C::MAX_CLUSTER; ++s)
            if (s < S)
              asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                           : "=f"(part[s].x), "=f"(part[s].y), "=f"(part[s].z), "=f"(part[s].w)
                           : "r"(recv_base + (uint32_t)((ui * S + s) * C::PART_BYTES + lane * 16)));
#pragma unroll
          for (int s = 0; s < C::MAX_CLUSTER; ++s)       // rank order: the result does not depend on timing
            if (s < S) { y[0] += part[s].x; y[1] += part[s].y; y[2] += part[s].z; y[3] += part[s].w; }
          float z[4] = {y[0], y[1], y[2], y[3]};
          if (R_intra != nullptr) {
            __syncwarp();
            asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(y_tile + lane * 16), "f"(y[0]), "f"(y[1]), "f"(y[2]), "f"(y[3]) : "memory");
            __syncwarp();
            intra_rotate_lane4(y_tile, rr, z);
          }
          quantize_lane4<FMT>(z, lane, 4 * c, live ? M : 0, blk_u, d, kb4, nvs, codes, scales);
        }
      }
    } else {
      float* y_s = reinterpret_cast<float*>(smem_gen + ntok * C::BF * 4 + (es * 4 + q) * C::Y_BYTES);
      const uint32_t p_saddr = smem_base;
      // lane l adds tokens (l / 8) + 4 j, j = 0..3, features 4 (l % 8) .. + 3 of the block, two tokens at a
      // time: their 2 S loads of 16 bytes go out before the first add, so a unit costs two round trips
      // through the cluster
      const int tr = lane >> 3, fc = (lane & 7) * 4;
#pragma unroll 1
      for (int pass = 0; pass < 2; ++pass) {
        const bool live = pass == 1;
        if (live) {
          acc_ok = mbar_wait(accf_bar, 0, cta_abort, err_word, SITE_EPI_ACC_FULL);
          acc_ok = __all_sync(0xFFFFFFFFu, acc_ok);
          if (acc_ok) {
            tc_fence_after_sync();
            float* prow = reinterpret_cast<float*>(smem_gen) + feature;     // partial tile [token][feature]
            for (int c0 = 16 * es; c0 < ntok; c0 += 16 * ESETS) {
              uint32_t v[16];
              tmem_ld_32x32_x16(tacc + c0, v);
              tmem_ld_wait();
#pragma unroll
              for (int j = 0; j < 16; ++j) prow[(c0 + j) * C::BF] = __uint_as_float(v[j]);
            }
          }
          tc_fence_before_sync();
          cluster_sync_all();                            // every CTA's partial tile is visible cluster-wide
        }
        uint32_t p_rank[C::MAX_CLUSTER];
#pragma unroll
        for (int s = 0; s < C::MAX_CLUSTER; ++s)
          p_rank[s] = s < S ? map_to_cta(p_saddr, live ? (uint32_t)s : (uint32_t)rank) : 0u;
        int g = rank + es * S;
        if (live && g >= groups && !together) cluster_arrive_relaxed();      // nothing to read
        for (; g < groups; g += S * ESETS) {
#pragma unroll
          for (int jh = 0; jh < 2; ++jh) {
            if (16 * g + 8 * jh >= M) break;      // rows 8 jh .. 8 jh + 7 of the group hold no token
            float4 part[2][C::MAX_CLUSTER];
#pragma unroll
            for (int j = 0; j < 2; ++j) {
              const uint32_t off = (uint32_t)(((16 * g + tr + 4 * (2 * jh + j)) * C::BF + q * 32 + fc) * 4);
#pragma unroll
              for (int s = 0; s < C::MAX_CLUSTER; ++s)
                if (s < S)
                  asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
                               : "=f"(part[j][s].x), "=f"(part[j][s].y), "=f"(part[j][s].z), "=f"(part[j][s].w)
                               : "r"(p_rank[s] + off));
            }
#pragma unroll
            for (int j = 0; j < 2; ++j) {
              float4 y = make_float4(0.f, 0.f, 0.f, 0.f);  // rank order: the result does not depend on timing
#pragma unroll
              for (int s = 0; s < C::MAX_CLUSTER; ++s)
                if (s < S) { y.x += part[j][s].x; y.y += part[j][s].y; y.z += part[j][s].z; y.w += part[j][s].w; }
              if (live) {                                // the y tile lies inside the stages: untouched while they are in use
                float* dst = y_s + (tr + 4 * (2 * jh + j)) * 33 + fc;
                dst[0] = y.x; dst[1] = y.y; dst[2] = y.z; dst[3] = y.w;
              }
            }
          }
          __syncwarp();
          if (live && g + S * ESETS >= groups && !together) cluster_arrive_relaxed();   // the last unit's partials are read
          uint32_t y[16];
#pragma unroll
          for (int n = 0; n < 4; ++n)
#pragma unroll
            for (int i = 0; i < 4; ++i)
              y[4 * n + i] = __float_as_uint(y_s[(r8 + 8 * (i >> 1)) * 33 + 8 * n + 2 * p + (i & 1)]);
          finish(y, g, live);
          __syncwarp();
        }
      }
    }
    // scale bytes of the rows no group covers, up to the last row of the 128-row scale tiles: zero
    if (rank == 0 && es == 0) {
      for (int row = q * 32 + lane; row < (M > 128 ? 256 : 128); row += 128) {
        if (row >= (PUSH ? units : 16 * groups)) {
          uint8_t* cell = scales + (size_t)(row >> 7) * kb4 * 512 + (row & 31) * 16 + ((row & 127) >> 5) * 4;
          if constexpr (FMT == FMT_NVFP4) {
            *reinterpret_cast<uint32_t*>(cell + (size_t)(2 * ft) * 512) = 0u;
            *reinterpret_cast<uint32_t*>(cell + (size_t)(2 * ft + 1) * 512) = 0u;
          } else {
            *reinterpret_cast<uint32_t*>(cell + (size_t)ft * 512) = 0u;
          }
        }
      }
    }
    tc_fence_before_sync();
  }
  if (PUSH) {
    if (warp < 2 && S > 1) cluster_wait();               // the epilogue warps have waited above
  } else {
    if (warp < 2) {                                      // as the epilogue warps in their pass 1
      tc_fence_before_sync();
      cluster_sync_all();
      if (!together) cluster_arrive_relaxed();
    }
    if (together) cluster_sync_all();                    // no CTA of the cluster reads this one's partial tile any more
    else cluster_wait();
  }

  // ------------------------------------------------------------------ teardown
  __syncthreads();
  // After a wait has given up, others may still push to this CTA: stay until they have left or given up as well (the
  // barrier does not count threads that have exited).
  if (PUSH && S > 1 && *cta_abort) cluster_sync_all();
  if (warp == 1) {
    tc_fence_after_sync();
    tmem_dealloc(tmem_base, tmem_cols);
  }
}

}  // namespace torq
