// C-ABI entry points of the library (see include/torq.h): argument validation, TMA descriptor
// encoding, kernel selection and launch.  Nothing here computes on the host.
#include <cuda.h>
#include <cuda_runtime.h>
#include <atomic>
#include <mutex>
#include <type_traits>

#include "../../include/torq.h"
#include "mxfp4_gemm_pair.cuh"
#include "mxfp4_gemm_wide.cuh"
#include "quantize.cuh"
#include "nvfp4_quantize.cuh"
#include "mxint4_quantize.cuh"
#include "rotate_quantize.cuh"
#include "rotate_quantize_pair.cuh"
#include "rotate_quantize_wide.cuh"
#include "rotate_fewtok.cuh"
#include "gemm_fewtok.cuh"
#include "rotate_structured.cuh"
#include "fp4_peak_probe.cuh"
#include "calibrate.cuh"
#include "wait_selftest.cuh"
#include "prepare_weights.cuh"
#include "sm100_ptx.cuh"

namespace torq {

__device__ int g_error_word = 0;

constexpr int kMaxDevices = 64;
struct DeviceState {
  bool ready = false;
  bool arch_ok = false;
  int sm_count = 0;
  int rot_pairs = 0;    // CTA pairs of the pair kernels that can be resident at once
  int gemm_pairs = 0;
  int few_fit[9] = {};  // clusters of S CTAs resident at once, one CTA per SM
  int push_fit[9] = {}; // the same of the few-token kernels that push, two CTAs per SM
  int* err_word = nullptr;
};
static DeviceState g_dev[kMaxDevices];
static std::mutex g_mutex;
static std::atomic<int64_t> g_launches{0};

using EncodeTiledFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*,
                                   const cuuint64_t*, const cuuint64_t*, const cuuint32_t*,
                                   const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                   CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
static EncodeTiledFn g_encode = nullptr;

template <typename K>
static bool opt_in_smem(K kernel, int bytes) {
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) ==
         cudaSuccess;
}

// How many clusters of `size` CTAs of `kernel` fit on the device at once (GPC boundaries can leave SMs unused).
template <typename K>
static int max_active_clusters(K kernel, int size, int threads, int smem, int sm_count) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(4 * sm_count / size * size), 1, 1);     // the answer never exceeds the grid
  cfg.blockDim = dim3((unsigned)threads, 1, 1);
  cfg.dynamicSmemBytes = (size_t)smem;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)size;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return n;
}
// Stands in for a few-token kernel in that question: of a kernel that allocates tensor memory the runtime counts one CTA per SM, whatever
// its shared memory.  Never launched.
__global__ void __launch_bounds__(RotFewCfg::THREADS, 2) fewtok_fit_kernel() {}

// The kernels of one format.
template <int FMT>
static bool opt_in_format() {
  constexpr int kWideSmem = 232448;                        // the widths share the kernels
  constexpr int few_rot = RotFewCfg::max_smem_bytes(), few_gemm = GemmFewCfg<FMT>::max_smem_bytes();
  return opt_in_smem(rotate_quantize_kernel<256, FMT>, RotCfg<256>::SMEM_BYTES) &&
         opt_in_smem(rotate_quantize_pair_kernel<FMT>, RotPairCfg::SMEM_BYTES) &&
         opt_in_smem(rotate_quantize_wide_kernel<FMT, 32>, kWideSmem) && opt_in_smem(rotate_quantize_wide_kernel<FMT, 128>, kWideSmem) &&
         opt_in_smem(rotate_quantize_wide_kernel<FMT, 256>, kWideSmem) && opt_in_smem(rotate_quantize_wide_kernel<FMT, 384>, kWideSmem) &&
         opt_in_smem(rotate_structured_kernel<FMT>, RotStructCfg::SMEM_BYTES) &&
         opt_in_smem(rotate_fewtok_kernel<FMT, 1, true>, few_rot) &&
         opt_in_smem(rotate_fewtok_kernel<FMT, 1, true, RotFewCfg::SHARED_STAGES>, few_rot) &&
         opt_in_smem(rotate_fewtok_kernel<FMT, 1, true, RotFewCfg::PUSH_STAGES>, few_rot) &&
         opt_in_smem(rotate_fewtok_kernel<FMT, 1, false, RotFewCfg::SHARED_STAGES>, few_rot) &&
         opt_in_smem(rotate_fewtok_kernel<FMT, 1>, few_rot) && opt_in_smem(rotate_fewtok_kernel<FMT, 2>, few_rot) &&
         opt_in_smem(mxfp4_gemm_pair_kernel<FMT>, GemmPairCfgT<FMT>::SMEM_BYTES) &&
         opt_in_smem(mxfp4_gemm_wide_kernel<FMT, 128>, kWideSmem) && opt_in_smem(mxfp4_gemm_wide_kernel<FMT, 256>, kWideSmem) &&
         opt_in_smem(mxfp4_gemm_wide_kernel<FMT, 384>, kWideSmem) && opt_in_smem(gemm_fewtok_kernel<FMT, 1, true>, few_gemm) &&
         opt_in_smem(gemm_fewtok_kernel<FMT, 1>, few_gemm) && opt_in_smem(gemm_fewtok_kernel<FMT, 2>, few_gemm);
}

// CTA pairs of a kernel that fills its SMs.
template <typename K>
static int max_active_pairs(K kernel, int threads, int smem, int sm_count) {
  const int n = max_active_clusters(kernel, 2, threads, smem, sm_count);
  return n < sm_count / 2 ? n : sm_count / 2;
}

// Per-device one-time set-up: architecture check, SM count, error-word address, shared-memory
// opt-in of the tensor-core kernels.  Returns nullptr when CUDA itself fails.
static DeviceState* device_state() {
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return nullptr;
  std::lock_guard<std::mutex> lock(g_mutex);
  DeviceState& st = g_dev[dev];
  if (st.ready) return &st;
  int major = 0;
  if (cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev) != cudaSuccess)
    return nullptr;
  if (cudaDeviceGetAttribute(&st.sm_count, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return nullptr;
  st.arch_ok = (major == 10);
  if (st.arch_ok) {
    if (cudaGetSymbolAddress(reinterpret_cast<void**>(&st.err_word), g_error_word) != cudaSuccess)
      return nullptr;
    if (!g_encode) {
      void* fn = nullptr;
      cudaDriverEntryPointQueryResult qres;
      if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &qres) !=
              cudaSuccess || qres != cudaDriverEntryPointSuccess || fn == nullptr)
        return nullptr;
      g_encode = reinterpret_cast<EncodeTiledFn>(fn);
    }
    const bool ok = opt_in_smem(fewtok_fit_kernel, RotFewCfg::max_smem_bytes()) && opt_in_format<FMT_MXFP4>() &&
                    opt_in_format<FMT_NVFP4>() && opt_in_format<FMT_MXINT4>() &&
                    opt_in_smem(rotate_quantize_kernel<256, FMT_F32OUT>, RotCfg<256>::SMEM_BYTES) &&
                    opt_in_smem(rotate_quantize_pair_kernel<FMT_F32OUT>, RotPairCfg::SMEM_BYTES);
    if (!ok) return nullptr;
    st.rot_pairs = max_active_pairs(rotate_quantize_pair_kernel<FMT_MXFP4>, RotPairCfg::THREADS,
                                    RotPairCfg::SMEM_BYTES, st.sm_count);
    st.gemm_pairs = max_active_pairs(mxfp4_gemm_pair_kernel<FMT_NVFP4>, GemmPairCfg::THREADS,
                                     GemmPairCfgT<FMT_NVFP4>::SMEM_BYTES, st.sm_count);
    if (st.rot_pairs < 1 || st.gemm_pairs < 1) return nullptr;
    for (int s = 1; s <= RotFewCfg::MAX_CLUSTER; ++s)
      st.few_fit[s] = max_active_clusters(rotate_fewtok_kernel<FMT_MXFP4, 2>, s, 320, RotFewCfg::smem_bytes(256, RotFewCfg::STAGES, false), st.sm_count);
    for (int s = 1; s <= RotFewCfg::MAX_CLUSTER; ++s)
      st.push_fit[s] = max_active_clusters(fewtok_fit_kernel, s, RotFewCfg::THREADS,
                                           RotFewCfg::smem_bytes(RotFewCfg::PUSH_NTOK, RotFewCfg::SHARED_STAGES, true), st.sm_count);
    cudaGetLastError();
  }
  st.ready = true;
  return &st;
}

// 2-D row-major tensor [rows, cols] of `elem_bytes`-byte elements, box [box_rows, box_cols],
// 128-byte swizzle, zero fill outside the tensor.
static bool encode_2d(CUtensorMap* map, CUtensorMapDataType dt, int elem_bytes, const void* base,
                      uint64_t rows, uint64_t cols, uint32_t box_rows, uint32_t box_cols,
                      CUtensorMapSwizzle swizzle = CU_TENSOR_MAP_SWIZZLE_128B) {
  cuuint64_t dims[2] = {cols, rows};
  cuuint64_t strides[1] = {cols * (uint64_t)elem_bytes};
  cuuint32_t box[2] = {box_cols, box_rows};
  cuuint32_t estr[2] = {1, 1};
  return g_encode(map, dt, 2, const_cast<void*>(base), dims, strides, box, estr,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle,
                  CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// X [M, d] bf16 seen as (position k: 32, token: M, block: d/32) with box (32, 1, 64): the box lands
// in shared memory as 64 rows (blocks) of 64 bytes (one token's 32 positions), 64-byte swizzle.
static bool encode_x_blocks_3d(CUtensorMap* map, const void* base, uint64_t M, uint64_t d) {
  cuuint64_t dims[3] = {32, M, d / 32};
  cuuint64_t strides[2] = {d * 2, 64};
  cuuint32_t box[3] = {32, 1, 64};
  cuuint32_t estr[3] = {1, 1, 1};
  return g_encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box, estr,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// X [M, d] bf16 seen as (K within a slab of 64, token, slab) with box (64, 128, slabs): each slab lands as 128 rows of 128 bytes,
// 128-byte swizzle, one slab behind the other.
static bool encode_x_slabs_3d(CUtensorMap* map, const void* base, uint64_t M, uint64_t d, uint32_t slabs) {
  cuuint64_t dims[3] = {64, M, d / 64};
  cuuint64_t strides[2] = {d * 2, 128};
  cuuint32_t box[3] = {64, 128, slabs};
  cuuint32_t estr[3] = {1, 1, 1};
  return g_encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box, estr,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

static inline bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }
static inline int ew_grid(int64_t items, int per_block, int sm_count) {
  int64_t blocks = (items + per_block - 1) / per_block;
  int64_t cap = (int64_t)sm_count * 16;
  return (int)(blocks < 1 ? 1 : (blocks > cap ? cap : blocks));
}
static inline torq_status launch_status() {
  g_launches.fetch_add(1, std::memory_order_relaxed);
  return cudaGetLastError() == cudaSuccess ? TORQ_OK : TORQ_ERR_LAUNCH;
}

// Launch of a persistent tensor-core kernel: `cluster` CTAs per cluster along x (1 or 2; the grid
// is a multiple of it) and programmatic stream serialization, so that the launch processing of
// this kernel overlaps the tail of the kernel before it (the kernel itself waits for that kernel
// to complete before it touches global memory).
template <typename... KArgs, typename... Args>
static void launch_tc(void (*kernel)(KArgs...), int cluster, int grid, int threads, int smem, cudaStream_t s,
                      Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid, 1, 1);
  cfg.blockDim = dim3((unsigned)threads, 1, 1);
  cfg.dynamicSmemBytes = (size_t)smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = (unsigned)cluster;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = cluster > 1 ? 2 : 1;
  cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

// What the workspace holds beyond the quantized activations: room that a rotation split over the SMs needs for its fp32
// partial tiles.  No kernel uses it any more; callers have sized and kept their workspaces by these functions.
static size_t spare_workspace_bytes(int64_t M, int64_t d) {
  const int64_t tiles = ((M + 127) / 128) * ((d + 255) / 256);
  if (2 * tiles > 160) return 0;
  int64_t s = 160 / tiles;
  s = s > 8 ? 8 : s;
  s = s > (d + 63) / 64 / 2 ? (d + 63) / 64 / 2 : s;
  return s < 2 ? 0 : (size_t)s * (size_t)((M + 127) / 128 * 128) * (size_t)d * sizeof(float);
}
constexpr int kRotFewMaxTokens = 256;    // up to here the rotation streams R_inter through the few-token kernel
constexpr int kGemmFewMaxTokens = 128;   // and the GEMM the weights
static_assert(kRotFewMaxTokens <= RotFewCfg::MAX_TOK && kGemmFewMaxTokens <= GemmFewCfg<FMT_MXFP4>::MAX_TOK, "few-token limits");
// Few-token kernels: tokens per instruction, and the cluster size S = number of K splits of one 128-feature
// tile: the largest S up to 8 within these bounds, each with both sides measured (us, cold operands):
//  * all clusters are resident at once.  `fit[S]` is what the runtime answers for one CTA per SM (148, 74, 45, 33,
//    26, 22, 15, 15: clusters do not cross GPCs); where two CTAs fit on an SM, twice that.  More in flight pays up
//    to there -- rotation d = 14336, M = 50: S = 2 (112 clusters) 63.6, S = 1 80.8; d = 7168: S = 4 (56) 20.3, S = 2
//    24.7; GEMM K = 14336, N = 6144: S = 4 (48) 11.5, S = 2 13.8 -- and a second wave costs more than it brings:
//    d = 5120, S = 7 (40, 30 fit) 20.7 against 13.5 at S = 6; d = 2048, M = 100: S = 8 (16, 15 fit) 14.1, S = 4 7.7;
//    With one CTA per SM, clusters of 5 that nearly fill the GPCs hinder the next kernel's: at 25 and 26 tiles (fit[5] = 26) S = 4
//    (d = 3328, 96 and 128 tokens: S = 5 13.7 and 12.8, S = 4 9.7 and 10.5; layer N = 3328, MXINT4, 96 tokens 22.0, GEMM K = 8192
//    N = 3200 7.7 and 7.4); clusters of 4, 6 and 8 fill them without harm.  Of 3 see fewtok_leave_together;
//  * above S = 4, at most 1.4 CTAs per SM, so that CTAs of the next kernel in the stream find room and send their
//    weight loads early (decode layer at d = N = 5120, M = 1: S = 5 17.86, S = 6 17.97, though the rotation by
//    itself is the faster one with S = 6), and `most`, so that a CTA has some K steps (the callers say how many): a longer
//    reduction has to be paid for by a shorter stream (rotation d = 2048, M = 50: S = 8 7.1, S = 4 6.5; GEMM K = 2048, N = 5120: S = 5
//    5.5, S = 4 5.1).  Above 128 tokens the reduction itself is shared out (up to 16 token groups), so there is no such bound (d = 1536:
//    S = 8 9.9, S = 4 11.3);
//  * no S above the smallest one with the same longest K range (GEMM K = 4096: S = 5 has ranges of 4 steps like S = 4).
static inline int fewtok_ntok(int64_t M) { return (int)((M + 15) / 16 * 16); }
static inline int fewtok_cluster(int64_t tiles, int64_t k_steps, int64_t most, int ctas_per_sm, int sm_count, const int* fit) {
  most = most < 4 ? 4 : (most > 8 ? 8 : most);
  int s = (int)(most < k_steps ? most : k_steps);
  while (s > 1 && (tiles > (int64_t)ctas_per_sm * fit[s] || (s > 4 && 10 * tiles * s > 14 * (int64_t)sm_count) ||
                   (s == 5 && ctas_per_sm == 1 && tiles > fit[5] - 2))) --s;
  while (s > 1 && (k_steps + s - 2) / (s - 1) == (k_steps + s - 1) / s) --s;      // fewer clusters' CTAs: they fit as well
  return s < 1 ? 1 : s;
}
// R_inter or W tiles (16 KiB) that all CTAs together ask the L2 for beyond their stages: 10 MB (us, 0 / 3 / 4 / 6 / 16 per CTA of 200,
// d = N = 5120, 1 token 14.8 / 14.3 / 14.25 / 14.4 / 15.7; of 192, 24 tokens d = 4096 NVFP4 3 / 4 / 6: 13.5 / 13.8 / 14.0; of 128, 100
// tokens d = 4096 0 / 3 / 5 / 8: 18.4 / 18.2 / 18.1 / 18.2).
constexpr int kAheadTiles = 640;
// Cluster size and stages of the few-token rotation.  65 to 128 tokens have an SM to themselves with four stages and share
// it with three.  Sharing wins where the K range of a CTA would be longer than 32 steps, that is where 148 CTAs are few for
// the tiles (us, alone / shared, 72 and 128 tokens: d = 5120, 27 steps 14.2 / 14.7 and 16.2 / 17.7; d = 6400, 50 steps 21.7 /
// 19.9 and 23.4 / 22.0; d = 8192 28.0 / 26.4 and 30.3 / 28.0; d = 11008, one CTA for each of 86 tiles 52.0 / 41.1 and 53.6 /
// 44.4; d = 14336 78 / 68 and 79 / 73).
struct FewRotation { int cluster, stages; bool push; };
static FewRotation fewtok_rotation(int64_t M, int64_t d, bool intra, const DeviceState* st) {
  const int ntok = fewtok_ntok(M);
  const int64_t tiles = d / 128, steps = d / 64;
  // Pushed partial sums make the reduction cheap: the largest cluster that leaves room for two more (push_fit: 148, 93, 71, 56, 45, 37, 33
  // clusters of 2 ... 8).  us, layers d = N, S = 4 / 6 / 8, 1 and 32 tokens: d = 1536 6.46 / 6.17 / 6.27 and 9.55 / 8.87 / 8.13, d = 2560
  // 8.29 / 7.57 / 7.23 and 10.7 / 10.35 / 9.49, d = 4096 11.2 / 10.5 / 10.6 and 14.5 / 13.6 / 12.7; without the room d = 4224 (33 tiles)
  // S = 7 / 8 11.3 / 11.8, d = 7168 (56 tiles) S = 4 / 5 23.2 / 23.6.  A fifth stage up to 16 tokens, but not on long K ranges (four /
  // five, 1 token: layer d = N = 5120 14.5 / 14.3; rotation d = 14336 59.4 / 60.7).  A rotation without R_intra keeps the clusters of the
  // rule below.  Above 32 tokens (three stages then) where clusters of eight fit, up to 56: us, layers, pulled / pushed, 40 tokens: 2048
  // -> 2048 10.65 / 10.1, 4096 -> 4096 15.85 / 15.1, 56 tokens 2560 -> 2560 13.25 / 12.15, 64 tokens 11.3 / 11.8 and 16.9 / 16.9; d =
  // 5120, S = 6, 50 tokens 19.4 / 19.8.  Above 48 from 20 tiles on (56 tokens NVFP4 2048 -> 2048 10.96 / 11.6).
  if (intra && (M <= 32 || (M <= (tiles < 20 ? 48 : RotFewCfg::PUSH_TOK) && tiles <= st->push_fit[RotFewCfg::MAX_CLUSTER] - 2))) {
    int S = (int)(steps < RotFewCfg::MAX_CLUSTER ? steps : RotFewCfg::MAX_CLUSTER);
    while (S > 1 && tiles > st->push_fit[S] - 2) --S;
    return {S, ntok > 32 ? RotFewCfg::SHARED_STAGES : (ntok <= 16 && steps <= 32 * S ? RotFewCfg::PUSH_STAGES : RotFewCfg::STAGES), true};
  }
  const int long_k = ntok > 128 ? 1 : 10, ctas = RotFewCfg::ctas_per_sm(ntok, RotFewCfg::STAGES, ntok <= 32);
  // 17 to 64 tokens: two steps less are enough for one more CTA (us, S = 4 / 5 at 48 steps, d = 3072, 24 and 64 tokens: 8.4 /
  // 7.7 and 9.8 / 9.0, the layer with N = 3072 12.7 / 11.2 and 15.1 / 14.6; S = 5 / 6 at 58, d = 3712: 9.6 / 8.9 and 11.0 / 10.6)
  int64_t most = (steps + (ntok > 16 && ntok <= 64 ? 2 : 0)) / long_k;
  // 65 to 96 tokens are five or six groups: a cluster of six, where it fits, has one unit per CTA, which pays from ranges of
  // four steps on (us, S = 4 or the one-wave kernel / S = 6, 65 and 96 tokens: d = 1536 7.4 / 6.1 and 7.4 / 6.5, MXINT4 7.6 / 6.2 and
  // 7.7 / 6.6, layer with N = 256 11.6 / 10.0 and 12.0 / 10.9; d = 2560 8.1 / 7.5 and 8.7 / 8.2).  At 23 and 24 tiles, where only five
  // fit, 96 tokens lose (d = 3072 9.3 / 9.6).
  if (ntok > 64 && ntok <= 96 && steps >= 24 && tiles <= st->few_fit[6] && most < 6) most = 6;
  const int S = fewtok_cluster(tiles, steps, most, ctas, st->sm_count, st->few_fit);
  if (ntok <= 16 && steps <= 32 * S) return {S, RotFewCfg::PUSH_STAGES, true};
  if (ctas > 1 || ntok > RotFewCfg::MAX_SHARED_TOK || steps <= 32 * S) return {S, RotFewCfg::STAGES, ntok <= 32};
  return {fewtok_cluster(tiles, steps, most, 2, st->sm_count, st->few_fit), RotFewCfg::SHARED_STAGES, false};
}
// Whether the CTAs of a cluster leave together instead of each when it has no more to do.  Alone on their SMs (65 tokens and
// more), clusters of 3 that nearly fill the GPCs (44 and 45 tiles, fit[3] = 45) hinder the clusters of the next kernel when
// they leave one by one (us, one by one / together: d = 5632, 96, 128 and 256 tokens 18.5 / 16.3, 19.1 / 18.0 and 28.1 / 22.9, layer
// with N = 256 and 256 tokens 36.0 / 29.9, with N = 5632 and 96 tokens 25.1 / 24.3; d = 5760 MXINT4, N = 5760, 128 tokens 35.1 /
// 31.9; only 129 tokens and more with many outputs lose, 31.1 / 31.8); elsewhere leaving early is the better (d = 4096, 96 tokens
// 11.1 / 11.8).
static bool fewtok_leave_together(int64_t M, int64_t tiles, FewRotation few, const DeviceState* st) {
  return M > 64 && few.stages == RotFewCfg::STAGES && few.cluster == 3 && tiles > st->few_fit[3] - 2;
}
// Cluster size of the few-token GEMM whose sums are pulled (17 tokens and more): above S = 4 three K steps per CTA, or two while the
// partial sums of all CTAs are few: 32 tokens per SM (us, S = 4 / 8, 17 and 64 tokens: N = 256, K = 4096 3.44 / 2.99 and 4.33 / 3.92,
// N = 1024 3.58 / 3.20 and 4.60 / 4.34; S = 4 / 6: 17 tokens N = 2048 3.75 / 3.47; beyond the line 64 tokens N = 2048 NVFP4 4.53 / 4.70).
static int fewtok_gemm_cluster(int ntok, int64_t tiles, int64_t steps, int ctas, const DeviceState* st) {
  const int S = fewtok_cluster(tiles, steps, steps / 2, ctas, st->sm_count, st->few_fit);
  if (tiles * S * ntok <= 32 * (int64_t)st->sm_count) return S;
  return fewtok_cluster(tiles, steps, steps / 3, ctas, st->sm_count, st->few_fit);
}
// Where the sums are pushed (M tokens), from the largest cluster down: above four CTAs where each keeps four K steps and has its SM to
// itself (a CTA's instructions wait for those of the other one on its SM), or with five and more steps; up to four where they have their
// SMs to themselves (a tenth may share), or with more than five steps.  us, layers, S = 3 / 4 / 5 / 8: 8 x 5120 -> 5120 (20 steps) 15.35
// / 14.5 / 15.0 / 15.2, 16 x 4096 -> 1024 (16) 12.0 / 10.0 / 10.2 / 10.8, 16 x 2048 -> 6144 (8) 8.06 / 8.36, 8 x 8192 -> 2048 (32) 28.0 /
// 27.1 / 26.4 / 24.4, 16 x 7168 -> 4096 (28), S = 4 / 6 23.25 / 22.3, 16 x 5120 -> 8192, S = 3 / 4 16.5 / 17.1; up to 4 tokens sharing
// costs less (1 x 5120 -> 5120 S = 4 / 5 14.4 / 14.3).  One or two steps are not split (16 tokens, N = 4096, K = 512 2.97 / 2.56; above
// 16 tokens there are nine and more).  Few tiles take as many CTAs as have two steps, while the sums are few as above, up to 16 tokens 8
// tokens per SM (us, S = 4 / 8: 1 token N = 256 2.96 / 2.58, N = 1024 3.10 / 2.82, the layer 11.2 / 10.9; beyond: N = 2048 the GEMM 3.62
// / 3.51, the layer of 16 tokens 13.2 / 13.5; S = 4 / 5 at K = 2560, N = 5120 the layer 11.0 / 11.5).
static int push_gemm_cluster(int64_t M, int64_t tiles, int64_t steps, const DeviceState* st) {
  if (steps >= 8) {
    const int S = fewtok_cluster(tiles, steps, steps / 2, 2, st->sm_count, st->few_fit);
    if (tiles * S * fewtok_ntok(M) <= (M > 16 ? 32 : 8) * (int64_t)st->sm_count) return S;
  }
  if (steps <= 2) return 1;
  for (int S = GemmFewCfg<>::MAX_CLUSTER; S > 1; --S) {
    if (S > steps || tiles > st->push_fit[S]) continue;
    const bool alone = 10 * tiles * S <= 11 * (int64_t)st->sm_count;
    if (S > 4 ? (steps >= 4 * S && (alone || M <= 4)) || 2 * steps >= 9 * S : alone || steps > 5 * S) {
      while (S > 1 && (steps + S - 2) / (S - 1) == (steps + S - 1) / S) --S;
      return S;
    }
  }
  return 1;
}
constexpr int kTailTiles = 8;              // a last wave of up to so many tiles leaves the pair rotation (below)
// A 192-column tile against a 256-column one: an instruction takes the larger of N / 2 cycles and 64 + N / 4, the reading of its A and B
// slices from shared memory (112 and 128 cycles; the bare loop of loads and instructions runs at 448 and 512 per K step).
constexpr double kNarrowTileCost = 0.88;

// Tile list of a pair kernel: `rows` 256-row tiles by `cols` columns on `max_pairs` CTA pairs, tiles dealt
// round robin.  When the 256-column tiles do not fill the last wave, trading three of them for four 192-column
// tiles (one unit) in some row tiles shortens that wave from one tile time to about three quarters.  The number
// of units is the one with the smallest longest-pair time, a narrow tile counted as `narrow_cost` wide tiles;
// zero unless it wins by at least 1 % (and always zero when the columns are not whole 256-column tiles).
static MixedTiles plan_pair_tiles(int rows, int64_t cols, int max_pairs, double narrow_cost) {
  const int wide_cols = (int)((cols + 255) / 256);
  if (cols % 256 != 0 || rows < 1) return mixed_tiles_make(rows < 1 ? 1 : rows, wide_cols, 0);
  struct Memo { int rows, wide_cols, max_pairs; double cost; int units; };
  static thread_local Memo memo[8] = {};
  static thread_local int memo_next = 0;
  for (const Memo& m : memo)
    if (m.rows == rows && m.wide_cols == wide_cols && m.max_pairs == max_pairs && m.cost == narrow_cost)
      return mixed_tiles_make(rows, wide_cols, m.units);
  auto longest = [&](int units) {
    const int wide = rows * wide_cols - 3 * units, narrow = 4 * units;
    const int P = wide + narrow < max_pairs ? wide + narrow : max_pairs;
    double worst = 0.0;
    for (int p = 0; p < P; ++p) {
      const int w = wide / P + (p < wide % P ? 1 : 0);
      // narrow tiles have the numbers wide .. wide + narrow - 1; pair p takes those congruent to p
      const int first = wide + ((p - wide) % P + P) % P;
      const int n = first < wide + narrow ? (wide + narrow - 1 - first) / P + 1 : 0;
      const double t = w + narrow_cost * n;
      if (t > worst) worst = t;
    }
    return worst;
  };
  const int max_units = rows * (wide_cols / 3);
  const double base = longest(0);
  double best = base;
  int best_units = 0;
  for (int u = 1; u <= max_units && 4 * u <= max_pairs + 8; ++u) {
    // the row tiles that trade one unit more must have the three wide tiles to give
    if (u % rows != 0 && 3 * (u / rows + 1) > wide_cols) break;
    const double t = longest(u);
    if (t < best - 1e-9) { best = t; best_units = u; }
  }
  if (best > 0.99 * base) best_units = 0;
  memo[memo_next] = Memo{rows, wide_cols, max_pairs, narrow_cost, best_units};
  memo_next = (memo_next + 1) % 8;
  return mixed_tiles_make(rows, wide_cols, best_units);
}

// The list of a GEMM whose weights have rows of `w_row_bytes`.  Every group of row tiles reads all of W once: many columns in groups of
// sixteen.  A long call runs at the power cap, where the traffic that this saves is clock, so loops of 0.9 s on each side in turn
// (us, eight / sixteen): 8192 x 51200, K = 5120 838 / 819, x 28672, K = 4096 388 / 378, x 14336 196 / 192, MXINT4 361 / 355, NVFP4 211 /
// 207, 4096 x 16384, K = 2048 69.1 / 68.6, 4096 x 10240, K = 8192 133 / 130, 8192 x 10240, K = 4096 139.3 / 139.0, x 8192, K = 8192 215.0 /
// 213.4.  Fewer columns or smaller weights lose: x 9216, K = 4096 125.0 / 125.3, 4500 x 8448 66.7 / 67.3, 8192 x 4096, K = 14336 179 /
// 181, x 28672, K = 256 102 / 103; the rotation loses too (d = 14336, 8192 tokens, the layer 2886 / 3062).
static MixedTiles plan_gemm_tiles(int64_t M, int64_t N, uint64_t w_row_bytes, int max_pairs) {
  MixedTiles t = plan_pair_tiles((int)((M + 255) / 256), N, max_pairs, kNarrowTileCost);
  if (N >= 8192 && (uint64_t)N * w_row_bytes >= (N >= 10240 ? 16u << 20 : 32u << 20)) t.group = 16;
  return t;
}

static int64_t write_tile_list(const MixedTiles& t, int32_t* out, int64_t cap) {
  for (int i = 0; out && i < t.total && i < cap; ++i) {
    int mp, col0;
    bool narrow;
    mixed_tile_coords(i, t, mp, col0, narrow);
    out[3 * i] = mp;
    out[3 * i + 1] = col0;
    out[3 * i + 2] = narrow ? kNarrowCols : 256;
  }
  return t.total;
}

static size_t quantized_bytes(int64_t M, int64_t d) {    // codes, then 256-byte aligned the scales
  return ((size_t)M * (size_t)(d / 2) + 255) / 256 * 256 + torq_scales_bytes(M, d);
}

static torq_status quantize_impl(DeviceState* st, const void* Z, torq_dtype dt, int64_t M, int64_t d,
                                 void* codes, void* scales, cudaStream_t s) {
  const int64_t kb4 = (d / 32 + 3) / 4;
  const int64_t items = ((M + 127) / 128 * 128) * ((kb4 * 128 + 255) / 256);   // warps
  const int grid = ew_grid(items, 8, st->sm_count);
  if (dt == TORQ_F32)
    quantize_kernel<float><<<grid, 256, 0, s>>>(static_cast<const float*>(Z), M, d,
                                                static_cast<uint8_t*>(codes), static_cast<uint8_t*>(scales));
  else
    quantize_kernel<__nv_bfloat16><<<grid, 256, 0, s>>>(static_cast<const __nv_bfloat16*>(Z), M, d,
                                                        static_cast<uint8_t*>(codes),
                                                        static_cast<uint8_t*>(scales));
  return launch_status();
}

}  // namespace torq

using namespace torq;

extern "C" {

size_t torq_scales_bytes(int64_t rows, int64_t k) {
  if (rows <= 0 || k <= 0) return 0;
  return (size_t)((rows + 127) / 128) * (size_t)((k / 32 + 3) / 4) * 512;
}

size_t torq_scale_offset(int64_t row, int64_t kblock, int64_t k) {
  return scale_offset(row, kblock, (k / 32 + 3) / 4);
}

size_t torq_workspace_bytes(int64_t M, int64_t d, int64_t N) {
  (void)N;
  if (M <= 0 || d <= 0) return 0;
  return quantized_bytes(M, d) + spare_workspace_bytes(M, d);
}

const char* torq_status_string(torq_status s) {
  switch (s) {
    case TORQ_OK: return "ok";
    case TORQ_ERR_NULL: return "null pointer";
    case TORQ_ERR_SHAPE: return "unsupported shape";
    case TORQ_ERR_ALIGN: return "pointer not 16-byte aligned";
    case TORQ_ERR_ARCH: return "device is not compute capability 10.x";
    case TORQ_ERR_LAUNCH: return "CUDA launch or descriptor error";
    case TORQ_ERR_TIMEOUT: return "a bounded device wait ran out";
    case TORQ_ERR_WORKSPACE: return "workspace missing or too small";
  }
  return "unknown";
}

int64_t torq_pair_tile_list(int64_t rows, int64_t cols, int32_t pairs, int32_t* out, int64_t cap) {
  if (rows < 1 || cols < 1 || pairs < 1 || rows > INT32_MAX / 2 || cols > INT32_MAX / 2) return -1;
  return write_tile_list(plan_pair_tiles((int)((rows + 255) / 256), cols, pairs, kNarrowTileCost), out, cap);
}

int64_t torq_gemm_tile_list(int64_t M, int64_t N, int64_t w_row_bytes, int32_t pairs, int32_t* out, int64_t cap) {
  if (M < 1 || N < 1 || w_row_bytes < 1 || pairs < 1 || M > INT32_MAX / 2 || N > INT32_MAX / 2 || w_row_bytes > INT32_MAX) return -1;
  return write_tile_list(plan_gemm_tiles(M, N, (uint64_t)w_row_bytes, pairs), out, cap);
}

int64_t torq_launch_count(void) { return g_launches.load(std::memory_order_relaxed); }

int torq_last_device_error(void* stream) {
  DeviceState* st = device_state();
  if (!st || !st->arch_ok) return 0;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if (cudaStreamSynchronize(s) != cudaSuccess) return TORQ_ERR_LAUNCH;
  int v = 0, zero = 0;
  if (cudaMemcpy(&v, st->err_word, sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess)
    return TORQ_ERR_LAUNCH;
  if (v != 0) cudaMemcpy(st->err_word, &zero, sizeof(int), cudaMemcpyHostToDevice);
  return v;
}

torq_status torq_quantize_mxfp4(const void* Z, torq_dtype z_dtype, int64_t M, int64_t d,
                                void* out_codes, void* out_scales, void* stream) {
  if (!Z || !out_codes || !out_scales) return TORQ_ERR_NULL;
  if (M < 1 || d < 32 || d % 32 != 0 || M > (1 << 30) || d > (1 << 30)) return TORQ_ERR_SHAPE;
  if (z_dtype != TORQ_F32 && z_dtype != TORQ_BF16) return TORQ_ERR_SHAPE;
  if (!aligned16(Z) || !aligned16(out_codes) || !aligned16(out_scales)) return TORQ_ERR_ALIGN;
  DeviceState* st = device_state();
  if (!st) return TORQ_ERR_LAUNCH;
  if (!st->arch_ok) return TORQ_ERR_ARCH;
  return quantize_impl(st, Z, z_dtype, M, d, out_codes, out_scales, static_cast<cudaStream_t>(stream));
}

// Width of the one-wave rotation's tiles, or 0 where another kernel is faster.  Times in us: once a fit to the rotation alone, since
// moved where both kernels were measured on either side of a line, so they say which kernel is the faster and not how long it takes.
// Of 202 rotations (d = 128 ... 14336, 1 to 4000 tokens, operands from HBM) these tiles are rated 7 % off in the median, a quarter low
// where a call runs at the power cap or d is above 8192; the few-token kernel is rated up to half low from d = 3072 on, where R_inter's
// stream sets its pace, and the pair kernel a quarter low at the power cap.  177 of them can run on either: 13 take the slower one,
// 300 x 6144 35.0 / 29.9, the others by up to 8 % (1 x 128 2.67 / 2.48, 777 x 3072 18.8 / 17.8, 777 x 4096 30.0 / 28.6).  f = filled part
// of a wave:
//  * here: 1.8 + 0.0155 per column (2 + 0.025 above 256 columns, 1.6 + 0.0155 up to 128) for launch and epilogue, from 177 to 256
//    tokens 1.6 + 0.022 (2 + 0.032, 1.4 + 0.022), what they were with warp-level instructions: the few-token kernel contracts K in
//    parts, which these tiles do in one accumulator, and a line that follows the shorter epilogue gives up precision for its 2 to 10 %
//    (codes that differ from those of 64-bit arithmetic, few tokens / here: 220 x 5504 6 / 51 of 1.2 M; layers with N = d 180 x 3072
//    18.5 / 16.7, 245 x 4096 22.85 / 21.6, 204 x 5120 27.2 / 28.15).  Then per K step of 64 the operand bytes, 0.17 +
//    0.0003 per column + 0.03 f (up to 128 columns, where a stage is two of these steps, 0.145 + 0.0003 per column + 0.035 f, but from d
//    = 6272 on, where R_inter's stream sets the pace), or the math, 0.00114 per column;
//  * few tokens: 3.1 / 4.4 / 5.6 up to 16 / 64 / 128 tokens, plus 0.22 / 0.2 / 0.36 per K step of the longest split; above, 6.4 (5.9 up
//    to 176 tokens: 160 x 2816 15.2 / 16.05 as layers) at 144 tokens and 0.025 per token more, 0.5 per CTA of a cluster above four, 0.42
//    per K step (us, few tokens / here: 144 tokens d = 2560 9.7 / 10.4, d = 4096 13.6 / 14.9; 208 d = 2560 12.6 / 10.4, d = 4096 15.0 /
//    15.0 (the layer with N = 6144 22.7 / 23.2), d = 5120 19.5 / 20.1; 256 d = 4096 16.2 / 15.1, d = 5120 20.9 / 20.0; 128 d = 2048 8.1 /
//    7.6).  Beside clusters of six (d = 2048 ... 2816, up to 192 tokens) this is a microsecond more than they take with cold operands,
//    and the line lies between what cold ones and an R_inter in the L2 ask for (layers with N = d, few tokens / here: 144 x 2432 cold
//    0.95 of the time, in the L2 1.11; 152 x 2560 0.93 and 1.09, 176 x 2560 0.97 and 1.11, 176 x 2816 0.97 and 1.06, 112 x 2176 0.95 and
//    1.04);
//  * few tokens whose sums are pushed: 2.7 + 0.22 per K step + 0.025 per token, 0.04 above 32 tokens (us, here / few tokens, 1, 16 and 32
//    tokens: d = 256 2.95 / 2.96, 2.95 / 3.21, 2.95 / 4.49; d = 512 3.97 / 3.08, 3.37 / 3.21, 3.46 / 3.60; d = 768 5.25 / 3.21, 4.24 /
//    3.37, 4.36 / 3.85);
//  * above 192 tokens a cluster of three has five units for its first CTA: 0.6 more (216 d = 4864 19.3 / 18.2);
//  * above d = 6144, where these tiles take up to 3 us less than the figures say: 7.0 up to 176 tokens, 7.6 up to 192, 10.5 above, 0.42
//    per K step (144 d = 6912 26.9 / 25.4, 150 d = 7040 28.2 / 26.3, 208 d = 7680 33.1 / 30.0);
//  * pair kernel: 6.8, plus per K step 0.32 for a wave and 0.2 + 0.14 f for the last, partly filled one (layers with N = d at 40 sizes
//    beside the line, 1772 to 4076 tokens, pair kernel / here: 0.99 to 1.6 of the time; 2540 x 2048 36.2 / 30.9, 2028 x 2048 25.3 / 25.05).
// The other formats follow the same figures, which were not fitted to them; wide_gemm_width says how that was checked.
// From 2048 x 4096 on a layer fills the pair kernel's waves and stays there: one-wave tiles would be wider than 384 columns (2048 x 4096
// measured 51.6 with 480 columns, 46.8 in the pair kernel).
static int wide_rotation_width(int64_t M, int64_t d, int few_steps, int few_S, bool push, int max_pairs) {
  const int64_t rows = (M + 255) / 256, steps = d / 64;
  // The line of 65 to 96 tokens, clusters of six, stays where it was, and so does that of an X below 128 KiB (up to 64 tokens; with
  // more, an X so small has a d that comes here by either figures), which these tiles read more slowly for a reason not found (us, few
  // tokens / here: d = 1024 63 tokens 5.7 / 5.8, 64 tokens 5.7 / 4.5; d = 1152 56 5.6 / 5.7, 60 5.7 / 4.7; d = 1536 40 5.9 / 9.3, 48
  // 6.0 / 5.6).
  const bool two_slabs = d <= 6144 && (M > 96 || (M <= 64 && M * d >= 65536));
  const bool against_parts = M > 176 && M <= kRotFewMaxTokens;
  const double column = against_parts ? 0.022 : 0.0155, column_wide = against_parts ? 0.032 : 0.025, fixed = against_parts ? 1.6 : 1.8;
  double best = 1e30;
  int width = 0;
  for (int w = 32; w <= RotWideCfg::MAX_WIDTH; w += 32) {
    if (rows * ((d + w - 1) / w) > max_pairs) continue;
    const double f = (double)(rows * ((d + w - 1) / w)) / max_pairs;
    const double bytes = (w <= 128 && two_slabs ? 0.145 + 0.035 * f : 0.17 + 0.03 * f) + 0.0003 * w, math = 0.00114 * w;
    const double ends = w > 256 ? 2.0 + column_wide * w : fixed - (w <= 128 && two_slabs ? 0.2 : 0.0) + column * w;
    const double t = ends + (double)steps * (bytes > math ? bytes : math);
    if (t < best) { best = t; width = w; }
  }
  double other;
  if (M <= kRotFewMaxTokens) {
    if (push) other = 2.7 + 0.22 * few_steps + (M <= 32 ? 0.025 : 0.04) * (double)M;
    else if (M <= 16) other = 3.1 + 0.22 * few_steps;
    else if (M <= 64) other = 4.4 + 0.2 * few_steps;
    else if (M <= 128) other = 5.6 + 0.36 * few_steps;
    else if (d > 6144) other = (M <= 176 ? 7.0 : (M <= 192 ? 7.6 : 10.5)) + 0.42 * few_steps;
    else other = (M <= 176 ? 5.9 : 6.4) + 0.025 * (double)(M - 144) + 0.42 * few_steps +
                 (few_S > 4 ? 0.5 * (few_S - 4) : (few_S == 3 && M > 192 ? 0.6 : 0.0));
  } else {
    const int64_t tiles = rows * ((d + 255) / 256);
    const int64_t full = tiles / max_pairs, rest = tiles % max_pairs;
    other = 6.8 + (double)steps * (0.32 * (double)full + (rest == 0 ? 0.0 : (full == 0 ? 0.32 : 0.2 + 0.14 * (double)rest / max_pairs)));
  }
  return best < 0.97 * other ? width : 0;
}

static torq_status rotate_wide(DeviceState* st, int fmt, const void* X, const void* R_inter, const void* R_intra, int64_t M,
                               int64_t d, uint8_t* codes, uint8_t* scales, float tensor_scale, int width, cudaStream_t s) {
  using C = RotWideCfg;
  CUtensorMap tmX, tmR, tmRt;
  const int tail = C::tail_cols(width);
  const uint32_t bk = (uint32_t)C::bk(width);
  if (!encode_x_slabs_3d(&tmX, X, (uint64_t)M, (uint64_t)d, bk / C::SLAB) ||
      !encode_2d(&tmR, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, R_inter, (uint64_t)d, (uint64_t)d, bk, 64) ||
      (tail && !encode_2d(&tmRt, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, R_inter, (uint64_t)d, (uint64_t)d, bk, (uint32_t)tail)))
    return TORQ_ERR_LAUNCH;
  if (!tail) tmRt = tmR;
  const int rows = (int)((M + 255) / 256), cols = (int)((d + width - 1) / width);
  auto launch = [&](auto format) {
    constexpr int F = decltype(format)::value;
    launch_tc(width > 256   ? rotate_quantize_wide_kernel<F, 384>
              : width > 128 ? rotate_quantize_wide_kernel<F, 256>
              : width > 32  ? rotate_quantize_wide_kernel<F, 128>
                            : rotate_quantize_wide_kernel<F, 32>,
              2, 2 * rows * cols, C::THREADS, C::smem_bytes(width), s, tmX, tmR, tmRt, static_cast<const __nv_bfloat16*>(R_intra),
              codes, scales, (int)M, (int)d, tensor_scale, rows, width, st->err_word);
  };
  if (fmt == FMT_MXINT4) launch(std::integral_constant<int, FMT_MXINT4>{});
  else if (fmt == FMT_NVFP4) launch(std::integral_constant<int, FMT_NVFP4>{});
  else launch(std::integral_constant<int, FMT_MXFP4>{});
  return launch_status();
}

// Few tokens: 128 features x all tokens per CTA, K split over a cluster, reduced through distributed shared memory; one
// launch, no scratch.  Feature tiles [ft0, ft0 + tiles) of all d / 128.
static torq_status rotate_fewtok(DeviceState* st, int fmt, const void* X, const void* R_inter, const void* R_intra, int64_t M,
                                 int64_t d, int ft0, int tiles, FewRotation few, uint8_t* codes, uint8_t* scales,
                                 float tensor_scale, cudaStream_t s) {
  CUtensorMap tmX, tmR;
  const int ntok = fewtok_ntok(M), S = few.cluster;
  if (!encode_2d(&tmX, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, X, (uint64_t)M, (uint64_t)d, (uint32_t)ntok, 64) ||
      !encode_2d(&tmR, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, R_inter, (uint64_t)d, (uint64_t)d, 64, 64))
    return TORQ_ERR_LAUNCH;
  const int smem = RotFewCfg::smem_bytes(ntok, few.stages, few.push);
  const float ts = fmt == FMT_NVFP4 ? tensor_scale : 0.0f;
  const __nv_bfloat16* ri = static_cast<const __nv_bfloat16*>(R_intra);
  // sums pushed, with five, four or three stages; pulled, two CTAs per SM: one set of epilogue warps; one CTA: two sets
  const bool share = few.stages == RotFewCfg::SHARED_STAGES, small = few.push || share || ntok <= 64;
  auto launch = [&](auto format) {
    constexpr int F = decltype(format)::value, P = RotFewCfg::PUSH_STAGES, NS = RotFewCfg::SHARED_STAGES;
    launch_tc(few.push ? (few.stages == P ? rotate_fewtok_kernel<F, 1, true, P>
                          : share         ? rotate_fewtok_kernel<F, 1, true, NS>
                                          : rotate_fewtok_kernel<F, 1, true>)
              : share  ? rotate_fewtok_kernel<F, 1, false, NS>
              : small  ? rotate_fewtok_kernel<F, 1>
                       : rotate_fewtok_kernel<F, 2>,
              S, tiles * S, small ? 192 : 320, smem, s, tmX, tmR, ri, codes, scales, (int)M, (int)d, ntok, S, ft0,
              fewtok_leave_together(M, tiles, few, st) ? 1 : 0, kAheadTiles / (tiles * S), ts, st->err_word);
  };
  if (fmt == FMT_MXINT4) launch(std::integral_constant<int, FMT_MXINT4>{});
  else if (fmt == FMT_NVFP4) launch(std::integral_constant<int, FMT_NVFP4>{});
  else launch(std::integral_constant<int, FMT_MXFP4>{});
  return launch_status();
}

// Steps 1-4.  `fmt` FMT_NVFP4 (with its tensor scale) needs R_inter.
// FMT_F32OUT: out_codes is float32 [M, d] and receives the rotated values (out_scales unused, may be
// NULL); `x_terms` > 1: X is [M, x_terms * d], the sum of its d-wide column groups is what is rotated.
static torq_status rotate_quantize_impl(const void* X, const void* R_inter, const void* R_intra, int64_t M,
                                        int64_t d, void* out_codes, void* out_scales, void* stream,
                                        int fmt = FMT_MXFP4, float tensor_scale = 0.0f, int x_terms = 1) {
  if (!X || !out_codes || (!out_scales && fmt != FMT_F32OUT)) return TORQ_ERR_NULL;
  if (fmt != FMT_MXFP4 && !R_inter) return TORQ_ERR_NULL;
  if (M < 1 || d < 32 || d % 32 != 0 || M > (1 << 30) || d > (1 << 24)) return TORQ_ERR_SHAPE;
  if (x_terms < 1 || x_terms > 4 || (x_terms > 1 && d % 64 != 0)) return TORQ_ERR_SHAPE;
  if (!aligned16(X) || !aligned16(out_codes) || (out_scales && !aligned16(out_scales)) ||
      (R_inter && !aligned16(R_inter)) || (R_intra && !aligned16(R_intra)))
    return TORQ_ERR_ALIGN;
  DeviceState* st = device_state();
  if (!st) return TORQ_ERR_LAUNCH;
  if (!st->arch_ok) return TORQ_ERR_ARCH;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  uint8_t* codes = static_cast<uint8_t*>(out_codes);
  uint8_t* scales = static_cast<uint8_t*>(out_scales);
  if (!R_inter) {
    if (!R_intra) return quantize_impl(st, X, TORQ_BF16, M, d, codes, scales, s);
    const int64_t items = ((M + 127) / 128 * 128) * (((d / 32 + 3) / 4) * 4);
    intra_quantize_kernel<<<ew_grid(items, 128, st->sm_count), 128, 0, s>>>(
        static_cast<const __nv_bfloat16*>(X), static_cast<const __nv_bfloat16*>(R_intra), M, d, codes,
        scales);
    return launch_status();
  }
  CUtensorMap tmX, tmR;
  if (d % 128 == 0 && x_terms == 1 && fmt != FMT_F32OUT) {
    int few_steps = 0;                                     // longest K range of the few-token kernel
    FewRotation few = {0, 0, false};
    if (M <= kRotFewMaxTokens) {
      few = fewtok_rotation(M, d, R_intra != nullptr, st);
      few_steps = (int)((d / 64 + few.cluster - 1) / few.cluster);
    }
    const int width = wide_rotation_width(M, d, few_steps, few.cluster, few.push && R_intra != nullptr, st->rot_pairs);
    if (width > 0) return rotate_wide(st, fmt, X, R_inter, R_intra, M, d, codes, scales, tensor_scale, width, s);
  }
  if (M <= kRotFewMaxTokens && d % 128 == 0 && x_terms == 1 && fmt != FMT_F32OUT)
    return rotate_fewtok(st, fmt, X, R_inter, R_intra, M, d, 0, (int)(d / 128), fewtok_rotation(M, d, R_intra != nullptr, st), codes,
                         scales, tensor_scale, s);
  if (!encode_2d(&tmX, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, X, (uint64_t)M, (uint64_t)d * x_terms, 128, 64) ||
      !encode_2d(&tmR, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, R_inter, (uint64_t)d, (uint64_t)d, 64, 64))
    return TORQ_ERR_LAUNCH;
  if (M > 128) {
    // CTA pairs: 256 x 256 tiles (the last wave 256 x 192 where that fills it better), one pair per two SMs.
    const int max_pairs = st->rot_pairs;
    CUtensorMap tmRn;                                      // second half of a narrow tile's 96 columns per CTA
    if (!encode_2d(&tmRn, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, R_inter, (uint64_t)d, (uint64_t)d, 64, 32))
      return TORQ_ERR_LAUNCH;
    MixedTiles tiles = plan_pair_tiles((int)((M + 255) / 256), d, max_pairs, kNarrowTileCost);
    // A last wave of a few tiles: the last `rest` column tiles of the first 256 tokens go to the few-token kernel instead, whose
    // K split puts up to 8 CTAs on each 128 features.  That is worth its launch where a wave is long (us, one list of tiles /
    // with this: 2048 x 14336 667 / 618 (the layer with N = 4096 686 / 658, again 723 / 671, a second copy of either side within
    // 0.4 %), 2048 x 4864 87.4 / 82.7, 2304 x 4352 77.5 / 75.1, 1024 x 9984 179 / 158, 4096 x 14336 1301 / 1249; and not up to d =
    // 4096: 3584 x 4096 85.9 / 86.0, 3328 x 3072 51.7 / 52.6).
    const int rest = (int)((M + 255) / 256 * (d / 256) % max_pairs), full = (int)((M + 255) / 256 * (d / 256) / max_pairs);
    if (full >= 2 && rest > 0 && rest <= kTailTiles && rest <= d / 256 - 1 && d > 4096 && d % 256 == 0 && x_terms == 1 && fmt != FMT_F32OUT) {
      tiles = mixed_tiles_make((int)((M + 255) / 256), (int)(d / 256), 0);
      tiles.rows_a = 1;
      tiles.less = rest;
      tiles.total -= rest;
      const int S = fewtok_cluster(2 * rest, d / 64, d / 64, 1, st->sm_count, st->few_fit);
      const torq_status rc = rotate_fewtok(st, fmt, X, R_inter, R_intra, 256, d, (int)(d / 128) - 2 * rest, 2 * rest,
                                           {S, RotFewCfg::STAGES, false}, codes, scales, tensor_scale, s);
      if (rc != TORQ_OK) return rc;
    }
    const int pairs = tiles.total < max_pairs ? tiles.total : max_pairs;
    if (fmt == FMT_MXINT4)
      launch_tc(rotate_quantize_pair_kernel<FMT_MXINT4>, 2, 2 * pairs, RotPairCfg::THREADS, RotPairCfg::SMEM_BYTES,
                s, tmX, tmR, tmRn, static_cast<const __nv_bfloat16*>(R_intra), codes, scales, (int)M, (int)d, 0.0f,
                x_terms, tiles, st->err_word);
    else if (fmt == FMT_NVFP4)
      launch_tc(rotate_quantize_pair_kernel<FMT_NVFP4>, 2, 2 * pairs, RotPairCfg::THREADS, RotPairCfg::SMEM_BYTES,
                s, tmX, tmR, tmRn, static_cast<const __nv_bfloat16*>(R_intra), codes, scales, (int)M, (int)d,
                tensor_scale, x_terms, tiles, st->err_word);
    else if (fmt == FMT_F32OUT)
      launch_tc(rotate_quantize_pair_kernel<FMT_F32OUT>, 2, 2 * pairs, RotPairCfg::THREADS, RotPairCfg::SMEM_BYTES,
                s, tmX, tmR, tmRn, static_cast<const __nv_bfloat16*>(R_intra), codes, scales, (int)M, (int)d, 0.0f,
                x_terms, tiles, st->err_word);
    else
      launch_tc(rotate_quantize_pair_kernel<FMT_MXFP4>, 2, 2 * pairs, RotPairCfg::THREADS, RotPairCfg::SMEM_BYTES,
                s, tmX, tmR, tmRn, static_cast<const __nv_bfloat16*>(R_intra), codes, scales, (int)M, (int)d, 0.0f,
                x_terms, tiles, st->err_word);
    return launch_status();
  }
  const int m_tiles = (int)((M + 127) / 128);
  const int tiles = m_tiles * (int)((d + 255) / 256);
  const int grid = tiles < st->sm_count ? tiles : st->sm_count;
  if (fmt == FMT_MXINT4)
    launch_tc(rotate_quantize_kernel<256, FMT_MXINT4>, 1, grid, RotCfg<256>::THREADS, RotCfg<256>::SMEM_BYTES, s,
              tmX, tmR, static_cast<const __nv_bfloat16*>(R_intra), codes, scales, (int)M, (int)d, 0.0f,
              x_terms, st->err_word);
  else if (fmt == FMT_NVFP4)
    launch_tc(rotate_quantize_kernel<256, FMT_NVFP4>, 1, grid, RotCfg<256>::THREADS, RotCfg<256>::SMEM_BYTES, s,
              tmX, tmR, static_cast<const __nv_bfloat16*>(R_intra), codes, scales, (int)M, (int)d, tensor_scale,
              x_terms, st->err_word);
  else if (fmt == FMT_F32OUT)
    launch_tc(rotate_quantize_kernel<256, FMT_F32OUT>, 1, grid, RotCfg<256>::THREADS, RotCfg<256>::SMEM_BYTES, s,
              tmX, tmR, static_cast<const __nv_bfloat16*>(R_intra), codes, scales, (int)M, (int)d, 0.0f,
              x_terms, st->err_word);
  else
    launch_tc(rotate_quantize_kernel<256>, 1, grid, RotCfg<256>::THREADS, RotCfg<256>::SMEM_BYTES, s, tmX, tmR,
              static_cast<const __nv_bfloat16*>(R_intra), codes, scales, (int)M, (int)d, 0.0f, x_terms,
              st->err_word);
  return launch_status();
}

torq_status torq_rotate_quantize(const void* X, const void* R_inter, const void* R_intra, int64_t M,
                                 int64_t d, void* out_codes, void* out_scales, void* stream) {
  return rotate_quantize_impl(X, R_inter, R_intra, M, d, out_codes, out_scales, stream);
}

static torq_status rotate_structured_impl(const void* X, const void* R_B, const void* R_intra, int64_t M, int64_t d,
                                          void* out_codes, void* out_scales, void* stream, int fmt,
                                          float tensor_scale) {
  if (!X || !R_B || !out_codes || !out_scales) return TORQ_ERR_NULL;
  if (M < 1 || d < 256 || d % 256 != 0 || M > (1 << 30) || d > (1 << 24)) return TORQ_ERR_SHAPE;
  if (!aligned16(X) || !aligned16(R_B) || !aligned16(out_codes) || !aligned16(out_scales) ||
      (R_intra && !aligned16(R_intra)))
    return TORQ_ERR_ALIGN;
  DeviceState* st = device_state();
  if (!st) return TORQ_ERR_LAUNCH;
  if (!st->arch_ok) return TORQ_ERR_ARCH;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const int64_t nb = d / 32;
  CUtensorMap tmRB, tmX3;
  if (!encode_2d(&tmRB, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, R_B, (uint64_t)nb, (uint64_t)nb, 128, 64) ||
      !encode_x_blocks_3d(&tmX3, X, (uint64_t)M, (uint64_t)d))
    return TORQ_ERR_LAUNCH;
  const int64_t tiles = ((nb + 127) / 128) * ((M + RotStructCfg::TOK - 1) / RotStructCfg::TOK);
  // Where a CTA can keep its rows of R_B, the grid is a multiple of the tiles that have others; where they do not fit (d >
  // 14336) they are loaded for every tile anyway and every SM works (d = 24576: 148 CTAs, as a multiple 144).
  const int64_t b_tiles = (nb + 127) / 128, k_slabs = (nb + RotStructCfg::BK - 1) / RotStructCfg::BK;
  const int64_t most = k_slabs <= RotStructCfg::RB_SLABS ? st->sm_count / b_tiles * b_tiles : st->sm_count;
  const int grid = (int)(tiles < most ? tiles : most);
  if (fmt == FMT_MXINT4)
    launch_tc(rotate_structured_kernel<FMT_MXINT4>, 1, grid, RotStructCfg::THREADS, RotStructCfg::SMEM_BYTES, s, tmRB,
              tmX3, static_cast<const __nv_bfloat16*>(R_B), static_cast<const __nv_bfloat16*>(R_intra), static_cast<uint8_t*>(out_codes),
              static_cast<uint8_t*>(out_scales), (int)M, (int)d, 0.0f, st->err_word);
  else if (fmt == FMT_NVFP4)
    launch_tc(rotate_structured_kernel<FMT_NVFP4>, 1, grid, RotStructCfg::THREADS, RotStructCfg::SMEM_BYTES, s, tmRB,
              tmX3, static_cast<const __nv_bfloat16*>(R_B), static_cast<const __nv_bfloat16*>(R_intra), static_cast<uint8_t*>(out_codes),
              static_cast<uint8_t*>(out_scales), (int)M, (int)d, tensor_scale, st->err_word);
  else
    launch_tc(rotate_structured_kernel<FMT_MXFP4>, 1, grid, RotStructCfg::THREADS, RotStructCfg::SMEM_BYTES, s, tmRB,
              tmX3, static_cast<const __nv_bfloat16*>(R_B), static_cast<const __nv_bfloat16*>(R_intra), static_cast<uint8_t*>(out_codes),
              static_cast<uint8_t*>(out_scales), (int)M, (int)d, 0.0f, st->err_word);
  return launch_status();
}

torq_status torq_rotate_quantize_structured(const void* X, const void* R_B, const void* R_intra, int64_t M,
                                            int64_t d, void* out_codes, void* out_scales, void* stream) {
  return rotate_structured_impl(X, R_B, R_intra, M, d, out_codes, out_scales, stream, FMT_MXFP4, 0.0f);
}

torq_status torq_rotate_quantize_structured_nvfp4(const void* X, const void* R_B, const void* R_intra, int64_t M,
                                                  int64_t d, float tensor_scale, void* out_codes, void* out_scales,
                                                  void* stream) {
  if (!(tensor_scale > 0.0f && tensor_scale <= 3.0e38f)) return TORQ_ERR_SHAPE;
  return rotate_structured_impl(X, R_B, R_intra, M, d, out_codes, out_scales, stream, FMT_NVFP4, tensor_scale);
}

}  // extern "C"

// Width of the one-wave GEMM's tiles, or 0 where another kernel is faster.  Times in us, fitted to MXFP4 with bf16 output
// at K = 128 ... 14336, N = 256 ... 12288, M = 17 ... 8000 (within 10 % of the kernels with one slab); f = filled part of a wave:
//  * here: 2 (1.8 / 1.5 up to 128 / 64 tokens) + 0.0062 per column + f for launch and epilogue, then per K step 0.24 or the
//    math, 0.0011 per column, + 0.025 f: with one slab of K per stage.  Up to 128 columns two take 0.15 to 0.19, which the figures
//    do not know: there they are high by up to a third (200 x 4096, K = 14336 17.3 modelled, 13.1 measured; 300 x 4096, K = 4096 7.8,
//    6.7) and take 192 columns in one slab where 128 in two would fit the pairs too (512 x 4096, K = 14336; 700 x 3072, K = 4096);
//  * few tokens (17 to 128, S CTAs per tile): 2.3 + 0.2 per K step of the longest split + per token 0.025 with S = 1 (the
//    accumulator goes to Y), else 0.012 + 0.035 / S.  With pulled sums; pushed ones (17 to 32 tokens, K > 2048) take less, and even by
//    these figures the one-wave kernel is 1.11 times and more their time at every size;
//  * pair kernel: one wave 4.1 + 0.9 f + (0.285 + 0.04 f) per K step, more (the last one as narrower tiles) 5.2 + per K step
//    0.325 for a full wave and 0.21 + 0.14 f for the last.
// The same figures choose for NVFP4, MXINT4 (twice the steps) and float32 output, which were not fitted.  A sweep of 5250 calls, the
// three formats and float32 output together, against the library without the one-wave kernels: 1.31 times as fast in the geometric
// mean; lost by this choice: MXFP4 1536 x 4096, K = 1024 6.78 / 6.88.
// Where it pays: 777 x 5120, K = 14336 (80 pair tiles) 34.7 -> 27.3, K = 4096 13.1 -> 11.2; 1280 x 4096, K = 14336 34.6 ->
// 27.8; short contractions: 40 x 4096, K = 512 4.0 -> 3.0; 100 x 4096, K = 512 5.1 -> 3.3; 3000 x 1024, K = 2048 7.1 -> 6.4.
static int wide_gemm_width(int64_t M, int64_t N, int64_t steps, int few_S, int max_pairs) {
  const int64_t rows = (M + 255) / 256;
  const double base = M <= 64 ? 1.5 : (M <= 128 ? 1.8 : 2.0);
  double best = 1e30;
  int width = 0;
  for (int w = 64; w <= GemmWideCfg<>::MAX_WIDTH; w += 64) {
    const int64_t tiles = rows * ((N + w - 1) / w);
    if (tiles > max_pairs) continue;
    const double f = (double)tiles / max_pairs, math = 0.0011 * w;
    const double t = base + 0.0062 * w + f + (double)steps * ((math > 0.24 ? math : 0.24) + 0.025 * f);
    if (t < best) { best = t; width = w; }
  }
  const int64_t tiles = rows * ((N + 255) / 256), full = tiles / max_pairs, rest = tiles % max_pairs;
  const double f = (double)rest / max_pairs;
  double other;
  if (few_S > 0)
    other = 2.3 + 0.2 * (double)((steps + few_S - 1) / few_S) + (double)M * (few_S == 1 ? 0.025 : 0.012 + 0.035 / few_S);
  else if (full == 0) other = 4.1 + 0.9 * f + (double)steps * (0.285 + 0.04 * f);
  else other = 5.2 + (double)steps * (0.325 * (double)full + (rest ? 0.21 + 0.14 * f : 0.0));
  return best < 0.97 * other ? width : 0;
}

template <int FMT>
static torq_status gemm_wide(DeviceState* st, const void* Aq, const void* As, const void* Wq, const void* Ws, int64_t M, int64_t N,
                             int64_t K, void* Y, torq_dtype y_dtype, float alpha, int width, cudaStream_t s) {
  using C = GemmWideCfg<FMT>;
  const uint64_t krow = (uint64_t)(FMT == FMT_MXINT4 ? K : K / 2);
  const uint64_t sf_words = (uint64_t)(K / (FMT == FMT_NVFP4 ? 64 : 128)) * 128;   // scale words per 128 rows
  const bool ybf = y_dtype == TORQ_BF16;
  CUtensorMap tmA, tmB, tmB1, tmSFA, tmSFB, tmY;
  if (!encode_2d(&tmA, CU_TENSOR_MAP_DATA_TYPE_UINT8, 1, Aq, (uint64_t)M, krow, 128, 128) ||
      !encode_2d(&tmB, CU_TENSOR_MAP_DATA_TYPE_UINT8, 1, Wq, (uint64_t)N, krow, (uint32_t)C::n0(width) / 2, 128) ||
      (width > 256 && !encode_2d(&tmB1, CU_TENSOR_MAP_DATA_TYPE_UINT8, 1, Wq, (uint64_t)N, krow, 64, 128)) ||
      !encode_2d(&tmSFA, CU_TENSOR_MAP_DATA_TYPE_UINT32, 4, As, (uint64_t)((M + 127) / 128), sf_words, 1, C::SF_BOX_WORDS,
                 CU_TENSOR_MAP_SWIZZLE_NONE) ||
      !encode_2d(&tmSFB, CU_TENSOR_MAP_DATA_TYPE_UINT32, 4, Ws, (uint64_t)((N + 127) / 128), sf_words, (uint32_t)C::chunks(width),
                 C::SF_BOX_WORDS, CU_TENSOR_MAP_SWIZZLE_NONE) ||
      !encode_2d(&tmY, ybf ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32, ybf ? 2 : 4, Y, (uint64_t)M,
                 (uint64_t)N, 32, ybf ? 64 : 32))
    return TORQ_ERR_LAUNCH;
  if (width <= 256) tmB1 = tmB;
  const int rows = (int)((M + 255) / 256), cols = (int)((N + width - 1) / width);
  const int range = C::range(width, C::two_slabs(M, K, (int64_t)rows * cols));
  launch_tc(range == 384 ? mxfp4_gemm_wide_kernel<FMT, 384> : (range == 256 ? mxfp4_gemm_wide_kernel<FMT, 256> : mxfp4_gemm_wide_kernel<FMT, 128>),
            2, 2 * rows * cols, C::THREADS, C::smem_bytes(width, range), s, tmA, tmB, tmB1, tmSFA, tmSFB, tmY, ybf ? 1 : 0, (int)M, (int)N, (int)K, rows, width, alpha,
            st->err_word);
  return launch_status();
}

// Step 5 for either format; `alpha` multiplies the NVFP4 result (product of the tensor scales).
template <int FMT>
static torq_status gemm_impl(const void* Aq, const void* As, const void* Wq, const void* Ws, int64_t M,
                             int64_t N, int64_t K, void* Y, torq_dtype y_dtype, float alpha, void* stream) {
  if (!Aq || !As || !Wq || !Ws || !Y) return TORQ_ERR_NULL;
  if (M < 1 || N < 8 || K < 128 || K % 128 != 0 || N % 8 != 0 || M > (1 << 30) || N > (1 << 30) ||
      K > (1 << 24))
    return TORQ_ERR_SHAPE;
  if (y_dtype != TORQ_F32 && y_dtype != TORQ_BF16) return TORQ_ERR_SHAPE;
  if (!aligned16(Aq) || !aligned16(As) || !aligned16(Wq) || !aligned16(Ws) || !aligned16(Y))
    return TORQ_ERR_ALIGN;
  DeviceState* st = device_state();
  if (!st) return TORQ_ERR_LAUNCH;
  if (!st->arch_ok) return TORQ_ERR_ARCH;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  constexpr int BN = 256;
  const uint64_t krow = (uint64_t)(FMT == FMT_MXINT4 ? K : K / 2);   // operand bytes per row
  CUtensorMap tmA, tmB;
  using FC = GemmFewCfg<FMT>;
  const int ntok = M <= kGemmFewMaxTokens ? fewtok_ntok(M) : 0;
  const int tiles = (int)((N + 127) / 128);
  // More tiles than CTAs that fit: every further wave of few-token CTAs starts with empty stages.  From 49 tokens on the
  // persistent pair kernels do better, half empty as their rows are (us, few-token against pairs: 100 tokens K = 4096,
  // N = 20480 20.4 / 12.9, N = 28672 21.4 / 16.3, N = 14336 10.9 / 11.1; 64 tokens, two CTAs per SM: K = 2048, N = 40960
  // 15.3 / 12.9, K = 4096, N = 28672 14.4 / 16.0; 40 tokens K = 5120, N = 51200 29.7 / 30.1).
  const bool many_waves = M > 48 && (int64_t)tiles > (int64_t)FC::ctas_per_sm((int)M, (int)K) * st->sm_count;
  if (ntok > 0 && !many_waves) {
    // Few tokens: 128 output features x all tokens per CTA, K split over a cluster, reduced through
    // distributed shared memory.
    const int64_t steps = (K + FC::BK - 1) / FC::BK;
    const bool push = FC::push((int)M, (int)K);
    const int ctas = FC::ctas_per_sm((int)M, (int)K);
    const int S = push ? push_gemm_cluster(M, tiles, steps, st) : fewtok_gemm_cluster(ntok, tiles, steps, ctas, st);
    const int width = M > 16 ? wide_gemm_width(M, N, steps, S, st->gemm_pairs) : 0;
    if (width > 0) return gemm_wide<FMT>(st, Aq, As, Wq, Ws, M, N, K, Y, y_dtype, alpha, width, s);
    if (!encode_2d(&tmB, CU_TENSOR_MAP_DATA_TYPE_UINT8, 1, Wq, (uint64_t)N, krow, 128, 128) ||
        !encode_2d(&tmA, CU_TENSOR_MAP_DATA_TYPE_UINT8, 1, Aq, (uint64_t)M, krow, (uint32_t)ntok, 128))
      return TORQ_ERR_LAUNCH;
    // sums pushed (FC::push); up to 64 tokens: one set of epilogue warps, two CTAs per SM; more: two sets.  65 to 80 tokens in
    // MXINT4 fit twice on an SM as well, and share it only where that gives them more K splits (us, shared / alone, 72 tokens:
    // N = 768, K = 3072 4.9 / 4.4, N = 1536 6.0 / 5.1, S = 8 either way; N = 6144, K = 4096, S = 4 and 1: 9.1 / 9.9).
    const bool small = ctas >= 2 && (ntok <= 64 || S > fewtok_gemm_cluster(ntok, tiles, steps, 1, st));
    launch_tc(push ? gemm_fewtok_kernel<FMT, 1, true> : (small ? gemm_fewtok_kernel<FMT, 1> : gemm_fewtok_kernel<FMT, 2>), S, tiles * S,
              small ? 192 : 320, FC::smem_bytes((int)M, (int)K), s, tmB, tmA, static_cast<const uint8_t*>(As),
              static_cast<const uint8_t*>(Ws), Y, y_dtype == TORQ_BF16 ? 1 : 0, (int)M, (int)N, (int)K, ntok, S,
              kAheadTiles / (tiles * S), alpha, st->err_word);
    return launch_status();
  }
  const int width = wide_gemm_width(M, N, (K + GemmWideCfg<FMT>::BK - 1) / GemmWideCfg<FMT>::BK, 0, st->gemm_pairs);
  if (width > 0) return gemm_wide<FMT>(st, Aq, As, Wq, Ws, M, N, K, Y, y_dtype, alpha, width, s);
  CUtensorMap tmSFA, tmSFB;
  const uint64_t kb4 = (uint64_t)(K / (FMT == FMT_NVFP4 ? 64 : 128));   // 512-byte scale chunks per row
  constexpr uint32_t sf_box = GemmPairCfgT<FMT>::SF_BOX_WORDS;
  if (!encode_2d(&tmA, CU_TENSOR_MAP_DATA_TYPE_UINT8, 1, Aq, (uint64_t)M, krow, 128, 128) ||
      !encode_2d(&tmB, CU_TENSOR_MAP_DATA_TYPE_UINT8, 1, Wq, (uint64_t)N, krow, BN / 2, 128) ||
      !encode_2d(&tmSFA, CU_TENSOR_MAP_DATA_TYPE_UINT32, 4, As, (uint64_t)((M + 127) / 128), kb4 * 128, 1, sf_box,
                 CU_TENSOR_MAP_SWIZZLE_NONE) ||
      !encode_2d(&tmSFB, CU_TENSOR_MAP_DATA_TYPE_UINT32, 4, Ws, (uint64_t)((N + 127) / 128), kb4 * 128, 2, sf_box,
                 CU_TENSOR_MAP_SWIZZLE_NONE))
    return TORQ_ERR_LAUNCH;
  CUtensorMap tmY;
  const bool ybf = y_dtype == TORQ_BF16;
  if (!encode_2d(&tmY, ybf ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32, ybf ? 2 : 4,
                 Y, (uint64_t)M, (uint64_t)N, 32, ybf ? 64 : 32))
    return TORQ_ERR_LAUNCH;
  CUtensorMap tmBn;                                      // half of a 192-column tile: 96 rows of W
  if (!encode_2d(&tmBn, CU_TENSOR_MAP_DATA_TYPE_UINT8, 1, Wq, (uint64_t)N, krow, kNarrowCols / 2, 128))
    return TORQ_ERR_LAUNCH;
  const int max_pairs = st->gemm_pairs;
  const MixedTiles list = plan_gemm_tiles(M, N, krow, max_pairs);
  const int pairs = list.total < max_pairs ? list.total : max_pairs;
  launch_tc(mxfp4_gemm_pair_kernel<FMT>, 2, 2 * pairs, GemmPairCfgT<FMT>::THREADS, GemmPairCfgT<FMT>::SMEM_BYTES, s,
            tmA, tmB, tmSFA, tmSFB, tmY, tmBn, list, ybf ? 1 : 0, (int)M, (int)N, (int)K, alpha, st->err_word);
  return launch_status();
}

extern "C" {

torq_status torq_mxfp4_gemm(const void* Aq, const void* As, const void* Wq, const void* Ws, int64_t M,
                            int64_t N, int64_t K, void* Y, torq_dtype y_dtype, void* stream) {
  return gemm_impl<FMT_MXFP4>(Aq, As, Wq, Ws, M, N, K, Y, y_dtype, 1.0f, stream);
}

static inline bool scale_ok(float s) { return s > 0.0f && s <= 3.0e38f; }   // positive, finite

torq_status torq_nvfp4_gemm(const void* Aq, const void* As, float a_tensor_scale, const void* Wq, const void* Ws,
                            float w_tensor_scale, int64_t M, int64_t N, int64_t K, void* Y, torq_dtype y_dtype,
                            void* stream) {
  if (!scale_ok(a_tensor_scale) || !scale_ok(w_tensor_scale)) return TORQ_ERR_SHAPE;
  return gemm_impl<FMT_NVFP4>(Aq, As, Wq, Ws, M, N, K, Y, y_dtype, a_tensor_scale * w_tensor_scale, stream);
}

size_t torq_nvfp4_scales_bytes(int64_t rows, int64_t k) {
  if (rows <= 0 || k <= 0) return 0;
  return (size_t)((rows + 127) / 128) * (size_t)((k / 16 + 3) / 4) * 512;
}

static size_t nvfp4_quantized_bytes(int64_t M, int64_t d) {
  return ((size_t)M * (size_t)(d / 2) + 255) / 256 * 256 + torq_nvfp4_scales_bytes(M, d);
}

size_t torq_nvfp4_workspace_bytes(int64_t M, int64_t d, int64_t N) {
  (void)N;
  if (M <= 0 || d <= 0) return 0;
  return nvfp4_quantized_bytes(M, d) + spare_workspace_bytes(M, d);
}

torq_status torq_expand_intra16(const void* R_intra16, int64_t d, void* R_intra32, void* stream) {
  if (!R_intra16 || !R_intra32) return TORQ_ERR_NULL;
  if (d < 32 || d % 32 != 0 || d > (1 << 24)) return TORQ_ERR_SHAPE;
  DeviceState* st = device_state();
  if (!st) return TORQ_ERR_LAUNCH;
  if (!st->arch_ok) return TORQ_ERR_ARCH;
  expand_intra16_kernel<<<ew_grid(d * 32, 256, st->sm_count), 256, 0, static_cast<cudaStream_t>(stream)>>>(
      static_cast<const __nv_bfloat16*>(R_intra16), d / 32, static_cast<__nv_bfloat16*>(R_intra32));
  return launch_status();
}

torq_status torq_quantize_nvfp4(const void* Z, torq_dtype z_dtype, int64_t M, int64_t d, float tensor_scale,
                                void* out_codes, void* out_scales, void* stream) {
  if (!Z || !out_codes || !out_scales) return TORQ_ERR_NULL;
  if (M < 1 || d < 16 || d % 16 != 0 || M > (1 << 30) || d > (1 << 30) || !scale_ok(tensor_scale))
    return TORQ_ERR_SHAPE;
  if (z_dtype != TORQ_F32 && z_dtype != TORQ_BF16) return TORQ_ERR_SHAPE;
  if (!aligned16(Z) || !aligned16(out_codes) || !aligned16(out_scales)) return TORQ_ERR_ALIGN;
  DeviceState* st = device_state();
  if (!st) return TORQ_ERR_LAUNCH;
  if (!st->arch_ok) return TORQ_ERR_ARCH;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const int64_t kb4 = (d / 16 + 3) / 4;
  const int64_t items = ((M + 127) / 128 * 128) * ((kb4 * 64 + 255) / 256);   // warps
  const int grid = ew_grid(items, 8, st->sm_count);
  if (z_dtype == TORQ_F32)
    nv_quantize_kernel<float><<<grid, 256, 0, s>>>(static_cast<const float*>(Z), M, d, tensor_scale,
                                                   static_cast<uint8_t*>(out_codes), static_cast<uint8_t*>(out_scales));
  else
    nv_quantize_kernel<__nv_bfloat16><<<grid, 256, 0, s>>>(static_cast<const __nv_bfloat16*>(Z), M, d, tensor_scale,
                                                           static_cast<uint8_t*>(out_codes),
                                                           static_cast<uint8_t*>(out_scales));
  return launch_status();
}

torq_status torq_rotate_quantize_nvfp4(const void* X, const void* R_inter, const void* R_intra32, int64_t M,
                                       int64_t d, float tensor_scale, void* out_codes, void* out_scales,
                                       void* stream) {
  if (!scale_ok(tensor_scale)) return TORQ_ERR_SHAPE;
  return rotate_quantize_impl(X, R_inter, R_intra32, M, d, out_codes, out_scales, stream, FMT_NVFP4,
                              tensor_scale);
}

torq_status torq_rotated_linear_nvfp4(const void* X, const void* R_inter, const void* R_intra32, float x_tensor_scale,
                                      const void* Wq, const void* Ws, float w_tensor_scale, int64_t M, int64_t d,
                                      int64_t N, void* Y, torq_dtype y_dtype, void* workspace, size_t workspace_bytes,
                                      void* dbg_codes, void* dbg_scales, void* stream) {
  if (!X || !R_inter || !Wq || !Ws || !Y) return TORQ_ERR_NULL;
  if (M < 1 || d < 128 || d % 128 != 0 || N < 8 || N % 8 != 0 || M > (1 << 30) || d > (1 << 24) ||
      !scale_ok(x_tensor_scale) || !scale_ok(w_tensor_scale))
    return TORQ_ERR_SHAPE;
  if (!workspace || workspace_bytes < torq_nvfp4_workspace_bytes(M, d, N)) return TORQ_ERR_WORKSPACE;
  if ((reinterpret_cast<uintptr_t>(workspace) & 255u) != 0) return TORQ_ERR_ALIGN;
  uint8_t* codes = static_cast<uint8_t*>(workspace);
  const size_t codes_bytes = (size_t)M * (size_t)(d / 2);
  uint8_t* scales = codes + (codes_bytes + 255) / 256 * 256;
  torq_status rc = rotate_quantize_impl(X, R_inter, R_intra32, M, d, codes, scales, stream, FMT_NVFP4, x_tensor_scale);
  if (rc != TORQ_OK) return rc;
  rc = torq_nvfp4_gemm(codes, scales, x_tensor_scale, Wq, Ws, w_tensor_scale, M, N, d, Y, y_dtype, stream);
  if (rc != TORQ_OK) return rc;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if (dbg_codes &&
      cudaMemcpyAsync(dbg_codes, codes, codes_bytes, cudaMemcpyDeviceToDevice, s) != cudaSuccess)
    return TORQ_ERR_LAUNCH;
  if (dbg_scales && cudaMemcpyAsync(dbg_scales, scales, torq_nvfp4_scales_bytes(M, d),
                                    cudaMemcpyDeviceToDevice, s) != cudaSuccess)
    return TORQ_ERR_LAUNCH;
  return TORQ_OK;
}

// ---- MXINT4 (format study of Section 6): integer codes, E8M0 scales, E4M3 operand bytes ----------

static size_t mxint4_quantized_bytes(int64_t M, int64_t d) {
  return ((size_t)M * (size_t)d + 255) / 256 * 256 + torq_scales_bytes(M, d);
}

size_t torq_mxint4_workspace_bytes(int64_t M, int64_t d, int64_t N) {
  (void)N;
  if (M <= 0 || d <= 0) return 0;
  return mxint4_quantized_bytes(M, d) + spare_workspace_bytes(M, d);
}

torq_status torq_quantize_mxint4(const void* Z, torq_dtype z_dtype, int64_t M, int64_t d, int packed, void* out_codes,
                                 void* out_scales, void* stream) {
  if (!Z || !out_codes || !out_scales) return TORQ_ERR_NULL;
  if (M < 1 || d < 32 || d % 32 != 0 || M > (1 << 30) || d > (1 << 30)) return TORQ_ERR_SHAPE;
  if (z_dtype != TORQ_F32 && z_dtype != TORQ_BF16) return TORQ_ERR_SHAPE;
  if (!aligned16(Z) || !aligned16(out_codes) || !aligned16(out_scales)) return TORQ_ERR_ALIGN;
  DeviceState* st = device_state();
  if (!st) return TORQ_ERR_LAUNCH;
  if (!st->arch_ok) return TORQ_ERR_ARCH;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const int64_t kb4 = (d / 32 + 3) / 4;
  const int64_t items = ((M + 127) / 128 * 128) * ((kb4 * 128 + 255) / 256);   // warps
  const int grid = ew_grid(items, 8, st->sm_count);
  uint8_t* c = static_cast<uint8_t*>(out_codes);
  uint8_t* sc = static_cast<uint8_t*>(out_scales);
  if (z_dtype == TORQ_F32) {
    const float* z = static_cast<const float*>(Z);
    if (packed) mxint4_quantize_kernel<float, true><<<grid, 256, 0, s>>>(z, M, d, c, sc);
    else mxint4_quantize_kernel<float, false><<<grid, 256, 0, s>>>(z, M, d, c, sc);
  } else {
    const __nv_bfloat16* z = static_cast<const __nv_bfloat16*>(Z);
    if (packed) mxint4_quantize_kernel<__nv_bfloat16, true><<<grid, 256, 0, s>>>(z, M, d, c, sc);
    else mxint4_quantize_kernel<__nv_bfloat16, false><<<grid, 256, 0, s>>>(z, M, d, c, sc);
  }
  return launch_status();
}

torq_status torq_mxint4_expand(const void* packed, int64_t rows, int64_t k, void* out_bytes, void* stream) {
  if (!packed || !out_bytes) return TORQ_ERR_NULL;
  if (rows < 1 || k < 32 || k % 32 != 0 || rows > (1 << 30) || k > (1 << 30)) return TORQ_ERR_SHAPE;
  if (!aligned16(packed) || !aligned16(out_bytes)) return TORQ_ERR_ALIGN;
  DeviceState* st = device_state();
  if (!st) return TORQ_ERR_LAUNCH;
  if (!st->arch_ok) return TORQ_ERR_ARCH;
  const int64_t words = rows * (k / 8);
  mxint4_expand_kernel<<<ew_grid(words, 256, st->sm_count), 256, 0, static_cast<cudaStream_t>(stream)>>>(
      static_cast<const uint32_t*>(packed), words, static_cast<uint2*>(out_bytes));
  return launch_status();
}

torq_status torq_rotate_quantize_mxint4(const void* X, const void* R_inter, const void* R_intra, int64_t M,
                                        int64_t d, void* out_bytes, void* out_scales, void* stream) {
  return rotate_quantize_impl(X, R_inter, R_intra, M, d, out_bytes, out_scales, stream, FMT_MXINT4,
                              0.0f);
}

torq_status torq_rotate_quantize_structured_mxint4(const void* X, const void* R_B, const void* R_intra, int64_t M,
                                                   int64_t d, void* out_bytes, void* out_scales, void* stream) {
  return rotate_structured_impl(X, R_B, R_intra, M, d, out_bytes, out_scales, stream, FMT_MXINT4, 0.0f);
}

torq_status torq_mxint4_gemm(const void* A8, const void* As, const void* W8, const void* Ws, int64_t M, int64_t N,
                             int64_t K, void* Y, torq_dtype y_dtype, void* stream) {
  return gemm_impl<FMT_MXINT4>(A8, As, W8, Ws, M, N, K, Y, y_dtype, 1.0f, stream);
}

torq_status torq_rotated_linear_mxint4(const void* X, const void* R_inter, const void* R_intra, const void* W8,
                                       const void* Ws, int64_t M, int64_t d, int64_t N, void* Y, torq_dtype y_dtype,
                                       void* workspace, size_t workspace_bytes, void* dbg_bytes, void* dbg_scales,
                                       void* stream) {
  if (!X || !R_inter || !W8 || !Ws || !Y) return TORQ_ERR_NULL;
  if (M < 1 || d < 128 || d % 128 != 0 || N < 8 || N % 8 != 0 || M > (1 << 30) || d > (1 << 24))
    return TORQ_ERR_SHAPE;
  if (!workspace || workspace_bytes < torq_mxint4_workspace_bytes(M, d, N)) return TORQ_ERR_WORKSPACE;
  if ((reinterpret_cast<uintptr_t>(workspace) & 255u) != 0) return TORQ_ERR_ALIGN;
  uint8_t* bytes = static_cast<uint8_t*>(workspace);
  const size_t n_bytes = (size_t)M * (size_t)d;
  uint8_t* scales = bytes + (n_bytes + 255) / 256 * 256;
  torq_status rc = rotate_quantize_impl(X, R_inter, R_intra, M, d, bytes, scales, stream, FMT_MXINT4, 0.0f);
  if (rc != TORQ_OK) return rc;
  rc = torq_mxint4_gemm(bytes, scales, W8, Ws, M, N, d, Y, y_dtype, stream);
  if (rc != TORQ_OK) return rc;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if (dbg_bytes && cudaMemcpyAsync(dbg_bytes, bytes, n_bytes, cudaMemcpyDeviceToDevice, s) != cudaSuccess)
    return TORQ_ERR_LAUNCH;
  if (dbg_scales &&
      cudaMemcpyAsync(dbg_scales, scales, torq_scales_bytes(M, d), cudaMemcpyDeviceToDevice, s) != cudaSuccess)
    return TORQ_ERR_LAUNCH;
  return TORQ_OK;
}

// Steps 1-5 with at least quantized_bytes(M, d) of workspace, checked by the caller: codes, then scales.
static torq_status rotated_linear_impl(const void* X, const void* R_inter, const void* R_intra, const void* Wq,
                                       const void* Ws, int64_t M, int64_t d, int64_t N, void* Y,
                                       torq_dtype y_dtype, void* workspace, void* dbg_codes, void* dbg_scales,
                                       void* stream) {
  uint8_t* codes = static_cast<uint8_t*>(workspace);
  const size_t codes_bytes = (size_t)M * (size_t)(d / 2);
  uint8_t* scales = codes + (codes_bytes + 255) / 256 * 256;
  torq_status rc = rotate_quantize_impl(X, R_inter, R_intra, M, d, codes, scales, stream);
  if (rc != TORQ_OK) return rc;
  rc = torq_mxfp4_gemm(codes, scales, Wq, Ws, M, N, d, Y, y_dtype, stream);
  if (rc != TORQ_OK) return rc;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if (dbg_codes &&
      cudaMemcpyAsync(dbg_codes, codes, codes_bytes, cudaMemcpyDeviceToDevice, s) != cudaSuccess)
    return TORQ_ERR_LAUNCH;
  if (dbg_scales && cudaMemcpyAsync(dbg_scales, scales, torq_scales_bytes(M, d),
                                    cudaMemcpyDeviceToDevice, s) != cudaSuccess)
    return TORQ_ERR_LAUNCH;
  return TORQ_OK;
}

torq_status torq_rotated_linear(const void* X, const void* R_inter, const void* R_intra, const void* Wq,
                                const void* Ws, int64_t M, int64_t d, int64_t N, void* Y,
                                torq_dtype y_dtype, void* workspace, size_t workspace_bytes,
                                void* dbg_codes, void* dbg_scales, void* stream) {
  if (!X || !Wq || !Ws || !Y) return TORQ_ERR_NULL;
  if (M < 1 || d < 128 || d % 128 != 0 || N < 8 || N % 8 != 0) return TORQ_ERR_SHAPE;
  if (!workspace || workspace_bytes < torq_workspace_bytes(M, d, N)) return TORQ_ERR_WORKSPACE;
  if ((reinterpret_cast<uintptr_t>(workspace) & 255u) != 0) return TORQ_ERR_ALIGN;
  return rotated_linear_impl(X, R_inter, R_intra, Wq, Ws, M, d, N, Y, y_dtype, workspace, dbg_codes, dbg_scales,
                             stream);
}

torq_status torq_rotated_linear_structured(const void* X, const void* R_B, const void* R_intra, const void* Wq,
                                           const void* Ws, int64_t M, int64_t d, int64_t N, void* Y,
                                           torq_dtype y_dtype, void* workspace, size_t workspace_bytes,
                                           void* dbg_codes, void* dbg_scales, void* stream) {
  if (!X || !R_B || !Wq || !Ws || !Y) return TORQ_ERR_NULL;
  if (M < 1 || d < 256 || d % 256 != 0 || N < 8 || N % 8 != 0) return TORQ_ERR_SHAPE;
  if (!workspace || workspace_bytes < quantized_bytes(M, d)) return TORQ_ERR_WORKSPACE;
  if ((reinterpret_cast<uintptr_t>(workspace) & 255u) != 0) return TORQ_ERR_ALIGN;
  uint8_t* codes = static_cast<uint8_t*>(workspace);
  const size_t codes_bytes = (size_t)M * (size_t)(d / 2);
  uint8_t* scales = codes + (codes_bytes + 255) / 256 * 256;
  torq_status rc = torq_rotate_quantize_structured(X, R_B, R_intra, M, d, codes, scales, stream);
  if (rc != TORQ_OK) return rc;
  rc = torq_mxfp4_gemm(codes, scales, Wq, Ws, M, N, d, Y, y_dtype, stream);
  if (rc != TORQ_OK) return rc;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if (dbg_codes &&
      cudaMemcpyAsync(dbg_codes, codes, codes_bytes, cudaMemcpyDeviceToDevice, s) != cudaSuccess)
    return TORQ_ERR_LAUNCH;
  if (dbg_scales && cudaMemcpyAsync(dbg_scales, scales, torq_scales_bytes(M, d),
                                    cudaMemcpyDeviceToDevice, s) != cudaSuccess)
    return TORQ_ERR_LAUNCH;
  return TORQ_OK;
}

// ---- the layer without any allocation -----------------------------------------------------------
// Scratch for torq_rotated_linear_static.  In host code this name is only a handle for the
// runtime's symbol table, not an address a kernel can use: the device address comes from
// cudaGetSymbolAddress, once per device, with that device current.
static __device__ __align__(256) uint8_t g_static_workspace[TORQ_STATIC_WORKSPACE_BYTES];
static void* g_static_workspace_addr[torq::kMaxDevices] = {};
static std::mutex g_static_workspace_mutex;

// Device address of the scratch array on the current device (nullptr when CUDA reports an error).
static void* static_workspace_address() {
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= torq::kMaxDevices) return nullptr;
  std::lock_guard<std::mutex> lock(g_static_workspace_mutex);
  if (!g_static_workspace_addr[dev]) {
    void* p = nullptr;
    if (cudaGetSymbolAddress(&p, g_static_workspace) != cudaSuccess || p == nullptr) {
      cudaGetLastError();                    // leave no sticky-looking error behind for the caller
      return nullptr;
    }
    g_static_workspace_addr[dev] = p;
  }
  return g_static_workspace_addr[dev];
}

torq_status torq_rotated_linear_static(const void* X, const void* R_inter, const void* R_intra,
                                       const void* Wq, const void* Ws, int64_t M, int64_t d,
                                       int64_t N, void* Y, torq_dtype y_dtype, void* stream) {
  if (!X || !Wq || !Ws || !Y) return TORQ_ERR_NULL;
  if (M < 1 || d < 128 || d % 128 != 0 || N < 8 || N % 8 != 0 || M > (1 << 30) || d > (1 << 24))
    return TORQ_ERR_SHAPE;
  if (quantized_bytes(M, d) > (size_t)TORQ_STATIC_WORKSPACE_BYTES) return TORQ_ERR_WORKSPACE;
  DeviceState* st = device_state();                // architecture first: another device has no image of the array
  if (!st) return TORQ_ERR_LAUNCH;
  if (!st->arch_ok) return TORQ_ERR_ARCH;
  void* scratch = static_workspace_address();
  if (!scratch) return TORQ_ERR_LAUNCH;
  return rotated_linear_impl(X, R_inter, R_intra, Wq, Ws, M, d, N, Y, y_dtype, scratch, nullptr, nullptr,
                             stream);
}

torq_status torq_probe_fp4_peak(int groups, double* tflops, void* stream) {
  if (!tflops) return TORQ_ERR_NULL;
  if (groups < 1 || groups > (1 << 24)) return TORQ_ERR_SHAPE;
  DeviceState* st = device_state();
  if (!st) return TORQ_ERR_LAUNCH;
  if (!st->arch_ok) return TORQ_ERR_ARCH;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if (!opt_in_smem(fp4_peak_probe_kernel, Fp4ProbeCfg::SMEM_BYTES)) return TORQ_ERR_LAUNCH;
  const int pairs = st->gemm_pairs;
  cudaEvent_t e0, e1;
  if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess) return TORQ_ERR_LAUNCH;
  launch_tc(fp4_peak_probe_kernel, 2, 2 * pairs, Fp4ProbeCfg::THREADS, Fp4ProbeCfg::SMEM_BYTES, s, 64, st->err_word);
  cudaEventRecord(e0, s);
  launch_tc(fp4_peak_probe_kernel, 2, 2 * pairs, Fp4ProbeCfg::THREADS, Fp4ProbeCfg::SMEM_BYTES, s, groups, st->err_word);
  cudaEventRecord(e1, s);
  g_launches.fetch_add(2, std::memory_order_relaxed);
  float ms = 0.f;
  const bool ok = cudaEventSynchronize(e1) == cudaSuccess && cudaEventElapsedTime(&ms, e0, e1) == cudaSuccess &&
                  cudaGetLastError() == cudaSuccess && ms > 0.f;
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  if (!ok) return TORQ_ERR_LAUNCH;
  *tflops = (double)pairs * groups * 4.0 * 2.0 * 256.0 * 256.0 * 64.0 / ((double)ms * 1e-3) / 1e12;
  return TORQ_OK;
}

torq_status torq_selftest_wait_timeout(uint64_t limit_ns, void* result_u64x3, void* stream) {
  if (!result_u64x3) return TORQ_ERR_NULL;
  if (limit_ns < 1000ull || limit_ns > 100000000ull) return TORQ_ERR_SHAPE;        // 1 us .. 100 ms
  if (!aligned16(result_u64x3)) return TORQ_ERR_ALIGN;
  DeviceState* st = device_state();
  if (!st) return TORQ_ERR_LAUNCH;
  if (!st->arch_ok) return TORQ_ERR_ARCH;
  wait_selftest_kernel<<<1, 64, 0, static_cast<cudaStream_t>(stream)>>>(
      (unsigned long long)limit_ns, st->err_word, static_cast<unsigned long long*>(result_u64x3));
  return launch_status();
}

torq_status torq_block_covariance(const void* X, int64_t T, int64_t d, void* Sigma_f64, void* stream) {
  if (!X || !Sigma_f64) return TORQ_ERR_NULL;
  if (T < 1 || d < 32 || d % 32 != 0 || T > (1 << 30) || d > (1 << 20)) return TORQ_ERR_SHAPE;
  if (!aligned16(X) || !aligned16(Sigma_f64)) return TORQ_ERR_ALIGN;
  DeviceState* st = device_state();
  if (!st) return TORQ_ERR_LAUNCH;
  if (!st->arch_ok) return TORQ_ERR_ARCH;
  const unsigned tiles = (unsigned)((d / 32 + 15) / 16);
  block_covariance_kernel<<<dim3(tiles, tiles, 1), 256, 0, static_cast<cudaStream_t>(stream)>>>(
      static_cast<const __nv_bfloat16*>(X), T, d, static_cast<double*>(Sigma_f64));
  return launch_status();
}

torq_status torq_givens_equalize(void* Sigma_f64, int64_t B, double eps, void* Q_f64, void* Q_bf16,
                                 void* n_rotations, void* stream) {
  if (!Sigma_f64 || !Q_f64) return TORQ_ERR_NULL;
  if (B < 1 || B > 32768 || !(eps >= 0.0)) return TORQ_ERR_SHAPE;
  if (!aligned16(Sigma_f64) || !aligned16(Q_f64) || (Q_bf16 && !aligned16(Q_bf16))) return TORQ_ERR_ALIGN;
  DeviceState* st = device_state();
  if (!st) return TORQ_ERR_LAUNCH;
  if (!st->arch_ok) return TORQ_ERR_ARCH;
  givens_equalize_kernel<<<1, 512, 0, static_cast<cudaStream_t>(stream)>>>(
      static_cast<double*>(Sigma_f64), (int)B, eps, static_cast<double*>(Q_f64), static_cast<__nv_bfloat16*>(Q_bf16),
      static_cast<int*>(n_rotations), (int)(4 * B));
  return launch_status();
}

torq_status torq_swizzle_scales(const void* linear_scales, int64_t rows, int64_t k, void* out,
                                void* stream) {
  if (!linear_scales || !out) return TORQ_ERR_NULL;
  if (rows < 1 || k < 32 || k % 32 != 0) return TORQ_ERR_SHAPE;
  DeviceState* st = device_state();
  if (!st) return TORQ_ERR_LAUNCH;
  if (!st->arch_ok) return TORQ_ERR_ARCH;
  const int64_t items = ((rows + 127) / 128 * 128) * (((k / 32 + 3) / 4) * 4);
  swizzle_scales_kernel<<<ew_grid(items, 256, st->sm_count), 256, 0, static_cast<cudaStream_t>(stream)>>>(
      static_cast<const uint8_t*>(linear_scales), rows, k / 32, static_cast<uint8_t*>(out));
  return launch_status();
}

// ---- offline weight side (Algorithm 3 step 5, option B) ------------------------------------------
// Workspace: the three-term bf16 split of W^T [N, 3 d], then (256-byte aligned) W' as float32 [N, d].
static size_t prep_split_bytes(int64_t d, int64_t N) { return ((size_t)N * (size_t)d * 6 + 255) / 256 * 256; }

size_t torq_prepare_weights_workspace_bytes(int64_t d, int64_t N) {
  if (d <= 0 || N <= 0) return 0;
  return prep_split_bytes(d, N) + (size_t)N * (size_t)d * 4;
}

// W' (float32 [N, d]) into the workspace; returns its address in *wp.
static torq_status rotate_weights(const void* W, const void* R_inter, const void* R_intra, int64_t d, int64_t N,
                                  void* workspace, size_t workspace_bytes, void* stream, float** wp) {
  if (!W || !R_inter) return TORQ_ERR_NULL;
  if (d < 64 || d % 64 != 0 || N < 1 || N > (1 << 30) || d > (1 << 24)) return TORQ_ERR_SHAPE;
  if (!workspace || workspace_bytes < torq_prepare_weights_workspace_bytes(d, N)) return TORQ_ERR_WORKSPACE;
  if ((reinterpret_cast<uintptr_t>(workspace) & 255u) != 0 || !aligned16(W)) return TORQ_ERR_ALIGN;
  DeviceState* st = device_state();
  if (!st) return TORQ_ERR_LAUNCH;
  if (!st->arch_ok) return TORQ_ERR_ARCH;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  __nv_bfloat16* T = static_cast<__nv_bfloat16*>(workspace);
  *wp = reinterpret_cast<float*>(static_cast<uint8_t*>(workspace) + prep_split_bytes(d, N));
  const int64_t tiles = ((N + 31) / 32) * ((d + 31) / 32);
  transpose_split3_kernel<<<ew_grid(tiles, 1, st->sm_count), 256, 0, s>>>(static_cast<const float*>(W), d, N, T);
  if (launch_status() != TORQ_OK) return TORQ_ERR_LAUNCH;
  return rotate_quantize_impl(T, R_inter, R_intra, N, d, *wp, nullptr, stream, FMT_F32OUT, 0.0f, 3);
}

torq_status torq_prepare_weights(const void* W, const void* R_inter, const void* R_intra, int64_t d, int64_t N,
                                 void* Wq, void* Ws, void* workspace, size_t workspace_bytes, void* stream) {
  if (!Wq || !Ws) return TORQ_ERR_NULL;
  float* wp = nullptr;
  const torq_status rc = rotate_weights(W, R_inter, R_intra, d, N, workspace, workspace_bytes, stream, &wp);
  if (rc != TORQ_OK) return rc;
  return torq_quantize_mxfp4(wp, TORQ_F32, N, d, Wq, Ws, stream);
}

torq_status torq_prepare_weights_nvfp4(const void* W, const void* R_inter, const void* R_intra32, int64_t d,
                                       int64_t N, void* Wq, void* Ws, float* tensor_scale, void* workspace,
                                       size_t workspace_bytes, void* stream) {
  if (!Wq || !Ws || !tensor_scale) return TORQ_ERR_NULL;
  float* wp = nullptr;
  torq_status rc = rotate_weights(W, R_inter, R_intra32, d, N, workspace, workspace_bytes, stream, &wp);
  if (rc != TORQ_OK) return rc;
  DeviceState* st = device_state();
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  // the split of W^T is no longer needed: its first word holds the running maximum
  unsigned int* amax_bits = static_cast<unsigned int*>(workspace);
  if (cudaMemsetAsync(amax_bits, 0, sizeof(unsigned int), s) != cudaSuccess) return TORQ_ERR_LAUNCH;
  absmax_kernel<<<ew_grid(N * d, 1024, st->sm_count), 256, 0, s>>>(wp, N * d, amax_bits);
  if (launch_status() != TORQ_OK) return TORQ_ERR_LAUNCH;
  float amax = 0.f;
  if (cudaMemcpyAsync(&amax, amax_bits, sizeof(float), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
      cudaStreamSynchronize(s) != cudaSuccess)
    return TORQ_ERR_LAUNCH;
  const float ts = amax / 2688.0f;                       // amax / (6 * 448), one float32 division
  if (!scale_ok(ts)) return TORQ_ERR_SHAPE;              // an all-zero (or non-finite) W' has no scale
  *tensor_scale = ts;
  return torq_quantize_nvfp4(wp, TORQ_F32, N, d, ts, Wq, Ws, stream);
}

torq_status torq_prepare_weights_mxint4(const void* W, const void* R_inter, const void* R_intra, int64_t d,
                                        int64_t N, void* Wn, void* W8, void* Ws, void* workspace,
                                        size_t workspace_bytes, void* stream) {
  if ((!Wn && !W8) || !Ws) return TORQ_ERR_NULL;
  float* wp = nullptr;
  torq_status rc = rotate_weights(W, R_inter, R_intra, d, N, workspace, workspace_bytes, stream, &wp);
  if (rc != TORQ_OK) return rc;
  if (Wn) {
    rc = torq_quantize_mxint4(wp, TORQ_F32, N, d, 1, Wn, Ws, stream);
    if (rc != TORQ_OK) return rc;
  }
  if (W8) return torq_quantize_mxint4(wp, TORQ_F32, N, d, 0, W8, Ws, stream);
  return TORQ_OK;
}

torq_status torq_merge_rotations_bf16(const void* R_inter, const void* R_intra, int64_t d, void* R_merged_bf16,
                                      void* stream) {
  if (!R_inter || !R_intra || !R_merged_bf16) return TORQ_ERR_NULL;
  if (d < 32 || d % 32 != 0 || d > (1 << 24)) return TORQ_ERR_SHAPE;
  DeviceState* st = device_state();
  if (!st) return TORQ_ERR_LAUNCH;
  if (!st->arch_ok) return TORQ_ERR_ARCH;
  merge_rotations_kernel<__nv_bfloat16><<<ew_grid(d * d, 256, st->sm_count), 256, 0, static_cast<cudaStream_t>(stream)>>>(
      static_cast<const __nv_bfloat16*>(R_inter), static_cast<const __nv_bfloat16*>(R_intra), d,
      static_cast<__nv_bfloat16*>(R_merged_bf16));
  return launch_status();
}

torq_status torq_merge_rotations(const void* R_inter, const void* R_intra, int64_t d, void* R_merged_f32,
                                 void* stream) {
  if (!R_inter || !R_intra || !R_merged_f32) return TORQ_ERR_NULL;
  if (d < 32 || d % 32 != 0 || d > (1 << 24)) return TORQ_ERR_SHAPE;
  DeviceState* st = device_state();
  if (!st) return TORQ_ERR_LAUNCH;
  if (!st->arch_ok) return TORQ_ERR_ARCH;
  merge_rotations_kernel<float><<<ew_grid(d * d, 256, st->sm_count), 256, 0, static_cast<cudaStream_t>(stream)>>>(
      static_cast<const __nv_bfloat16*>(R_inter), static_cast<const __nv_bfloat16*>(R_intra), d,
      static_cast<float*>(R_merged_f32));
  return launch_status();
}

}  // extern "C"

