// tcgen05 GEMM for the transformer sublayers run on the kept rows (Fig. 3b: "Attention or FFN layers
// using FastVAR"): out = epilogue(A[M,K] * W[N,K]^T + bias), bf16 operands, fp32 accumulation in TMEM.
//
// Persistent kernel: one CTA per SM walks over 128 x BN output tiles (tile t = blockIdx.x + i*gridDim.x,
// m fastest so that the CTAs running together share W tiles in L2).  Warp roles:
//   warp 0   : TMA producer -- streams 128x64 A tiles and BNx64 W tiles (128-byte swizzle) through a
//              ring of shared-memory stages guarded by full/empty mbarriers; the ring runs across tiles.
//   warp 1   : allocates TMEM (two accumulators of BN columns), and one lane issues tcgen05.mma
//              (M=128, N=BN, K=16) four times per stage; tcgen05.commit releases the stage and, after
//              the last k-block of a tile, signals that tile's accumulator.
//   warps 2-5: epilogue -- tcgen05.ld the accumulator (thread = row, 32 columns at a time), fuse bias /
//              GELU / gate+residual / the Q | K-cache | V^T-cache split, and store; the accumulator is
//              handed back as soon as it is in registers, so the epilogue of tile i runs under the
//              MMAs of tile i+1.  (Residual epilogues: warps 2-9, gemm_epilogue.cuh.)
// BN (128 / 192 / 256) is picked per shape on the host to minimise rounds x tile width on the SM count.
// Shapes with too few tiles to occupy the GPU (the small scale steps, where the GEMM is a stream of weights) split K over the CTAs of a
// cluster (gemm_cluster.cu).
// Every wait is bounded; on expiry a code is written to the status word and the CTA unwinds normally.
#include <cuda.h>
#include <cuda_bf16.h>

#include <mutex>

#include "gemm_choice.h"
#include "gemm_epilogue.cuh"
#include "internal.h"
#include "sm100.cuh"

namespace fv {

using namespace gemm_detail;

namespace {

constexpr int BM = 128;
constexpr int BK = 64;
constexpr int kATileBytes = BM * BK * 2;  // 16 KB

// kKps: k-blocks per pipeline stage.  The producer and the MMA issuer both pay a fixed price per stage (a barrier's wait, a
// commit or an expect), which for tiles of up to 128 columns exceeds the time of one k-block's MMAs: the producer alone takes
// 394 clocks per k-block with one of them per stage and 282 with two.  The wider tiles keep one k-block per stage: their MMAs
// take that long anyway, and two k-blocks would leave two stages (398 -> 537 clocks for 192-wide tiles).
template <int BN> struct GemmCfg {
  static constexpr int kKps = (BN <= 128) ? 2 : 1;
  static constexpr int kBTileBytes = BN * BK * 2;
  static constexpr int kSubBytes = kATileBytes + kBTileBytes;   // one k-block: A tile, then W tile
  static constexpr int kStageBytes = kKps * kSubBytes;
  static constexpr int kStages = (BN == 256) ? 4 : (BN == 192 ? 5 : (BN == 128 ? 3 : 4));
  static constexpr int kTmemCols = (BN <= 64) ? 128 : ((BN == 128) ? 256 : 512);  // two accumulators, power of two
  static constexpr int kAccStride = (BN <= 64) ? 64 : ((BN == 128) ? 128 : 256);  // column offset of the second accumulator
  // operand stages | per-warp bias slices | barriers | (residual-epilogue kernels only) one turning tile per warp
  static constexpr int smem_bytes(bool resid) {
    return kStages * kStageBytes + (resid ? kResidBiasBytes + kResidSmemBytes : kBiasSmemBytes) + 256 /*barriers*/ + 1024 /*alignment slack*/;
  }
};

// KIND 1 / 3 (RESID): the instantiations launched for the residual epilogue of an fp32 / a bf16 stream, 5 / 7 for rows of a map.  They are kernels of their own because
// that epilogue takes eight warps and more registers per thread; the others stay small enough for a bandwidth-bound kernel of another
// stream (the restoration of the rows that were not kept) to share the SMs with them.
template <int BN, int KIND>
__device__ __forceinline__ void gemm_body(const CUtensorMap& tmA, const CUtensorMap& tmB, const GemmDev p) {
  using Cfg = GemmCfg<BN>;
  constexpr int STAGES = Cfg::kStages;
  constexpr int KPS = Cfg::kKps;
  constexpr bool RESID = is_resid(KIND);   // KIND 2: the QKV projection with cosine attention / rotary positions on Q and K
  constexpr bool XB = is_resid_bf16(KIND), MAP = is_resid_map(KIND);
  constexpr int kBiasBytes = RESID ? kResidBiasBytes : kBiasSmemBytes;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint4* bias_s = reinterpret_cast<uint4*>(smem + STAGES * Cfg::kStageBytes);   // per-warp bias slice of the tile
  uint64_t* full_bar = reinterpret_cast<uint64_t*>(smem + STAGES * Cfg::kStageBytes + kBiasBytes);
  float* resid_s = reinterpret_cast<float*>(smem + STAGES * Cfg::kStageBytes + kBiasBytes + 256);   // RESID: one tile per warp
  uint64_t* empty_bar = full_bar + STAGES;
  uint64_t* acc_full = empty_bar + STAGES;   // [2]
  uint64_t* acc_empty = acc_full + 2;        // [2]
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_empty + 2);

  pdl_trigger();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int tiles_m = (p.M + BM - 1) / BM;
  const int tiles_n = (p.N + BN - 1) / BN;
  const int total_tiles = tiles_m * tiles_n;
  const int num_kb = (p.K + BK - 1) / BK;

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) { mbar_init(&full_bar[s], 1); mbar_init(&empty_bar[s], 1); }
    for (int s = 0; s < 2; ++s) { mbar_init(&acc_full[s], 1); mbar_init(&acc_empty[s], gemm_threads(KIND) - 64); }
    mbar_fence_init();
    tma_prefetch_desc(&tmA);
    tma_prefetch_desc(&tmB);
  }
  if (warp == 1) { tmem_alloc(tmem_slot, Cfg::kTmemCols); tmem_relinquish(); }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  // Set-up above overlaps the previous kernel.  Activations and outputs are touched only after
  // pdl_wait(); the weight tiles (never written by a kernel of the step) are requested before it.

  if (warp == 0) {
    if (lane == 0) {
      uint32_t it = 0;
      bool ok = true;
      int pre = 0;  // stages of the first tile whose W tile is already on its way
      if ((int)blockIdx.x < total_tiles) {
        const int n0 = ((int)blockIdx.x / tiles_m) * BN;
        pre = min(STAGES, (num_kb + KPS - 1) / KPS);
        for (int i = 0; i < pre; ++i) {
          mbar_expect_tx(&full_bar[i], Cfg::kStageBytes);
          for (int u = 0; u < KPS; ++u)   // (a k-block beyond K reads zeros)
            tma_load_2d(smem + i * Cfg::kStageBytes + u * Cfg::kSubBytes + kATileBytes, &tmB, (KPS * i + u) * BK, n0, &full_bar[i]);
        }
      }
      pdl_wait();
      for (int tile = blockIdx.x; ok && tile < total_tiles; tile += gridDim.x) {
        const int m0 = (tile % tiles_m) * BM, n0 = (tile / tiles_m) * BN;
        for (int kb = 0; kb < num_kb; kb += KPS, ++it) {   // one stage: KPS k-blocks
          const int s = it % STAGES;
          uint8_t* a_s = smem + s * Cfg::kStageBytes;
          if ((int)it < pre) {  // W tiles requested before the wait: only the activations are missing
            for (int u = 0; u < KPS; ++u) tma_load_2d(a_s + u * Cfg::kSubBytes, &tmA, (kb + u) * BK, m0, &full_bar[s]);
            continue;
          }
          const uint32_t ph = (it / STAGES) & 1;
          if (!mbar_wait(&empty_bar[s], ph ^ 1)) { report(p.status, DEV_TIMEOUT_TMA); ok = false; break; }
          mbar_expect_tx(&full_bar[s], Cfg::kStageBytes);
          for (int u = 0; u < KPS; ++u) {
            tma_load_2d(a_s + u * Cfg::kSubBytes, &tmA, (kb + u) * BK, m0, &full_bar[s]);
            tma_load_2d(a_s + u * Cfg::kSubBytes + kATileBytes, &tmB, (kb + u) * BK, n0, &full_bar[s]);
          }
        }
      }
    }
  } else if (warp == 1) {
    pdl_wait();
    {
      constexpr uint32_t idesc = umma_idesc_bf16(BM, BN);
      const bool leader = elect_one();
      uint32_t lt = 0, s = 0, ph = 0;   // tile count; ring stage and its phase
      bool ok = true;
      for (int tile = blockIdx.x; ok && tile < total_tiles; tile += gridDim.x, ++lt) {
        const uint32_t buf = lt & 1;
        if (!mbar_wait(&acc_empty[buf], ((lt >> 1) & 1) ^ 1)) { report(p.status, DEV_TIMEOUT_MMA); ok = false; break; }
        tc_fence_after();
        const uint32_t d = tmem_base + buf * Cfg::kAccStride;
        for (int kb = 0; kb < num_kb; kb += KPS) {
          if (!mbar_wait(&full_bar[s], ph)) { report(p.status, DEV_TIMEOUT_MMA); ok = false; break; }
          tc_fence_after();
          const uint64_t desc = umma_desc_k_sw128(smem_u32(smem + s * Cfg::kStageBytes));
          if (leader) {
#pragma unroll
            for (int u = 0; u < KPS; ++u) {
              const uint64_t adesc = desc + u * (Cfg::kSubBytes >> 4), bdesc = adesc + (kATileBytes >> 4);
#pragma unroll
              for (int kk = 0; kk < BK / 16; ++kk)
                umma_bf16(d, adesc + 2 * kk, bdesc + 2 * kk, idesc, (kb | u | kk) != 0);
            }
            umma_commit(&empty_bar[s]);
          }
          if (++s == STAGES) { s = 0; ph ^= 1; }
        }
        if (ok && leader) umma_commit(&acc_full[buf]);
      }
    }
  } else {
    // ---- epilogue: thread = one accumulator row, 32 fp32 columns per tcgen05.ld ----
    pdl_wait();
    const int quarter = warp & 3;
    const uint32_t lane_off = uint32_t(quarter * 32) << 16;
    uint32_t lt = 0;
    [[maybe_unused]] bool ok = true;
    for (int tile = blockIdx.x; tile < total_tiles; tile += gridDim.x, ++lt) {
      const uint32_t buf = lt & 1;
      const int m0 = (tile % tiles_m) * BM, n0 = (tile / tiles_m) * BN;
      const int row = m0 + quarter * 32 + lane;
      const bool row_ok = row < p.M;
      uint4* bias_w = bias_s + (RESID ? warp - 2 : quarter) * 32;
      stage_bias(p, bias_w, lane, n0, BN);
      const uint32_t t0 = tmem_base + lane_off + buf * Cfg::kAccStride;
      if constexpr (RESID) {
        const int half = (warp - 2) >> 2;
        const auto release = [&] { tc_fence_before(); mbar_arrive(&acc_empty[buf]); };
        // the first chunk of `out` is on its way while the accumulator is computed
        const bool turned = p.rows_per_image >= 32 || p.epilogue == EPI_F32;   // (images of fewer than 32 rows take the row-per-thread path)
        ResidRows<MAP> rr;
        typename ResidX<XB>::Raw x[8];
        if (turned) {
          rr = resid_rows<MAP>(p, lane, m0 + quarter * 32);
          residual_load_x<XB, MAP>(p, rr, x, lane, n0 + 32 * half);
        }
        if (ok && !mbar_wait(&acc_full[buf], (lt >> 1) & 1)) { report(p.status, DEV_TIMEOUT_EPI); ok = false; }
        ok = __all_sync(0xffffffffu, ok);
        if (!MAP && !ok) break;
        tc_fence_after();
        if constexpr (MAP) {        // (images of at least 128 rows)
          if (ok) residual_tile<XB, true, BN>(p, rr, x, t0, half, lane, n0, bias_w, resid_s + (warp - 2) * kResidTileFloats, release);
          residual_tile_sums<BN>(p, resid_s, (int)threadIdx.x - 64, m0, n0, ok);
        } else if (turned) {
          residual_tile<XB, false, BN>(p, rr, x, t0, half, lane, n0, bias_w, resid_s + (warp - 2) * kResidTileFloats, release);
        } else {
          const int img = row_ok ? row / p.rows_per_image : 0, jrow = row_ok ? row - img * p.rows_per_image : 0;
#pragma unroll 1
          for (int c0 = 32 * half; c0 < BN; c0 += 64) {
            uint32_t r[32];
            tmem_ld32(t0 + c0, r);
            tmem_wait_ld();
            if (c0 + 64 >= BN) release();
            if (row_ok && n0 + c0 < p.N) epilogue_chunk(p, r, row, img, jrow, n0 + c0, bias_w + c0 / 8);
          }
        }
        continue;
      }
      if (!mbar_wait(&acc_full[buf], (lt >> 1) & 1)) { report(p.status, DEV_TIMEOUT_EPI); break; }
      tc_fence_after();
      const int img = row_ok ? row / p.rows_per_image : 0;
      const int jrow = row_ok ? row - img * p.rows_per_image : 0;
      if (KIND == 2) {
        qkv_extras_tile<BN>(p, t0, row, row_ok, img, jrow, n0, bias_w);
        tc_fence_before();
        mbar_arrive(&acc_empty[buf]);
      } else {
#pragma unroll 1
        for (int c0 = 0; c0 < BN; c0 += 64) {
          // two chunks in flight: the second load overlaps the first chunk's stores
          uint32_t r0[32], r1[32];
          tmem_ld32(t0 + c0, r0);
          tmem_ld32(t0 + c0 + 32, r1);
          tmem_wait_ld();
          if (c0 + 64 >= BN) {  // accumulator fully in registers: hand the buffer back to the MMA warp
            tc_fence_before();
            mbar_arrive(&acc_empty[buf]);
          }
          const int col = n0 + c0;
          if (row_ok && col < p.N) epilogue_chunk(p, r0, row, img, jrow, col, bias_w + c0 / 8);
          if (row_ok && col + 32 < p.N) epilogue_chunk(p, r1, row, img, jrow, col + 32, bias_w + c0 / 8 + 4);
        }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    __syncwarp();
    tmem_dealloc(tmem_base, Cfg::kTmemCols);
  }
}

template <int BN, int KIND>
__global__ void __launch_bounds__(gemm_threads(KIND), 1)
gemm_bf16_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, const GemmDev p) { gemm_body<BN, KIND>(tmA, tmB, p); }

// The kept rows of a large map on 64-wide tiles (gemm_leaves_room): this kernel's CTAs come early, before all CTAs of the restoration of the other rows
// are placed, and wait.  Ten warps put three on a scheduler, so 3 x R registers a lane and two warps of the restoration (80) fit the scheduler's 512 up
// to R = 117; with 158 the restoration had to crowd on the SMs left (56 ... 60 us instead of 38 ... 44 behind two images of 64 x 64 tokens, C 2048, 143 kept
// rows; us per block there 285 -> 250; one image, C 1920, 400 rows 191 -> 170; 80 x 80, C 1920, 300 rows 191 -> 171; 96 x 96, C 2048, 300 rows 314 -> 284).
template <int KIND>
__global__ void __maxnreg__(112)
gemm_beside_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, const GemmDev p) { gemm_body<64, KIND>(tmA, tmB, p); }

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                  const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeTiledFn g_encode = nullptr;
int g_num_sms = 148;
std::once_flag g_encode_once;

void load_encode() {
  void* fn = nullptr;
  cudaDriverEntryPointQueryResult qres;
  if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &qres) == cudaSuccess &&
      qres == cudaDriverEntryPointSuccess)
    g_encode = reinterpret_cast<EncodeTiledFn>(fn);
}

template <int BN, int KIND> cudaError_t set_attr() {
  return cudaFuncSetAttribute(gemm_bf16_kernel<BN, KIND>, cudaFuncAttributeMaxDynamicSharedMemorySize, GemmCfg<BN>::smem_bytes(is_resid(KIND)));
}

}  // namespace

bool make_tmap_bf16_2d(void* tmap_out, const void* base, uint64_t rows, uint64_t cols, uint32_t box_rows) {
  std::call_once(g_encode_once, load_encode);
  if (!g_encode) return false;
  cuuint64_t dims[2] = {cols, rows};
  cuuint64_t strides[1] = {cols * 2};
  cuuint32_t box[2] = {64, box_rows};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = g_encode(static_cast<CUtensorMap*>(tmap_out), CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims,
                        strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                        CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}

cudaError_t gemm_init() {
  cudaError_t e = set_attr<128, 0>();
  if (e == cudaSuccess) e = set_attr<192, 0>();
  if (e == cudaSuccess) e = set_attr<256, 0>();
  if (e == cudaSuccess) e = set_attr<128, 1>();
  if (e == cudaSuccess) e = set_attr<192, 1>();
  if (e == cudaSuccess) e = set_attr<256, 1>();
  if (e == cudaSuccess) e = set_attr<64, 0>();
  if (e == cudaSuccess) e = set_attr<64, 1>();
  if (e == cudaSuccess) e = cudaFuncSetAttribute(gemm_beside_kernel<5>, cudaFuncAttributeMaxDynamicSharedMemorySize, GemmCfg<64>::smem_bytes(true));
  if (e == cudaSuccess) e = cudaFuncSetAttribute(gemm_beside_kernel<7>, cudaFuncAttributeMaxDynamicSharedMemorySize, GemmCfg<64>::smem_bytes(true));
  if (e == cudaSuccess) e = set_attr<64, 5>();
  if (e == cudaSuccess) e = set_attr<128, 5>();
  if (e == cudaSuccess) e = set_attr<192, 5>();
  if (e == cudaSuccess) e = set_attr<256, 5>();
  if (e == cudaSuccess) e = set_attr<64, 7>();
  if (e == cudaSuccess) e = set_attr<128, 7>();
  if (e == cudaSuccess) e = set_attr<192, 7>();
  if (e == cudaSuccess) e = set_attr<256, 7>();
  if (e == cudaSuccess) e = set_attr<64, 3>();
  if (e == cudaSuccess) e = set_attr<128, 3>();
  if (e == cudaSuccess) e = set_attr<192, 3>();
  if (e == cudaSuccess) e = set_attr<256, 3>();
  if (e == cudaSuccess) e = set_attr<128, 2>();
  if (e == cudaSuccess) e = set_attr<192, 2>();
  if (e == cudaSuccess) e = set_attr<256, 2>();
  if (e == cudaSuccess) e = gemm_pair_init();
  if (e == cudaSuccess) e = gemm_cluster_init();
  if (e != cudaSuccess) return e;
  int dev = 0;
  e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  return cudaDeviceGetAttribute(&g_num_sms, cudaDevAttrMultiProcessorCount, dev);
}

// Size that scratch for a K split through global memory had.  No shape takes one any more (clusters do it, without scratch); callers may
// still ask for the size and pass the buffer.
size_t gemm_splitk_ws_bytes() { return 4096 + (size_t)2 * 148 * BM * 128 * sizeof(float); }

template <int BN>
static cudaError_t launch_bn(const GemmArgs& g, const GemmDev& p, int tiles_m, cudaStream_t st) {
  alignas(64) CUtensorMap tmA, tmB;
  if (!make_tmap_bf16_2d(&tmA, g.a, g.M, g.K, BM)) return cudaErrorInvalidValue;
  if (!make_tmap_bf16_2d(&tmB, g.w, g.N, g.K, BN)) return cudaErrorInvalidValue;
  const long tiles = (long)tiles_m * ((g.N + BN - 1) / BN);
  const int grid = (int)(tiles < g_num_sms ? tiles : g_num_sms);
  if constexpr (BN == 64)
    if (p.row_idx && gemm_leaves_room(g.M, g.rows_per_image, g.map_tokens, g.N))
      return launch_pdl(p.epilogue == EPI_RESIDUAL ? gemm_beside_kernel<5> : gemm_beside_kernel<7>, dim3(grid), dim3(gemm_threads(5)), GemmCfg<BN>::smem_bytes(true), st, tmA, tmB, p);
  if (p.row_idx && p.epilogue == EPI_RESIDUAL)
    return launch_pdl(gemm_bf16_kernel<BN, 5>, dim3(grid), dim3(gemm_threads(5)), GemmCfg<BN>::smem_bytes(true), st, tmA, tmB, p);
  if (p.row_idx)
    return launch_pdl(gemm_bf16_kernel<BN, 7>, dim3(grid), dim3(gemm_threads(7)), GemmCfg<BN>::smem_bytes(true), st, tmA, tmB, p);
  if (p.epilogue == EPI_RESIDUAL || p.epilogue == EPI_F32)
    return launch_pdl(gemm_bf16_kernel<BN, 1>, dim3(grid), dim3(gemm_threads(1)), GemmCfg<BN>::smem_bytes(true), st, tmA, tmB, p);
  if (p.epilogue == EPI_RESIDUAL_XBF16)
    return launch_pdl(gemm_bf16_kernel<BN, 3>, dim3(grid), dim3(gemm_threads(3)), GemmCfg<BN>::smem_bytes(true), st, tmA, tmB, p);
  if constexpr (BN < 128)
    if (p.epilogue == EPI_QKV_SPLIT && (p.qk_scale || p.rope_table)) return cudaErrorInvalidValue;   // never chosen for them
  if constexpr (BN >= 128)
    if (p.epilogue == EPI_QKV_SPLIT && (p.qk_scale || p.rope_table))
      return launch_pdl(gemm_bf16_kernel<BN, 2>, dim3(grid), dim3(gemm_threads(2)), GemmCfg<BN>::smem_bytes(false), st, tmA, tmB, p);
  return launch_pdl(gemm_bf16_kernel<BN, 0>, dim3(grid), dim3(gemm_threads(0)), GemmCfg<BN>::smem_bytes(false), st, tmA, tmB, p);
}

// Bytes of the operands and results of a GEMM: A, W, and what its epilogue reads and writes (a residual epilogue the stream both ways, a copy of the branch
// output beside it, the column sums of the rows of a map).
static double operand_bytes(const GemmArgs& g) {
  const double mn = (double)g.M * g.N;
  double out = mn * (g.epilogue == EPI_RESIDUAL ? 8.0 : (g.epilogue == EPI_RESIDUAL_XBF16 || g.epilogue == EPI_F32 ? 4.0 : 2.0));
  if (g.aux && (g.epilogue == EPI_RESIDUAL || g.epilogue == EPI_RESIDUAL_XBF16)) out += 2.0 * mn;
  if (g.colsum)
    for (int img = 0; img < g.M / g.rows_per_image; ++img) out += 4.0 * g.N * map_colsum_count(img, g.rows_per_image);
  return 2.0 * ((double)g.M * g.K + (double)g.N * g.K) + out;
}

static int g_force_path = 0;
void gemm_force_path(int path) { g_force_path = path; }

fv_status launch_gemm(const GemmArgs& g, cudaStream_t st) {
  if (g.M <= 0 || g.N <= 0 || g.K <= 0 || (g.K % 8) || (g.N % 8) || !g.a || !g.w) return FV_ERR_INVALID_ARG;
  if (g.rows_per_image <= 0) return FV_ERR_INVALID_ARG;
  if (g.epilogue == EPI_QKV_SPLIT && (g.C % 128 || g.q_cols % 128)) return FV_ERR_UNSUPPORTED;
  const int tiles_m = (g.M + BM - 1) / BM;
  // Q / K extras (cosine attention, rotary positions): one-CTA tiles that hold whole heads, no K split
  const bool qk_extras = g.epilogue == EPI_QKV_SPLIT && (g.qk_scale || g.rope_table);
  if (qk_extras && g.head_dim != 64 && g.head_dim != 128) return FV_ERR_UNSUPPORTED;
  // rows of a map: a tile's 128 rows hold at most two images, and the tile is one CTA's or a pair's
  const bool map = g.row_idx != nullptr;
  if (map && ((g.epilogue != EPI_RESIDUAL && g.epilogue != EPI_RESIDUAL_XBF16) || !g.row_inv || g.map_tokens <= 0 || g.rows_per_image < kMinMapRows || g.aux))
    return FV_ERR_UNSUPPORTED;
  TileChoice tc = pick_tile(g.M, g.N, g.K, g_num_sms, qk_extras ? g.head_dim : 0, !map);
  const TileChoice picked = tc;
  if (g_force_path == 1 && tc.pair) tc = TileChoice{256, false, 1};
  if (g_force_path == 2) tc = TileChoice{256, true, 1};
  if (g_force_path == 3) tc = TileChoice{128, true, 1};
  if (g_force_path >= 4 && g_force_path <= 6) tc = TileChoice{128 + 64 * (g_force_path - 4), false, 1};
  if (g_force_path == 7) tc = TileChoice{64, false, 1};
  if (qk_extras) {   // (a forced tile is widened until it is allowed)
    if (tc.pair) tc = TileChoice{256, false, 1};
    if (tc.bn < 128) tc.bn = 128;            // the extras exist for tiles of at least 128 columns
    if (tc.bn % g.head_dim) tc.bn = 256;
  }
  int bn = tc.bn;
  GemmDev p;
  p.kb_per_split = 0;   // (clusters)
  p.bias = static_cast<const __nv_bfloat16*>(g.bias);
  p.M = g.M; p.N = g.N; p.K = g.K; p.epilogue = g.epilogue; p.out = g.out; p.aux = g.aux; p.gamma = g.gamma;
  if (g.epilogue == EPI_F32) { p.aux = nullptr; p.gamma = nullptr; }
  p.mod_stride = g.mod_stride; p.rows_per_image = g.rows_per_image; p.q_cols = g.q_cols; p.C = g.C;
  p.k_cache = static_cast<__nv_bfloat16*>(g.k_cache); p.vt_cache = static_cast<__nv_bfloat16*>(g.vt_cache);
  p.kv_capacity = g.kv_capacity; p.kv_offset = g.kv_offset; p.status = g.status;
  p.qk_scale = qk_extras ? g.qk_scale : nullptr;
  p.rope_table = qk_extras ? reinterpret_cast<const float2*>(g.rope_table) : nullptr;
  p.rope_idx = qk_extras ? g.rope_idx : nullptr;
  p.head_dim = g.head_dim;
  p.row_idx = g.row_idx; p.row_inv = g.row_inv; p.map_tokens = g.map_tokens; p.colsum = g.colsum; p.colsum_slots = map_colsum_slots(g.rows_per_image);
  // K split over the CTAs of a cluster, the partials reduced through distributed shared memory.  Up to 48 rows two CTAs
  // share an SM (gemm_cluster.cu): 8 slices while the CTAs stay within one per SM, else 4 within two, else 2 (us at M 8, weights from HBM,
  // 8 / 4 / 2 slices: N 2048 K 2048 3.9 / 4.6 / 6.4; N 6144 9.1 / 6.7 / 8.0; N 8192 10.1 / 7.6 / 8.9; N 2048 K 8192 9.0 / 11.9 / 20;
  // 1024-wide models N 3072 3.7 / 3.6 / 4.2; N 1024 K 4096 4.6 / 6.4 / 10.3).  From 64 rows on the other tiles are as fast or faster.
  int cluster_slices = 0, cluster_bn = 0;
  if (g_force_path == 0 && !qk_extras && !map) {
    const long t128 = (g.N + 127) / 128;
    if (g.M <= 48 && g.K > 7 * BK && t128 <= g_num_sms) { cluster_bn = 128; cluster_slices = t128 * 8 <= g_num_sms ? 8 : (t128 * 4 <= 2 * g_num_sms ? 4 : 2); }
    else if (picked.slices > 1) { cluster_bn = picked.bn; cluster_slices = picked.slices; }
  }
  if (g_force_path >= 8 && g_force_path <= 11 && !qk_extras && !map) {   // 8: 128 wide x 4 slices, 9: 128 x 2, 10: 64 x 4, 11: 64 x 2
    cluster_bn = g_force_path <= 9 ? 128 : 64;
    cluster_slices = (g_force_path & 1) ? 2 : 4;
  }
  if (g_force_path == 12 && !qk_extras && !map && g.M <= 48) { cluster_bn = 128; cluster_slices = 8; }   // (few rows only)
  if (cluster_slices) {
    const int num_kb = (g.K + BK - 1) / BK;
    p.kb_per_split = (num_kb + cluster_slices - 1) / cluster_slices;
    p.kb_per_split += p.kb_per_split & 1;   // even: a pipeline stage of the cluster kernel may hold two k-blocks of ONE slice
  }
  LaunchScope scope(KC_GEMM, 1, 2.0 * g.M * (double)g.N * g.K, operand_bytes(g), st);
  if (cluster_slices) return launch_gemm_cluster(g, p, cluster_bn, cluster_slices, st) == cudaSuccess ? FV_OK : FV_ERR_CUDA;
  if (tc.pair) {
    cudaError_t e2 = launch_gemm_pair(g, p, bn, st);
    return e2 == cudaSuccess ? FV_OK : FV_ERR_CUDA;
  }
  cudaError_t e = bn == 256 ? launch_bn<256>(g, p, tiles_m, st)
                : (bn == 192 ? launch_bn<192>(g, p, tiles_m, st) : (bn == 64 ? launch_bn<64>(g, p, tiles_m, st) : launch_bn<128>(g, p, tiles_m, st)));
  return e == cudaSuccess ? FV_OK : FV_ERR_CUDA;
}

}  // namespace fv
