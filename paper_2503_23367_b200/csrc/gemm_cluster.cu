// K split inside a thread-block cluster: the GEMMs of the small scale steps (few rows against a large weight
// matrix) have too few output tiles to occupy the GPU, so S CTAs of one cluster share a tile and each takes
// 1/S of its k-blocks.  The partial accumulators never go through global memory: every CTA writes the rows
// that another CTA owns straight into that CTA's shared memory (distributed shared memory), one cluster
// barrier later every CTA adds the S partials of its own 128/S rows in rank order and runs the epilogue for
// them -- a reduce-scatter, so the work after the barrier shrinks with S instead of growing, and the result
// does not depend on timing.  No scratch buffer, no arrival counters.
//
// One tile per cluster, one accumulator of BN columns in TMEM per CTA; warp roles as in gemm.cu (warp 0 TMA
// producer, warp 1 MMA issuer, warps 2-5 accumulator readers / epilogue).  Every mbarrier wait is bounded; a
// CTA whose wait expires reports it and still takes part in the cluster barrier, so the others never hang.
#include <cuda.h>
#include <cuda_bf16.h>

#include "gemm_epilogue.cuh"
#include "internal.h"
#include "sm100.cuh"

namespace fv {

using namespace gemm_detail;

namespace {

constexpr int BM = 128;
constexpr int BK = 64;
constexpr int kThreads = 192;

// Up to 48 rows (FLIP) the operands change places: 128 rows of W are the M side of the MMA and the ROWS rows of A its N side, so the
// accumulator is the tile transposed.  An MMA reads its M operand whole, 128 rows of it, whatever the GEMM's own rows: with A there, 64-wide
// tiles cost 64 clocks per 16 of K, most of them for rows that do not exist, and the MMAs of a slice were the longest part of a launch
// (M 4, K 4096 in four slices: 4500 of 7000 clocks).  Us per launch of a chain, weights from HBM, before -> after: M 4 N 6144 K 2048
// 8.3 -> 6.6 (the weights alone take 3.8), N 2048 K 2048 4.5 -> 3.8, N 8192 K 2048 9.0 -> 7.4, N 2048 K 8192 9.9 -> 9.0; M 32 7.8 -> 6.9,
// 4.8 -> 4.5, 8.8 -> 7.8, 10.3 -> 9.7; 1024-wide models M 25 4.1 -> 3.9, 3.4 -> 3.4, 4.7 -> 4.4, 5.4 -> 4.9.  At 64 rows the two are even:
// the transposed accumulator goes to its owners one word per lane and row.  (Reducing and finishing it four rows at a time,
// in wide words, costs more in the epilogue than it saves there: M 32 N 6144 6.9 -> 7.3.)
//
// The builds for few rows stay under 113 KB of shared memory, ring and reduce buffer together, and under 168 registers (the launch bounds say
// so: two slices of 64 rows took 190 without, and one CTA per SM: M 40 N 16384 K 2048 19.6 us, 14.1 now), so that TWO CTAs share an SM:
// the CTAs of the next GEMM of the step start (programmatic launch) beside those of this one and fetch their first
// weights while this one computes, and outputs of up to 8192 columns fit the GPU in four slices.
//
// kKps: k-blocks per pipeline stage.  Producer and MMA issuer pay a fixed price per stage (a barrier's wait, a commit or an
// expect) that exceeds the time of one k-block's MMAs of a 64-wide tile: with two k-blocks behind one barrier it is paid half as
// often.  128-wide tiles keep one (two cost a stage of ring: M 32 N 2048 K 8192 9.7 -> 10.3).
constexpr int kFlipRows = 48;   // most rows of the builds with W on the M side
template <int BN, int ROWS> struct ClusterCfg {
  static constexpr bool kFlip = ROWS < 128;
  static constexpr int kKps = BN == 128 ? 1 : 2;
  static constexpr int kATile = ROWS * BK * 2;
  static constexpr int kBTileBytes = BN * BK * 2;
  static constexpr int kSubBytes = kATile + kBTileBytes;       // one k-block: A tile, then W tile
  static constexpr int kStageBytes = kKps * kSubBytes;
  static constexpr int kStages = kFlip ? (ROWS == 32 ? 4 : 3) : (BN == 128 ? 4 : 3);
  static constexpr int kTmemCols = kFlip ? ROWS : BN;       // one accumulator (powers of two)
  static constexpr int kRedPitch = BN + 4;                  // floats per row of the reduce buffer (bank spread)
  static constexpr int kRedBytes = ROWS * kRedPitch * 4;    // [S sources][ROWS/S rows][pitch] = ROWS rows in all
  // operand stages | per-warp bias slices | barriers | reduce buffer
  static constexpr int kSmemBytes = kStages * kStageBytes + kBiasSmemBytes + 256 + kRedBytes + 1024 /*alignment slack*/;
  static_assert(!kFlip || (BN == 128 && kSmemBytes <= 113 * 1024), "two CTAs per SM");
};

__device__ __forceinline__ uint32_t map_to_cta(uint32_t local, uint32_t cta) {
  uint32_t remote;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(local), "r"(cta));
  return remote;
}
__device__ __forceinline__ void st_cluster_f4(uint32_t addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
  asm volatile("st.shared::cluster.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(a), "r"(b), "r"(c), "r"(d) : "memory");
}

__device__ __forceinline__ void st_cluster_f1(uint32_t addr, uint32_t a) {
  asm volatile("st.shared::cluster.b32 [%0], %1;" ::"r"(addr), "r"(a) : "memory");
}

template <int BN, int S, int ROWS>
__global__ void __launch_bounds__(kThreads, ClusterCfg<BN, ROWS>::kFlip ? 2 : 1)
gemm_cluster_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, const GemmDev p) {
  using Cfg = ClusterCfg<BN, ROWS>;
  constexpr bool FLIP = Cfg::kFlip;
  constexpr int kATileBytes = Cfg::kATile;
  constexpr int STAGES = Cfg::kStages;
  constexpr int KPS = Cfg::kKps;
  constexpr int ROWS_PER = ROWS / S;      // rows of the tile each CTA finishes
  // The CTA finishes ROWS_PER x BN values, four consecutive columns per epilogue thread and turn: lanes along the columns, so that a
  // warp stores whole lines; along the rows where the columns are V's (its cache is transposed: a key's neighbours are rows).
  // What a residual stream or gate contributes does not depend on the product and is fetched before the barriers, up to PRE turns
  // of it: read after the reduction it cost two dependent trips to L2, 1.7 us of a 6.4 us launch.
  constexpr int QUADS = BN / 4;
  constexpr int TURNS = ROWS_PER * QUADS / 128;
  constexpr int PRE = TURNS < 8 ? TURNS : 8;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint4* bias_s = reinterpret_cast<uint4*>(smem + STAGES * Cfg::kStageBytes);
  uint64_t* full_bar = reinterpret_cast<uint64_t*>(smem + STAGES * Cfg::kStageBytes + kBiasSmemBytes);
  uint64_t* empty_bar = full_bar + STAGES;
  uint64_t* acc_full = empty_bar + STAGES;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_full + 1);
  float* red = reinterpret_cast<float*>(smem + STAGES * Cfg::kStageBytes + kBiasSmemBytes + 256);   // [S][ROWS_PER][pitch]

  pdl_trigger();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cluster_ctarank();
  const int tile = blockIdx.x / S;
  const int tiles_m = (p.M + BM - 1) / BM;
  const int m0 = (tile % tiles_m) * BM, n0 = (tile / tiles_m) * BN;
  const int num_kb = (p.K + BK - 1) / BK;
  const int kb0 = min(num_kb, (int)rank * p.kb_per_split), kb1 = min(num_kb, kb0 + p.kb_per_split);

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) { mbar_init(&full_bar[s], 1); mbar_init(&empty_bar[s], 1); }
    mbar_init(acc_full, 1);
    mbar_fence_init();
    tma_prefetch_desc(&tmA);
    tma_prefetch_desc(&tmB);
  }
  if (warp == 1) { tmem_alloc(tmem_slot, Cfg::kTmemCols); tmem_relinquish(); }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  // first half of the "every CTA of the cluster has started" barrier; the second half precedes the first
  // store into another CTA's shared memory (a rank with an empty K slice gets there almost at once)
  cluster_arrive_relaxed();

  const bool v_tile = p.epilogue == EPI_QKV_SPLIT && n0 >= p.q_cols + p.C;
  const bool x_f32 = p.epilogue == EPI_RESIDUAL, x_b16 = p.epilogue == EPI_RESIDUAL_XBF16;
  const int et = (int)threadIdx.x - 64;                   // 0..127 among the epilogue threads
  auto place = [&](int i, int& lrow, int& quad) {
    const int f = et + 128 * i;
    lrow = v_tile ? f % ROWS_PER : f / QUADS;
    quad = v_tile ? f / ROWS_PER : f % QUADS;
  };
  float4 xv[PRE], gv[PRE];
  auto fetch = [&](int i, int slot) {   // stream and gate of turn i
    int lrow, quad;
    place(i, lrow, quad);
    const int row = m0 + (int)rank * ROWS_PER + lrow, col = n0 + 4 * quad;
    gv[slot] = make_float4(1.f, 1.f, 1.f, 1.f);
    if (row >= p.M || col >= p.N) return;
    const size_t at = (size_t)row * p.N + col;
    if (x_f32) {
      xv[slot] = *reinterpret_cast<const float4*>(static_cast<const float*>(p.out) + at);
    } else {
      const uint2 u = *reinterpret_cast<const uint2*>(static_cast<const __nv_bfloat16*>(p.out) + at);
      xv[slot] = make_float4(__uint_as_float(u.x << 16), __uint_as_float(u.x & 0xFFFF0000u), __uint_as_float(u.y << 16), __uint_as_float(u.y & 0xFFFF0000u));
    }
    if (p.gamma) gv[slot] = *reinterpret_cast<const float4*>(p.gamma + (size_t)(row / p.rows_per_image) * p.mod_stride + col);
  };

  if (warp == 0) {
    if (lane == 0) {
      // the weight tiles (never written by a kernel of the step) are requested before the dependency wait
      const int nst = (kb1 - kb0 + KPS - 1) / KPS;    // stages of KPS k-blocks; a k-block beyond K reads zeros
      const int pre = min(STAGES, nst);
      for (int i = 0; i < pre; ++i) {
        mbar_expect_tx(&full_bar[i], Cfg::kStageBytes);
        for (int u = 0; u < KPS; ++u)
          tma_load_2d(smem + i * Cfg::kStageBytes + u * Cfg::kSubBytes + kATileBytes, &tmB, (kb0 + KPS * i + u) * BK, n0, &full_bar[i]);
      }
      pdl_wait();
      for (int it = 0; it < nst; ++it) {
        const int s = it % STAGES;
        const int kb = kb0 + KPS * it;
        uint8_t* a_s = smem + s * Cfg::kStageBytes;
        if (it < pre) {
          for (int u = 0; u < KPS; ++u) tma_load_2d(a_s + u * Cfg::kSubBytes, &tmA, (kb + u) * BK, m0, &full_bar[s]);
          continue;
        }
        const uint32_t ph = (it / STAGES) & 1;
        if (!mbar_wait(&empty_bar[s], ph ^ 1)) { report(p.status, DEV_TIMEOUT_TMA); break; }
        mbar_expect_tx(&full_bar[s], Cfg::kStageBytes);
        for (int u = 0; u < KPS; ++u) {
          tma_load_2d(a_s + u * Cfg::kSubBytes, &tmA, (kb + u) * BK, m0, &full_bar[s]);
          tma_load_2d(a_s + u * Cfg::kSubBytes + kATileBytes, &tmB, (kb + u) * BK, n0, &full_bar[s]);
        }
      }
    }
  } else if (warp == 1) {
    pdl_wait();
    {
      constexpr uint32_t idesc = FLIP ? umma_idesc_bf16(BN, ROWS) : umma_idesc_bf16(BM, BN);
      const bool leader = elect_one();
      uint32_t s = 0, ph = 0;   // ring stage and its phase
      bool ok = true;
      const int nst = (kb1 - kb0 + KPS - 1) / KPS;
      for (int it = 0; it < nst; ++it) {
        if (!mbar_wait(&full_bar[s], ph)) { report(p.status, DEV_TIMEOUT_MMA); ok = false; break; }
        tc_fence_after();
        const uint64_t desc = umma_desc_k_sw128(smem_u32(smem + s * Cfg::kStageBytes));
        if (leader) {
#pragma unroll
          for (int u = 0; u < KPS; ++u) {
            const uint64_t adesc = desc + u * (Cfg::kSubBytes >> 4), bdesc = adesc + (kATileBytes >> 4);
#pragma unroll
            for (int kk = 0; kk < BK / 16; ++kk)
              umma_bf16(tmem_base, (FLIP ? bdesc : adesc) + 2 * kk, (FLIP ? adesc : bdesc) + 2 * kk, idesc, (it | u | kk) != 0);
          }
          umma_commit(&empty_bar[s]);
        }
        if (++s == STAGES) { s = 0; ph ^= 1; }
      }
      if (ok && leader && kb1 > kb0) umma_commit(acc_full);
    }
  } else {
    // ---- accumulator readers: thread = one row of the tile (FLIP: one column); a row's partial goes to the CTA that owns the row ----
    pdl_wait();                             // (the bias may be a product of the kernel before, like A and the stream)
    if (x_f32 || x_b16) {
#pragma unroll
      for (int i = 0; i < PRE; ++i) fetch(i, i);
    }
    stage_bias(p, bias_s + (warp & 3) * 32, lane, n0, BN);
    const int quarter = warp & 3;
    bool have = kb1 > kb0;
    if (have && !mbar_wait(acc_full, 0)) { report(p.status, DEV_TIMEOUT_EPI); have = false; }
    have = __all_sync(0xffffffffu, have);   // the TMEM loads below are warp-wide
    tc_fence_after();
    cluster_wait();                         // every CTA of the cluster is running: its shared memory may be written
    const uint32_t t0 = tmem_base + (uint32_t(quarter * 32) << 16);
    const int t = quarter * 32 + lane;      // accumulator lane
#pragma unroll 1
    for (int c0 = 0; c0 < (FLIP ? min(ROWS, p.M) : BN); c0 += 32) {
      uint32_t r[32];
      if (have) {            // uniform over the warp
        tmem_ld32(t0 + c0, r);
        tmem_wait_ld();
      } else {
#pragma unroll
        for (int i = 0; i < 32; ++i) r[i] = 0u;   // a slice without k-blocks (or an expired wait) adds nothing
      }
      if constexpr (FLIP) {  // rows c0 .. c0 + 31 of column t: a warp stores 32 consecutive columns of a row at a time
        const uint32_t local = smem_u32(red + (size_t)rank * ROWS_PER * Cfg::kRedPitch + t);
#pragma unroll
        for (int i = 0; i < 32; ++i) {
          const int row = c0 + i;
          if (row < p.M) st_cluster_f1(map_to_cta(local + (row % ROWS_PER) * (Cfg::kRedPitch * 4), row / ROWS_PER), r[i]);
        }
      } else if (m0 + t < p.M) {
        const uint32_t dst = map_to_cta(smem_u32(red + ((size_t)rank * ROWS_PER + t % ROWS_PER) * Cfg::kRedPitch + c0), t / ROWS_PER);
#pragma unroll
        for (int g = 0; g < 8; ++g) st_cluster_f4(dst + 16 * g, r[4 * g], r[4 * g + 1], r[4 * g + 2], r[4 * g + 3]);
      }
    }
    tc_fence_before();
  }
  // Every thread of every CTA of the cluster: the partials are in place after this barrier, and no CTA is
  // written to afterwards (so each may finish and exit on its own).
  __syncwarp();
  if (warp < 2) cluster_wait();             // completes these warps' half of the start-up barrier
  cluster_sync_all();
  if (warp >= 2) {
    const uint2* bias_w = reinterpret_cast<const uint2*>(bias_s + (warp & 3) * 32);
#pragma unroll 1
    for (int i0 = 0; i0 < TURNS; i0 += PRE) {
      if (i0 > 0 && (x_f32 || x_b16)) {
#pragma unroll
        for (int u = 0; u < PRE; ++u) fetch(i0 + u, u);
      }
      float4 v[PRE];                       // the sums of all turns first: their shared-memory reads do not wait for one another
#pragma unroll
      for (int u = 0; u < PRE; ++u) {
        int lrow, quad;
        place(i0 + u, lrow, quad);
        const float* src = red + (size_t)lrow * Cfg::kRedPitch + 4 * quad;
        v[u] = *reinterpret_cast<const float4*>(src);
#pragma unroll
        for (int s = 1; s < S; ++s) {      // rank order: the sum does not depend on timing
          const float4 w = *reinterpret_cast<const float4*>(src + (size_t)s * ROWS_PER * Cfg::kRedPitch);
          v[u].x += w.x; v[u].y += w.y; v[u].z += w.z; v[u].w += w.w;
        }
        if (p.bias) {
          const uint2 bb = bias_w[quad];
          v[u].x += __uint_as_float(bb.x << 16); v[u].y += __uint_as_float(bb.x & 0xFFFF0000u);
          v[u].z += __uint_as_float(bb.y << 16); v[u].w += __uint_as_float(bb.y & 0xFFFF0000u);
        }
      }
      if (x_f32 || x_b16) {
#pragma unroll
        for (int u = 0; u < PRE; ++u) {
          int lrow, quad;
          place(i0 + u, lrow, quad);
          const int row = m0 + (int)rank * ROWS_PER + lrow, col = n0 + 4 * quad;
          if (row >= p.M || col >= p.N) continue;
          const size_t at = (size_t)row * p.N + col;
          const float4 g = gv[u];
          float4 x = xv[u];
          x.x = fmaf(g.x, v[u].x, x.x); x.y = fmaf(g.y, v[u].y, x.y); x.z = fmaf(g.z, v[u].z, x.z); x.w = fmaf(g.w, v[u].w, x.w);
          if (x_f32) *reinterpret_cast<float4*>(static_cast<float*>(p.out) + at) = x;
          else *reinterpret_cast<uint2*>(static_cast<__nv_bfloat16*>(p.out) + at) = make_uint2(pack_bf16x2(x.x, x.y), pack_bf16x2(x.z, x.w));
          if (p.aux) *reinterpret_cast<uint2*>(static_cast<__nv_bfloat16*>(p.aux) + at) = make_uint2(pack_bf16x2(v[u].x, v[u].y), pack_bf16x2(v[u].z, v[u].w));
        }
      } else if (v_tile) {
#pragma unroll
        for (int u = 0; u < PRE; ++u) {
          int lrow, quad;
          place(i0 + u, lrow, quad);
          const int row = m0 + (int)rank * ROWS_PER + lrow, col = n0 + 4 * quad;
          if (row >= p.M || col >= p.N) continue;
          const int img = row / p.rows_per_image, jrow = row - img * p.rows_per_image;
          __nv_bfloat16* dst = p.vt_cache + ((size_t)img * p.C + (col - p.q_cols - p.C)) * p.kv_capacity + p.kv_offset + jrow;
          dst[0] = __float2bfloat16_rn(v[u].x);
          dst[p.kv_capacity] = __float2bfloat16_rn(v[u].y);
          dst[2 * (size_t)p.kv_capacity] = __float2bfloat16_rn(v[u].z);
          dst[3 * (size_t)p.kv_capacity] = __float2bfloat16_rn(v[u].w);
        }
      } else {
        // rows of bf16 (or fp32) values; the K columns of a QKV projection belong to the cache
        const bool k_tile = p.epilogue == EPI_QKV_SPLIT && n0 >= p.q_cols, f32 = p.epilogue == EPI_F32, gelu = p.epilogue == EPI_GELU_BF16;
        const int ld = p.epilogue == EPI_QKV_SPLIT ? p.q_cols : p.N;
#pragma unroll
        for (int u = 0; u < PRE; ++u) {
          int lrow, quad;
          place(i0 + u, lrow, quad);
          const int row = m0 + (int)rank * ROWS_PER + lrow, col = n0 + 4 * quad;
          if (row >= p.M || col >= p.N) continue;
          if (gelu) { v[u].x = gelu_tanh_fast(v[u].x); v[u].y = gelu_tanh_fast(v[u].y); v[u].z = gelu_tanh_fast(v[u].z); v[u].w = gelu_tanh_fast(v[u].w); }
          if (f32) {
            *reinterpret_cast<float4*>(static_cast<float*>(p.out) + (size_t)row * ld + col) = v[u];
            continue;
          }
          __nv_bfloat16* dst = static_cast<__nv_bfloat16*>(p.out) + (size_t)row * ld + col;
          if (k_tile) {
            const int img = row / p.rows_per_image, jrow = row - img * p.rows_per_image;
            dst = p.k_cache + ((size_t)img * p.kv_capacity + p.kv_offset + jrow) * p.C + (col - p.q_cols);
          }
          *reinterpret_cast<uint2*>(dst) = make_uint2(pack_bf16x2(v[u].x, v[u].y), pack_bf16x2(v[u].z, v[u].w));
        }
      }
    }
  }
  __syncthreads();
  if (warp == 1) {
    __syncwarp();
    tmem_dealloc(tmem_base, Cfg::kTmemCols);
  }
}

template <int BN, int S, int ROWS> cudaError_t set_attr() {
  return cudaFuncSetAttribute(gemm_cluster_kernel<BN, S, ROWS>, cudaFuncAttributeMaxDynamicSharedMemorySize, ClusterCfg<BN, ROWS>::kSmemBytes);
}

template <int BN, int S, int ROWS>
cudaError_t launch(const GemmArgs& g, const GemmDev& p, long tiles, cudaStream_t st) {
  alignas(64) CUtensorMap tmA, tmB;
  if (!make_tmap_bf16_2d(&tmA, g.a, g.M, g.K, ROWS)) return cudaErrorInvalidValue;
  if (!make_tmap_bf16_2d(&tmB, g.w, g.N, g.K, BN)) return cudaErrorInvalidValue;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)(tiles * S)); cfg.blockDim = dim3(kThreads); cfg.dynamicSmemBytes = ClusterCfg<BN, ROWS>::kSmemBytes; cfg.stream = st;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  at[1].id = cudaLaunchAttributeClusterDimension;
  at[1].val.clusterDim.x = S; at[1].val.clusterDim.y = 1; at[1].val.clusterDim.z = 1;
  cfg.attrs = at; cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, gemm_cluster_kernel<BN, S, ROWS>, tmA, tmB, p);
}

}  // namespace

cudaError_t gemm_cluster_init() {
  cudaError_t e = set_attr<128, 2, 128>();
  if (e == cudaSuccess) e = set_attr<128, 4, 128>();
  if (e == cudaSuccess) e = set_attr<64, 2, 128>();
  if (e == cudaSuccess) e = set_attr<64, 4, 128>();
  if (e == cudaSuccess) e = set_attr<128, 2, 32>();
  if (e == cudaSuccess) e = set_attr<128, 4, 32>();
  if (e == cudaSuccess) e = set_attr<128, 8, 32>();
  if (e == cudaSuccess) e = set_attr<128, 2, 64>();
  if (e == cudaSuccess) e = set_attr<128, 4, 64>();
  if (e == cudaSuccess) e = set_attr<128, 8, 64>();
  return e;
}

// bn in {64, 128}, slices in {2, 4} (few rows: bn 128, slices in {2, 4, 8}); p.kb_per_split k-blocks per CTA.
cudaError_t launch_gemm_cluster(const GemmArgs& g, const GemmDev& p, int bn, int slices, cudaStream_t st) {
  const long tiles = (long)((g.M + BM - 1) / BM) * ((g.N + bn - 1) / bn);
  if (g.M <= kFlipRows && bn == 128) {
    const bool few = g.M <= 32;
    if (slices == 2) return few ? launch<128, 2, 32>(g, p, tiles, st) : launch<128, 2, 64>(g, p, tiles, st);
    if (slices == 4) return few ? launch<128, 4, 32>(g, p, tiles, st) : launch<128, 4, 64>(g, p, tiles, st);
    if (slices == 8) return few ? launch<128, 8, 32>(g, p, tiles, st) : launch<128, 8, 64>(g, p, tiles, st);
  }
  if (bn == 128 && slices == 2) return launch<128, 2, 128>(g, p, tiles, st);
  if (bn == 128 && slices == 4) return launch<128, 4, 128>(g, p, tiles, st);
  if (bn == 64 && slices == 2) return launch<64, 2, 128>(g, p, tiles, st);
  if (bn == 64 && slices == 4) return launch<64, 4, 128>(g, p, tiles, st);
  return cudaErrorInvalidValue;
}

}  // namespace fv
