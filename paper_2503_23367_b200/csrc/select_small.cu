// What happens between two branches of a pruned scale step on a SMALL token map, in one launch per sublayer: Cached Token Restoration of
// the previous sublayer (Eq. 6: kept rows from its output, the others from its cache, with gate and residual), Pivotal Token
// Selection of this one (Eq. 4-5, exact top-k, ties to the lowest index, ascending) and the gather + LayerNorm + modulation of
// the kept rows.
//
// A cluster of CTAs owns an image, every CTA a run of consecutive rows; a thread owns 8 channels of up to kRows of them and keeps those
// values in registers from the restoration to the LayerNorm.  The CTAs exchange three things through distributed shared memory,
// each behind a cluster barrier or two: column sums (-> mean token), score keys (-> ranks, by counting: every key against every other), kept
// flags (-> positions).  Nothing crosses L2 on the way, which is what the separate kernels (restoration on two streams, column-sum
// fold, scoring with arrival counters, ranking, gather) spend their time on when the map is small: dependent round trips of about
// a microsecond.  Separately they take, 8 images of 256 tokens, C 1024: 9 + 11 + 4.5 us in three launches beside a side stream; here
// one image takes about 12 us (device timestamps: 3-4 restoration, 2 column sums, 1 + 2.5 mean and scores, 1 + 2 ranks and positions,
// 1-2 LayerNorm), each cluster barrier 0.7-1 us of it.
// All sums have a fixed order; a map larger than the registers hold is read again from L2 in every phase.
#include <cuda_bf16.h>

#include "internal.h"
#include "sm100.cuh"

namespace fv {

namespace {

constexpr int kThreads = 512;
constexpr int kWarps = kThreads / 32;
constexpr int kRows = 8;              // rows of a chunk per thread
constexpr int kMaxCluster = 16;
static_assert(2 * kWarps <= kRows * kWarps, "the near-tie count reduces in the words of the partial scores");
static_assert(2048 / 4 <= kThreads, "one thread per four channels");

struct SmallArgs {
  void* x;
  const uint4* y;                     // output of the previous sublayer's branch on its kept rows, or null (nothing to restore)
  const uint4* cache;
  const int32_t* inv_prev;
  const float* gamma_prev;
  int n, C, k, h, w, hc, wc, mod_stride;
  int32_t *idx, *inv;
  float* score;                       // [B, n] or null
  int32_t* near_tie;                  // [B] or null
  const float *sigma, *beta;
  uint2* a_out;
  int rows_per_cta;                   // R
  bool early;                         // gate and modulation may be read before the dependency wait
};

// shared memory of a CTA, in 4-byte words
struct SmallSmem {
  int part, mean, mod, colred, keys, flags, red, row, total;
};
__host__ __device__ inline SmallSmem small_smem(int n, int C, int R) {
  SmallSmem s;
  int off = 0;
  s.part = off; off += C;                            // every CTA's column sums over this CTA's slice of the channels
  s.mean = off; off += C;
  s.mod = off; off += 2 * C;                         // sigma, beta
  s.colred = off; off += kThreads * 8;               // column sums of the CTA's thread groups
  s.keys = off; off += (n + 3) / 4 * 4;
  s.flags = off; off += (n + 15) / 16 * 4;           // one byte per token
  s.red = off; off += kRows * kWarps;                // per row of a chunk and warp: a partial score
  s.row = off; off += 2 * ((R + 3) / 4 * 4);         // per own row: source, score -> position
  s.total = off;
  return s;
}

__device__ __forceinline__ uint32_t remote_addr(const void* p, uint32_t cta) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(smem_u32(p)), "r"(cta));
  return r;
}
__device__ __forceinline__ uint32_t cluster_size() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_nctaid.x;" : "=r"(r));
  return r;
}
// Through L2 and in program order: the row may have been written by another thread of this CTA, or by the kernel before this one.
__device__ __forceinline__ uint4 load16(const void* p) {
  uint4 v;
  asm volatile("ld.global.cg.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ int load_index(const int32_t* p) {
  int v;
  asm volatile("ld.global.cg.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void unpack8(const uint4& u, float (&f)[8]) {
  const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) { f[2 * i] = __uint_as_float(w[i] << 16); f[2 * i + 1] = __uint_as_float(w[i] & 0xFFFF0000u); }
}
__device__ __forceinline__ void load_row8(const float* p, float (&f)[8]) {
  const uint4 a = load16(p), b = load16(p + 4);
  f[0] = __uint_as_float(a.x); f[1] = __uint_as_float(a.y); f[2] = __uint_as_float(a.z); f[3] = __uint_as_float(a.w);
  f[4] = __uint_as_float(b.x); f[5] = __uint_as_float(b.y); f[6] = __uint_as_float(b.z); f[7] = __uint_as_float(b.w);
}
__device__ __forceinline__ void load_row8(const __nv_bfloat16* p, float (&f)[8]) { unpack8(load16(p), f); }

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// STEP: the build a scale step launches (restoration before, gather and LayerNorm after); the other is a selection alone, which may count
// near-ties: code that the step's build had to carry too cost it 0.4 % of a schedule of small maps.
template <typename XT, bool STEP>
__global__ void __launch_bounds__(kThreads, 1) select_small_kernel(const SmallArgs a) {
  extern __shared__ __align__(16) float sm[];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, b = blockIdx.y;
  const uint32_t rank = cluster_ctarank(), cl = cluster_size();
  const int n = a.n, C = a.C, C8 = C / 8, R = a.rows_per_cta;
  const SmallSmem at = small_smem(n, C, R);
  float* part = sm + at.part;
  float* mean = sm + at.mean;
  float4* mod = reinterpret_cast<float4*>(sm + at.mod);
  float* colred = sm + at.colred;
  uint32_t* keys = reinterpret_cast<uint32_t*>(sm + at.keys);
  uint8_t* flags = reinterpret_cast<uint8_t*>(sm + at.flags);
  float* red = sm + at.red;
  const int RP = (R + 3) / 4 * 4;
  int* s_src = reinterpret_cast<int*>(sm + at.row);        // kept row's index j, or ~(source row of the cache)
  float* s_score = sm + at.row + RP;
  int* s_pos = reinterpret_cast<int*>(s_score);            // (the score is on its way to the others by then)
  const int r0 = min(n, (int)rank * R), own = min(n, r0 + R) - r0;
  // thread group g of G, GW threads wide (whole warps), works on the rows g, g + G, ...
  const int GW = (C8 + 31) & ~31, G = kThreads / GW, g = tid / GW, ct = tid - g * GW, WG = GW / 32;
  const bool live = g < G && ct < C8;
  const int chunk_rows = kRows * G, chunks = max(1, (own + chunk_rows - 1) / chunk_rows);
  XT* xb = static_cast<XT*>(a.x) + (size_t)b * n * C + ct * 8;

  pdl_trigger();
  cluster_arrive_relaxed();
  for (int i = tid; i < (n + 15) / 16 * 4; i += kThreads) reinterpret_cast<uint32_t*>(flags)[i] = 0u;
  // gate and modulation vectors: behind the wait when the kernel before may have produced them (a step in place), else at once
  const bool lookup = a.y && tid < own, modulate = a.sigma && tid < C / 4;   // (own <= R and C / 4 are at most kThreads)
  float4 sg = make_float4(0.f, 0.f, 0.f, 0.f), bt = sg;
  float gam[8];
#pragma unroll
  for (int e = 0; e < 8; ++e) gam[e] = 1.f;
  auto fetch_mod = [&] {
    if (live && a.y && a.gamma_prev) load_row8(a.gamma_prev + (size_t)b * a.mod_stride + ct * 8, gam);
    if (modulate) {
      sg = x_load4(a.sigma + (size_t)b * a.mod_stride + tid * 4);
      bt = x_load4(a.beta + (size_t)b * a.mod_stride + tid * 4);
    }
  };
  if (STEP && a.early) fetch_mod();
  pdl_wait();
  float v[kRows][8];
#pragma unroll
  for (int u = 0; u < 4; ++u)            // the first rows are fetched while the sources of all rows are looked up
    if (live && u * G + g < own) load_row8(xb + (size_t)(r0 + u * G + g) * C, v[u]);
  int j = 0;
  if (lookup) j = load_index(a.inv_prev + (size_t)b * n + r0 + tid);
  if (STEP && !a.early) fetch_mod();
  if (lookup) {
    const int t = r0 + tid, yy = t / a.w, xx = t - yy * a.w;
    s_src[tid] = j >= 0 ? j : ~((yy * a.hc) / a.h * a.wc + (xx * a.wc) / a.w);
  }
  if (modulate) { mod[tid] = sg; mod[C / 4 + tid] = bt; }
  __syncthreads();

  // ---- restoration of the previous sublayer, column sums of the restored rows
  float acc[8];
#pragma unroll
  for (int e = 0; e < 8; ++e) acc[e] = 0.f;
#pragma unroll 1
  for (int q = 0; q < chunks; ++q) {
#pragma unroll
    for (int u0 = 0; u0 < kRows; u0 += 4) {   // four rows in flight
      uint4 src[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int i = q * chunk_rows + (u0 + u) * G + g;
        if (live && i < own) {
          if (u0 > 0 || q > 0) load_row8(xb + (size_t)(r0 + i) * C, v[u0 + u]);
          if (a.y) {
            const int s = s_src[i];
            src[u] = load16(s >= 0 ? a.y + ((size_t)b * a.k + s) * C8 + ct : a.cache + ((size_t)b * a.hc * a.wc + ~s) * C8 + ct);
          }
        }
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int i = q * chunk_rows + (u0 + u) * G + g;
        if (live && i < own) {
          if (a.y) {
            float f[8];
            unpack8(src[u], f);
#pragma unroll
            for (int e = 0; e < 8; ++e) v[u0 + u][e] = fmaf(gam[e], f[e], v[u0 + u][e]);
            x_store8(xb + (size_t)(r0 + i) * C, v[u0 + u]);
          }
#pragma unroll
          for (int e = 0; e < 8; ++e) acc[e] += v[u0 + u][e];
        }
      }
    }
  }
  if (live) {
    float4* dst = reinterpret_cast<float4*>(colred + g * C + ct * 8);
    dst[0] = make_float4(acc[0], acc[1], acc[2], acc[3]);
    dst[1] = make_float4(acc[4], acc[5], acc[6], acc[7]);
  }
  __syncthreads();
  cluster_wait();              // every CTA of the cluster is running: its shared memory may be written
  // CTA o owns slice o of the channels: it receives every CTA's sums over it, adds them in rank order and hands the mean back to all
  const int C4 = C / 4, S4 = C4 / (int)cl;
  if (tid < C4) {
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int q = 0; q < G; ++q) {
      const float4 p = reinterpret_cast<const float4*>(colred + q * C)[tid];
      s.x += p.x; s.y += p.y; s.z += p.z; s.w += p.w;
    }
    const int o = tid / S4;
    asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};"
                 ::"r"(remote_addr(reinterpret_cast<float4*>(part) + (int)rank * S4 + tid - o * S4, (uint32_t)o)), "f"(s.x), "f"(s.y), "f"(s.z), "f"(s.w) : "memory");
  }
  cluster_sync_all();

  // ---- mean token (Eq. 4), scores (Eq. 5)
  if (tid < C4) {                        // one (receiver, four channels) per thread
    const int o = tid / S4, c = tid - o * S4;
    const float fn = (float)n;
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int q = 0; q < kMaxCluster; ++q)
      if (q < (int)cl) {
        const float4 p = reinterpret_cast<const float4*>(part)[q * S4 + c];
        s.x += p.x; s.y += p.y; s.z += p.z; s.w += p.w;
      }
    asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};"
                 ::"r"(remote_addr(reinterpret_cast<float4*>(mean) + (int)rank * S4 + c, (uint32_t)o)), "f"(s.x / fn), "f"(s.y / fn), "f"(s.z / fn), "f"(s.w / fn) : "memory");
  }
  cluster_sync_all();
  float m[8];
#pragma unroll
  for (int e = 0; e < 8; ++e) m[e] = live ? mean[ct * 8 + e] : 0.f;
  const int gw = warp - g * WG;          // this warp inside its group
#pragma unroll 1
  for (int q = 0; q < chunks; ++q) {
    if (chunks > 1) {
#pragma unroll
      for (int u = 0; u < kRows; ++u) {
        const int i = q * chunk_rows + u * G + g;
        if (live && i < own) load_row8(xb + (size_t)(r0 + i) * C, v[u]);
      }
    }
    float sc[kRows];
#pragma unroll
    for (int u = 0; u < kRows; ++u) {
      sc[u] = 0.f;
      if (live && q * chunk_rows + u * G + g < own) {
#pragma unroll
        for (int e = 0; e < 8; ++e) { const float d = v[u][e] - m[e]; sc[u] = fmaf(d, d, sc[u]); }
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
      for (int u = 0; u < kRows; ++u) sc[u] += __shfl_xor_sync(0xffffffffu, sc[u], o);
    if (lane == 0 && g < G) {
#pragma unroll
      for (int u = 0; u < kRows; ++u) red[(u * G + g) * WG + gw] = sc[u];
    }
    __syncthreads();
    if (tid < chunk_rows && q * chunk_rows + tid < own) {
      float sc = 0.f;
      for (int w = 0; w < WG; ++w) sc += red[tid * WG + w];
      s_score[q * chunk_rows + tid] = sc;
      if (a.score) a.score[(size_t)b * n + r0 + q * chunk_rows + tid] = sc;
    }
    __syncthreads();
  }
  for (int f = tid; f < own * (int)cl; f += kThreads) {    // the scores' keys (bit patterns of non-negative values) to every CTA
    const int i = f / (int)cl, o = f - i * (int)cl;
    const uint32_t key = __float_as_uint(s_score[i]) & 0x7FFFFFFFu;
    asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(remote_addr(keys + r0 + i, (uint32_t)o)), "r"(key) : "memory");
  }
  cluster_sync_all();

  // ---- rank of every own token among all: keys above it, and equal keys of lower tokens; kept if fewer than k
  for (int i = warp; i < own; i += kWarps) {
    const int t = r0 + i;
    const uint32_t key = keys[t];
    int before = 0;
    for (int j = lane * 4; j < n; j += 128) {
      const uint4 o = *reinterpret_cast<const uint4*>(keys + j);
      const uint32_t k4[4] = {o.x, o.y, o.z, o.w};
#pragma unroll
      for (int e = 0; e < 4; ++e)
        if (j + e < n) before += (k4[e] > key) || (k4[e] == key && j + e < t);
    }
    before = __reduce_add_sync(0xffffffffu, before);
    if (before < a.k && lane < (int)cl)
      asm volatile("st.shared::cluster.u8 [%0], %1;" ::"r"(remote_addr(flags + t, (uint32_t)lane)), "r"(1u) : "memory");
  }
  cluster_sync_all();          // no CTA is written to after this barrier

  // ---- positions (kept tokens below), outputs of the selection
  for (int i = warp; i < own; i += kWarps) {
    const int t = r0 + i;
    int below = 0;
    for (int j = lane; j * 4 < t; j += 32) {
      uint32_t f = reinterpret_cast<const uint32_t*>(flags)[j];
      if (j * 4 + 4 > t) f &= (1u << (8 * (t - 4 * j))) - 1u;
      below += __popc(f);
    }
    below = __reduce_add_sync(0xffffffffu, below);
    if (lane == 0) {
      const int pos = flags[t] ? below : -1;
      s_pos[i] = pos;
      if (a.inv) a.inv[(size_t)b * n + t] = pos;
      if (pos >= 0) a.idx[(size_t)b * a.k + pos] = t;
    }
  }
  if (!STEP && a.near_tie && rank == 0) {   // tokens within 1e-5 of the threshold, the smallest kept key (all keys and flags are here)
    uint32_t* r = reinterpret_cast<uint32_t*>(red);
    uint32_t tau = 0xFFFFFFFFu;
    for (int j = tid; j < n; j += kThreads)
      if (flags[j]) tau = min(tau, keys[j]);
    tau = __reduce_min_sync(0xffffffffu, tau);
    if (lane == 0) r[warp] = tau;
    __syncthreads();
    for (int w = 0; w < kWarps; ++w) tau = min(tau, r[w]);
    const float tau_f = __uint_as_float(tau), band = 1e-5f * tau_f;
    uint32_t near = 0;
    for (int j = tid; j < n; j += kThreads) near += fabsf(__uint_as_float(keys[j]) - tau_f) <= band;
    near = __reduce_add_sync(0xffffffffu, near);
    if (lane == 0) r[kWarps + warp] = near;
    __syncthreads();
    if (tid == 0) {
      for (int w = 1; w < kWarps; ++w) near += r[kWarps + w];
      a.near_tie[b] = (int32_t)near;
    }
  }
  if (!STEP) return;
  __syncthreads();

  // ---- LayerNorm + modulation of the kept rows -> bf16 A operand; a warp per row, the arithmetic (and bits) of gather_ln_kernel
  constexpr int kVec = 16;
  for (int i = warp; i < own; i += kWarps) {
    const int pos = s_pos[i];
    if (pos < 0) continue;
    const XT* row = static_cast<const XT*>(a.x) + ((size_t)b * n + r0 + i) * C;
    float4 r[kVec];
    float sum = 0.f;
#pragma unroll
    for (int j = 0; j < kVec; ++j)
      if (lane + 32 * j < C4) r[j] = x_load4(row + (size_t)(lane + 32 * j) * 4);
#pragma unroll
    for (int j = 0; j < kVec; ++j)
      if (lane + 32 * j < C4) sum += (r[j].x + r[j].y) + (r[j].z + r[j].w);
    sum = warp_sum(sum);
    const float inv_c = 1.0f / (float)(C4 * 4);
    const float mu = sum * inv_c;
    float var = 0.f;
#pragma unroll
    for (int j = 0; j < kVec; ++j)
      if (lane + 32 * j < C4) {
        const float dx = r[j].x - mu, dy = r[j].y - mu, dz = r[j].z - mu, dw = r[j].w - mu;
        var += (dx * dx + dy * dy) + (dz * dz + dw * dw);
      }
    var = warp_sum(var);
    const float rstd = rsqrtf(var * inv_c + 1e-6f);
    uint2* dst = a.a_out + ((size_t)b * a.k + pos) * C4;
#pragma unroll
    for (int j = 0; j < kVec; ++j) {
      const int c4 = lane + 32 * j;
      if (c4 >= C4) break;
      float4 o = make_float4((r[j].x - mu) * rstd, (r[j].y - mu) * rstd, (r[j].z - mu) * rstd, (r[j].w - mu) * rstd);
      if (a.sigma) {
        const float4 sg = mod[c4], bt = mod[C4 + c4];
        o.x = fmaf(o.x, 1.f + sg.x, bt.x); o.y = fmaf(o.y, 1.f + sg.y, bt.y); o.z = fmaf(o.z, 1.f + sg.z, bt.z); o.w = fmaf(o.w, 1.f + sg.w, bt.w);
      }
      dst[c4] = make_uint2(pack_bf16x2(o.x, o.y), pack_bf16x2(o.z, o.w));
    }
  }
}

int g_clusters[2] = {0, 0};     // clusters of 8 / of 16 CTAs the GPU holds at once

template <typename XT, bool STEP> cudaError_t attr() {
  cudaError_t e = cudaFuncSetAttribute(select_small_kernel<XT, STEP>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(select_small_kernel<XT, STEP>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  return e;
}

}  // namespace

static cudaError_t init_once() {
  cudaError_t e = attr<float, true>();
  if (e == cudaSuccess) e = attr<float, false>();
  if (e == cudaSuccess) e = attr<__nv_bfloat16, true>();
  if (e == cudaSuccess) e = attr<__nv_bfloat16, false>();
  if (e != cudaSuccess) return e;
  for (int i = 0; i < 2; ++i) {
    const int cl = kMaxCluster / 2 << i;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(cl); cfg.blockDim = dim3(kThreads); cfg.dynamicSmemBytes = 200 * 1024;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = cl; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
    cfg.attrs = at; cfg.numAttrs = 1;
    int clusters = 0;
    if (cudaOccupancyMaxActiveClusters(&clusters, select_small_kernel<float, true>, &cfg) == cudaSuccess) g_clusters[i] = clusters;
    else (void)cudaGetLastError();
  }
  return cudaSuccess;
}
cudaError_t select_small_init() {
  static const cudaError_t e = init_once();
  return e;
}

// CTAs per image, or 0: the map is not for this kernel.  16 while the GPU holds a cluster of them per image, else 8 while it holds one of
// those: images that wait for a second round of clusters pay the whole chain again (16 x 16 tokens, C 1024, us a selection alone, separate kernels ->
// this one: 12 images 14.2 -> 10.3, 16 images 15.0 -> 19.0, 64 images 27.5 -> 47.6; us per block of a step 114 -> 107, 125 -> 149, 352 -> 434).  A CTA works
// through its rows alone, so the gain over the separate kernels (some 9 ... 12 us per sublayer on the smallest maps) is used up
// at about 50 rows, or 200 KB of them.  Measured, us per block of 2 sublayers (3 at C 2048), separate kernels -> this one: 16 rows C 1024
// 91 -> 69, C 2048 161 -> 137; 32 rows (clusters of 8) C 1024 107 -> 94; 21 rows C 1920 179 -> 170; 25 rows C 2048 183 -> 190; 36 rows
// C 256 74 -> 63, C 512 84 -> 80, C 1024 bf16 stream 119 -> 107; 64 rows C 256 76 -> 78, C 512 90 -> 98, C 1024 bf16 148 -> 155.  (Against separate
// kernels with a launch for the kept rows, which images of fewer than 128 of them still take.)
static int small_cluster(int B, int n, int C, bool x_bf16) {
  if (C % 128 || C > 2048) return 0;
  const int cl = g_clusters[1] >= B ? 16 : (g_clusters[0] >= B ? 8 : 0);
  if (cl == 0) return 0;
  const int R = (n + cl - 1) / cl;
  if (R > 40 || (size_t)R * C * (x_bf16 ? 2 : 4) > 176 * 1024 || (size_t)small_smem(n, C, R).total * 4 > 200 * 1024) return 0;
  return cl;
}
bool select_small_supported(int B, int n, int C, bool x_bf16) { return small_cluster(B, n, C, x_bf16) > 0; }

// Inside a step, between two sublayers whose last GEMM could restore the kept rows itself (128 of them per image): that route's selection has no
// restoration in front of it and beats the one launch unless a CTA has very little to work through.  Us per block of 2 sublayers (3 at C 2048), this kernel ->
// that route, one / two / four images.  16 rows: C 256 50 -> 55 / 50 -> 56 / 54 -> 58, C 512 59 -> 63 / 59 -> 64 / 66 -> 65, C 768 63 -> 70 / 71 -> 69 / 71 -> 74, C 1024 67 -> 74 / 75 -> 76 /
// 80 -> 82, C 1152 82 -> 78 / 82 -> 82 / 87 -> 88, C 1536 92 -> 89 / 98 -> 92 / 108 -> 102, C 2048 153 -> 146 / 164 -> 152 / 193 -> 185.  From 17 rows on a thread has a second
// chunk of them: 18 rows C 512 64 -> 62 / 63 -> 64 / 67 -> 66, C 1024 73 -> 73 / 80 -> 77 / 85 -> 86, C 1536 102 -> 90 / 108 -> 94 / 120 -> 105.  Narrow models have so
// little to move that it stays ahead: 23 rows C 128 52 -> 55 / 52 -> 55 / 55 -> 57, C 256 54 -> 57 / 57 -> 58 / 57 -> 58, C 384 57 -> 60 / 59 -> 61 / 65 -> 64; 28 rows C 128 54 -> 55 / 55 -> 55 /
// 58 -> 58, C 256 57 -> 58 / 59 -> 60 / 63 -> 60, C 384 61 -> 62 / 62 -> 63 / 70 -> 66; 33 rows C 256 62 -> 60 / 63 -> 60 / 67 -> 63.  A bf16 stream has its lines in the same places.
bool select_small_in_step(int B, int n, int C, bool x_bf16, bool gemm_could_restore) {
  const int cl = small_cluster(B, n, C, x_bf16);
  return cl > 0 && (!gemm_could_restore || (C <= 1024 && (n + cl - 1) / cl <= (C <= 384 ? 24 : 16)));
}

cudaError_t launch_select_small(const SmallSelect& f, cudaStream_t st) {
  const int cl = small_cluster(f.B, f.n, f.C, f.x_bf16);
  if (cl == 0) return cudaErrorInvalidConfiguration;
  SmallArgs a{};
  a.x = f.x; a.y = static_cast<const uint4*>(f.y); a.cache = static_cast<const uint4*>(f.cache); a.inv_prev = f.inv_prev; a.gamma_prev = f.gamma_prev;
  a.n = f.n; a.C = f.C; a.k = f.k; a.h = f.h; a.w = f.w; a.hc = f.hc; a.wc = f.wc; a.mod_stride = f.mod_stride;
  a.idx = f.idx; a.inv = f.inv; a.score = f.score; a.near_tie = f.near_tie; a.early = f.early; a.sigma = f.sigma; a.beta = f.beta; a.a_out = static_cast<uint2*>(f.a_out);
  a.rows_per_cta = (f.n + cl - 1) / cl;
  // algorithmic bytes: the map read (and written where it is restored from y and the cache), indices, the kept rows' bf16 copy
  const double es = f.x_bf16 ? 2.0 : 4.0;
  const double bytes = (double)f.B * f.C * (f.n * es * (f.y ? 2.0 : 1.0) + (f.y ? 2.0 * f.k + 2.0 * f.hc * f.wc : 0.0) + (f.a_out ? 2.0 * f.k : 0.0)) + 4.0 * f.B * ((double)f.k + f.n);
  LaunchScope scope(KC_SELECT, 1, bytes, bytes, st);
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(cl, f.B); cfg.blockDim = dim3(kThreads); cfg.dynamicSmemBytes = (size_t)small_smem(f.n, f.C, a.rows_per_cta).total * 4; cfg.stream = st;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  at[1].id = cudaLaunchAttributeClusterDimension;
  at[1].val.clusterDim.x = cl; at[1].val.clusterDim.y = 1; at[1].val.clusterDim.z = 1;
  cfg.attrs = at; cfg.numAttrs = 2;
  auto go = [&](auto* step, auto* alone) { return cudaLaunchKernelEx(&cfg, f.a_out ? step : alone, a); };
  return f.x_bf16 ? go(select_small_kernel<__nv_bfloat16, true>, select_small_kernel<__nv_bfloat16, false>) : go(select_small_kernel<float, true>, select_small_kernel<float, false>);
}

}  // namespace fv
