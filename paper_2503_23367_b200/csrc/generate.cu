// The generation loop around the scale step (Sec. 3.1, Eq. 2-3): output head + token choice, residual
// accumulation r_k = interpolate(r_{k-1}) + codebook[id], and the token map entering the next scale.
// The head's contraction is the library's tcgen05 GEMM with an fp32 epilogue; the rest is memory-bound
// and lives here: a row-wise argmax (one warp per row of logits), a gather-and-add over the codebook, and
// the small d -> C map (d <= 64: a dot product per output element, no tensor-core shape).
#include <cuda_runtime.h>

#include <algorithm>
#include <climits>
#include <cstdint>
#include <vector>

#include "internal.h"
#include "sm100.cuh"   // the device status codes

namespace fv {
namespace {

// ---- ids[r] = argmax_v (logits[r, v] + tau * noise[r, v]), lowest v on ties; one warp per row ----
__global__ void __launch_bounds__(256) argmax_rows_kernel(const float4* logits, const float4* noise, float tau,
                                                          int rows, int V4, int32_t* __restrict__ ids) {
  pdl_trigger();
  const int lane = threadIdx.x & 31;
  const int row = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  pdl_wait();
  if (row >= rows) return;
  const float4* lp = logits + (size_t)row * V4;
  const float4* np = noise ? noise + (size_t)row * V4 : nullptr;
  float best = -INFINITY;
  int bi = INT_MAX;
  for (int j0 = 0; j0 < V4; j0 += 128) {   // four loads per lane in flight
    float4 z[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int j = j0 + lane + 32 * i;
      z[i] = j < V4 ? __ldcs(lp + j) : make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
    }
    if (np) {
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int j = j0 + lane + 32 * i;
        if (j < V4) {
          const float4 g = __ldcs(np + j);
          z[i].x = fmaf(tau, g.x, z[i].x); z[i].y = fmaf(tau, g.y, z[i].y); z[i].z = fmaf(tau, g.z, z[i].z); z[i].w = fmaf(tau, g.w, z[i].w);
        }
      }
    }
    // indices grow within a lane, so a strict comparison keeps the first occurrence
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int j = j0 + lane + 32 * i;
      if (z[i].x > best) { best = z[i].x; bi = 4 * j; }
      if (z[i].y > best) { best = z[i].y; bi = 4 * j + 1; }
      if (z[i].z > best) { best = z[i].z; bi = 4 * j + 2; }
      if (z[i].w > best) { best = z[i].w; bi = 4 * j + 3; }
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float ov = __shfl_xor_sync(0xFFFFFFFFu, best, o);
    const int oi = __shfl_xor_sync(0xFFFFFFFFu, bi, o);
    if (ov > best || (ov == best && oi < bi)) { best = ov; bi = oi; }
  }
  if (lane == 0) ids[row] = bi == INT_MAX ? 0 : bi;   // a row of NaN / -inf: id 0
}

// ---- Eq. 2: r_out[b,t,:] = (r_prev ? r_prev[b, src(t), :] : 0) + codebook[ids[b,t], :] ----
__global__ void __launch_bounds__(256) residual_accumulate_kernel(const int32_t* ids, const float4* codebook,
                                                                  const float4* r_prev, int hp, int wp, int B, int h,
                                                                  int w, int d4, int V, float4* __restrict__ r_out, int32_t* status) {
  pdl_trigger();
  pdl_wait();
  const int n = h * w;
  const long total = (long)B * n * d4;
  for (long i = (long)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (long)gridDim.x * blockDim.x) {
    const int c = (int)(i % d4);
    const long tok = i / d4;
    const int t = (int)(tok % n), b = (int)(tok / n);
    int id = dep_load(ids + tok);
    if (id < 0 || id >= V) {
      if (status) atomicCAS(status, 0, DEV_BAD_TOKEN_ID);
      id = id < 0 ? 0 : V - 1;
    }
    float4 f = dep_load4(codebook + (size_t)id * d4 + c);
    if (r_prev) {
      const int y = t / w, x = t - y * w;
      const int src = (int)(((long)y * hp) / h) * wp + (int)(((long)x * wp) / w);
      const float4 p = dep_load4(r_prev + ((size_t)b * hp * wp + src) * d4 + c);
      f.x += p.x; f.y += p.y; f.z += p.z; f.w += p.w;
    }
    r_out[i] = f;
  }
}

// ---- x[b,t,:] = r[b, src(t), :] * W_in^T + b_in + pos[t,:] ----
// CTA = 64 tokens of the map r x 256 channels, thread = 8 tokens x 8 channels (two groups of four: a warp stores 512 contiguous bytes
// at a time).  The product belongs to the SOURCE token, of which the next map has several copies (nearest interpolation), so it
// is computed once and written, with each copy's own embedding, to all of them.  Up to 32 code channels at a time lie in
// shared memory, W_in as [j][channel] and the tokens' vectors as [j][token]; the shared-memory port hands a warp one word per
// lane and clock, a broadcast word included, so a thread tile of T x C costs T + C of its clocks for T C / 4 of an SM's multiply-adds: 8 x 8
// balances the two, and two channels go through one packed multiply-add.  A warp then walks the copies of its own tokens, whose
// products its lanes hold in registers, the embedding rows of two copies in flight.  Measured for 2 x 48 x 48 -> 64 x 64 tokens, C 2048, d 32
// (map written + embedding read: 16 us), back to back: 41 us (38 while W_in was read before the dependency wait); 45.5 with single multiply-adds, the products passed through shared
// memory to be indexed by copy and the embedding rows prefetched into L2 (which gives nothing); a product per target token in 8 x 8 tiles 52,
// and with one channel per thread 73.  Two rounds of CTAs, each a chain of loads (embedding rows 11 us in all), products (8) and
// stores (6); CTAs of 32 or 16 tokens, four or eight to an SM, do not overlap them better (40, 52).  The additions keep their order (j
// ascending, bias, embedding).
// TW: tokens per warp.  One instead of eight where tiles of 64 tokens leave the GPU to a few CTAs, each of which then takes its warps' tokens one
// after the other (launch_next_input draws the line).
constexpr int kNextChannels = 256;      // one per thread while W_in is staged
// Four floats at an address that is 16-byte aligned (vec) or not.
__device__ __forceinline__ float4 load4_any(const float* p, int vec) {
  return vec ? dep_load4(p) : make_float4(dep_load(p), dep_load(p + 1), dep_load(p + 2), dep_load(p + 3));
}
template <int D, int TW>
__global__ void __launch_bounds__(256, 2) next_input_kernel(const float* r, int h, int w, int h2, int w2, const float* w_in,
                                                            const float* b_in, const float* pos, int C, int B, int vec, int slice,
                                                            float* __restrict__ x_out) {
  constexpr int DC = D < 32 ? D : 32;
  constexpr int kNextTokens = 8 * TW;
  __shared__ __align__(16) float w_s[DC][kNextChannels];
  __shared__ __align__(16) float r_s[DC][kNextTokens];
  __shared__ int s_first[kNextTokens], s_nx[kNextTokens], s_cnt[kNextTokens];   // a token's copies: first one, copies per row of the next map, all
  __shared__ long s_img[kNextTokens], s_row[kNextTokens];                       // first row of its image in x_out; its row of r, or -1
  pdl_trigger();
  const int hu = min(h, h2), wu = min(w, w2), nu = hu * wu;   // along an axis that shrinks only the tokens that have a target take part
  const long rows = (long)B * nu;
  const int cblocks = (C + kNextChannels - 1) / kNextChannels;
  const long row0 = (long)(blockIdx.x / cblocks) * kNextTokens;
  const int c0 = (int)(blockIdx.x % cblocks) * kNextChannels;
  const int tid = threadIdx.x;
  if (tid < kNextTokens) {   // token (y, x) is the source of the targets y2 with floor(y2 h / h2) = y, and x2 likewise
    const long row = row0 + tid;
    int first = 0, nx = 0, ny = 0;
    long src = -1;
    if (row < rows) {
      const int b = (int)(row / nu), t = (int)(row - (long)b * nu), i = t / wu, j = t - i * wu;
      const int y0 = h2 <= h ? i : (int)(((long)i * h2 + h - 1) / h), x0 = w2 <= w ? j : (int)(((long)j * w2 + w - 1) / w);
      ny = h2 <= h ? 1 : (int)(((long)(i + 1) * h2 + h - 1) / h) - y0;
      nx = w2 <= w ? 1 : (int)(((long)(j + 1) * w2 + w - 1) / w) - x0;
      first = y0 * w2 + x0;
      src = (long)b * h * w + (h2 <= h ? (long)i * h / h2 : i) * w + (w2 <= w ? (long)j * w / w2 : j);
      s_img[tid] = (long)b * h2 * w2;
    }
    s_first[tid] = first; s_nx[tid] = nx; s_cnt[tid] = nx * ny; s_row[tid] = src;
  }
  uint64_t acc2[TW][4];   // channel pairs
#pragma unroll
  for (int t = 0; t < TW; ++t)
#pragma unroll
    for (int e = 0; e < 4; ++e) acc2[t][e] = 0ull;
  const int lane = tid & 31, warp = tid >> 5;
  const int tl = warp * TW;              // this thread's tokens inside the tile; its channels are 4 lane .. and 128 + 4 lane ..
  const int ca = c0 + 4 * lane, cb = ca + 128;
  __syncthreads();
  pdl_wait();                            // W_in, b_in and pos are the caller's like r: any of them may come from the kernel before
  // embedding rows of the copies k0 and k0 + 1 of a token
  float4 pa[2], pb[2];
  int t2[2];
  auto fetch = [&](int k0, int cnt, int nx, int first) {
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int d = min(k0 + u, cnt - 1), yy = d / nx;
      t2[u] = first + yy * w2 + (d - yy * nx);
      pa[u] = pb[u] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (pos && k0 + u < cnt) {
        const float* q = pos + (size_t)t2[u] * C;
        if (ca < C) pa[u] = load4_any(q + ca, vec);
        if (cb < C) pb[u] = load4_any(q + cb, vec);
      }
    }
  };
  const int k_first = (int)blockIdx.y * slice;   // this slice's copies
  auto k_end = [&](int t) { return (int)min((long)s_cnt[tl + t], ((long)blockIdx.y + 1) * slice); };
  if (TW == 1 && k_first < k_end(0)) fetch(k_first, k_end(0), s_nx[tl], s_first[tl]);   // on their way beside W_in and r
  for (int d0 = 0; d0 < D; d0 += DC) {
    if (d0) __syncthreads();             // the chunk before has been used
    {   // all of a thread's loads are requested before the first is stored: one round trip for W_in, one for r
      float4 q[DC / 4];                  // channel c0 + tid
#pragma unroll
      for (int i = 0; i < DC / 4; ++i) {
        q[i] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (c0 + tid < C) q[i] = dep_load4(w_in + (size_t)(c0 + tid) * D + d0 + 4 * i);
      }
#pragma unroll
      for (int i = 0; i < DC / 4; ++i) { w_s[4 * i][tid] = q[i].x; w_s[4 * i + 1][tid] = q[i].y; w_s[4 * i + 2][tid] = q[i].z; w_s[4 * i + 3][tid] = q[i].w; }
    }
    if constexpr (TW == 8) {
      constexpr int JP = DC / 4;         // four threads per token
      const int t = tid >> 2, j0 = (tid & 3) * JP;
      const long src = s_row[t];
      float v[JP];
#pragma unroll
      for (int u = 0; u < JP; ++u) v[u] = src >= 0 ? dep_load(r + src * D + d0 + j0 + u) : 0.f;
#pragma unroll
      for (int u = 0; u < JP; ++u) r_s[j0 + u][t] = v[u];
    } else if (tid < kNextTokens * DC) { // at most one word per thread
      const int t = tid / DC, j = tid - t * DC;
      r_s[j][t] = s_row[t] >= 0 ? dep_load(r + s_row[t] * D + d0 + j) : 0.f;
    }
    __syncthreads();
#pragma unroll 2
    for (int j = 0; j < DC; ++j) {
      const ulonglong2 wa = *reinterpret_cast<const ulonglong2*>(&w_s[j][4 * lane]), wb = *reinterpret_cast<const ulonglong2*>(&w_s[j][128 + 4 * lane]);
      const uint64_t wv[4] = {wa.x, wa.y, wb.x, wb.y};
      float rv[TW];
      if constexpr (TW == 8) {
        const float4 ra = *reinterpret_cast<const float4*>(&r_s[j][tl]), rb = *reinterpret_cast<const float4*>(&r_s[j][tl + 4]);
        rv[0] = ra.x; rv[1] = ra.y; rv[2] = ra.z; rv[3] = ra.w; rv[4] = rb.x; rv[5] = rb.y; rv[6] = rb.z; rv[7] = rb.w;
      } else {
        rv[0] = r_s[j][tl];
      }
#pragma unroll
      for (int t = 0; t < TW; ++t) {
        uint64_t rr;
        asm("mov.b64 %0, {%1, %1};" : "=l"(rr) : "f"(rv[t]));
#pragma unroll
        for (int e = 0; e < 4; ++e) asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc2[t][e]) : "l"(rr), "l"(wv[e]));
      }
    }
  }
  float acc[TW][8];
#pragma unroll
  for (int t = 0; t < TW; ++t)
#pragma unroll
    for (int e = 0; e < 4; ++e) asm("mov.b64 {%0, %1}, %2;" : "=f"(acc[t][2 * e]), "=f"(acc[t][2 * e + 1]) : "l"(acc2[t][e]));
  // the copies of the warp's tokens, two at a time
  float4 bias[2];
#pragma unroll
  for (int g = 0; g < 2; ++g) {
    const int c = g ? cb : ca;
    bias[g] = b_in && c < C ? load4_any(b_in + c, 0) : make_float4(0.f, 0.f, 0.f, 0.f);
  }
#pragma unroll
  for (int t = 0; t < TW; ++t) {
    const int cnt = k_end(t), nx = s_nx[tl + t], first = s_first[tl + t];
    const float4 va = make_float4(acc[t][0] + bias[0].x, acc[t][1] + bias[0].y, acc[t][2] + bias[0].z, acc[t][3] + bias[0].w);
    const float4 vb = make_float4(acc[t][4] + bias[1].x, acc[t][5] + bias[1].y, acc[t][6] + bias[1].z, acc[t][7] + bias[1].w);
    float* img = x_out + (cnt ? s_img[tl + t] : 0) * C;
    for (int k0 = k_first; k0 < cnt; k0 += 2) {
      if (TW > 1 || k0 > k_first) fetch(k0, cnt, nx, first);
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        if (k0 + u >= cnt) break;
        float* dst = img + (size_t)t2[u] * C;
        const float4 oa = make_float4(va.x + pa[u].x, va.y + pa[u].y, va.z + pa[u].z, va.w + pa[u].w);
        const float4 ob = make_float4(vb.x + pb[u].x, vb.y + pb[u].y, vb.z + pb[u].z, vb.w + pb[u].w);
        if (vec) {
          if (ca < C) *reinterpret_cast<float4*>(dst + ca) = oa;
          if (cb < C) *reinterpret_cast<float4*>(dst + cb) = ob;
        } else {
          if (ca < C) { dst[ca] = oa.x; dst[ca + 1] = oa.y; dst[ca + 2] = oa.z; dst[ca + 3] = oa.w; }
          if (cb < C) { dst[cb] = ob.x; dst[cb + 1] = ob.y; dst[cb + 2] = ob.z; dst[cb + 3] = ob.w; }
        }
      }
    }
  }
}

struct HeadLayout { size_t a, logits, total; };
HeadLayout head_layout(int rows, int C, int V, bool own_logits) {
  HeadLayout l{};
  size_t off = 0;
  l.a = off; off = align_up(off + (size_t)rows * C * 2, 256);
  l.logits = off; if (own_logits) off = align_up(off + (size_t)rows * V * 4, 256);
  l.total = off;
  return l;
}

}  // namespace

cudaError_t launch_argmax_rows(const float* logits, const float* noise, float tau, int rows, int V, int32_t* ids, cudaStream_t st) {
  const double bytes = (double)rows * V * 4.0 * (noise ? 2.0 : 1.0) + 4.0 * rows;
  LaunchScope scope(KC_SELECT, 1, bytes, bytes, st);
  return launch_pdl(argmax_rows_kernel, dim3((rows + 7) / 8), dim3(256), 0, st, reinterpret_cast<const float4*>(logits),
                    reinterpret_cast<const float4*>(noise), tau, rows, V / 4, ids);
}

cudaError_t launch_residual_accumulate(const int32_t* ids, int B, int h, int w, const float* codebook, int V, int d, const float* r_prev,
                                       int hp, int wp, float* r_out, int32_t* status, cudaStream_t st) {
  const long total = (long)B * h * w * (d / 4);
  const double bytes = (double)B * h * w * (4.0 + (r_prev ? 3.0 : 2.0) * d * 4.0);
  LaunchScope scope(KC_RESTORE, 1, bytes, bytes, st);
  const long blocks = (total + 255) / 256;
  return launch_pdl(residual_accumulate_kernel, dim3((unsigned)(blocks < 148 * 16 ? blocks : 148 * 16)), dim3(256), 0, st, ids,
                    reinterpret_cast<const float4*>(codebook), reinterpret_cast<const float4*>(r_prev), hp, wp, B, h, w, d / 4, V,
                    reinterpret_cast<float4*>(r_out), status);
}

cudaError_t launch_next_input(const float* r, int B, int h, int w, int d, int h2, int w2, const float* w_in, const float* b_in,
                              const float* pos, int C, float* x_out, cudaStream_t st) {
  const long rows = (long)B * h2 * w2;
  const double bytes = (double)rows * C * (pos ? 8.0 : 4.0) + (double)rows * d * 4.0;
  LaunchScope scope(KC_RESTORE, 1, bytes, bytes, st);
  // Token tiles x channel blocks along x.  A warp takes its tokens one after the other and writes the copies of each two at a time: eight tokens per warp
  // use the GPU best, but where their tiles would not even give every second SM a CTA, one per warp is sooner done (us, eight -> one: 8 x 8 -> 10 x 10
  // tokens, C 256 8.3 -> 3.4; 16 x 16 -> 20 x 20 twice, C 1024 11.4 -> 10.4; 20 x 20 -> 24 x 24, C 2048 14.0 -> 10.6; with 100 tiles 24.9 -> 34.1, with 128
  // 16.4 -> 24.5).  Where a few tokens become many the copies of a token are cut into slices along y, as many as run at once at two CTAs per
  // SM, each with the product computed again (8 x 8 -> 64 x 64, C 2048: 18 us in 37 slices, 24 in 16).
  const long tokens = (long)B * std::min(h, h2) * std::min(w, w2), cblocks = (C + kNextChannels - 1) / kNextChannels;
  const int tw = 2 * ((tokens + 63) / 64 * cblocks) < 148 ? 1 : 8;
  const long ctas = (tokens + 8 * tw - 1) / (8 * tw) * cblocks;
  const long copies = (long)(h2 > h ? (h2 + h - 1) / h : 1) * (w2 > w ? (w2 + w - 1) / w : 1);   // most copies of a token
  const long slices = std::max(1L, std::min((copies + 1) / 2, 2L * 148 / ctas));
  const int slice = (int)((copies + slices - 1) / slices);
  if (ctas > INT_MAX) return cudaErrorInvalidValue;
  const dim3 grid((unsigned)ctas, (unsigned)((copies + slice - 1) / slice));
  const int vec = ((reinterpret_cast<uintptr_t>(x_out) | reinterpret_cast<uintptr_t>(pos)) & 15u) == 0;   // C is a multiple of 4
  auto go = [&](auto* one, auto* eight) {
    return launch_pdl(tw == 1 ? one : eight, grid, dim3(256), 0, st, r, h, w, h2, w2, w_in, b_in, pos, C, B, vec, slice, x_out);
  };
  switch (d) {
    case 8: return go(next_input_kernel<8, 1>, next_input_kernel<8, 8>);
    case 16: return go(next_input_kernel<16, 1>, next_input_kernel<16, 8>);
    case 32: return go(next_input_kernel<32, 1>, next_input_kernel<32, 8>);
    case 64: return go(next_input_kernel<64, 1>, next_input_kernel<64, 8>);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace fv

using namespace fv;

namespace {
bool al16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }
fv_status cu(cudaError_t e) { return e == cudaSuccess ? FV_OK : FV_ERR_CUDA; }
}  // namespace

extern "C" {

size_t fv_head_workspace_bytes(int32_t rows, int32_t C, int32_t V) {
  if (rows <= 0 || C <= 0 || V <= 0) return 0;
  return head_layout(rows, C, V, true).total;
}

fv_status fv_argmax_rows(const float* logits_dev, const float* noise_dev, float tau, int32_t rows, int32_t V, int32_t* ids_out_dev,
                         void* stream) {
  if (!logits_dev || !ids_out_dev || rows <= 0 || V <= 0 || (V % 4) || !al16(logits_dev) || (noise_dev && !al16(noise_dev)))
    return FV_ERR_INVALID_ARG;
  return cu(launch_argmax_rows(logits_dev, noise_dev, tau, rows, V, ids_out_dev, static_cast<cudaStream_t>(stream)));
}

fv_status fv_head_tokens(const float* y_dev, int32_t B, int32_t n, int32_t C, const float* mod_head_dev, const void* w_head_dev,
                         const void* b_head_dev, int32_t V, const float* noise_dev, float tau, int32_t* ids_out_dev,
                         float* logits_out_dev, void* workspace_dev, size_t workspace_bytes, int32_t* status_dev, void* stream) {
  if (!y_dev || !mod_head_dev || !w_head_dev || !ids_out_dev || !workspace_dev || B <= 0 || n <= 0) return FV_ERR_INVALID_ARG;
  if (C <= 0 || (C % 8) || C > 2048 || V <= 0 || (V % 8)) return FV_ERR_INVALID_ARG;
  if ((reinterpret_cast<uintptr_t>(workspace_dev) & 255u) || (logits_out_dev && !al16(logits_out_dev))) return FV_ERR_INVALID_ARG;
  const int rows = B * n;
  const HeadLayout l = head_layout(rows, C, V, logits_out_dev == nullptr);
  if (workspace_bytes < l.total) return FV_ERR_CAPACITY;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  char* ws = static_cast<char*>(workspace_dev);
  float* logits = logits_out_dev ? logits_out_dev : reinterpret_cast<float*>(ws + l.logits);
  fv_status s = fv_gather_ln(y_dev, nullptr, B, n, n, C, mod_head_dev, mod_head_dev + C, 2 * C, ws + l.a, status_dev, stream);
  if (s != FV_OK) return s;
  s = fv_gemm_bf16(ws + l.a, w_head_dev, b_head_dev, rows, V, C, EPI_F32, logits, nullptr, nullptr, 0, n, status_dev, nullptr, 0, stream);
  if (s != FV_OK) return s;
  return cu(launch_argmax_rows(logits, noise_dev, tau, rows, V, ids_out_dev, st));
}

fv_status fv_residual_accumulate(const int32_t* ids_dev, int32_t B, int32_t h, int32_t w, const float* codebook_dev, int32_t V, int32_t d,
                                 const float* r_prev_dev, int32_t hp, int32_t wp, float* r_out_dev, int32_t* status_dev, void* stream) {
  if (!ids_dev || !codebook_dev || !r_out_dev || B <= 0 || h <= 0 || w <= 0 || V <= 0 || d <= 0 || (d % 4)) return FV_ERR_INVALID_ARG;
  if (r_prev_dev && (hp <= 0 || wp <= 0 || r_prev_dev == r_out_dev)) return FV_ERR_INVALID_ARG;
  if (!al16(codebook_dev) || !al16(r_out_dev) || (r_prev_dev && !al16(r_prev_dev))) return FV_ERR_INVALID_ARG;
  return cu(launch_residual_accumulate(ids_dev, B, h, w, codebook_dev, V, d, r_prev_dev, hp, wp, r_out_dev, status_dev,
                                       static_cast<cudaStream_t>(stream)));
}

fv_status fv_next_scale_input(const float* r_dev, int32_t B, int32_t h, int32_t w, int32_t d, int32_t h2, int32_t w2, const float* w_in_dev,
                              const float* b_in_dev, const float* pos_dev, int32_t C, float* x_out_dev, void* stream) {
  if (!r_dev || !w_in_dev || !x_out_dev || B <= 0 || h <= 0 || w <= 0 || h2 <= 0 || w2 <= 0 || C <= 0 || (C % 4)) return FV_ERR_INVALID_ARG;
  if (d != 8 && d != 16 && d != 32 && d != 64) return FV_ERR_UNSUPPORTED;
  if (!al16(w_in_dev)) return FV_ERR_INVALID_ARG;
  return cu(launch_next_input(r_dev, B, h, w, d, h2, w2, w_in_dev, b_in_dev, pos_dev, C, x_out_dev, static_cast<cudaStream_t>(stream)));
}

namespace {
struct GenLayout { size_t status, x, y, r0, r1, head, total; };
GenLayout gen_layout(const fv_config& c, const fv_generator& g) {
  int n_max = 0;
  for (int i = 0; i < c.n_steps; ++i) n_max = n_max > c.h[i] * c.w[i] ? n_max : c.h[i] * c.w[i];
  const size_t rows = (size_t)c.B_max * n_max;
  GenLayout l{};
  size_t off = 0;
  l.status = off; off = align_up(off + 256, 1024);
  l.x = off; off = align_up(off + rows * c.C * 4, 1024);
  l.y = off; off = align_up(off + rows * c.C * 4, 1024);
  l.r0 = off; off = align_up(off + rows * g.d * 4, 1024);
  l.r1 = off; off = align_up(off + rows * g.d * 4, 1024);
  l.head = off; off = align_up(off + head_layout((int)rows, c.C, g.V, true).total, 1024);
  l.total = off;
  return l;
}
}  // namespace

size_t fv_generate_workspace_bytes(const fv_ctx* ctx, const fv_generator* gen) {
  if (!ctx || !gen || gen->V <= 0 || gen->d <= 0) return 0;
  return gen_layout(*ctx_config(ctx), *gen).total;
}

fv_status fv_generate(fv_ctx* ctx, const fv_generator* gen, const float* start_dev, int32_t B, const double* keep_host,
                      const float* const* noise_host, int32_t* ids_out_dev, float* r_out_dev, void* workspace_dev, size_t workspace_bytes,
                      void* stream) {
  if (!ctx || !gen || !start_dev || !keep_host || !ids_out_dev || !r_out_dev || !workspace_dev) return FV_ERR_INVALID_ARG;
  if (!gen->codebook_dev || !gen->w_head_dev || !gen->mod_head_dev || !gen->w_in_dev) return FV_ERR_INVALID_ARG;
  const fv_config& c = *ctx_config(ctx);
  if (B <= 0 || B > c.B_max || (reinterpret_cast<uintptr_t>(workspace_dev) & 1023u)) return FV_ERR_INVALID_ARG;
  if (c.resid_dtype != 0) return FV_ERR_UNSUPPORTED;   // the head reads an fp32 token map
  const GenLayout l = gen_layout(c, *gen);
  if (workspace_bytes < l.total) return FV_ERR_CAPACITY;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  char* ws = static_cast<char*>(workspace_dev);
  // the head GEMM and Eq. 2 report into the context's own status word, which fv_device_status reads
  int32_t* status = ctx_status_word(ctx);
  float* x = reinterpret_cast<float*>(ws + l.x);
  float* y = reinterpret_cast<float*>(ws + l.y);
  float* r[2] = {reinterpret_cast<float*>(ws + l.r0), reinterpret_cast<float*>(ws + l.r1)};
  const size_t head_bytes = l.total - l.head;
  fv_status s = fv_reset(ctx);
  if (s != FV_OK) return s;
  (void)st;
  const int K = c.n_steps;
  size_t id_off = 0;
  for (int k = 0; k < K; ++k) {
    const int h = c.h[k], w = c.w[k], n = h * w;
    const float* xin = k == 0 ? start_dev : x;
    s = fv_var_step(ctx, xin, B, k, keep_host[k], y, nullptr, nullptr, stream);
    if (s != FV_OK) return s;
    int32_t* ids = ids_out_dev + id_off;
    s = fv_head_tokens(y, B, n, c.C, gen->mod_head_dev, gen->w_head_dev, gen->b_head_dev, gen->V,
                       noise_host ? noise_host[k] : nullptr, gen->tau, ids, nullptr, ws + l.head, head_bytes, status, stream);
    if (s != FV_OK) return s;
    float* r_cur = (k + 1 == K) ? r_out_dev : r[k & 1];
    const float* r_prev = k ? r[(k - 1) & 1] : nullptr;
    s = fv_residual_accumulate(ids, B, h, w, gen->codebook_dev, gen->V, gen->d, r_prev, k ? c.h[k - 1] : 0, k ? c.w[k - 1] : 0, r_cur,
                               status, stream);
    if (s != FV_OK) return s;
    if (k + 1 < K) {
      s = fv_next_scale_input(r_cur, B, h, w, gen->d, c.h[k + 1], c.w[k + 1], gen->w_in_dev, gen->b_in_dev,
                              gen->pos_dev ? gen->pos_dev[k + 1] : nullptr, c.C, x, stream);
      if (s != FV_OK) return s;
    }
    id_off += (size_t)B * n;
  }
  return FV_OK;
}

}  // extern "C"
