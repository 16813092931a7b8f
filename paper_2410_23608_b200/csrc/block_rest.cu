// The rest of the pre-norm transformer block around SPA (Sec. 3.2: selected tokens go through attention, the
// others straight to the feed-forward network): LayerNorm over the channels and the GELU (by erff), forward and
// backward.  The two feed-forward products are the library's linear layers run over all B*N tokens.
// Row-wise streaming kernels: one warp per token row, 16-byte accesses, fp32 arithmetic; the per-channel sums
// of the LayerNorm backward are taken per CTA in a fixed order and combined by the shared reduction kernel.
#include "spa_common.cuh"

namespace spa {
namespace {

constexpr int kRestThreads = 256;
constexpr int kLnChunks = 4;  // 16-byte chunks of a row per lane: C <= 128 chunks (1024 bf16 / 512 fp32 channels)

// LayerNorm of every token row.  kGate: the SPA gate reads the normalised (rounded) row from the same registers - scores
// and mask as spa_gate writes them - and the row itself is passed on to `copy` (the residual stream that the attention
// adds to): one pass over x instead of three kernels that read x or its normalisation again.
template <typename T, bool kGate>
__global__ void __launch_bounds__(kRestThreads)
layer_norm_kernel(const uint4* x16, const T* gamma, const T* beta, float eps,
                  int rows, int C, uint4* __restrict__ y16, float* __restrict__ mean, float* __restrict__ rstd,
                  const T* w_g, float b_g, float tau, float* __restrict__ scores, uint8_t* __restrict__ mask,
                  uint4* __restrict__ copy16) {
  pdl_entry();
  constexpr int E = Vec16<T>::kElems;
  const int lane = threadIdx.x & 31, Q = C / E;
  const int warps = gridDim.x * (kRestThreads / 32);
  const uint4* g16 = reinterpret_cast<const uint4*>(gamma);
  const uint4* b16 = reinterpret_cast<const uint4*>(beta);
  const uint4* w16 = reinterpret_cast<const uint4*>(w_g);
  for (int t = blockIdx.x * (kRestThreads / 32) + (threadIdx.x >> 5); t < rows; t += warps) {
    float v[kLnChunks][E];
    float s = 0.f;
#pragma unroll
    for (int k = 0; k < kLnChunks; ++k) {
      const int q = lane + 32 * k;
      if (q < Q) {
        const uint4 raw = ld_stream16(x16 + (long long)t * Q + q);
        if (kGate) copy16[(long long)t * Q + q] = raw;
        Vec16<T>::to_float(raw, v[k]);
#pragma unroll
        for (int e = 0; e < E; ++e) s += v[k][e];
      }
    }
    const float mu = warp_sum(s) / C;
    float ss = 0.f;
#pragma unroll
    for (int k = 0; k < kLnChunks; ++k)
      if (lane + 32 * k < Q) {
#pragma unroll
        for (int e = 0; e < E; ++e) { const float d = v[k][e] - mu; ss = fmaf(d, d, ss); }
      }
    const float rs = rsqrtf(warp_sum(ss) / C + eps);
    if (lane == 0) { mean[t] = mu; rstd[t] = rs; }
    float dot = 0.f;
#pragma unroll
    for (int k = 0; k < kLnChunks; ++k) {
      const int q = lane + 32 * k;
      if (q < Q) {
        float o[E], g[E], b[E];
        Vec16<T>::to_float(g16[q], g);
        Vec16<T>::to_float(b16[q], b);
#pragma unroll
        for (int e = 0; e < E; ++e) o[e] = (v[k][e] - mu) * rs * g[e] + b[e];
        const uint4 out = Vec16<T>::from_float(o);
        y16[(long long)t * Q + q] = out;
        if (kGate) {
          Vec16<T>::to_float(out, o);
          Vec16<T>::to_float(w16[q], g);
#pragma unroll
          for (int e = 0; e < E; ++e) dot = fmaf(o[e], g[e], dot);
        }
      }
    }
    if (kGate) {
      const float sc = warp_sum(dot) + b_g;
      if (lane == 0) { scores[t] = sc; mask[t] = sc > tau ? 1 : 0; }
    }
  }
}

// dx = rstd (g - mean(g) - xh mean(g xh)), g = dy gamma, xh = (x - mean) rstd; optionally + add (the residual
// branch's gradient).  Per-CTA sums of dy xh (dgamma) and dy (dbeta) go to part[blockIdx][2C].
// kCh = 16-byte chunks of a row per lane (ceil(C / (32 chunks))): sized exactly, so that narrow rows do not
// carry the registers of wide ones.
// dy_row (optional): row t of dy is packed row dy_row[t], or zero where that is negative (the gradient reaches selected
// tokens only).  dz_row / dz16 (optional): dx row t goes to packed row dz_row[t] as well, where that is not negative.
// Bound by the latency of a row (its loads, two sums over the warp, its store), so all loads of a row go out together, as
// raw chunks, and there are two CTAs per SM of a row or a few per warp: 8 192 rows of 768, three arrays of 12.6 MB in and one
// out, with the reduction that follows: 30.7 -> 16.9 us (the residual was read behind the row's sums, four rows per warp, the
// CTA's sums met bank conflicts of eight, the reduction read a sector for every value).
template <typename T, int kCh>
__global__ void __launch_bounds__(kRestThreads, kCh <= 3 ? 2 : 1)
layer_norm_bwd_kernel(const uint4* dy16, const uint4* x16, const T* gamma,
                      const float* mean, const float* rstd, const uint4* add16, int rows,
                      int C, uint4* dx16, float* __restrict__ part, const int32_t* dy_row,
                      const int32_t* dz_row, uint4* __restrict__ dz16) {
  pdl_entry();
  constexpr int E = Vec16<T>::kElems;
  extern __shared__ __align__(16) float acc_s[];  // [8 warps][2C]
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, Q = C / E;
  float ag[kCh][E], ab[kCh][E];
#pragma unroll
  for (int k = 0; k < kCh; ++k)
#pragma unroll
    for (int e = 0; e < E; ++e) { ag[k][e] = 0.f; ab[k][e] = 0.f; }
  const int warps = gridDim.x * (kRestThreads / 32);
  for (int t = blockIdx.x * (kRestThreads / 32) + warp; t < rows; t += warps) {
    const int src = dy_row != nullptr ? ld_dep(dy_row + t) : t;
    const int dz = dz_row != nullptr ? ld_dep(dz_row + t) : -1;
    const uint4 zero = make_uint4(0u, 0u, 0u, 0u);
    uint4 xr[kCh], ar[kCh], dr[kCh];
#pragma unroll
    for (int k = 0; k < kCh; ++k) {
      const int q = lane + 32 * k;
      xr[k] = q < Q ? ld_stream16(x16 + (long long)t * Q + q) : zero;
      ar[k] = q < Q && add16 != nullptr ? add16[(long long)t * Q + q] : zero;
    }
    const float mu = mean[t], rs = rstd[t];
#pragma unroll
    for (int k = 0; k < kCh; ++k) {
      const int q = lane + 32 * k;
      dr[k] = q < Q && src >= 0 ? ld_stream16(dy16 + (long long)src * Q + q) : zero;
    }
    if (src < 0) {  // no gradient into this row: what the residual branch brings, or nothing
#pragma unroll
      for (int k = 0; k < kCh; ++k) {
        const int q = lane + 32 * k;
        if (q < Q) {
          dx16[(long long)t * Q + q] = ar[k];
          if (dz >= 0) dz16[(long long)dz * Q + q] = ar[k];
        }
      }
      continue;
    }
    float s1 = 0.f, s2 = 0.f;
#pragma unroll
    for (int k = 0; k < kCh; ++k) {
      const int q = lane + 32 * k;
      if (q < Q) {
        float dy[E], xv[E], gm[E];
        Vec16<T>::to_float(dr[k], dy);
        Vec16<T>::to_float(xr[k], xv);
        Vec16<T>::to_float(reinterpret_cast<const uint4*>(gamma)[q], gm);
#pragma unroll
        for (int e = 0; e < E; ++e) {
          const float xh = (xv[e] - mu) * rs, g = dy[e] * gm[e];
          s1 += g;
          s2 = fmaf(g, xh, s2);
          ag[k][e] = fmaf(dy[e], xh, ag[k][e]);
          ab[k][e] += dy[e];
        }
      }
    }
    const float m1 = warp_sum(s1) / C, m2 = warp_sum(s2) / C;
#pragma unroll
    for (int k = 0; k < kCh; ++k) {
      const int q = lane + 32 * k;
      if (q < Q) {
        float dy[E], xv[E], gm[E], a[E];
        Vec16<T>::to_float(dr[k], dy);
        Vec16<T>::to_float(xr[k], xv);
        Vec16<T>::to_float(ar[k], a);
        Vec16<T>::to_float(reinterpret_cast<const uint4*>(gamma)[q], gm);
#pragma unroll
        for (int e = 0; e < E; ++e) {
          const float xh = (xv[e] - mu) * rs, g = dy[e] * gm[e];
          a[e] = (g - m1 - xh * m2) * rs + a[e];
        }
        const uint4 v = Vec16<T>::from_float(a);
        dx16[(long long)t * Q + q] = v;
        if (dz >= 0) dz16[(long long)dz * Q + q] = v;
      }
    }
  }
  float* mine = acc_s + warp * 2 * C;
#pragma unroll
  for (int k = 0; k < kCh; ++k) {
    const int q = lane + 32 * k;
    if (q < Q) {
#pragma unroll
      for (int e = 0; e < E; e += 4) {
        *reinterpret_cast<float4*>(mine + q * E + e) = make_float4(ag[k][e], ag[k][e + 1], ag[k][e + 2], ag[k][e + 3]);
        *reinterpret_cast<float4*>(mine + C + q * E + e) = make_float4(ab[k][e], ab[k][e + 1], ab[k][e + 2], ab[k][e + 3]);
      }
    }
  }
  __syncthreads();
  for (int c = threadIdx.x; c < 2 * C; c += kRestThreads) {
    float s = 0.f;
#pragma unroll
    for (int w = 0; w < kRestThreads / 32; ++w) s += acc_s[w * 2 * C + c];
    part[(long long)blockIdx.x * 2 * C + c] = s;
  }
}

// out = gelu(u) (kBwd = false) or out = dh * gelu'(u) (kBwd = true), over `total` 16-byte chunks
template <typename T, bool kBwd>
__global__ void __launch_bounds__(kRestThreads)
gelu_kernel(const uint4* u16, const uint4* dh16, long long total, uint4* out16) {
  pdl_entry();
  constexpr int E = Vec16<T>::kElems;
  for (long long k = (long long)blockIdx.x * kRestThreads + threadIdx.x; k < total; k += (long long)gridDim.x * kRestThreads) {
    float u[E], o[E];
    Vec16<T>::to_float(ld_stream16(u16 + k), u);
    if (kBwd) {
      float d[E];
      Vec16<T>::to_float(dh16[k], d);
#pragma unroll
      for (int e = 0; e < E; ++e) o[e] = d[e] * gelu_grad_f(u[e]);
    } else {
#pragma unroll
      for (int e = 0; e < E; ++e) o[e] = gelu_f(u[e]);
    }
    out16[k] = Vec16<T>::from_float(o);
  }
}

// Both kernels are bound by the latency of a row rather than by bandwidth: the forward takes two rows per warp and up; the
// backward one and up, with as many CTAs as fit at once (each adds a line of partial sums to combine).
int ln_grid(int rows) {
  int g = (rows + 15) / 16;
  if (g > kNumSMs * 6) g = kNumSMs * 6;
  return g < 1 ? 1 : g;
}
int ln_bwd_grid(int rows) {
  const int g = (rows + 7) / 8;
  return g < 1 ? 1 : (g > kNumSMs * 2 ? kNumSMs * 2 : g);
}

}  // namespace

size_t layer_norm_workspace_bytes(const spa_params& p) { return (size_t)ln_bwd_grid(p.B * p.N) * 2 * p.C * sizeof(float) + 256; }

bool layer_norm_supported(const spa_params& p) { return p.C / (p.dtype == SPA_F32 ? 4 : 8) <= 32 * kLnChunks; }

int launch_layer_norm(const spa_params& p, const void* x, const void* gamma, const void* beta, float eps, void* y,
                      float* mean, float* rstd, cudaStream_t st) {
  return launch_layer_norm_gate(p, x, gamma, beta, eps, y, mean, rstd, nullptr, 0.f, nullptr, nullptr, nullptr, st);
}

int launch_layer_norm_gate(const spa_params& p, const void* x, const void* gamma, const void* beta, float eps, void* y,
                           float* mean, float* rstd, const void* w_g, float b_g, float* scores, uint8_t* mask, void* copy,
                           cudaStream_t st) {
  const int rows = p.B * p.N;
  if (rows == 0) return SPA_OK;
  if (!layer_norm_supported(p)) return SPA_ERR_UNSUPPORTED;
#define SPA_LN(T, G)                                                                                                  \
  launch_pdl(layer_norm_kernel<T, G>, ln_grid(rows), kRestThreads, 0, st, (const uint4*)x, (const T*)gamma,           \
             (const T*)beta, eps, rows, p.C, (uint4*)y, mean, rstd, (const T*)w_g, b_g, p.tau, scores, mask, (uint4*)copy)
  if (p.dtype == SPA_F32) { if (w_g != nullptr) SPA_LN(float, true); else SPA_LN(float, false); }
  else { if (w_g != nullptr) SPA_LN(__nv_bfloat16, true); else SPA_LN(__nv_bfloat16, false); }
#undef SPA_LN
  SPA_CUDA_CHECK_LAUNCH("layer_norm_kernel");
  return SPA_OK;
}

int launch_layer_norm_bwd(const spa_params& p, const void* dy, const void* x, const void* gamma, const float* mean,
                          const float* rstd, const void* add, void* dx, float* dgamma, float* dbeta, void* workspace,
                          cudaStream_t st, const int32_t* dy_row, const int32_t* dz_row, void* dz) {
  const int rows = p.B * p.N;
  if (rows == 0) return SPA_OK;
  if (!layer_norm_supported(p)) return SPA_ERR_UNSUPPORTED;
  const int grid = ln_bwd_grid(rows);
  const size_t smem = (size_t)(kRestThreads / 32) * 2 * p.C * sizeof(float);
  float* part = reinterpret_cast<float*>(workspace);
  const int chunks = (p.C / (p.dtype == SPA_F32 ? 4 : 8) + 31) / 32;  // 1..4 (layer_norm_supported)
  cudaError_t e = cudaSuccess;
#define SPA_LN_BWD(T, CH)                                                                                             \
  do {                                                                                                                \
    auto kern = layer_norm_bwd_kernel<T, CH>;                                                                         \
    static DeviceOnce attr;                                                                                           \
    e = attr.run([&] { return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 64 * 1024); }); \
    if (e == cudaSuccess)                                                                                             \
      launch_pdl(kern, grid, kRestThreads, smem, st, (const uint4*)dy, (const uint4*)x, (const T*)gamma, mean, rstd, \
                 (const uint4*)add, rows, p.C, (uint4*)dx, part, dy_row, dz_row, (uint4*)dz);                          \
  } while (0)
#define SPA_LN_BWD_T(T)                                                                                               \
  do {                                                                                                                \
    if (chunks <= 1) SPA_LN_BWD(T, 1); else if (chunks == 2) SPA_LN_BWD(T, 2); else if (chunks == 3) SPA_LN_BWD(T, 3); \
    else SPA_LN_BWD(T, 4);                                                                                            \
  } while (0)
  if (p.dtype == SPA_F32) SPA_LN_BWD_T(float); else SPA_LN_BWD_T(__nv_bfloat16);
#undef SPA_LN_BWD_T
#undef SPA_LN_BWD
  if (e != cudaSuccess) { set_cuda_error(e, "layer_norm_bwd_kernel"); return SPA_ERR_CUDA; }
  SPA_CUDA_CHECK_LAUNCH("layer_norm_bwd_kernel");
  // dgamma = columns [0, C) of the per-CTA sums, dbeta = columns [C, 2C): one reduction launch for both
  return launch_partial_sum(part, grid, 2 * p.C, p.C, dgamma, p.C, dbeta, st);
}

int launch_gelu(const spa_params& p, const void* u, const void* dh, int n_cols, void* out, cudaStream_t st) {
  const int E = p.dtype == SPA_F32 ? 4 : 8;
  const long long total = (long long)p.B * p.N * n_cols / E;
  if (total == 0) return SPA_OK;
  long long g = (total + kRestThreads * 4 - 1) / (kRestThreads * 4);
  if (g > kNumSMs * 8) g = kNumSMs * 8;
  const int grid = g < 1 ? 1 : (int)g;
  if (p.dtype == SPA_F32) {
    if (dh) launch_pdl(gelu_kernel<float, true>, grid, kRestThreads, 0, st, (const uint4*)u, (const uint4*)dh, total, (uint4*)out);
    else launch_pdl(gelu_kernel<float, false>, grid, kRestThreads, 0, st, (const uint4*)u, (const uint4*)dh, total, (uint4*)out);
  } else {
    if (dh) launch_pdl(gelu_kernel<__nv_bfloat16, true>, grid, kRestThreads, 0, st, (const uint4*)u, (const uint4*)dh, total, (uint4*)out);
    else launch_pdl(gelu_kernel<__nv_bfloat16, false>, grid, kRestThreads, 0, st, (const uint4*)u, (const uint4*)dh, total, (uint4*)out);
  }
  SPA_CUDA_CHECK_LAUNCH("gelu_kernel");
  return SPA_OK;
}

}  // namespace spa
