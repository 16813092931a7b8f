// Tensor-core (tcgen05 / TMEM / TMA) kernels for bf16 problems: entry points used by the dispatcher.
#pragma once

#include "spa_common.cuh"

namespace spa {

// The same on the device, for eight bf16 values of a row at element offset `at` of the result: `fetch` ahead of time what the
// result is combined with, `finish` behind the product.  One kind per kernel: a second set of fetched values spills, and a
// result that is not known to be apart from what it is combined with costs the plain products 1 us.  kEpiOwn: the result as
// it is, or joined to what `out` holds (other = out).  gelu reads the rounded result, as spa_gelu would; that call takes erff,
// this one normal_cdf_pdf, so the two may differ by a rounding.
enum EpiKind { kEpiOwn, kEpiAdd, kEpiGeluGrad, kEpiGelu };
template <int kKind> struct RowEpilogue {
  __nv_bfloat16* other;  // out or null; add; u; h
  __device__ __forceinline__ bool combines() const { return kKind == kEpiAdd || kKind == kEpiGeluGrad || (kKind == kEpiOwn && other != nullptr); }
  __device__ __forceinline__ void fetch(const __nv_bfloat16* out, uint4& a, long long at) const {
    if (combines()) a = *reinterpret_cast<const uint4*>((kKind == kEpiOwn ? out : other) + at);
  }
  __device__ __forceinline__ void finish(__nv_bfloat16* out, long long at, uint4 v, const uint4& a) const {
    if (combines()) {
      float f[8], g[8];
      Vec16<__nv_bfloat16>::to_float(v, f);
      Vec16<__nv_bfloat16>::to_float(a, g);
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        if (kKind != kEpiGeluGrad) {
          f[e] += g[e];
        } else {
          float cdf, pdf;
          normal_cdf_pdf(g[e], cdf, pdf);
          f[e] *= fmaf(g[e], pdf, cdf);
        }
      }
      v = Vec16<__nv_bfloat16>::from_float(f);
    }
    *reinterpret_cast<uint4*>(out + at) = v;
    if (kKind == kEpiGelu) {
      float f[8];
      Vec16<__nv_bfloat16>::to_float(v, f);
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        float cdf, pdf;
        normal_cdf_pdf(f[e], cdf, pdf);
        f[e] *= cdf;
      }
      *reinterpret_cast<uint4*>(other + at) = Vec16<__nv_bfloat16>::from_float(f);
    }
  }
};

size_t tc_linear_workspace_bytes(const spa_params& p);
size_t tc_weight_grad_workspace_bytes(const spa_params& p, int n_in, int n_out);
size_t tc_attention_workspace_bytes(const spa_params& p);

bool tc_linear_supported(int n_in, int n_out);
// row_map (optional): output row i is written to row row_map[i] of `out`, added to its contents if `accumulate`.
int launch_linear_fwd_tc(const spa_params& p, const void* a, const void* W, const void* bias, int n_in, int n_out,
                         const int32_t* cu, void* out, int32_t* d_status, cudaStream_t st,
                         const int32_t* row_map = nullptr, const LinearEpilogue& epi = {});
int launch_linear_bwd_tc(const spa_params& p, const void* a, const void* W, const void* dout, int n_in, int n_out,
                         const int32_t* cu, void* da, float* dW, float* db, void* workspace, int32_t* d_status,
                         cudaStream_t st, const int32_t* row_map = nullptr, const LinearEpilogue& epi = {});

// CTA-pair variants (cta_group::2, 256 x 256 tiles) of the forward product and the input gradient
bool tc_pair_linear_supported(const spa_params& p, int n_in, int n_out, int n_cols);  // n_cols: width of the result
int launch_linear_fwd_pair(const spa_params& p, const void* a, const void* W, const void* bias, int n_in, int n_out,
                           const int32_t* cu, void* out, int32_t* d_status, cudaStream_t st, const int32_t* row_map,
                           const LinearEpilogue& epi);
int launch_linear_dgrad_pair(const spa_params& p, const void* W, const void* dout, int n_in, int n_out, const int32_t* cu,
                             void* da, int32_t* d_status, cudaStream_t st, const int32_t* row_map, const LinearEpilogue& epi);

// weight gradient on CTA pairs: `splits` partial tiles [splits][n_out][n_in] and, with part_b, splits * tiles_n partial bias
// gradients [.][n_out]; the splits that have rows (at most the number of 64-row blocks) are written
struct PairWgradPlan { int splits, tiles_n, tiles; };
PairWgradPlan pair_wgrad_plan(int capacity, int n_in, int n_out);
int launch_wgrad_pair(const spa_params& p, const void* a, const void* dout, int n_in, int n_out, const int32_t* cu, float* part,
                      float* part_b, const PairWgradPlan& pl, int32_t* d_status, cudaStream_t st);

// weight gradient (and db unless NULL) of the narrower layers, K split over clusters, no scratch
int launch_wgrad_cluster(const spa_params& p, const void* a, const void* dout, int n_in, int n_out, const int32_t* cu, float* dW,
                         float* db, int32_t* d_status, cudaStream_t st);

bool tc_attention_fwd_supported(const spa_params& p);
int launch_attention_fwd_tc(const spa_params& p, const void* qkv, const int32_t* seg, int n_seg, void* ao, float* lse,
                            int32_t* d_status, cudaStream_t st);
bool tc_attention_bwd_supported(const spa_params& p);
int launch_attention_bwd_tc(const spa_params& p, const void* qkv, const void* ao, const float* lse, const void* dao,
                            const int32_t* seg, int n_seg, void* dqkv, void* workspace, int32_t* d_status,
                            cudaStream_t st);
// Device address, on the current device, of the SPA_STATIC_SCRATCH_BYTES array built into the library.
int static_attention_scratch(void** out);

}  // namespace spa
