// C boundary: argument validation and dispatch to the kernels.  Nothing here computes.
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

#include <atomic>
#include <new>

#include "spa_common.cuh"
#include "spa_tc.cuh"

namespace spa {

static thread_local char g_cuda_error[256] = "";

void set_cuda_error(cudaError_t e, const char* where) {
  snprintf(g_cuda_error, sizeof(g_cuda_error), "%s: %s", where, cudaGetErrorString(e));
}

bool pdl_enabled() {
  static const bool on = []() { const char* e = getenv("SPA_PDL"); return !(e != nullptr && e[0] == '0'); }();
  return on;
}

static std::atomic<unsigned long long> g_launches{0};
void count_launch() { g_launches.fetch_add(1, std::memory_order_relaxed); }

namespace {

inline bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

int check_params(const spa_params* p) {
  if (p == nullptr) return SPA_ERR_INVALID_ARG;
  if (p->B < 0 || p->N <= 0 || p->C <= 0 || p->H <= 0) return SPA_ERR_INVALID_ARG;
  if ((long long)p->B * p->N > (1LL << 20)) return SPA_ERR_UNSUPPORTED;
  if (p->capacity < 1 || (long long)p->capacity > (long long)(p->B > 0 ? p->B : 1) * p->N) return SPA_ERR_INVALID_ARG;
  if (p->dtype != SPA_F32 && p->dtype != SPA_BF16) return SPA_ERR_UNSUPPORTED;
  if (p->C % p->H != 0) return SPA_ERR_INVALID_ARG;
  const int es = p->dtype == SPA_F32 ? 4 : 2;
  if ((p->C * es) % 16 != 0 || p->C > 8192) return SPA_ERR_UNSUPPORTED;
  // the kernels take row maxima before scaling, which needs a scale that is positive (0 selects 1/sqrt(d))
  if (!(p->softmax_scale >= 0.f) || !(p->softmax_scale <= 3.0e38f)) return SPA_ERR_INVALID_ARG;
  return SPA_OK;
}

int check_heads(const spa_params* p) {
  const int d = p->C / p->H;
  return (d == 32 || d == 64) ? SPA_OK : SPA_ERR_UNSUPPORTED;
}

// bf16 problems run on the tensor-core kernels unless the caller asks for the fp32-FMA ones
inline bool use_tc(const spa_params* p) { return p->dtype == SPA_BF16 && !(p->flags & SPA_FLAG_SIMT_ONLY); }

// linear layers that the bf16 tensor-core kernels do not take: fp32 data, or bf16 on the fp32-FMA kernels
int linear_fwd_other(const spa_params& p, const void* a, const void* W, const void* bias, int n_in, int n_out, const int32_t* cu,
                     void* out, int32_t* d_status, void* stream, const int32_t* row_map = nullptr, bool accumulate = false) {
  cudaStream_t st = (cudaStream_t)stream;
  return p.dtype == SPA_F32 ? launch_linear_fwd_f32(p, a, W, bias, n_in, n_out, cu, out, d_status, st, row_map, {accumulate ? out : nullptr})
                            : launch_linear_fwd_simt(p, a, W, bias, n_in, n_out, cu, out, st, row_map, accumulate);
}
int linear_bwd_other(const spa_params& p, const void* a, const void* W, const void* dout, int n_in, int n_out, const int32_t* cu,
                     void* da, float* dW, float* db, int32_t* d_status, void* stream, const int32_t* row_map = nullptr,
                     bool accumulate = false) {
  cudaStream_t st = (cudaStream_t)stream;
  return p.dtype == SPA_F32 ? launch_linear_bwd_f32(p, a, W, dout, n_in, n_out, cu, da, dW, db, d_status, st, row_map, {accumulate ? da : nullptr})
                            : launch_linear_bwd_simt(p, a, W, dout, n_in, n_out, cu, da, dW, db, st, row_map, accumulate);
}

#define SPA_REQUIRE(cond, code) do { if (!(cond)) return (code); } while (0)
#define SPA_PTR(ptr) SPA_REQUIRE((ptr) != nullptr && aligned16(ptr), SPA_ERR_INVALID_ARG)
#define SPA_OPT_PTR(ptr) SPA_REQUIRE((ptr) == nullptr || aligned16(ptr), SPA_ERR_INVALID_ARG)

}  // namespace
}  // namespace spa

using namespace spa;

extern "C" {

size_t spa_workspace_bytes(const spa_params* p) {
  if (check_params(p) != SPA_OK) return 0;
  const size_t a = tc_linear_workspace_bytes(*p), b = tc_attention_workspace_bytes(*p);
  return a > b ? a : b;
}

int spa_gate(const spa_params* p, const void* x, const void* w_g, float b_g, const float* s_up, float* scores,
             uint8_t* mask, void* stream) {
  int rc = check_params(p);
  if (rc != SPA_OK) return rc;
  SPA_PTR(x); SPA_PTR(w_g); SPA_PTR(scores); SPA_PTR(mask); SPA_OPT_PTR(s_up);
  return launch_gate(*p, x, w_g, b_g, s_up, scores, mask, nullptr, (cudaStream_t)stream);
}

int spa_gate_prefill(const spa_params* p, const void* x, const void* w_g, float b_g, const float* s_up, float* scores,
                     uint8_t* mask, void* y, void* stream) {
  int rc = check_params(p);
  if (rc != SPA_OK) return rc;
  SPA_PTR(x); SPA_PTR(w_g); SPA_PTR(scores); SPA_PTR(mask); SPA_PTR(y); SPA_OPT_PTR(s_up);
  return launch_gate(*p, x, w_g, b_g, s_up, scores, mask, y == x ? nullptr : y, (cudaStream_t)stream);
}

int spa_select_pack(const spa_params* p, const void* x, const uint8_t* mask, const float* scores, void* x_packed,
                    int32_t* idx, int32_t* inv, int32_t* cu_seqlens, int32_t* d_status, void* stream) {
  int rc = check_params(p);
  if (rc != SPA_OK) return rc;
  SPA_PTR(x); SPA_PTR(mask); SPA_PTR(x_packed); SPA_PTR(idx); SPA_PTR(cu_seqlens); SPA_OPT_PTR(inv);
  if (p->flags & SPA_FLAG_GATE_SCALE) SPA_PTR(scores);
  if (p->B == 0) {
    cudaError_t e = cudaMemsetAsync(cu_seqlens, 0, sizeof(int32_t), (cudaStream_t)stream);
    if (e != cudaSuccess) { set_cuda_error(e, "spa_select_pack"); return SPA_ERR_CUDA; }
    return SPA_OK;
  }
  return launch_select_pack(*p, x, mask, scores, nullptr, x_packed, idx, inv, cu_seqlens, d_status, (cudaStream_t)stream);
}

size_t spa_pack_state_bytes(const spa_params* p) {
  if (check_params(p) != SPA_OK) return 0;
  return gate_pack_state_bytes(*p);
}

int spa_gate_select_pack_supported(const spa_params* p) {
  return (check_params(p) == SPA_OK && gate_pack_supported(*p)) ? 1 : 0;
}

int spa_gate_select_pack(const spa_params* p, const void* x, const void* w_g, float b_g, const float* s_up,
                         float* scores, uint8_t* mask, void* y, void* x_packed, int32_t* idx, int32_t* inv,
                         int32_t* cu_seqlens, void* pack_state, int32_t* d_status, void* stream) {
  int rc = check_params(p);
  if (rc != SPA_OK) return rc;
  SPA_PTR(x); SPA_PTR(w_g); SPA_PTR(scores); SPA_PTR(mask); SPA_PTR(x_packed); SPA_PTR(idx); SPA_PTR(cu_seqlens);
  SPA_PTR(pack_state); SPA_OPT_PTR(s_up); SPA_OPT_PTR(inv); SPA_OPT_PTR(y);
  if (!gate_pack_supported(*p)) return SPA_ERR_UNSUPPORTED;
  if (p->B == 0) {
    cudaError_t e = cudaMemsetAsync(cu_seqlens, 0, sizeof(int32_t), (cudaStream_t)stream);
    if (e != cudaSuccess) { set_cuda_error(e, "spa_gate_select_pack"); return SPA_ERR_CUDA; }
    return SPA_OK;
  }
  return launch_gate_pack(*p, x, w_g, b_g, s_up, scores, mask, y == x ? nullptr : y, x_packed, idx, inv, cu_seqlens,
                          pack_state, d_status, (cudaStream_t)stream);
}

int spa_select_pack_ordered(const spa_params* p, const void* x, const uint8_t* mask, const float* scores,
                            const int32_t* order, void* x_packed, int32_t* idx, int32_t* inv, int32_t* cu_seqlens,
                            int32_t* d_status, void* stream) {
  if (order == nullptr) return SPA_ERR_INVALID_ARG;
  int rc = check_params(p);
  if (rc != SPA_OK) return rc;
  SPA_PTR(x); SPA_PTR(mask); SPA_PTR(x_packed); SPA_PTR(idx); SPA_PTR(cu_seqlens); SPA_OPT_PTR(inv);
  if (p->flags & SPA_FLAG_GATE_SCALE) SPA_PTR(scores);
  if (p->B == 0) {
    cudaError_t e = cudaMemsetAsync(cu_seqlens, 0, sizeof(int32_t), (cudaStream_t)stream);
    if (e != cudaSuccess) { set_cuda_error(e, "spa_select_pack_ordered"); return SPA_ERR_CUDA; }
    return SPA_OK;
  }
  return launch_select_pack(*p, x, mask, scores, order, x_packed, idx, inv, cu_seqlens, d_status, (cudaStream_t)stream);
}

int32_t spa_container_max_segments(const spa_params* p, int32_t L) {
  if (check_params(p) != SPA_OK || L < 1) return 0;
  return p->B + p->capacity / L;
}

int spa_container_offsets(const spa_params* p, const int32_t* cu_seqlens, int32_t L, int32_t* seg_offsets,
                          void* stream) {
  int rc = check_params(p);
  if (rc != SPA_OK) return rc;
  if (cu_seqlens == nullptr || seg_offsets == nullptr || L < 1) return SPA_ERR_INVALID_ARG;
  return launch_container_offsets(*p, cu_seqlens, L, spa_container_max_segments(p, L), seg_offsets, (cudaStream_t)stream);
}

int spa_packed_qkv(const spa_params* p, const void* x_packed, const void* W_qkv, const void* b_qkv,
                   const int32_t* cu_seqlens, void* qkv, int32_t* d_status, void* stream) {
  int rc = check_params(p);
  if (rc != SPA_OK) return rc;
  SPA_PTR(x_packed); SPA_PTR(W_qkv); SPA_PTR(cu_seqlens); SPA_PTR(qkv); SPA_OPT_PTR(b_qkv);
  if (use_tc(p) && tc_linear_supported(p->C, 3 * p->C)) {
    rc = launch_linear_fwd_tc(*p, x_packed, W_qkv, b_qkv, p->C, 3 * p->C, cu_seqlens, qkv, d_status,
                              (cudaStream_t)stream);
    if (rc != SPA_ERR_UNSUPPORTED) return rc;  // geometry the TMA path cannot describe: fp32-FMA kernels
  }
  return linear_fwd_other(*p, x_packed, W_qkv, b_qkv, p->C, 3 * p->C, cu_seqlens, qkv, d_status, stream);
}

int spa_packed_proj(const spa_params* p, const void* a, const void* W_o, const void* b_o, const int32_t* cu_seqlens,
                    void* z, int32_t* d_status, void* stream) {
  int rc = check_params(p);
  if (rc != SPA_OK) return rc;
  SPA_PTR(a); SPA_PTR(W_o); SPA_PTR(cu_seqlens); SPA_PTR(z); SPA_OPT_PTR(b_o);
  if (use_tc(p) && tc_linear_supported(p->C, p->C)) {
    rc = launch_linear_fwd_tc(*p, a, W_o, b_o, p->C, p->C, cu_seqlens, z, d_status, (cudaStream_t)stream);
    if (rc != SPA_ERR_UNSUPPORTED) return rc;
  }
  return linear_fwd_other(*p, a, W_o, b_o, p->C, p->C, cu_seqlens, z, d_status, stream);
}

int spa_packed_attention_fwd(const spa_params* p, const void* qkv, const int32_t* seg_offsets, int32_t n_seg,
                             void* attn_out, float* lse, int32_t* d_status, void* stream) {
  int rc = check_params(p);
  if (rc != SPA_OK) return rc;
  rc = check_heads(p);
  if (rc != SPA_OK) return rc;
  SPA_PTR(qkv); SPA_PTR(seg_offsets); SPA_PTR(attn_out); SPA_PTR(lse);
  SPA_REQUIRE(n_seg >= 0, SPA_ERR_INVALID_ARG);
  if (use_tc(p) && tc_attention_fwd_supported(*p)) {
    rc = launch_attention_fwd_tc(*p, qkv, seg_offsets, n_seg, attn_out, lse, d_status, (cudaStream_t)stream);
    if (rc != SPA_ERR_UNSUPPORTED) return rc;
  }
  return launch_attention_fwd_simt(*p, qkv, seg_offsets, n_seg, attn_out, lse, (cudaStream_t)stream);
}

int spa_packed_attention_bwd(const spa_params* p, const void* qkv, const void* attn_out, const float* lse,
                             const void* d_attn_out, const int32_t* seg_offsets, int32_t n_seg, void* dqkv,
                             void* workspace, int32_t* d_status, void* stream) {
  int rc = check_params(p);
  if (rc != SPA_OK) return rc;
  rc = check_heads(p);
  if (rc != SPA_OK) return rc;
  SPA_PTR(qkv); SPA_PTR(attn_out); SPA_PTR(lse); SPA_PTR(d_attn_out); SPA_PTR(seg_offsets); SPA_PTR(dqkv);
  SPA_OPT_PTR(workspace);
  SPA_REQUIRE(n_seg >= 0, SPA_ERR_INVALID_ARG);
  if (use_tc(p) && tc_attention_bwd_supported(*p) && workspace != nullptr) {
    rc = launch_attention_bwd_tc(*p, qkv, attn_out, lse, d_attn_out, seg_offsets, n_seg, dqkv, workspace, d_status,
                                 (cudaStream_t)stream);
    if (rc != SPA_ERR_UNSUPPORTED) return rc;
  }
  return launch_attention_bwd_simt(*p, qkv, attn_out, lse, d_attn_out, seg_offsets, n_seg, dqkv,
                                   (cudaStream_t)stream);
}

int spa_packed_attention_bwd_static(const spa_params* p, const void* qkv, const void* attn_out, const float* lse,
                                    const void* d_attn_out, const int32_t* seg_offsets, int32_t n_seg, void* dqkv,
                                    int32_t* d_status, void* stream) {
  int rc = check_params(p);
  if (rc != SPA_OK) return rc;
  rc = check_heads(p);
  if (rc != SPA_OK) return rc;
  SPA_PTR(qkv); SPA_PTR(attn_out); SPA_PTR(lse); SPA_PTR(d_attn_out); SPA_PTR(seg_offsets); SPA_PTR(dqkv);
  SPA_REQUIRE(n_seg >= 0, SPA_ERR_INVALID_ARG);
  if (!use_tc(p) || !tc_attention_bwd_supported(*p)) return SPA_ERR_UNSUPPORTED;
  if ((unsigned long long)p->H * (unsigned long long)p->capacity * sizeof(float) > SPA_STATIC_SCRATCH_BYTES)
    return SPA_ERR_SCRATCH;
  void* scratch = nullptr;  // the array inside the library image: nothing is allocated here
  rc = static_attention_scratch(&scratch);
  if (rc != SPA_OK) return rc;
  return launch_attention_bwd_tc(*p, qkv, attn_out, lse, d_attn_out, seg_offsets, n_seg, dqkv, scratch, d_status,
                                 (cudaStream_t)stream);
}

int spa_unpack_scatter(const spa_params* p, const void* z_packed, const void* x, const int32_t* idx,
                       const int32_t* inv, const int32_t* cu_seqlens, void* y, int32_t* d_status, void* stream) {
  (void)d_status;
  int rc = check_params(p);
  if (rc != SPA_OK) return rc;
  SPA_PTR(z_packed); SPA_PTR(cu_seqlens); SPA_PTR(y);
  if (p->flags & SPA_FLAG_INPLACE) {
    SPA_PTR(idx);
    SPA_REQUIRE(x == nullptr || x == y, SPA_ERR_INVALID_ARG);
    x = y;
  } else {
    SPA_PTR(x); SPA_PTR(inv);
    SPA_REQUIRE(x != y, SPA_ERR_INVALID_ARG);
  }
  if (p->B == 0) return SPA_OK;
  return launch_unpack_scatter(*p, z_packed, x, idx, inv, cu_seqlens, y, (cudaStream_t)stream);
}

int spa_unpack_scatter_bwd(const spa_params* p, const void* dY, const int32_t* idx, const int32_t* inv,
                           const int32_t* cu_seqlens, void* dz_packed, void* dX, void* stream) {
  int rc = check_params(p);
  if (rc != SPA_OK) return rc;
  SPA_PTR(dY); SPA_PTR(inv); SPA_PTR(cu_seqlens); SPA_PTR(dz_packed); SPA_OPT_PTR(dX);
  if (p->B == 0) return SPA_OK;
  return launch_unpack_scatter_bwd(*p, dY, idx, inv, cu_seqlens, dz_packed, dX, (cudaStream_t)stream);
}

int spa_select_pack_bwd(const spa_params* p, const void* dx_packed, const void* dY, const int32_t* idx,
                        const int32_t* cu_seqlens, void* dX, void* stream) {
  int rc = check_params(p);
  if (rc != SPA_OK) return rc;
  SPA_PTR(dx_packed); SPA_PTR(idx); SPA_PTR(cu_seqlens); SPA_PTR(dX);
  if (p->flags & SPA_FLAG_RESIDUAL) SPA_PTR(dY);
  if (p->B == 0) return SPA_OK;
  return launch_select_pack_bwd(*p, dx_packed, dY, idx, cu_seqlens, dX, (cudaStream_t)stream);
}

int spa_packed_linear_bwd(const spa_params* p, const void* a, const void* W, const void* dout, int32_t n_in,
                          int32_t n_out, const int32_t* cu_seqlens, void* da, float* dW, float* db, void* workspace,
                          int32_t* d_status, void* stream) {
  int rc = check_params(p);
  if (rc != SPA_OK) return rc;
  SPA_PTR(dout); SPA_PTR(cu_seqlens);
  SPA_OPT_PTR(da); SPA_OPT_PTR(dW); SPA_OPT_PTR(db); SPA_OPT_PTR(workspace);
  if (da != nullptr) SPA_PTR(W);
  if (dW != nullptr) SPA_PTR(a);
  SPA_REQUIRE(n_in > 0 && n_out > 0, SPA_ERR_INVALID_ARG);
  const int es = p->dtype == SPA_F32 ? 4 : 2;
  SPA_REQUIRE((n_in * es) % 16 == 0 && (n_out * es) % 16 == 0, SPA_ERR_UNSUPPORTED);
  if (use_tc(p) && tc_linear_supported(n_in, n_out) && workspace != nullptr) {
    rc = launch_linear_bwd_tc(*p, a, W, dout, n_in, n_out, cu_seqlens, da, dW, db, workspace, d_status,
                              (cudaStream_t)stream);
    if (rc != SPA_ERR_UNSUPPORTED) return rc;
  }
  return linear_bwd_other(*p, a, W, dout, n_in, n_out, cu_seqlens, da, dW, db, d_status, stream);
}

int spa_fused_scatter_supported(const spa_params* p) {
  if (check_params(p) != SPA_OK) return 0;
  return (use_tc(p) && tc_linear_supported(p->C, p->C) && tc_linear_supported(p->C, 3 * p->C)) ? 1 : 0;
}

int spa_unpack_prefill(const spa_params* p, const void* src, void* dst, void* stream) {
  int rc = check_params(p);
  if (rc != SPA_OK) return rc;
  SPA_PTR(src); SPA_PTR(dst);
  if (src == dst || p->B == 0) return SPA_OK;
  return launch_copy_tokens(*p, src, dst, (cudaStream_t)stream);
}

int spa_packed_proj_scatter(const spa_params* p, const void* a, const void* W_o, const void* b_o, const int32_t* idx,
                            const int32_t* cu_seqlens, void* y, int32_t* d_status, void* stream) {
  int rc = check_params(p);
  if (rc != SPA_OK) return rc;
  SPA_PTR(a); SPA_PTR(W_o); SPA_PTR(idx); SPA_PTR(cu_seqlens); SPA_PTR(y); SPA_OPT_PTR(b_o);
  if (!spa_fused_scatter_supported(p)) return SPA_ERR_UNSUPPORTED;
  return launch_linear_fwd_tc(*p, a, W_o, b_o, p->C, p->C, cu_seqlens, y, d_status, (cudaStream_t)stream, idx,
                              {(p->flags & SPA_FLAG_RESIDUAL) ? y : nullptr});
}

int spa_packed_linear_bwd_scatter(const spa_params* p, const void* a, const void* W, const void* dout, int32_t n_in,
                                  int32_t n_out, const int32_t* idx, const int32_t* cu_seqlens, void* dX, float* dW,
                                  float* db, void* workspace, int32_t* d_status, void* stream) {
  int rc = check_params(p);
  if (rc != SPA_OK) return rc;
  SPA_PTR(dout); SPA_PTR(W); SPA_PTR(idx); SPA_PTR(cu_seqlens); SPA_PTR(dX);
  SPA_OPT_PTR(dW); SPA_OPT_PTR(db); SPA_OPT_PTR(workspace);
  if (dW != nullptr) SPA_PTR(a);
  SPA_REQUIRE(n_in == p->C && n_out > 0, SPA_ERR_INVALID_ARG);  // rows of dX are C wide
  SPA_REQUIRE(n_out % 8 == 0, SPA_ERR_UNSUPPORTED);
  if (!spa_fused_scatter_supported(p) || !tc_linear_supported(n_in, n_out)) return SPA_ERR_UNSUPPORTED;
  if ((dW != nullptr || db != nullptr) && workspace == nullptr) return SPA_ERR_INVALID_ARG;
  return launch_linear_bwd_tc(*p, a, W, dout, n_in, n_out, cu_seqlens, dX, dW, db, workspace, d_status,
                              (cudaStream_t)stream, idx, {(p->flags & SPA_FLAG_RESIDUAL) ? dX : nullptr});
}

size_t spa_train_workspace_bytes(const spa_params* p) {
  if (check_params(p) != SPA_OK) return 0;
  return train_workspace_bytes(*p);
}

int spa_score_pool(const float* scores_prev, int32_t B, int32_t rows, int32_t cols, float* s_up, void* stream) {
  if (B < 0 || rows <= 0 || cols <= 0 || (long long)B * rows * cols > (1LL << 28)) return SPA_ERR_INVALID_ARG;
  if (scores_prev == nullptr || s_up == nullptr) return SPA_ERR_INVALID_ARG;
  return launch_score_pool(scores_prev, B, rows, cols, s_up, (cudaStream_t)stream);
}

int spa_select_loss(const spa_params* p, const float* scores, const uint8_t* labels, float alpha, float* ds,
                    float* loss, void* workspace, void* stream) {
  int rc = check_params(p);
  if (rc != SPA_OK) return rc;
  if (scores == nullptr || ds == nullptr || workspace == nullptr) return SPA_ERR_INVALID_ARG;
  return launch_select_loss(*p, scores, labels, alpha, ds, loss, workspace, (cudaStream_t)stream);
}

int spa_select_pack_bwd_gated(const spa_params* p, const void* dx_packed, const void* x, const float* scores,
                              const void* dY, const int32_t* idx, const int32_t* cu_seqlens, void* dX, float* ds,
                              void* stream) {
  int rc = check_params(p);
  if (rc != SPA_OK) return rc;
  SPA_PTR(dx_packed); SPA_PTR(x); SPA_PTR(idx); SPA_PTR(cu_seqlens); SPA_PTR(dX);
  if (scores == nullptr || ds == nullptr) return SPA_ERR_INVALID_ARG;
  if (p->flags & SPA_FLAG_RESIDUAL) SPA_PTR(dY);
  if (p->B == 0) return SPA_OK;
  return launch_pack_bwd_gated(*p, dx_packed, x, scores, dY, idx, cu_seqlens, dX, ds, (cudaStream_t)stream);
}

int spa_gate_bwd(const spa_params* p, const void* x, const void* w_g, const float* scores, const float* s_up,
                 const float* ds, void* dX, float* dw_g, float* db_g, float* ds_up, void* workspace, void* stream) {
  int rc = check_params(p);
  if (rc != SPA_OK) return rc;
  SPA_PTR(x); SPA_PTR(w_g); SPA_PTR(dX);
  if (scores == nullptr || ds == nullptr || dw_g == nullptr || workspace == nullptr) return SPA_ERR_INVALID_ARG;
  return launch_gate_bwd(*p, x, w_g, scores, s_up, ds, dX, dw_g, db_g, ds_up, workspace, (cudaStream_t)stream);
}

int spa_packed_linear(const spa_params* p, const void* a, const void* W, const void* b, int32_t n_in, int32_t n_out,
                      const int32_t* cu_seqlens, void* out, int32_t accumulate, int32_t* d_status, void* stream) {
  int rc = check_params(p);
  if (rc != SPA_OK) return rc;
  SPA_PTR(a); SPA_PTR(W); SPA_PTR(cu_seqlens); SPA_PTR(out); SPA_OPT_PTR(b);
  SPA_REQUIRE(n_in > 0 && n_out > 0, SPA_ERR_INVALID_ARG);
  const int es = p->dtype == SPA_F32 ? 4 : 2;
  SPA_REQUIRE((n_in * es) % 16 == 0 && (n_out * es) % 16 == 0, SPA_ERR_UNSUPPORTED);
  if (use_tc(p) && tc_linear_supported(n_in, n_out)) {
    rc = launch_linear_fwd_tc(*p, a, W, b, n_in, n_out, cu_seqlens, out, d_status, (cudaStream_t)stream, nullptr,
                              {accumulate != 0 ? out : nullptr});
    if (rc != SPA_ERR_UNSUPPORTED) return rc;
  }
  return linear_fwd_other(*p, a, W, b, n_in, n_out, cu_seqlens, out, d_status, stream, nullptr, accumulate != 0);
}

int spa_layer_norm(const spa_params* p, const void* x, const void* gamma, const void* beta, float eps, void* y,
                   float* mean, float* rstd, void* stream) {
  int rc = check_params(p);
  if (rc != SPA_OK) return rc;
  SPA_PTR(x); SPA_PTR(gamma); SPA_PTR(beta); SPA_PTR(y);
  if (mean == nullptr || rstd == nullptr || !(eps > 0.f)) return SPA_ERR_INVALID_ARG;
  return launch_layer_norm(*p, x, gamma, beta, eps, y, mean, rstd, (cudaStream_t)stream);
}

int spa_layer_norm_bwd(const spa_params* p, const void* dy, const void* x, const void* gamma, const float* mean,
                       const float* rstd, const void* add, void* dx, float* dgamma, float* dbeta, void* workspace,
                       void* stream) {
  int rc = check_params(p);
  if (rc != SPA_OK) return rc;
  SPA_PTR(dy); SPA_PTR(x); SPA_PTR(gamma); SPA_PTR(dx); SPA_OPT_PTR(add);
  if (mean == nullptr || rstd == nullptr || dgamma == nullptr || dbeta == nullptr || workspace == nullptr)
    return SPA_ERR_INVALID_ARG;
  return launch_layer_norm_bwd(*p, dy, x, gamma, mean, rstd, add, dx, dgamma, dbeta, workspace, (cudaStream_t)stream);
}

int spa_gelu(const spa_params* p, const void* u, int32_t n_cols, void* h, void* stream) {
  int rc = check_params(p);
  if (rc != SPA_OK) return rc;
  SPA_PTR(u); SPA_PTR(h);
  SPA_REQUIRE(n_cols > 0 && (n_cols * (p->dtype == SPA_F32 ? 4 : 2)) % 16 == 0, SPA_ERR_INVALID_ARG);
  return launch_gelu(*p, u, nullptr, n_cols, h, (cudaStream_t)stream);
}

int spa_gelu_bwd(const spa_params* p, const void* dh, const void* u, int32_t n_cols, void* du, void* stream) {
  int rc = check_params(p);
  if (rc != SPA_OK) return rc;
  SPA_PTR(dh); SPA_PTR(u); SPA_PTR(du);
  SPA_REQUIRE(n_cols > 0 && (n_cols * (p->dtype == SPA_F32 ? 4 : 2)) % 16 == 0, SPA_ERR_INVALID_ARG);
  return launch_gelu(*p, u, dh, n_cols, du, (cudaStream_t)stream);
}

// ---- the block as one unit: sequencing only ------------------------------------------------------------------
struct spa_overlap {
  cudaStream_t side, side2;
  cudaEvent_t fork, join;
};

int spa_overlap_create(spa_overlap** out) {
  if (out == nullptr) return SPA_ERR_INVALID_ARG;
  spa_overlap* ov = new (std::nothrow) spa_overlap{nullptr, nullptr, nullptr, nullptr};
  if (ov == nullptr) return SPA_ERR_INVALID_ARG;
  cudaError_t e = cudaStreamCreateWithFlags(&ov->side, cudaStreamNonBlocking);
  if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&ov->side2, cudaStreamNonBlocking);
  if (e == cudaSuccess) e = cudaEventCreateWithFlags(&ov->fork, cudaEventDisableTiming);
  if (e == cudaSuccess) e = cudaEventCreateWithFlags(&ov->join, cudaEventDisableTiming);
  if (e != cudaSuccess) {
    set_cuda_error(e, "spa_overlap_create");
    spa_overlap_destroy(ov);
    return SPA_ERR_CUDA;
  }
  *out = ov;
  return SPA_OK;
}

int spa_overlap_destroy(spa_overlap* ov) {
  if (ov == nullptr) return SPA_OK;
  if (ov->join != nullptr) cudaEventDestroy(ov->join);
  if (ov->fork != nullptr) cudaEventDestroy(ov->fork);
  if (ov->side2 != nullptr) cudaStreamDestroy(ov->side2);
  if (ov->side != nullptr) cudaStreamDestroy(ov->side);
  delete ov;
  return SPA_OK;
}

namespace {
inline bool block_fused(const spa_params* p) { return !(p->flags & SPA_FLAG_UNFUSED); }
// The two products that scatter their rows to the tokens: tensor-core problems, else the fp32-FMA kernels.
int proj_scatter(const spa_params* p, const spa_block_buffers* b, void* y, void* stream) {
  if (spa_fused_scatter_supported(p))
    return spa_packed_proj_scatter(p, b->attn_out, b->W_o, b->b_o, b->idx, b->cu_seqlens, y, b->d_status, stream);
  SPA_PTR(b->attn_out); SPA_PTR(b->W_o); SPA_PTR(b->idx); SPA_PTR(b->cu_seqlens); SPA_PTR(y); SPA_OPT_PTR(b->b_o);
  return linear_fwd_other(*p, b->attn_out, b->W_o, b->b_o, p->C, p->C, b->cu_seqlens, y, b->d_status, stream, b->idx,
                          (p->flags & SPA_FLAG_RESIDUAL) != 0);
}
int qkv_bwd_scatter(const spa_params* p, const spa_block_buffers* b, float* dW, float* db, void* ws, void* stream) {
  if (spa_fused_scatter_supported(p))
    return spa_packed_linear_bwd_scatter(p, b->x_packed, b->W_qkv, b->dqkv, p->C, 3 * p->C, b->idx, b->cu_seqlens, b->dX, dW, db,
                                         ws, b->d_status, stream);
  SPA_PTR(b->dqkv); SPA_PTR(b->W_qkv); SPA_PTR(b->x_packed); SPA_PTR(b->idx); SPA_PTR(b->cu_seqlens); SPA_PTR(b->dX);
  SPA_OPT_PTR(dW); SPA_OPT_PTR(db);
  return linear_bwd_other(*p, b->x_packed, b->W_qkv, b->dqkv, p->C, 3 * p->C, b->cu_seqlens, b->dX, dW, db, b->d_status, stream,
                          b->idx, (p->flags & SPA_FLAG_RESIDUAL) != 0);
}
inline bool is_recorded(cudaStream_t st) {
  cudaStreamCaptureStatus s = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(st, &s) == cudaSuccess) return s == cudaStreamCaptureStatusActive;
  cudaGetLastError();
  return false;
}
// `side` (a stream of ov) starts after everything enqueued on the main stream so far
inline int fork_side(const spa_overlap* ov, cudaStream_t main, cudaStream_t side) {
  cudaError_t e = cudaEventRecord(ov->fork, main);
  if (e == cudaSuccess) e = cudaStreamWaitEvent(side, ov->fork, 0);
  if (e != cudaSuccess) { set_cuda_error(e, "spa_block_bwd: fork"); return SPA_ERR_CUDA; }
  return SPA_OK;
}
inline int join_side(const spa_overlap* ov, cudaStream_t main, cudaStream_t side) {
  cudaError_t e = cudaEventRecord(ov->join, side);
  if (e == cudaSuccess) e = cudaStreamWaitEvent(main, ov->join, 0);
  if (e != cudaSuccess) { set_cuda_error(e, "spa_block_bwd: join"); return SPA_ERR_CUDA; }
  return SPA_OK;
}
#define SPA_STEP(call) do { rc = (call); if (rc != SPA_OK) return rc; } while (0)
}  // namespace

int spa_block_fwd(const spa_params* p, const spa_block_buffers* b, void* stream) {
  int rc = check_params(p);
  if (rc != SPA_OK) return rc;
  if (b == nullptr) return SPA_ERR_INVALID_ARG;
  const bool inplace = (p->flags & SPA_FLAG_INPLACE) != 0;
  const bool fused = block_fused(p);
  void* y = inplace ? const_cast<void*>(b->x) : b->y;
  SPA_REQUIRE(!inplace || b->y == nullptr || b->y == b->x, SPA_ERR_INVALID_ARG);
  // gate (Eq. 4) and hard selection; on the fused path it also writes the pass-through rows y = x
  const bool one_pass = b->pack_state != nullptr && b->order == nullptr && gate_pack_supported(*p);
  if (one_pass)  // gate, selection and packing read x once
    SPA_STEP(spa_gate_select_pack(p, b->x, b->w_g, b->b_g, b->s_up, b->scores, b->mask, (fused && !inplace) ? y : nullptr,
                                  b->x_packed, b->idx, b->inv, b->cu_seqlens, b->pack_state, b->d_status, stream));
  else if (fused && !inplace) SPA_STEP(spa_gate_prefill(p, b->x, b->w_g, b->b_g, b->s_up, b->scores, b->mask, y, stream));
  else SPA_STEP(spa_gate(p, b->x, b->w_g, b->b_g, b->s_up, b->scores, b->mask, stream));
  // token packing
  if (one_pass) {
  } else if (b->order == nullptr)
    SPA_STEP(spa_select_pack(p, b->x, b->mask, b->scores, b->x_packed, b->idx, b->inv, b->cu_seqlens, b->d_status, stream));
  else
    SPA_STEP(spa_select_pack_ordered(p, b->x, b->mask, b->scores, b->order, b->x_packed, b->idx, b->inv, b->cu_seqlens,
                                     b->d_status, stream));
  if (b->container_len > 0) {  // the paper's containers: cuts built on the device from the selection just packed
    SPA_REQUIRE(b->seg_offsets != nullptr, SPA_ERR_INVALID_ARG);
    SPA_STEP(spa_container_offsets(p, b->cu_seqlens, b->container_len, const_cast<int32_t*>(b->seg_offsets), stream));
  }
  SPA_STEP(spa_packed_qkv(p, b->x_packed, b->W_qkv, b->b_qkv, b->cu_seqlens, b->qkv, b->d_status, stream));
  const int32_t* seg = b->seg_offsets != nullptr ? b->seg_offsets : b->cu_seqlens;
  const int32_t n_seg = b->container_len > 0 ? spa_container_max_segments(p, b->container_len)
                                             : (b->seg_offsets != nullptr ? b->n_seg : p->B);
  SPA_STEP(spa_packed_attention_fwd(p, b->qkv, seg, n_seg, b->attn_out, b->lse, b->d_status, stream));
  if (fused) return proj_scatter(p, b, y, stream);
  SPA_STEP(spa_packed_proj(p, b->attn_out, b->W_o, b->b_o, b->cu_seqlens, b->z, b->d_status, stream));
  return spa_unpack_scatter(p, b->z, inplace ? nullptr : b->x, b->idx, b->inv, b->cu_seqlens, y, b->d_status, stream);
}

int spa_block_bwd(const spa_params* p, const spa_block_buffers* b, void* stream) {
  int rc = check_params(p);
  if (rc != SPA_OK) return rc;
  if (b == nullptr) return SPA_ERR_INVALID_ARG;
  const int C = p->C;
  cudaStream_t main = (cudaStream_t)stream;
  // the weight gradients feed nothing downstream: with `overlap` they run on the second stream, with a scratch
  // area of their own, beside the attention backward and the input gradients.
  const spa_overlap* ov = b->overlap;
  SPA_REQUIRE(ov == nullptr || b->workspace_side != nullptr || spa_workspace_bytes(p) == 0, SPA_ERR_INVALID_ARG);
  const bool fused = block_fused(p) && !b->trainable;
  const int32_t* seg = b->seg_offsets != nullptr ? b->seg_offsets : b->cu_seqlens;
  const int32_t n_seg = (b->container_len > 0 && b->seg_offsets != nullptr)
                            ? spa_container_max_segments(p, b->container_len)
                            : (b->seg_offsets != nullptr ? b->n_seg : p->B);
  void* side = ov != nullptr ? (void*)ov->side : nullptr;

  if (b->trainable)
    SPA_STEP(spa_select_loss(p, b->scores, b->labels, b->alpha, b->ds, b->loss, b->train_workspace, stream));
  // dz = rows of dY at the selected tokens; dX = dY on the tokens that passed through
  SPA_STEP(spa_unpack_scatter_bwd(p, b->dY, b->idx, b->inv, b->cu_seqlens, b->dz, b->dX, stream));
  // In a recorded step the QKV layer's weight gradient has a stream of its own, with scratch of its own: `workspace`, whose
  // D_i the attention backward in front of it was the last to read.  Behind the projection's on one stream it would have two
  // predecessors, and such a kernel of a graph is not launched early (programmatic launch).  One graph per step, 64 images
  // of 196 tokens of 384 channels 127.6 -> 122.0 us, 2 of 4 200 of 256 133.0 -> 126.6, 128 of 196 of 768 245 -> 242.5.  The
  // second fork and join cost 2 us, more than that gives on small batches (16 images of 196 tokens of 768 channels 98 ->
  // 100, of 384 76.5 -> 75.0) and 1 to 2 us in a step that is not recorded.
  const bool apart = ov != nullptr && b->workspace != nullptr && p->capacity >= 4096 && is_recorded(main);
  cudaStream_t side_qkv = ov == nullptr ? nullptr : (apart ? ov->side2 : ov->side);
  bool forked = false, forked_qkv = false;
  int rc_side = SPA_OK;
  if (ov == nullptr) {
    SPA_STEP(spa_packed_linear_bwd(p, b->attn_out, b->W_o, b->dz, C, C, b->cu_seqlens, b->d_attn_out, b->dW_o, b->db_o,
                                   b->workspace, b->d_status, stream));
  } else {
    SPA_STEP(fork_side(ov, main, ov->side));
    forked = true;
    rc_side = spa_packed_linear_bwd(p, b->attn_out, b->W_o, b->dz, C, C, b->cu_seqlens, nullptr, b->dW_o, b->db_o,
                                    b->workspace_side, b->d_status, side);
    rc = spa_packed_linear_bwd(p, b->attn_out, b->W_o, b->dz, C, C, b->cu_seqlens, b->d_attn_out, nullptr, nullptr,
                               b->workspace, b->d_status, stream);
  }
  if (rc == SPA_OK && rc_side == SPA_OK)
    rc = spa_packed_attention_bwd(p, b->qkv, b->attn_out, b->lse, b->d_attn_out, seg, n_seg, b->dqkv, b->workspace,
                                  b->d_status, stream);
  if (rc == SPA_OK && rc_side == SPA_OK) {
    if (ov != nullptr) {
      // it reads dqkv: behind the attention backward
      rc_side = fork_side(ov, main, side_qkv);
      forked_qkv = rc_side == SPA_OK;
      if (rc_side == SPA_OK)
        rc_side = spa_packed_linear_bwd(p, b->x_packed, b->W_qkv, b->dqkv, C, 3 * C, b->cu_seqlens, nullptr, b->dW_qkv,
                                        b->db_qkv, apart ? b->workspace : b->workspace_side, b->d_status, (void*)side_qkv);
    }
    float* dW = ov != nullptr ? nullptr : b->dW_qkv;
    float* db = ov != nullptr ? nullptr : b->db_qkv;
    void* ws = ov != nullptr ? nullptr : b->workspace;
    if (fused) {
      // the input gradient scatters its rows to the selected tokens itself: no packed dx, no scatter kernel
      rc = qkv_bwd_scatter(p, b, dW, db, ws, stream);
    } else {
      rc = spa_packed_linear_bwd(p, b->x_packed, b->W_qkv, b->dqkv, C, 3 * C, b->cu_seqlens, b->dx_packed, dW, db,
                                 ov != nullptr ? b->workspace : ws, b->d_status, stream);
      if (rc == SPA_OK) {
        if (b->trainable && (p->flags & SPA_FLAG_GATE_SCALE))
          rc = spa_select_pack_bwd_gated(p, b->dx_packed, b->x, b->scores, b->dY, b->idx, b->cu_seqlens, b->dX, b->ds,
                                         stream);
        else
          rc = spa_select_pack_bwd(p, b->dx_packed, b->dY, b->idx, b->cu_seqlens, b->dX, stream);
      }
    }
  }
  if (rc == SPA_OK && rc_side == SPA_OK && b->trainable)
    rc = spa_gate_bwd(p, b->x, b->w_g, b->scores, b->s_up, b->ds, b->dX, b->dw_g, b->db_g, b->ds_up, b->train_workspace, stream);
  if (forked) {  // joined on every path, so that a recording stream is never left forked
    int rj = join_side(ov, main, ov->side);
    if (forked_qkv && side_qkv != ov->side) {
      const int rq = join_side(ov, main, side_qkv);
      if (rj == SPA_OK) rj = rq;
    }
    if (rc == SPA_OK) rc = rc_side != SPA_OK ? rc_side : rj;
  }
  return rc;
}
namespace {
// A linear layer whose result goes through `epi` on its way out, whichever kernels the problem takes: where they cannot
// (bf16 on fp32 FMAs), the same as calls of their own.
int linear_fwd_epi(const spa_params* p, const void* a, const void* W, const void* bias, int n_in, int n_out, const int32_t* cu,
                   void* out, const LinearEpilogue& epi, int32_t* d_status, void* stream) {
  SPA_PTR(a); SPA_PTR(W); SPA_PTR(cu); SPA_PTR(out); SPA_OPT_PTR(bias); SPA_OPT_PTR(epi.add); SPA_OPT_PTR(epi.h);
  const int es = p->dtype == SPA_F32 ? 4 : 2;
  SPA_REQUIRE(n_in > 0 && n_out > 0, SPA_ERR_INVALID_ARG);
  SPA_REQUIRE((n_in * es) % 16 == 0 && (n_out * es) % 16 == 0, SPA_ERR_UNSUPPORTED);
  cudaStream_t st = (cudaStream_t)stream;
  if (p->dtype == SPA_F32) return launch_linear_fwd_f32(*p, a, W, bias, n_in, n_out, cu, out, d_status, st, nullptr, epi);
  if (use_tc(p) && tc_linear_supported(n_in, n_out)) {
    const int rc = launch_linear_fwd_tc(*p, a, W, bias, n_in, n_out, cu, out, d_status, st, nullptr, epi);
    if (rc != SPA_ERR_UNSUPPORTED) return rc;
  }
  if (epi.add != nullptr && epi.add != out) {
    const int rc = spa_unpack_prefill(p, epi.add, out, stream);
    if (rc != SPA_OK) return rc;
  }
  const int rc = launch_linear_fwd_simt(*p, a, W, bias, n_in, n_out, cu, out, st, nullptr, epi.add != nullptr);
  return rc != SPA_OK || epi.h == nullptr ? rc : launch_gelu(*p, out, nullptr, n_out, epi.h, st);
}
// ... and the gradients of one; da *= gelu'(u)
int linear_bwd_gelu(const spa_params* p, const void* a, const void* W, const void* dout, int n_in, int n_out, const int32_t* cu,
                    void* da, const void* u, float* dW, float* db, void* workspace, int32_t* d_status, void* stream) {
  SPA_PTR(a); SPA_PTR(W); SPA_PTR(dout); SPA_PTR(cu); SPA_PTR(da); SPA_PTR(u); SPA_OPT_PTR(dW); SPA_OPT_PTR(db); SPA_OPT_PTR(workspace);
  const int es = p->dtype == SPA_F32 ? 4 : 2;
  SPA_REQUIRE(n_in > 0 && n_out > 0, SPA_ERR_INVALID_ARG);
  SPA_REQUIRE((n_in * es) % 16 == 0 && (n_out * es) % 16 == 0, SPA_ERR_UNSUPPORTED);
  cudaStream_t st = (cudaStream_t)stream;
  LinearEpilogue epi;
  epi.u = u;
  if (p->dtype == SPA_F32) return launch_linear_bwd_f32(*p, a, W, dout, n_in, n_out, cu, da, dW, db, d_status, st, nullptr, epi);
  if (use_tc(p) && tc_linear_supported(n_in, n_out) && workspace != nullptr) {
    const int rc = launch_linear_bwd_tc(*p, a, W, dout, n_in, n_out, cu, da, dW, db, workspace, d_status, st, nullptr, epi);
    if (rc != SPA_ERR_UNSUPPORTED) return rc;
  }
  const int rc = launch_linear_bwd_simt(*p, a, W, dout, n_in, n_out, cu, da, dW, db, st);
  return rc != SPA_OK ? rc : launch_gelu(*p, u, da, n_in, da, st);
}
int check_layer(const spa_params* p, const spa_layer_buffers* l) {
  const int rc = check_params(p);
  if (rc != SPA_OK) return rc;
  if (l == nullptr || l->blk == nullptr) return SPA_ERR_INVALID_ARG;
  SPA_PTR(l->x); SPA_PTR(l->g1); SPA_PTR(l->be1); SPA_PTR(l->g2); SPA_PTR(l->be2);
  SPA_PTR(l->z); SPA_PTR(l->y1); SPA_PTR(l->t); SPA_PTR(l->out); SPA_PTR(l->u); SPA_PTR(l->h);
  SPA_REQUIRE(l->m1 != nullptr && l->r1 != nullptr && l->m2 != nullptr && l->r2 != nullptr && l->eps > 0.f, SPA_ERR_INVALID_ARG);
  SPA_REQUIRE((p->flags & SPA_FLAG_RESIDUAL) != 0, SPA_ERR_INVALID_ARG);
  return SPA_OK;
}
}  // namespace

size_t spa_layer_workspace_bytes(const spa_params* p, int32_t hidden, int32_t side) {
  if (check_params(p) != SPA_OK || hidden <= 0) return 0;
  size_t most = 0;
  auto at_least = [&](size_t bytes) { most = bytes > most ? bytes : most; };
  if (side != 0) {  // the weight gradients
    const int layers[4][2] = {{hidden, p->C}, {p->C, hidden}, {p->C, p->C}, {p->C, 3 * p->C}};
    for (const auto& l : layers) at_least(tc_weight_grad_workspace_bytes(*p, l[0], l[1]));
  } else {  // D_i of the attention backward, the per-CTA sums of the LayerNorm backward
    at_least(tc_attention_workspace_bytes(*p));
    at_least(layer_norm_workspace_bytes(*p));
  }
  return (most + 255) & ~(size_t)255;
}

// Eight kernels instead of the twelve that the calls one by one take (a kernel boundary costs 2.6 us, more than the work of
// most of them on a small batch): LN1 also writes the gate's scores and the residual stream, the first feed-forward product
// writes its activation too, the second adds the residual from where it lies.  8 x 196 tokens of 384 channels: 78 -> 67 us.
int spa_layer_fwd(const spa_params* p, const spa_layer_buffers* l, void* stream) {
  int rc = check_layer(p, l);
  if (rc != SPA_OK) return rc;
  const spa_block_buffers* b = l->blk;
  const int C = p->C, Hd = l->hidden;
  SPA_PTR(b->w_g); SPA_PTR(b->scores); SPA_PTR(b->mask);
  if (p->B == 0) return SPA_OK;
  SPA_STEP(launch_layer_norm_gate(*p, l->x, l->g1, l->be1, l->eps, l->z, l->m1, l->r1, b->w_g, b->b_g, b->scores, b->mask, l->y1,
                                  (cudaStream_t)stream));
  SPA_STEP(spa_select_pack(p, l->z, b->mask, b->scores, b->x_packed, b->idx, b->inv, b->cu_seqlens, b->d_status, stream));
  SPA_STEP(spa_packed_qkv(p, b->x_packed, b->W_qkv, b->b_qkv, b->cu_seqlens, b->qkv, b->d_status, stream));
  SPA_STEP(spa_packed_attention_fwd(p, b->qkv, b->cu_seqlens, p->B, b->attn_out, b->lse, b->d_status, stream));
  if (block_fused(p)) {
    SPA_STEP(proj_scatter(p, b, l->y1, stream));  // joins the residual stream that LN1 has copied
  } else {
    SPA_STEP(spa_packed_proj(p, b->attn_out, b->W_o, b->b_o, b->cu_seqlens, b->z, b->d_status, stream));
    SPA_STEP(spa_unpack_scatter(p, b->z, l->x, b->idx, b->inv, b->cu_seqlens, l->y1, b->d_status, stream));
  }
  SPA_STEP(launch_layer_norm(*p, l->y1, l->g2, l->be2, l->eps, l->t, l->m2, l->r2, (cudaStream_t)stream));
  LinearEpilogue up, down;
  up.h = l->h;
  down.add = l->y1;
  SPA_STEP(linear_fwd_epi(p, l->t, l->W1, l->b1, C, Hd, l->cu_all, l->u, up, b->d_status, stream));
  return linear_fwd_epi(p, l->h, l->W2, l->b2, Hd, C, l->cu_all, l->out, down, b->d_status, stream);
}

// The activation's derivative rides on the input gradient of the second product, dz on LN2's backward, and LN1's backward
// gathers its rows from the packed input gradient: no pass over the hidden gradient, no zeroed and scattered dZ.
int spa_layer_bwd(const spa_params* p, const spa_layer_buffers* l, void* stream) {
  int rc = check_layer(p, l);
  if (rc != SPA_OK) return rc;
  const spa_block_buffers* b = l->blk;
  const int C = p->C, Hd = l->hidden;
  cudaStream_t st = (cudaStream_t)stream;
  SPA_PTR(l->d_out); SPA_PTR(l->dh); SPA_PTR(l->dt); SPA_PTR(l->dy1); SPA_PTR(l->dX); SPA_PTR(b->dz); SPA_PTR(b->dx_packed);
  SPA_PTR(b->inv);
  SPA_REQUIRE(l->dg1 != nullptr && l->dbe1 != nullptr && l->dg2 != nullptr && l->dbe2 != nullptr && l->workspace != nullptr,
              SPA_ERR_INVALID_ARG);
  if (p->B == 0) return SPA_OK;
  // the weight gradients on the second stream where there is one, each beside the input gradient of its layer and what
  // follows (as in spa_block_bwd)
  const spa_overlap* ov = l->workspace_side != nullptr ? b->overlap : nullptr;
  void* side = ov != nullptr ? (void*)ov->side : stream;
  void* ws_side = ov != nullptr ? l->workspace_side : l->workspace;
  bool forked = false;
  auto fork = [&]() -> int {
    if (ov == nullptr) return SPA_OK;
    forked = true;
    return fork_side(ov, st, ov->side);
  };
  auto run = [&]() -> int {
    SPA_STEP(fork());
    SPA_STEP(spa_packed_linear_bwd(p, l->h, l->W2, l->d_out, Hd, C, l->cu_all, nullptr, l->dW2, l->db2, ws_side, b->d_status, side));
    SPA_STEP(linear_bwd_gelu(p, l->h, l->W2, l->d_out, Hd, C, l->cu_all, l->dh, l->u, nullptr, nullptr, l->workspace, b->d_status, stream));
    SPA_STEP(fork());
    SPA_STEP(spa_packed_linear_bwd(p, l->t, l->W1, l->dh, C, Hd, l->cu_all, nullptr, l->dW1, l->db1, ws_side, b->d_status, side));
    SPA_STEP(spa_packed_linear_bwd(p, l->t, l->W1, l->dh, C, Hd, l->cu_all, l->dt, nullptr, nullptr, l->workspace, b->d_status, stream));
    SPA_STEP(launch_layer_norm_bwd(*p, l->dt, l->y1, l->g2, l->m2, l->r2, l->d_out, l->dy1, l->dg2, l->dbe2, l->workspace, st, nullptr,
                                   b->inv, b->dz));
    SPA_STEP(fork());
    SPA_STEP(spa_packed_linear_bwd(p, b->attn_out, b->W_o, b->dz, C, C, b->cu_seqlens, nullptr, b->dW_o, b->db_o, ws_side, b->d_status,
                                   side));
    SPA_STEP(spa_packed_linear_bwd(p, b->attn_out, b->W_o, b->dz, C, C, b->cu_seqlens, b->d_attn_out, nullptr, nullptr, l->workspace,
                                   b->d_status, stream));
    SPA_STEP(spa_packed_attention_bwd(p, b->qkv, b->attn_out, b->lse, b->d_attn_out, b->cu_seqlens, p->B, b->dqkv, l->workspace,
                                      b->d_status, stream));
    SPA_STEP(fork());
    SPA_STEP(spa_packed_linear_bwd(p, b->x_packed, b->W_qkv, b->dqkv, C, 3 * C, b->cu_seqlens, nullptr, b->dW_qkv, b->db_qkv, ws_side,
                                   b->d_status, side));
    SPA_STEP(spa_packed_linear_bwd(p, b->x_packed, b->W_qkv, b->dqkv, C, 3 * C, b->cu_seqlens, b->dx_packed, nullptr, nullptr,
                                   l->workspace, b->d_status, stream));
    return launch_layer_norm_bwd(*p, b->dx_packed, l->x, l->g1, l->m1, l->r1, l->dy1, l->dX, l->dg1, l->dbe1, l->workspace, st, b->inv);
  };
  rc = run();
  if (forked) {  // joined on every path, so that a recording stream is never left forked
    const int rj = join_side(ov, st, ov->side);
    if (rc == SPA_OK) rc = rj;
  }
  return rc;
}
#undef SPA_STEP

int spa_read_status(const int32_t* d_status, void* stream) {
  if (d_status == nullptr) return SPA_ERR_INVALID_ARG;
  int32_t v = 0;
  cudaError_t e = cudaMemcpyAsync(&v, d_status, sizeof(v), cudaMemcpyDeviceToHost, (cudaStream_t)stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize((cudaStream_t)stream);
  if (e != cudaSuccess) { set_cuda_error(e, "spa_read_status"); return SPA_ERR_CUDA; }
  return v;
}

const char* spa_status_string(int status) {
  switch (status) {
    case SPA_OK: return "ok";
    case SPA_ERR_INVALID_ARG: return "invalid argument";
    case SPA_ERR_UNSUPPORTED: return "unsupported dtype, head dimension or size";
    case SPA_ERR_CAPACITY: return "more selected tokens than the packed capacity";
    case SPA_ERR_CUDA: return "CUDA runtime error";
    case SPA_ERR_TIMEOUT: return "a bounded device-side wait expired";
    case SPA_ERR_SCRATCH: return "the problem needs more scratch than the built-in array holds";
    default: return "unknown status";
  }
}

const char* spa_last_cuda_error(void) { return g_cuda_error; }

unsigned long long spa_launch_count(void) { return g_launches.load(std::memory_order_relaxed); }

}  // extern "C"
