// Shared device/host helpers of the SPA kernels (sm_100a).
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>

#include "spa.h"

namespace spa {

constexpr int kNumSMs = 148;  // B200: two dies of 74 SMs

// Under programmatic dependent launch whoever wrote a kernel's operands may still run when the kernel starts, and they may
// be read behind pdl_wait() only.  So no kernel reads global memory by what the compiler may move above that wait or serve
// from the read-only path: no ld.global.nc, no __ldg, no cache-hint intrinsics (they are not ordered with the wait), no
// pointer that is read and __restrict__.  What is left: plain loads through ordinary pointers, and the loads below, which
// are volatile, as the wait is.  ld_dep: ordered with this kernel's other accesses too.  One exception: the bias of a linear
// layer, which no kernel of this library writes and which is read under a branch on the row count that came from behind
// the wait; behind plain loads the epilogues wait for it (14 413 x 768 x 256: 15.6 -> 16.8 us).
__device__ __forceinline__ int32_t ld_dep(const int32_t* p) {
  int32_t v;
  asm volatile("ld.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ uint32_t ld_dep(const uint8_t* p) {
  uint32_t v;
  asm volatile("ld.global.u8 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ uint4 ld_dep16(const void* p) {
  uint4 v;
  asm volatile("ld.global.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p) : "memory");
  return v;
}

// Number of valid packed rows: the device-resident total, clamped to the allocated rows.
__device__ __forceinline__ int packed_rows(const int32_t* offsets, int n_seg, int capacity) {
  int n = ld_dep(offsets + n_seg);
  return n < capacity ? n : capacity;
}

__device__ __forceinline__ void record_status(int32_t* d_status, int code) {
  if (d_status != nullptr) atomicCAS(d_status, 0, code);
}

// Programmatic dependent launch: every kernel lets its successor in the stream start being scheduled at
// once, and itself waits for its predecessor's results before touching global memory.  Launch
// latency and CTA ramp-up of the next kernel overlap the tail of this one.
__device__ __forceinline__ void pdl_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_entry() { pdl_launch_dependents(); pdl_wait(); }

// ---- 16-byte vector access, converted to fp32 ------------------------------------------------
template <typename T> struct Vec16;
template <> struct Vec16<float> {
  static constexpr int kElems = 4;
  __device__ static __forceinline__ void to_float(const uint4& v, float* f) {
    f[0] = __uint_as_float(v.x); f[1] = __uint_as_float(v.y);
    f[2] = __uint_as_float(v.z); f[3] = __uint_as_float(v.w);
  }
  __device__ static __forceinline__ uint4 from_float(const float* f) {
    return make_uint4(__float_as_uint(f[0]), __float_as_uint(f[1]), __float_as_uint(f[2]), __float_as_uint(f[3]));
  }
};
template <> struct Vec16<__nv_bfloat16> {
  static constexpr int kElems = 8;
  __device__ static __forceinline__ void to_float(const uint4& v, float* f) {
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {  // a bf16 is the high half of an fp32
      f[2 * i] = __uint_as_float(w[i] << 16);
      f[2 * i + 1] = __uint_as_float(w[i] & 0xffff0000u);
    }
  }
  __device__ static __forceinline__ uint4 from_float(const float* f) {
    uint32_t w[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      __nv_bfloat162 h = __floats2bfloat162_rn(f[2 * i], f[2 * i + 1]);
      w[i] = *reinterpret_cast<uint32_t*>(&h);
    }
    return make_uint4(w[0], w[1], w[2], w[3]);
  }
};

template <typename T> __device__ __forceinline__ float to_f32(T v);
template <> __device__ __forceinline__ float to_f32<float>(float v) { return v; }
template <> __device__ __forceinline__ float to_f32<__nv_bfloat16>(__nv_bfloat16 v) { return __bfloat162float(v); }

template <typename T> __device__ __forceinline__ T from_f32(float v);
template <> __device__ __forceinline__ float from_f32<float>(float v) { return v; }
template <> __device__ __forceinline__ __nv_bfloat16 from_f32<__nv_bfloat16>(float v) { return __float2bfloat16_rn(v); }

__device__ __forceinline__ uint4 ld_stream16(const void* p) {  // 16 bytes that are read once
  uint4 v;
  asm volatile("ld.global.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
  return v;
}

// 32 bytes in one store where they are a whole sector, else two of 16
__device__ __forceinline__ void st_global32(void* p, const uint4& a, const uint4& b, bool sector) {
  if (!sector) {
    static_cast<uint4*>(p)[0] = a;
    static_cast<uint4*>(p)[1] = b;
    return;
  }
  asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};"
               ::"l"(p), "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w), "r"(b.x), "r"(b.y), "r"(b.z), "r"(b.w) : "memory");
}
__device__ __forceinline__ void prefetch_l1(const void* p) { asm volatile("prefetch.global.L1 [%0];" ::"l"(p)); }

// The exact (erf) GELU and its derivative
__device__ __forceinline__ float gelu_f(float u) { return 0.5f * u * (1.f + erff(u * 0.70710678118654752f)); }
__device__ __forceinline__ float gelu_grad_f(float u) {
  return 0.5f * (1.f + erff(u * 0.70710678118654752f)) + u * 0.3989422804014327f * __expf(-0.5f * u * u);
}

// Standard normal distribution function and density, Phi(u) and phi(u), from Abramowitz and Stegun 7.1.26: erfc(x) =
// t (a1 + t (a2 + t (a3 + t (a4 + t a5)))) e^(-x^2), t = 1 / (1 + 0.3275911 x), x >= 0, |error| <= 1.5e-7 (Phi: 7e-8, in fp32
// 3e-7; by erff 6e-8).  For results stored as bf16, whose rounding is 2e-3 of them: gelu and gelu' come out the same but for 2
// and 0 of the 3 064 bf16 values of 0.001 < |u| < 4, with the same error; below, the tail's relative error grows (5e-5 at u =
// -3, 5e-4 at -4, 4e-3 at -6, 1e-2 at -8), less than that of 1 + erff, which has no digits left there.  About half of erff's
// instructions: 8 192 x 3 072 forward and backward in a layer's training, 509 -> 518 us by erff.
__device__ __forceinline__ void normal_cdf_pdf(float u, float& cdf, float& pdf) {
  const float x = fabsf(u) * 0.70710678118654752f;
  const float e = __expf(-x * x);
  const float t = __fdividef(1.f, fmaf(0.3275911f, x, 1.f));
  const float tail = 0.5f * t * fmaf(t, fmaf(t, fmaf(t, fmaf(t, 1.061405429f, -1.453152027f), 1.421413741f), -0.284496736f), 0.254829592f) * e;
  cdf = u < 0.f ? tail : 1.f - tail;
  pdf = 0.3989422804014327f * e;
}

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Segment containing packed row i: the s with offsets[s] <= i < offsets[s+1] (empty segments are skipped).
__device__ __forceinline__ int find_segment(const int32_t* offsets, int n_seg, int i) {
  int lo = 0, hi = n_seg;  // invariant: offsets[lo] <= i < offsets[hi]
  while (hi - lo > 1) {
    int mid = (lo + hi) >> 1;
    if (ld_dep(offsets + mid) <= i) lo = mid; else hi = mid;
  }
  return lo;
}

struct RowSeg { int lo, hi; };

// Segment bounds of packed row i (hi clamped to the valid rows); rows >= Np get an empty range.
__device__ __forceinline__ RowSeg row_segment(const int32_t* seg, int n_seg, int Np, int i) {
  RowSeg r{0, 0};
  if (i < Np) {
    const int s = find_segment(seg, n_seg, i);
    r.lo = ld_dep(seg + s);
    const int hi = ld_dep(seg + s + 1);
    r.hi = hi < Np ? hi : Np;
  }
  return r;
}

// ---- host side -------------------------------------------------------------------------------
void set_cuda_error(cudaError_t e, const char* where);
void count_launch();  // one more kernel of this library was enqueued (host-side tally)
#define SPA_CUDA_CHECK_LAUNCH(where)                                   \
  do {                                                                 \
    cudaError_t e__ = cudaGetLastError();                              \
    if (e__ != cudaSuccess) { ::spa::set_cuda_error(e__, where); return SPA_ERR_CUDA; } \
    ::spa::count_launch();                                             \
  } while (0)

// Set-up that a kernel needs once on every device that runs it (the opt-in to more than 48 KB of dynamic shared
// memory is a per-device attribute of the function).  run(fn) calls fn with the current device the first time that
// device is seen and never again once fn has returned cudaSuccess; safe to call from several host threads.
class DeviceOnce {
 public:
  template <typename F> cudaError_t run(F&& fn) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const unsigned long long bit = 1ull << (dev & 63);
    if (done_.load(std::memory_order_acquire) & bit) return cudaSuccess;
    e = fn();
    if (e == cudaSuccess) done_.fetch_or(bit, std::memory_order_release);
    return e;
  }
 private:
  std::atomic<unsigned long long> done_{0};
};

bool pdl_enabled();  // programmatic dependent launch is on unless the environment sets SPA_PDL=0

// Launch `kern` on `st`, allowing it to overlap the tail of the previous kernel of the stream.
template <typename... KArgs, typename... Args>
cudaError_t launch_pdl(void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl_enabled() ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kern, static_cast<KArgs>(args)...);
}

// launchers implemented per .cu file; every one enqueues on `st` and returns a spa_status
int launch_gate(const spa_params& p, const void* x, const void* w_g, float b_g, const float* s_up,
                float* scores, uint8_t* mask, void* y, cudaStream_t st);
int launch_select_pack(const spa_params& p, const void* x, const uint8_t* mask, const float* scores,
                       const int32_t* order, void* xp, int32_t* idx, int32_t* inv, int32_t* cu, int32_t* d_status,
                       cudaStream_t st);
// gate + selection + packing in one kernel (gate_pack.cu); y may be NULL (no pass-through copy)
bool gate_pack_supported(const spa_params& p);
size_t gate_pack_state_bytes(const spa_params& p);
int launch_gate_pack(const spa_params& p, const void* x, const void* w_g, float b_g, const float* s_up, float* scores,
                     uint8_t* mask, void* y, void* xp, int32_t* idx, int32_t* inv, int32_t* cu, void* state,
                     int32_t* d_status, cudaStream_t st);
int launch_container_offsets(const spa_params& p, const int32_t* cu, int L, int n_max, int32_t* out, cudaStream_t st);
int launch_unpack_scatter(const spa_params& p, const void* z, const void* x, const int32_t* idx,
                          const int32_t* inv, const int32_t* cu, void* y, cudaStream_t st);
int launch_unpack_scatter_bwd(const spa_params& p, const void* dY, const int32_t* idx, const int32_t* inv,
                              const int32_t* cu, void* dz, void* dX, cudaStream_t st);
int launch_select_pack_bwd(const spa_params& p, const void* dxp, const void* dY, const int32_t* idx,
                           const int32_t* cu, void* dX, cudaStream_t st);
// trainable selection (select_train.cu)
size_t train_workspace_bytes(const spa_params& p);
int launch_score_pool(const float* prev, int B, int rows, int cols, float* s_up, cudaStream_t st);
int launch_select_loss(const spa_params& p, const float* scores, const uint8_t* labels, float alpha, float* ds,
                       float* loss, void* workspace, cudaStream_t st);
int launch_pack_bwd_gated(const spa_params& p, const void* dxp, const void* x, const float* scores, const void* dY,
                          const int32_t* idx, const int32_t* cu, void* dX, float* ds, cudaStream_t st);
int launch_gate_bwd(const spa_params& p, const void* x, const void* w_g, const float* scores, const float* s_up,
                    const float* ds, void* dX, float* dw_g, float* db_g, float* ds_up, void* workspace,
                    cudaStream_t st);
// out[j] = sum over blocks (fixed order) of part[block * stride + j], j < n_out; the next n_out2 columns go to out2
int launch_partial_sum(const float* part, int n_blocks, int stride, int n_out, float* out, int n_out2, float* out2,
                       cudaStream_t st);
// the rest of the transformer block (block_rest.cu)
size_t layer_norm_workspace_bytes(const spa_params& p);
bool layer_norm_supported(const spa_params& p);
int launch_layer_norm(const spa_params& p, const void* x, const void* gamma, const void* beta, float eps, void* y,
                      float* mean, float* rstd, cudaStream_t st);
// with the gate on the normalised rows (scores, mask) and a copy of x
int launch_layer_norm_gate(const spa_params& p, const void* x, const void* gamma, const void* beta, float eps, void* y,
                           float* mean, float* rstd, const void* w_g, float b_g, float* scores, uint8_t* mask, void* copy,
                           cudaStream_t st);
// dy_row (optional): row t of dy is dy[dy_row[t]], zero where negative; dz_row, dz (optional): dz[dz_row[t]] = dx[t] too
int launch_layer_norm_bwd(const spa_params& p, const void* dy, const void* x, const void* gamma, const float* mean,
                          const float* rstd, const void* add, void* dx, float* dgamma, float* dbeta, void* workspace,
                          cudaStream_t st, const int32_t* dy_row = nullptr, const int32_t* dz_row = nullptr,
                          void* dz = nullptr);
int launch_gelu(const spa_params& p, const void* u, const void* dh, int n_cols, void* out, cudaStream_t st);
int launch_copy_tokens(const spa_params& p, const void* src, void* dst, cudaStream_t st);  // dst[B*N][C] = src

// What a linear layer's result goes through on its way out, row by row (rows as they are written, after row_map):
//   add   result += add                 (a residual branch; may be `out` itself)
//   u     result *= gelu'(u)            (the input gradient through the activation; u has the result's shape)
//   h     h = gelu(result) beside it    (h has the result's shape)
struct LinearEpilogue { const void* add = nullptr; const void* u = nullptr; void* h = nullptr; };

// out[M][n_out] = a[M][n_in] W[n_out][n_in]^T + bias, M = packed rows (device); row_map: output row i is written to row
// row_map[i] of `out`.  _simt: bf16 data on fp32 FMAs; _f32: fp32 data.
int launch_linear_fwd_simt(const spa_params& p, const void* a, const void* W, const void* bias, int n_in,
                           int n_out, const int32_t* cu, void* out, cudaStream_t st, const int32_t* row_map = nullptr,
                           bool accumulate = false);
int launch_linear_bwd_simt(const spa_params& p, const void* a, const void* W, const void* dout, int n_in,
                           int n_out, const int32_t* cu, void* da, float* dW, float* db, cudaStream_t st,
                           const int32_t* row_map = nullptr, bool accumulate = false);
int launch_colsum_simt(const spa_params& p, const void* dout, int n_out, const int32_t* cu, float* db, cudaStream_t st);
int launch_linear_fwd_f32(const spa_params& p, const void* a, const void* W, const void* bias, int n_in, int n_out,
                          const int32_t* cu, void* out, int32_t* d_status, cudaStream_t st,
                          const int32_t* row_map = nullptr, const LinearEpilogue& epi = {});
int launch_linear_bwd_f32(const spa_params& p, const void* a, const void* W, const void* dout, int n_in, int n_out,
                          const int32_t* cu, void* da, float* dW, float* db, int32_t* d_status, cudaStream_t st,
                          const int32_t* row_map = nullptr, const LinearEpilogue& epi = {});
int launch_attention_fwd_simt(const spa_params& p, const void* qkv, const int32_t* seg, int n_seg, void* ao,
                              float* lse, cudaStream_t st);
int launch_attention_bwd_simt(const spa_params& p, const void* qkv, const void* ao, const float* lse,
                              const void* dao, const int32_t* seg, int n_seg, void* dqkv, cudaStream_t st);

inline float softmax_scale_of(const spa_params& p) {
  return p.softmax_scale != 0.f ? p.softmax_scale : 1.0f / sqrtf((float)(p.C / p.H));
}

}  // namespace spa
