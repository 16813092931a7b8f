// Staging of operand tiles as fp32 in shared memory for the fp32-FMA kernels: asynchronous 16-byte copies where the
// source is fp32, load - convert - store where it is bf16.  Also the cluster helpers of their split sums.
#pragma once

#include "spa_common.cuh"

namespace spa {

// 16 bytes global -> shared without passing through registers; zero-filled when `in` is false (nothing is read then).
__device__ __forceinline__ void cp_async16(void* dst_smem, const void* src, bool in) {
  const uint32_t d = static_cast<uint32_t>(__cvta_generic_to_shared(dst_smem));
  const int n = in ? 16 : 0;
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(n) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// One 16-byte chunk of T at `src` (a valid address when `in`) to Vec16<T>::kElems floats at `dst`; zeros otherwise.
// `base` is any readable address: the source operand of a copy that reads nothing.
template <typename T> __device__ __forceinline__ void stage16(float* dst, const T* src, bool in, const T* base);
template <> __device__ __forceinline__ void stage16<float>(float* dst, const float* src, bool in, const float* base) {
  cp_async16(dst, in ? src : base, in);
}
template <>
__device__ __forceinline__ void stage16<__nv_bfloat16>(float* dst, const __nv_bfloat16* src, bool in, const __nv_bfloat16*) {
  float f[8] = {};
  if (in) Vec16<__nv_bfloat16>::to_float(*reinterpret_cast<const uint4*>(src), f);
  *reinterpret_cast<float4*>(dst) = make_float4(f[0], f[1], f[2], f[3]);
  *reinterpret_cast<float4*>(dst + 4) = make_float4(f[4], f[5], f[6], f[7]);
}

__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// the same variable in the shared memory of CTA `rank` of this cluster
__device__ __forceinline__ float ld_dsmem(const float* p, int rank) {
  uint32_t a;
  float v;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(static_cast<uint32_t>(__cvta_generic_to_shared(p))), "r"(rank));
  asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ float4 ld_dsmem4(const float* p, int rank) {
  uint32_t a;
  float4 v;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(static_cast<uint32_t>(__cvta_generic_to_shared(p))), "r"(rank));
  asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(a) : "memory");
  return v;
}
// Sum of the same variable over the first `split` <= 8 CTAs of the cluster, in their order, all loads in flight together
// (one after the other they took 4 700 of the 7 000 clocks behind a product's last k-block).
__device__ __forceinline__ float4 sum_dsmem4(const float* p, int split) {
  float4 w[8];
#pragma unroll
  for (int s = 0; s < 8; ++s)
    if (s < split) w[s] = ld_dsmem4(p, s);
  float4 v = w[0];
#pragma unroll
  for (int s = 1; s < 8; ++s)
    if (s < split) { v.x += w[s].x; v.y += w[s].y; v.z += w[s].z; v.w += w[s].w; }
  return v;
}
__device__ __forceinline__ float sum_dsmem(const float* p, int split) {
  float w[8];
#pragma unroll
  for (int s = 0; s < 8; ++s)
    if (s < split) w[s] = ld_dsmem(p, s);
  float v = w[0];
#pragma unroll
  for (int s = 1; s < 8; ++s)
    if (s < split) v += w[s];
  return v;
}

}  // namespace spa
