// fp32 linear layers on the packed tokens (QKV / output projection and their gradients; the 3LC^2 and NC^2 terms of
// Eq. 9) on the tensor cores, at fp32 accuracy.
//
// An fp32 value is the exact sum of three bf16 values (8 + 8 + 8 bits of its 24): x = x0 + x1 + x2.  Of the nine
// products of two such sums the six largest are formed - x0 y0; x0 y1, x1 y0, x0 y2, x1 y1, x2 y0 - and what is left
// out lies below 2^-26 of |x||y|, under the rounding of an fp32 product.  x0 y0 has an accumulator of its own: the
// small terms then add no rounding steps at the magnitude of the result; the two are added at the end.  (The method:
// Henry, Tang, Heinecke, "Leveraging the bfloat16 Artificial Intelligence Datatype For Higher-Precision Computations", 2019.)
//   forward  A = a (K contiguous),     B = W (K contiguous),   M = packed rows (device)
//   dgrad    A = dout (K contiguous),  B = W (N contiguous),   M = packed rows (device)
//   wgrad    A = dout (M contiguous),  B = a (N contiguous),   K = packed rows (device)
// One tile of 128 x BN per CTA.  Eight warps load fp32 lines (64 contiguous values) one k-block ahead, split them and
// write three bf16 operand tiles under the 128-byte swizzle; either memory order keeps its lines, K-major or MN-major
// operands follow from it.  A ninth warp issues the products.  The finished tile goes through shared memory, where a
// cluster that splits K adds its partial tiles in a fixed order over distributed shared memory: no scratch in global
// memory, bitwise reproducible.
// Infinities: an infinite part times a zero part is NaN where the product of the values is not, and a finite value next to
// fp32's largest rounds to an infinite first part.  Either leaves an infinity or NaN in the result, so results that are not
// finite are formed again as a chain of fp32 FMAs over K (fma_chain), which is what they are by definition.
// Bound: 24 products per 64-k block and tile (1 650 clocks at BN = 128) against about 800 issue clocks of splitting.
// 1 568 x 1 152 x 384: forward 18, dgrad 23, wgrad 23 us, where fp32 FMAs on 64 x 64 tiles took 73, 99 and 141; error
// against fp64 1e-7 to 5e-7 relative, that of the FMA kernels 2e-7 to 1e-6.
#include <math_constants.h>

#include "simt_stage.cuh"
#include "sm100_ptx.cuh"
#include "spa_common.cuh"

namespace spa {
namespace {

constexpr int BM = 128, BK = 64;
constexpr int kWorkers = 256;              // threads that load, split and store
constexpr int kThreads = kWorkers + 32;    // and the warp that issues the products
constexpr int kStages = 2;
constexpr int kMaxSplit = 8;               // portable cluster size
constexpr int kAPlane = BM * 128;          // one bf16 operand tile: 128-byte lines
template <int BN> constexpr int kBPlane = BN * 128;
template <int BN> constexpr int kStageBytes = 3 * (kAPlane + kBPlane<BN>);
template <int BN> constexpr int kLdT = BN + 4;  // finished tile in shared memory, fp32
template <int BN> constexpr int kSmem = kStages * kStageBytes<BN> + 1024 + 64;

__device__ __forceinline__ float4 ld_values(const float* p) {
  const uint4 v = ld_dep16(p);
  return make_float4(__uint_as_float(v.x), __uint_as_float(v.y), __uint_as_float(v.z), __uint_as_float(v.w));
}

struct Tile8 { float4 a, b; };  // eight consecutive values of a line

// Two values into their three bf16 parts, packed pairwise.  An infinite first part has no rest.
__device__ __forceinline__ void split2(float x, float y, uint32_t& p0, uint32_t& p1, uint32_t& p2) {
  auto pack = [](float u, float v) { __nv_bfloat162 h = __floats2bfloat162_rn(u, v); return *reinterpret_cast<uint32_t*>(&h); };
  auto rest = [](float v, uint32_t part) { return (part & 0x7f800000u) != 0x7f800000u ? v - __uint_as_float(part) : 0.f; };
  p0 = pack(x, y);
  x = rest(x, p0 << 16);
  y = rest(y, p0 & 0xffff0000u);
  p1 = pack(x, y);
  x -= __uint_as_float(p1 << 16);
  y -= __uint_as_float(p1 & 0xffff0000u);
  p2 = pack(x, y);
}

// Operand tile of R rows (m or n) x BK: unit u = (line, 16-byte chunk of the bf16 line).  K contiguous: line = row.
// Rows contiguous: line = k, 64 rows per box.  A worker takes units tid, tid + 256, ...
template <int R, bool kMn> struct Operand {
  static constexpr int kUnits = R * 8 / kWorkers;
  __device__ static __forceinline__ void place(int u, int& row, int& k, uint32_t& off) {
    const int chunk = u & 7, line = u >> 3;
    if (!kMn) { row = line; k = chunk * 8; off = line * 128 + ((chunk ^ (line & 7)) << 4); }
    else { const int kl = line & 63, box = line >> 6; row = box * 64 + chunk * 8; k = kl; off = box * 8192 + kl * 128 + ((chunk ^ (kl & 7)) << 4); }
  }
  __device__ static __forceinline__ void load(Tile8* t, const float* src, long long ld, int r0, int rows, int k0,
                                              int k_end, int tid) {
#pragma unroll
    for (int i = 0; i < kUnits; ++i) {
      int row, k;
      uint32_t off;
      place(tid + i * kWorkers, row, k, off);
      row += r0; k += k0;
      const float* p = src + (kMn ? (long long)k * ld + row : (long long)row * ld + k);
      const bool in0 = row < rows && k < k_end, in1 = kMn ? (row + 4 < rows && k < k_end) : (row < rows && k + 4 < k_end);
      t[i].a = in0 ? ld_values(p) : make_float4(0.f, 0.f, 0.f, 0.f);
      t[i].b = in1 ? ld_values(p + 4) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
  }
  __device__ static __forceinline__ void store(const Tile8* t, uint8_t* plane0, int tid) {
    constexpr int kPlane = R * 128;
#pragma unroll
    for (int i = 0; i < kUnits; ++i) {
      int row, k;
      uint32_t off;
      place(tid + i * kWorkers, row, k, off);
      uint4 p0, p1, p2;
      split2(t[i].a.x, t[i].a.y, p0.x, p1.x, p2.x);
      split2(t[i].a.z, t[i].a.w, p0.y, p1.y, p2.y);
      split2(t[i].b.x, t[i].b.y, p0.z, p1.z, p2.z);
      split2(t[i].b.z, t[i].b.w, p0.w, p1.w, p2.w);
      *reinterpret_cast<uint4*>(plane0 + off) = p0;
      *reinterpret_cast<uint4*>(plane0 + kPlane + off) = p1;
      *reinterpret_cast<uint4*>(plane0 + 2 * kPlane + off) = p2;
    }
  }
};

__device__ __forceinline__ uint64_t operand_desc(uint32_t addr, int k, bool mn) {
  return mn ? ptx::smem_desc_sw128(addr + k * 2048, BK * 128, 1024) : ptx::smem_desc_sw128(addr + k * 32, 16, 1024);
}

// Results m, n .. n + 3 as chains of FMAs over K, for those that the three parts leave infinite or NaN: rare, so not inlined.
// Chains that are all NaN stay NaN.
template <bool kAMn, bool kBMn>
__device__ __noinline__ float4 fma_chain(const float* A, long long lda, const float* B, long long ldb, int m, int n, int K) {
  float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
  for (int k = 0; k < K; ++k) {
    const float a = A[kAMn ? (long long)k * lda + m : (long long)m * lda + k];
    float b[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) b[j] = B[kBMn ? (long long)k * ldb + n + j : (long long)(n + j) * ldb + k];
    v.x = fmaf(a, b[0], v.x);
    v.y = fmaf(a, b[1], v.y);
    v.z = fmaf(a, b[2], v.z);
    v.w = fmaf(a, b[3], v.w);
    if (v.x != v.x && v.y != v.y && v.z != v.z && v.w != v.w) break;
  }
  return v;
}

// dyn_which: 1 = M is the device-side packed row count, 2 = K is.
// row_map (optional): output row i goes to row row_map[i] of `out`; add, u, h: LinearEpilogue.
// colsum (optional, wgrad): colsum[m] = sum_k A(m,k), by the CTAs of the first column of tiles from the lines they load.
template <int BN, bool kAMn, bool kBMn>
__global__ void __launch_bounds__(kThreads, 1)
gemm_f32_kernel(const float* A, long long lda, const float* Bm, long long ldb,
                const float* bias, float* out, long long ldo, int M, int N, int K,
                const int32_t* cu, int n_seg, int capacity, int dyn_which, const float* add, const float* u, float* h,
                const int32_t* row_map, float* __restrict__ colsum, int32_t* d_status) {
  using OpA = Operand<BM, kAMn>;
  using OpB = Operand<BN, kBMn>;
  constexpr uint32_t kIdesc = ptx::idesc_bf16_f32(BM, BN, kAMn, kBMn);
  constexpr uint32_t kCols = 2 * BN;  // x0 y0 in columns [0, BN), the five small products in [BN, 2 BN)
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t smem_base = (ptx::smem_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t* smem_al = smem_raw + (smem_base - ptx::smem_u32(smem_raw));
  const uint32_t bar_base = smem_base + kStages * kStageBytes<BN>;
  auto full_bar = [&](int s) { return bar_base + 8u * s; };
  auto empty_bar = [&](int s) { return bar_base + 8u * (kStages + s); };
  const uint32_t done_bar = bar_base + 8u * 2 * kStages;
  volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(smem_al + kStages * kStageBytes<BN> + 48);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(smem_al + kStages * kStageBytes<BN> + 52);
  if (tid == 0) {
    for (int s = 0; s < kStages; ++s) { ptx::mbar_init(full_bar(s), kWorkers / 32); ptx::mbar_init(empty_bar(s), 1); }
    ptx::mbar_init(done_bar, 1);
    *abort_flag = 0;
    ptx::fence_mbar_init();
  }
  pdl_entry();
  {
    const int rows = packed_rows(cu, n_seg, capacity);
    if (dyn_which == 1) M = rows; else K = rows;
  }
  const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
  if (m0 >= M || n0 >= N) return;  // the same for all CTAs of a cluster
  const int split = gridDim.z, z = blockIdx.z;
  const int k_blocks = (K + BK - 1) / BK;
  const int mine = z < k_blocks ? (k_blocks - z + split - 1) / split : 0;  // k-blocks z, z + split, ... are this CTA's
  const bool sums = kAMn && colsum != nullptr && blockIdx.x == 0;
  if (warp == kWorkers / 32) ptx::tmem_alloc(ptx::smem_u32(const_cast<uint32_t*>(tmem_slot)), kCols);
  ptx::tc_fence_before_sync();
  __syncthreads();
  ptx::tc_fence_after_sync();
  const uint32_t tmem = *tmem_slot;
  float asum[2][8] = {};  // wgrad: this worker's share of the column sums (its chunk of both boxes of A)

  if (warp < kWorkers / 32) {
    Tile8 a[OpA::kUnits], b[OpB::kUnits];
    auto load = [&](Tile8* ta, Tile8* tb, int i) {
      const int k0 = (z + i * split) * BK;
      OpA::load(ta, A, lda, m0, M, k0, K, tid);
      OpB::load(tb, Bm, ldb, n0, N, k0, K, tid);
    };
    if (mine > 0) load(a, b, 0);
    bool ok = true;
    for (int i = 0; i < mine; ++i) {
      Tile8 an[OpA::kUnits], bn[OpB::kUnits];
      if (i + 1 < mine) load(an, bn, i + 1);
      const int s = i % kStages;
      if (i >= kStages) ok = __all_sync(0xffffffffu, ok && ptx::mbar_wait(empty_bar(s), ((i / kStages) - 1) & 1)) != 0;
      if (!ok) {
        if (lane == 0) { record_status(d_status, SPA_ERR_TIMEOUT); *abort_flag = 1; }
        break;
      }
      uint8_t* st = smem_al + s * kStageBytes<BN>;
      OpA::store(a, st, tid);
      OpB::store(b, st + 3 * kAPlane, tid);
      ptx::fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0) ptx::mbar_arrive(full_bar(s));
      if (kAMn && sums) {
#pragma unroll
        for (int u = 0; u < OpA::kUnits; ++u) {
          float* d = asum[u / (OpA::kUnits / 2)];
          d[0] += a[u].a.x; d[1] += a[u].a.y; d[2] += a[u].a.z; d[3] += a[u].a.w;
          d[4] += a[u].b.x; d[5] += a[u].b.y; d[6] += a[u].b.z; d[7] += a[u].b.w;
        }
      }
#pragma unroll
      for (int u = 0; u < OpA::kUnits; ++u) a[u] = an[u];
#pragma unroll
      for (int u = 0; u < OpB::kUnits; ++u) b[u] = bn[u];
    }
  } else {
    // x0 y0 first, then the small terms: planes of A and B of each product
    bool ok = true;
    for (int i = 0; ok && i < mine; ++i) {
      const int s = i % kStages;
      ok = __all_sync(0xffffffffu, ptx::mbar_wait(full_bar(s), (i / kStages) & 1)) != 0 && *abort_flag == 0;
      ok = __all_sync(0xffffffffu, ok) != 0;
      if (!ok) {
        if (lane == 0) { record_status(d_status, SPA_ERR_TIMEOUT); *abort_flag = 1; }
        if (ptx::elect_one()) ptx::mma_commit(done_bar);  // the products issued so far
        __syncwarp();
        break;
      }
      ptx::tc_fence_after_sync();
      const uint32_t as = smem_base + s * kStageBytes<BN>, bs = as + 3 * kAPlane;
      if (ptx::elect_one()) {
#pragma unroll
        for (int q = 0; q < 6; ++q) {
          constexpr int pa[6] = {0, 0, 1, 0, 1, 2}, pb[6] = {0, 1, 0, 2, 1, 0};
#pragma unroll
          for (int k = 0; k < BK / 16; ++k)
            ptx::mma_bf16(tmem + (q == 0 ? 0 : BN), operand_desc(as + pa[q] * kAPlane, k, kAMn),
                          operand_desc(bs + pb[q] * kBPlane<BN>, k, kBMn), kIdesc, (i > 0 || k > 0 || q > 1) ? 1u : 0u);
        }
        ptx::mma_commit(empty_bar(s));
        if (i == mine - 1) ptx::mma_commit(done_bar);
      }
      __syncwarp();
    }
  }
  // every product that was issued has completed: the finished tile takes the stages' memory
  float* tile = reinterpret_cast<float*>(smem_al);
  constexpr int kLd = kLdT<BN>;
  static_assert((BM * kLd + BM) * 4 <= kStages * kStageBytes<BN> && 32 * 128 * 4 <= kStageBytes<BN>, "fits the stages");
  float* tile_sum = tile + BM * kLd;  // column sums, one per row of the tile
  __syncwarp();
  if (mine > 0 && !__all_sync(0xffffffffu, ptx::mbar_wait(done_bar, 0))) {
    if (lane == 0) { record_status(d_status, SPA_ERR_TIMEOUT); *abort_flag = 1; }
  }
  __syncthreads();
  if (kAMn && sums) {  // 32 workers per chunk of 8 rows, added up in a fixed order through the stages' memory
    if (tid < kWorkers) {
#pragma unroll
      for (int j = 0; j < 2; ++j)
#pragma unroll
        for (int e = 0; e < 8; ++e) tile[(tid >> 3) * BM + j * 64 + (tid & 7) * 8 + e] = asum[j][e];
    }
    __syncthreads();
    float v = 0.f;
    if (tid < BM)
      for (int r = 0; r < 32; ++r) v += tile[r * BM + tid];
    __syncthreads();
    if (tid < BM) tile_sum[tid] = v;
  }
  ptx::tc_fence_after_sync();
  if (warp < kWorkers / 32) {
    const int quarter = warp & 3, half = warp >> 2;
    float* row = tile + (quarter * 32 + lane) * kLd + half * (BN / 2);
#pragma unroll
    for (int c = 0; c < BN / 2; c += 32) {
      uint32_t r[32], r2[32];
      if (mine > 0) {
        const uint32_t at = tmem + ((uint32_t)(quarter * 32) << 16) + half * (BN / 2) + c;
        ptx::tmem_ld_32x32(at, r);
        ptx::tmem_ld_32x32(at + BN, r2);
        ptx::tmem_ld_wait();
      } else {
#pragma unroll
        for (int e = 0; e < 32; ++e) r[e] = r2[e] = 0u;
      }
#pragma unroll
      for (int e = 0; e < 32; e += 4)
        *reinterpret_cast<float4*>(row + c + e) =
            make_float4(__uint_as_float(r[e]) + __uint_as_float(r2[e]), __uint_as_float(r[e + 1]) + __uint_as_float(r2[e + 1]),
                        __uint_as_float(r[e + 2]) + __uint_as_float(r2[e + 2]), __uint_as_float(r[e + 3]) + __uint_as_float(r2[e + 3]));
    }
  }
  ptx::tc_fence_before_sync();
  if (split > 1) cluster_sync_all(); else __syncthreads();
  // rows z, z + split, ... of the tile: the partial tiles of the cluster added in the order of z, whole lines stored
  const int rows = M - m0 < BM ? M - m0 : BM;
  const int my_rows = (rows - z + split - 1) / split;
  if (!*abort_flag) {
    for (int e = tid; e < my_rows * (BN / 4); e += kThreads) {
      const int r = z + (e / (BN / 4)) * split, c = (e % (BN / 4)) * 4;
      if (n0 + c >= N) continue;
      const float* src = tile + r * kLd + c;
      float4 v = split > 1 ? sum_dsmem4(src, split) : *reinterpret_cast<const float4*>(src);
      if (!(fabsf(v.x) + fabsf(v.y) + fabsf(v.z) + fabsf(v.w) < CUDART_INF_F)) v = fma_chain<kAMn, kBMn>(A, lda, Bm, ldb, m0 + r, n0 + c, K);
      if (bias != nullptr) {
        const float4 w = ld_values(bias + n0 + c);
        v.x += w.x; v.y += w.y; v.z += w.z; v.w += w.w;
      }
      const int m = m0 + r;
      const long long at = (row_map != nullptr ? (long long)ld_dep(row_map + m) : (long long)m) * ldo + n0 + c;
      if (add != nullptr) {
        const float4 w = *reinterpret_cast<const float4*>(add + at);
        v.x += w.x; v.y += w.y; v.z += w.z; v.w += w.w;
      }
      if (u != nullptr) {
        const float4 w = *reinterpret_cast<const float4*>(u + at);
        v.x *= gelu_grad_f(w.x); v.y *= gelu_grad_f(w.y); v.z *= gelu_grad_f(w.z); v.w *= gelu_grad_f(w.w);
      }
      *reinterpret_cast<float4*>(out + at) = v;
      if (h != nullptr)
        *reinterpret_cast<float4*>(h + at) = make_float4(gelu_f(v.x), gelu_f(v.y), gelu_f(v.z), gelu_f(v.w));
    }
    if (kAMn && sums)
      for (int e = tid; e < my_rows; e += kThreads) {
        const int r = z + e * split;
        colsum[m0 + r] = split > 1 ? sum_dsmem(tile_sum + r, split) : tile_sum[r];
      }
  }
  if (split > 1) cluster_sync_all(); else __syncthreads();  // nobody leaves while a partial tile is still being read
  if (warp == kWorkers / 32) {
    ptx::tc_fence_after_sync();
    ptx::tmem_dealloc(tmem, kCols);
  }
}

struct Gemm {
  const void *A, *B, *bias;
  void* out;
  long long lda, ldb, ldo;
  int M, N, K, dyn_which;
  LinearEpilogue epi;
  const int32_t *cu, *row_map;
  int n_seg, capacity;
  float* colsum;
  int32_t* d_status;
};

template <int BN, bool kAMn, bool kBMn> int launch_tile(const Gemm& g, int split, cudaStream_t st, const char* what) {
  auto kern = gemm_f32_kernel<BN, kAMn, kBMn>;
  static DeviceOnce attr_once;  // per instantiation and device
  cudaError_t e = attr_once.run([&] { return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem<BN>); });
  if (e != cudaSuccess) { set_cuda_error(e, what); return SPA_ERR_CUDA; }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((g.N + BN - 1) / BN, (g.M + BM - 1) / BM, split);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = kSmem<BN>;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  int n = 0;
  if (pdl_enabled()) {
    attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[n++].val.programmaticStreamSerializationAllowed = 1;
  }
  if (split > 1) {
    attr[n].id = cudaLaunchAttributeClusterDimension;
    attr[n].val.clusterDim.x = 1;
    attr[n].val.clusterDim.y = 1;
    attr[n++].val.clusterDim.z = split;
  }
  cfg.attrs = attr;
  cfg.numAttrs = n;
  e = cudaLaunchKernelEx(&cfg, kern, (const float*)g.A, g.lda, (const float*)g.B, g.ldb, (const float*)g.bias, (float*)g.out, g.ldo,
                         g.M, g.N, g.K, g.cu, g.n_seg, g.capacity, g.dyn_which, (const float*)g.epi.add, (const float*)g.epi.u, (float*)g.epi.h, g.row_map, g.colsum, g.d_status);
  if (e != cudaSuccess) { set_cuda_error(e, what); return SPA_ERR_CUDA; }
  SPA_CUDA_CHECK_LAUNCH(what);
  return SPA_OK;
}

// Tile width and split of K by estimated clocks: waves of one CTA per SM, each with its k-blocks (1 650 clocks at
// BN = 128; 1 250 at BN = 64, whose products are bound by the operand reads), its start and end, and the exchange of
// a split.  M (or K) is only known on the device: half of the allocated rows stands for it.
template <bool kAMn, bool kBMn> int launch_gemm(const Gemm& g, cudaStream_t st, const char* what) {
  const int m = g.dyn_which == 1 ? (g.M + 1) / 2 : g.M, k = g.dyn_which == 2 ? (g.K + 1) / 2 : g.K;
  const int k_blocks = (k + BK - 1) / BK;
  int bn = 64, split = 1;
  long long best = -1;
  for (int b = 64; b <= 128; b += 64)
    for (int s = 1; s <= kMaxSplit && s <= k_blocks; s *= 2) {
      const long long ctas = (long long)((m + BM - 1) / BM) * ((g.N + b - 1) / b) * s;
      const long long cost = ((ctas + kNumSMs - 1) / kNumSMs) * (((k_blocks + s - 1) / s) * (b == 128 ? 1650 : 1250) + 4500 + (s > 1 ? 1500 : 0));
      if (best < 0 || cost < best) { best = cost; bn = b; split = s; }
    }
  return bn == 128 ? launch_tile<128, kAMn, kBMn>(g, split, st, what) : launch_tile<64, kAMn, kBMn>(g, split, st, what);
}

}  // namespace

int launch_linear_fwd_f32(const spa_params& p, const void* a, const void* W, const void* bias, int n_in, int n_out,
                          const int32_t* cu, void* out, int32_t* d_status, cudaStream_t st, const int32_t* row_map,
                          const LinearEpilogue& epi) {
  const Gemm g{a, W, bias, out, n_in, n_in, n_out, p.capacity, n_out, n_in, 1, epi, cu, row_map, p.B, p.capacity, nullptr, d_status};
  return launch_gemm<false, false>(g, st, "gemm_f32_kernel(fwd)");
}

int launch_linear_bwd_f32(const spa_params& p, const void* a, const void* W, const void* dout, int n_in, int n_out,
                          const int32_t* cu, void* da, float* dW, float* db, int32_t* d_status, cudaStream_t st,
                          const int32_t* row_map, const LinearEpilogue& epi) {
  if (da != nullptr) {  // da[m][j] = sum_o dout[m][o] W[o][j]
    const Gemm g{dout, W, nullptr, da, n_out, n_in, n_in, p.capacity, n_in, n_out, 1, epi, cu, row_map, p.B, p.capacity, nullptr, d_status};
    const int rc = launch_gemm<false, true>(g, st, "gemm_f32_kernel(dgrad)");
    if (rc != SPA_OK) return rc;
  }
  if (dW != nullptr) {  // dW[o][j] = sum_i dout[i][o] a[i][j]; db beside it
    const Gemm g{dout, a, nullptr, dW, n_out, n_in, n_in, n_out, n_in, p.capacity, 2, {}, cu, nullptr, p.B, p.capacity, db, d_status};
    return launch_gemm<true, true>(g, st, "gemm_f32_kernel(wgrad)");
  }
  return db != nullptr ? launch_colsum_simt(p, dout, n_out, cu, db, st) : SPA_OK;
}

}  // namespace spa
