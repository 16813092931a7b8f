// bf16 weight and bias gradients of the narrower packed layers (Sec. 3.2; the backward of the 3LC^2 and NC^2 terms of
// Eq. 9) in one kernel: dW[n_out][n_in] = dout^T a, db[m] = sum_k dout[k][m], K = the device-side packed row count.
//
// A cluster owns one 128 x 128 tile of dW and deals its CTAs the 64-row blocks of K in turn.  Every CTA accumulates its
// share in TMEM, turns it out to shared memory, and the cluster's CTAs add up the partial tiles - rows z, z + S, ... by
// CTA z, in the order of the CTAs - over distributed shared memory: dW is written once, no partial tile and no second
// kernel touches global memory, and the sums have a fixed order.  The bias gradient is the product with a matrix of
// ones (16 columns behind the tile's in TMEM) in the clusters of the first column of tiles.
// Split-K through global memory (up to 31 partial tiles per layer, a column-sum kernel and a reduction kernel) took
// 29.6 us for 768 x 256 over 15 120 rows, 14.3 us for 384 x 384 over 6 272 and 8.9 us for 1 152 x 384 over 98.
#include "simt_stage.cuh"
#include "sm100_ptx.cuh"
#include "spa_tc.cuh"

namespace spa {
namespace {

constexpr int kT = 128, BK = 64;     // tile of dW, rows of a k-block
constexpr int kOp = kT * BK * 2;     // one operand of a stage: two boxes of 64 columns x 64 rows (128-byte lines)
constexpr int kThreads = 192;        // warp 0: TMA, warp 1: MMA and TMEM, warps 2-5: accumulator to shared memory
constexpr int kLd = kT + 4;          // finished tile in shared memory, fp32
template <int kStages> constexpr int kSmem = kStages * 2 * kOp + 1024 /* ones */ + 1024 /* alignment */ + 128 /* barriers */ + kT * 4 /* sums */;
static_assert(kT * kLd * 4 <= 3 * 2 * kOp, "the finished tile takes the stages' memory");

// kStages = 3: two CTAs per SM, so that one's start and end run under the other's loop; 6: one CTA per SM with the same
// 192 KB of copies in flight (what the loop is bound by), where no more CTAs than SMs are launched.
template <int kStages>
__global__ void __launch_bounds__(kThreads, kStages == 3 ? 2 : 1)
wgrad_cluster_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, float* __restrict__ dW,
                     float* __restrict__ db, int M, int N, const int32_t* cu, int n_seg, int capacity,
                     uint32_t wait_limit, int32_t* d_status) {
  constexpr uint32_t kIdesc = ptx::idesc_bf16_f32(kT, kT, true, true);
  constexpr uint32_t kIdescOnes = ptx::idesc_bf16_f32(kT, 16, true, false);
  extern __shared__ uint8_t smem_raw[];
  const uint32_t smem_base = (ptx::smem_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t* smem_al = smem_raw + (smem_base - ptx::smem_u32(smem_raw));
  constexpr int kOnes = kStages * 2 * kOp, kBars = kOnes + 1024;
  const uint32_t bar_base = smem_base + kBars;
  auto full_bar = [&](int s) { return bar_base + 8u * s; };
  auto empty_bar = [&](int s) { return bar_base + 8u * (kStages + s); };
  const uint32_t done_bar = bar_base + 8u * 2 * kStages, drain_bar = done_bar + 8;
  constexpr int kSlot = 112;  // TMEM address, abort flag
  static_assert(8 * (2 * kStages + 2) <= kSlot, "the barriers end in front of the words behind them");
  volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(smem_al + kBars + kSlot);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(smem_al + kBars + kSlot + 4);
  float* tile = reinterpret_cast<float*>(smem_al);
  float* sums = reinterpret_cast<float*>(smem_al + kBars + 128);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  pdl_launch_dependents();
  if (tid == 0) {
    ptx::prefetch_tensormap(&tmA);
    ptx::prefetch_tensormap(&tmB);
    for (int s = 0; s < kStages; ++s) { ptx::mbar_init(full_bar(s), 1); ptx::mbar_init(empty_bar(s), 1); }
    ptx::mbar_init(done_bar, 1);
    ptx::mbar_init(drain_bar, 1);
    *abort_flag = 0;
    ptx::fence_mbar_init();
  }
  if (warp == 2) {  // 16 rows of 32 ones in whole lines: the same under any swizzle (8 lines serve as both row groups)
    for (int i = lane; i < 64; i += 32)
      *reinterpret_cast<uint4*>(smem_al + kOnes + i * 16) = make_uint4(0x3f803f80u, 0x3f803f80u, 0x3f803f80u, 0x3f803f80u);
    ptx::fence_proxy_async_smem();
  }
  if (warp == 1) ptx::tmem_alloc(ptx::smem_u32(const_cast<uint32_t*>(tmem_slot)), 2 * kT);
  ptx::tc_fence_before_sync();
  __syncthreads();
  ptx::tc_fence_after_sync();
  const uint32_t tmem = *tmem_slot;

  pdl_wait();
  const int K = packed_rows(cu, n_seg, capacity);
  const int n0 = blockIdx.x * kT, m0 = blockIdx.y * kT, split = gridDim.z, z = blockIdx.z;
  const int k_blocks = (K + BK - 1) / BK;
  const int mine = z < k_blocks ? (k_blocks - z + split - 1) / split : 0;  // k-blocks z, z + split, ...
  const bool with_sums = db != nullptr && blockIdx.x == 0;
  auto wait = [&](uint32_t bar, uint32_t parity) { return ptx::mbar_wait_or_abort(bar, parity, bar_base + kSlot + 4, d_status, SPA_ERR_TIMEOUT, wait_limit); };

  int issued = 0;  // the producer's: k-blocks whose copies have been issued
  if (warp == 0) {
    if (lane == 0) {
      int i = 0;
      for (; i < mine; ++i) {
        const int s = i % kStages, k0 = (z + i * split) * BK;
        if (i >= kStages && !wait(empty_bar(s), ((i / kStages) - 1) & 1)) break;
        const uint32_t a_dst = smem_base + s * 2 * kOp, b_dst = a_dst + kOp;
        ptx::mbar_expect_tx(full_bar(s), 2 * kOp);
#pragma unroll
        for (int j = 0; j < 2; ++j) ptx::tma_load_2d(a_dst + j * (BK * 128), &tmA, full_bar(s), m0 + 64 * j, k0);
#pragma unroll
        for (int j = 0; j < 2; ++j) ptx::tma_load_2d(b_dst + j * (BK * 128), &tmB, full_bar(s), n0 + 64 * j, k0);
      }
      issued = i;
    }
    __syncwarp();
  } else if (warp == 1) {
    // both 8-row groups of the ones operand are the same eight lines: a stride of zero between them
    const uint64_t ones_desc = ptx::smem_desc_sw128(smem_base + kOnes, 16, 0);
    bool live = true;  // every wait of this lane has been satisfied
    for (int i = 0; i < mine; ++i) {
      const int s = i % kStages;
      live = wait(full_bar(s), (i / kStages) & 1) && live;
      __syncwarp();
      const int k_valid = K - (z + i * split) * BK;
      if (k_valid < BK) {  // lines of the four boxes past the last packed row
        for (int line = k_valid + (lane >> 3); line < BK; line += 4)
#pragma unroll
          for (int box = 0; box < 4; ++box)
            *reinterpret_cast<uint4*>(smem_al + s * 2 * kOp + box * (BK * 128) + line * 128 + (lane & 7) * 16) = make_uint4(0, 0, 0, 0);
        ptx::fence_proxy_async_smem();
        __syncwarp();
      }
      ptx::tc_fence_after_sync();
      const uint32_t a_src = smem_base + s * 2 * kOp, b_src = a_src + kOp;
      if (ptx::elect_one()) {
#pragma unroll
        for (int k = 0; k < BK / 16; ++k)
          ptx::mma_bf16(tmem, ptx::smem_desc_sw128(a_src + k * 2048, BK * 128, 1024),
                        ptx::smem_desc_sw128(b_src + k * 2048, BK * 128, 1024), kIdesc, (i > 0 || k > 0) ? 1u : 0u);
        if (with_sums) {
#pragma unroll
          for (int k = 0; k < BK / 16; ++k)
            ptx::mma_bf16(tmem + kT, ptx::smem_desc_sw128(a_src + k * 2048, BK * 128, 1024), ones_desc, kIdescOnes, (i > 0 || k > 0) ? 1u : 0u);
        }
        if (live) ptx::mma_commit(empty_bar(s));
        if (i == mine - 1) ptx::mma_commit(done_bar);
      }
      __syncwarp();
    }
  } else {
    if (mine > 0) wait(done_bar, 0);
    __syncwarp();
    ptx::tc_fence_after_sync();
    const int q = warp & 3;
    float* row = tile + (q * 32 + lane) * kLd;
    const uint32_t at = tmem + ((uint32_t)(q * 32) << 16);
#pragma unroll
    for (int c = 0; c < kT; c += 64) {
      uint32_t r[64];
      if (mine > 0) {
        ptx::tmem_ld_32x32(at + c, r);
        ptx::tmem_ld_32x32(at + c + 32, r + 32);
        ptx::tmem_ld_wait();
      } else {
#pragma unroll
        for (int e = 0; e < 64; ++e) r[e] = 0u;
      }
#pragma unroll
      for (int e = 0; e < 64; e += 4) *reinterpret_cast<uint4*>(row + c + e) = make_uint4(r[e], r[e + 1], r[e + 2], r[e + 3]);
    }
    if (with_sums) {
      uint32_t r[16];
      r[0] = 0u;
      if (mine > 0) {
        ptx::tmem_ld_32x16(at + kT, r);
        ptx::tmem_ld_wait();
      }
      sums[q * 32 + lane] = __uint_as_float(r[0]);
    }
    ptx::tc_fence_before_sync();
  }
  __syncwarp();
  if (split > 1) cluster_sync_all(); else __syncthreads();
  const bool failed = *abort_flag != 0;
  if (!failed) {
    const int rows = M - m0 < kT ? M - m0 : kT, my_rows = rows > z ? (rows - z + split - 1) / split : 0;
    for (int e = tid; e < my_rows * (kT / 4); e += kThreads) {
      const int r = z + (e / (kT / 4)) * split, c = (e % (kT / 4)) * 4;
      if (n0 + c >= N) continue;
      const float* src = tile + r * kLd + c;
      float4 v = split > 1 ? sum_dsmem4(src, split) : *reinterpret_cast<const float4*>(src);
      *reinterpret_cast<float4*>(dW + (long long)(m0 + r) * N + n0 + c) = v;
    }
    if (with_sums)
      for (int e = tid; e < my_rows; e += kThreads) {
        const int r = z + e * split;
        db[m0 + r] = split > 1 ? sum_dsmem(sums + r, split) : sums[r];
      }
  }
  if (split > 1) cluster_sync_all(); else __syncthreads();  // nobody leaves while a partial tile is still being read
  if (__builtin_expect(failed, 0)) ptx::drain_cta(issued, kStages, full_bar(0), drain_bar);
  if (warp == 1) {
    ptx::tc_fence_after_sync();
    ptx::tmem_dealloc(tmem, 2 * kT);
  }
}

}  // namespace

namespace {
template <int kStages>
int launch_stages(dim3 grid, const CUtensorMap& tmA, const CUtensorMap& tmB, float* dW, float* db, int n_out, int n_in,
                  const int32_t* cu, const spa_params& p, int32_t* d_status, cudaStream_t st) {
  auto kern = wgrad_cluster_kernel<kStages>;
  static DeviceOnce once;  // per instantiation and device
  cudaError_t e = once.run([&] { return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem<kStages>); });
  if (e != cudaSuccess) { set_cuda_error(e, "wgrad_cluster_kernel"); return SPA_ERR_CUDA; }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = kSmem<kStages>;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  int n = 0;
  if (pdl_enabled()) {
    attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[n++].val.programmaticStreamSerializationAllowed = 1;
  }
  if (grid.z > 1) {
    attr[n].id = cudaLaunchAttributeClusterDimension;
    attr[n].val.clusterDim.x = 1;
    attr[n].val.clusterDim.y = 1;
    attr[n++].val.clusterDim.z = grid.z;
  }
  cfg.attrs = attr;
  cfg.numAttrs = n;
  e = cudaLaunchKernelEx(&cfg, kern, tmA, tmB, dW, db, n_out, n_in, cu, p.B, p.capacity, ptx::wait_limit(p.flags), d_status);
  if (e != cudaSuccess) { set_cuda_error(e, "wgrad_cluster_kernel"); return SPA_ERR_CUDA; }
  SPA_CUDA_CHECK_LAUNCH("wgrad_cluster_kernel");
  return SPA_OK;
}
}  // namespace

// K is split while the clusters still run all at once - clusters of 4 and 8 fill about seven eighths of the GPU - and
// every CTA keeps two k-blocks (when half of the capacity is in use).  Up to two CTAs per SM: a k-block of 128 x 128 takes
// an SM 530 clocks with two of them and 760 with one (shared memory takes 32 KB of copies in and 32 KB of operand
// reads, 512 clocks, for 280 clocks of products).
int launch_wgrad_cluster(const spa_params& p, const void* a, const void* dout, int n_in, int n_out, const int32_t* cu, float* dW,
                         float* db, int32_t* d_status, cudaStream_t st) {
  CUtensorMap tmA, tmB;
  if (!make_tmap_bf16_2d(&tmA, dout, n_out, p.capacity, (uint64_t)n_out * 2, 64, BK) ||
      !make_tmap_bf16_2d(&tmB, a, n_in, p.capacity, (uint64_t)n_in * 2, 64, BK))
    return SPA_ERR_UNSUPPORTED;
  const int tn = (n_in + kT - 1) / kT, tm = (n_out + kT - 1) / kT;
  int split = 1;
  while (split < 8 && tn * tm * split * 2 <= 256 && p.capacity / 2 >= split * 2 * 2 * BK) split *= 2;
  const dim3 grid(tn, tm, split);
  return tn * tm * split <= (split < 4 ? kNumSMs : 128) ? launch_stages<6>(grid, tmA, tmB, dW, db, n_out, n_in, cu, p, d_status, st)
                                    : launch_stages<3>(grid, tmA, tmB, dW, db, n_out, n_in, cu, p, d_status, st);
}

}  // namespace spa
