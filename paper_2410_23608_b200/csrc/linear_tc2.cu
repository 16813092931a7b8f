// bf16 linear layers on CTA pairs: the forward product and the input gradient of the wide layers
// (the 3LC^2 and NC^2 terms of Eq. 9 at C >= 512) with one tcgen05.mma spanning two SMs.
//
// A 128 x 128 tile per CTA needs 32 KB of operands for every 2 x 128 x 128 x 64 flops and is bound by the
// L2-to-SM operand feed at about half of the tensor pipe.  Here two CTAs of a cluster share one
// 256 x 256 tile: CTA r holds rows [128 r, 128 r + 128) of A and of the accumulator, and one half
// (128 of the 256 N positions) of B; the pair's MMA (cta_group::2, M = 256, N = 256) reads both
// halves of B from the two CTAs' shared memory.  Per CTA that is the same 32 KB per k-block for
// twice the flops.  Operand stages are filled by each CTA's own TMA loads (no multicast); all
// transaction bytes are counted on the leader CTA's barrier, whose MMA warp issues for the pair;
// tcgen05.commit releases the stage in both CTAs.  Two 256-column accumulators per CTA (all 512 TMEM
// columns) let the epilogue of one tile run under the main loop of the next.
//
// Barriers (s = stage, a = accumulator):
//   full[s]        leader only, 2 arrivals (one expect_tx per CTA) + the bytes of both CTAs' loads
//   empty[s]       both CTAs, 1 arrival: commit of the MMAs that read stage s (multicast to the pair)
//   tmem_full[a]   both CTAs, 1 arrival: commit after the last k-block of a tile (multicast)
//   tmem_empty[a]  leader only, 16 arrivals: the eight epilogue warps of each CTA
// Every wait is bounded; the cluster-wide barriers (after set-up, before exit, and a third where a wait has run out)
// are reached by every thread on every path, so a CTA never leaves while its peer may still touch its shared memory.
#include "sm100_ptx.cuh"
#include "spa_tc.cuh"

namespace spa {
namespace {

namespace ptx2 {
__device__ __forceinline__ uint32_t cluster_ctarank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// shared::cluster address of the same variable in CTA `rank` of the cluster
__device__ __forceinline__ uint32_t map_to_cta(uint32_t smem_addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(smem_addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// arrive (and add expected bytes) on a barrier that may live in the peer CTA
__device__ __forceinline__ void mbar_expect_tx_cluster(uint32_t cluster_bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cluster.b64 _, [%0], %1;" ::"r"(cluster_bar), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ int ld_peer_s32(uint32_t cluster_addr) {
  int v;
  asm volatile("ld.shared::cluster.s32 %0, [%1];" : "=r"(v) : "r"(cluster_addr) : "memory");
  return v;
}
__device__ __forceinline__ void st_peer_s32(uint32_t cluster_addr, int v) {
  asm volatile("st.shared::cluster.s32 [%0], %1;" ::"r"(cluster_addr), "r"(v) : "memory");
}
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t cluster_bar) {
  asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" ::"r"(cluster_bar) : "memory");
}
__device__ __forceinline__ void mbar_arrive_release_cluster(uint32_t cluster_bar) {  // publishes this CTA's writes to the pair
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_bar) : "memory");
}
// tiled load into this CTA's shared memory, completion counted on a barrier of the pair (leader's)
__device__ __forceinline__ void tma_load_2d_pair(uint32_t dst, const CUtensorMap* tm, uint32_t cluster_bar, int x, int y) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
      ::"r"(dst), "l"(reinterpret_cast<uint64_t>(tm)), "r"(cluster_bar), "r"(x), "r"(y) : "memory");
}
__device__ __forceinline__ void tmem_alloc_pair(uint32_t dst_smem, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(dst_smem), "r"(ncols) : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc_pair(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
// D[tmem, both CTAs] (+)= A * B with A, B in the shared memory of both CTAs; issued by one thread of the leader
__device__ __forceinline__ void mma_bf16_pair(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                              uint32_t accumulate) {
  const uint32_t z = 0;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, {%5, %5, %5, %5, %5, %5, %5, %5}, p;\n\t}"
      ::"r"(tmem_d), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate), "r"(z) : "memory");
}
// arrive on the barrier at this offset in both CTAs once every MMA issued so far has completed
__device__ __forceinline__ void mma_commit_pair(uint32_t bar) {
  const uint16_t mask = 3;
  asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
               ::"r"(bar), "h"(mask) : "memory");
}
}  // namespace ptx2

constexpr int PM = 128;            // rows of A and of the accumulator per CTA
constexpr int PN = 256;            // N of the pair's tile; each CTA stages PN / 2 positions of B
constexpr int PK = 64;             // k-block
constexpr int kPairStages = 5;
constexpr int kPairEpiWarps = 8;   // two per TMEM lane quarter: they split the 32-column groups of a tile
constexpr int kPairThreads = 64 + 32 * kPairEpiWarps;  // warp 0: TMA, warp 1: MMA (leader) + TMEM owner, then the epilogue warps
constexpr int kPairStage = PM * PK * 2 + (PN / 2) * PK * 2;  // 32 KB
constexpr int kPairSmem = kPairStages * kPairStage + 1024 + 256 + kPairEpiWarps * 4096;  // ring, alignment slack, barriers, transposition

// Where a wait has run out in either CTA of a pair, by all threads of both: the copies and products in flight complete
// (each wait with a limit) before the CTAs' memory goes away.  `issued` k-blocks of a CTA have been reported to the leader's
// full barriers, stage by stage, each phase of which takes one report of either CTA and the bytes of both.  A stage is
// refilled only behind the products that read it, so the two counts differ by the number of stages at most: the CTA that
// is behind reports the rest without bytes, and then the last phase of every stage completes when its copies have landed.
//   issued_s: a word in shared memory; full0: the first full barrier; drain: a barrier of one arrival that nothing else
//   uses; tail_bar (or 0): a barrier of this CTA with copies in flight, and the parity of its phase
// Not inlined: inside the kernels this code cost every launch 0.1 us.
__device__ __noinline__ void drain_pair(uint32_t rank, uint32_t issued_s, uint32_t full0, uint32_t drain,
                                        uint32_t tail_bar, uint32_t tail_parity) {
  if (threadIdx.x == 0) {
    const int mine = ptx::lds_s32(issued_s), peers = ptx2::ld_peer_s32(ptx2::map_to_cta(issued_s, rank ^ 1));
    const int all = mine > peers ? mine : peers;
    for (int it = mine; it < all; ++it) ptx2::mbar_arrive_cluster(ptx2::map_to_cta(full0 + 8u * (it % kPairStages), 0));
    if (tail_bar != 0) ptx::mbar_wait(tail_bar, tail_parity);
    if (rank == 0)
      for (int it = all > kPairStages ? all - kPairStages : 0; it < all; ++it)
        ptx::mbar_wait(full0 + 8u * (it % kPairStages), (it / kPairStages) & 1);
  }
  __syncwarp();
  if (threadIdx.x / 32 == 1) {  // the warp that issues the leader's products: they complete in both CTAs
    if (rank == 0 && ptx::elect_one()) ptx2::mma_commit_pair(drain);
    __syncwarp();
    ptx::mbar_wait(drain, 0);
  }
  __syncthreads();
  ptx2::cluster_sync();
}

// The end of a pair kernel: nobody leaves while the peer may still read this CTA's operands or signal its barriers; a
// failure of one CTA (its abort flag) becomes the peer's too.
__device__ __forceinline__ void leave_pair(uint32_t rank, uint32_t abort_s, uint32_t issued_s, uint32_t full0, uint32_t drain,
                                           uint32_t tail_bar = 0, uint32_t tail_parity = 0) {
  if ((threadIdx.x & 31) == 0 && ptx::lds_s32(abort_s) != 0) ptx2::st_peer_s32(ptx2::map_to_cta(abort_s, rank ^ 1), 1);
  ptx::tc_fence_before_sync();
  ptx2::cluster_sync();  // every thread of both CTAs
  if (__builtin_expect(ptx::lds_s32(abort_s) != 0, 0)) drain_pair(rank, issued_s, full0, drain, tail_bar, tail_parity);
}

// kBMn: B = W is MN-major (input gradient: K = n_out rows of W, N = n_in contiguous); otherwise K-major
// (forward: N = n_out rows of W, K = n_in contiguous).  A is always K-major, the output bf16.
// M is the device-side packed row count.  row_map and epi as in the single-CTA kernel.
template <bool kBMn, int kKind>
__global__ void __launch_bounds__(kPairThreads)
gemm_pair_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                 const __nv_bfloat16* bias, __nv_bfloat16* __restrict__ out, long long ldo, int N, int K,
                 const int32_t* cu, int n_seg, int capacity, const int32_t* row_map,
                 RowEpilogue<kKind> epi, uint32_t wait_limit, int32_t* d_status) {
  constexpr uint32_t kIdesc = ptx::idesc_bf16_f32(2 * PM, PN, false, kBMn);
  pdl_launch_dependents();

  extern __shared__ uint8_t smem_raw[];
  const uint32_t smem_base = (ptx::smem_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t* smem_al = smem_raw + (smem_base - ptx::smem_u32(smem_raw));
  const uint32_t bar_base = smem_base + kPairStages * kPairStage;
  auto full_bar = [&](int s) { return bar_base + 8u * s; };
  auto empty_bar = [&](int s) { return bar_base + 8u * (kPairStages + s); };
  auto tmem_full_bar = [&](int a) { return bar_base + 8u * (2 * kPairStages + a); };
  auto tmem_empty_bar = [&](int a) { return bar_base + 8u * (2 * kPairStages + 2 + a); };
  const uint32_t drain_bar = bar_base + 8u * (2 * kPairStages + 4);
  volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(smem_al + kPairStages * kPairStage + 192);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(smem_al + kPairStages * kPairStage + 196);
  const uint32_t abort_s = bar_base + 196, issued_s = bar_base + 200;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = ptx2::cluster_ctarank();   // 0 = leader
  const int pair = blockIdx.x >> 1, n_pairs = gridDim.x >> 1;
  if (threadIdx.x == 0) {
    ptx::prefetch_tensormap(&tmA);
    ptx::prefetch_tensormap(&tmB);
    for (int s = 0; s < kPairStages; ++s) {
      ptx::mbar_init(full_bar(s), 2);
      ptx::mbar_init(empty_bar(s), 1);
    }
    for (int a = 0; a < 2; ++a) { ptx::mbar_init(tmem_full_bar(a), 1); ptx::mbar_init(tmem_empty_bar(a), 2 * kPairEpiWarps); }
    ptx::mbar_init(drain_bar, 1);
    *abort_flag = 0;
    ptx::fence_mbar_init();
  }
  if (warp == 1) ptx2::tmem_alloc_pair(ptx::smem_u32(const_cast<uint32_t*>(tmem_slot)), 2 * PN);
  ptx::tc_fence_before_sync();
  __syncthreads();
  ptx2::cluster_sync();  // both CTAs' barriers exist before either signals the other
  ptx::tc_fence_after_sync();
  const uint32_t tmem_base = *tmem_slot;

  pdl_wait();  // everything above touched no global memory
  const int M = packed_rows(cu, n_seg, capacity);
  const int tiles_n = (N + PN - 1) / PN;
  const int tiles_m = (M + 2 * PM - 1) / (2 * PM);
  const int total = tiles_m * tiles_n;
  const int k_blocks = (K + PK - 1) / PK;
  auto wait_lane = [&](uint32_t bar, uint32_t parity) { return ptx::mbar_wait_or_abort(bar, parity, abort_s, d_status, SPA_ERR_TIMEOUT, wait_limit); };
  auto wait = [&](uint32_t bar, uint32_t parity) { return ptx::mbar_wait_or_abort_warp(bar, parity, abort_s, d_status, SPA_ERR_TIMEOUT, wait_limit); };

  if (warp == 0) {
    // ------------------------------------------------------------------ TMA producer (one per CTA)
    if (lane == 0) {
      int it = 0;
      bool live = true;
      for (int tile = pair; tile < total && live && !*abort_flag; tile += n_pairs) {
        const int m0 = (tile / tiles_n) * 2 * PM + (int)rank * PM;
        const int n0 = (tile % tiles_n) * PN + (int)rank * (PN / 2);
        for (int kb = 0; kb < k_blocks; ++kb, ++it) {
          const int s = it % kPairStages;
          if (it >= kPairStages && !wait_lane(empty_bar(s), ((it / kPairStages) - 1) & 1)) { live = false; break; }
          const uint32_t a_dst = smem_base + s * kPairStage, b_dst = a_dst + PM * PK * 2;
          const uint32_t lead_full = ptx2::map_to_cta(full_bar(s), 0);
          ptx2::mbar_expect_tx_cluster(lead_full, kPairStage);
          const int k0 = kb * PK;
          ptx2::tma_load_2d_pair(a_dst, &tmA, lead_full, k0, m0);
          if (!kBMn) {
            ptx2::tma_load_2d_pair(b_dst, &tmB, lead_full, k0, n0);
          } else {
#pragma unroll
            for (int j = 0; j < PN / 2 / 64; ++j)
              ptx2::tma_load_2d_pair(b_dst + j * (PK * 128), &tmB, lead_full, n0 + 64 * j, k0);
          }
        }
      }
      ptx::sts_s32(issued_s, it);
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer: the leader's, for the pair
    if (rank == 0) {
      int it = 0, tl = 0;
      bool live = true;  // every wait of this lane has been satisfied
      for (int tile = pair; tile < total && !__any_sync(0xffffffffu, *abort_flag != 0); tile += n_pairs, ++tl) {
        const int acc = tl & 1;
        if (tl >= 2) live = wait(tmem_empty_bar(acc), ((tl >> 1) - 1) & 1) && live;
        ptx::tc_fence_after_sync();
        const uint32_t tmem_d = tmem_base + acc * PN;
        for (int kb = 0; kb < k_blocks; ++kb, ++it) {
          const int s = it % kPairStages;
          live = wait(full_bar(s), (it / kPairStages) & 1) && live;
          ptx::tc_fence_after_sync();
          const uint32_t a_src = smem_base + s * kPairStage, b_src = a_src + PM * PK * 2;
          if (ptx::elect_one()) {
#pragma unroll
            for (int k = 0; k < PK / 16; ++k) {
              const uint64_t adesc = ptx::smem_desc_sw128(a_src + k * 32, 16, 1024);
              const uint64_t bdesc = kBMn ? ptx::smem_desc_sw128(b_src + k * 2048, PK * 128, 1024)
                                          : ptx::smem_desc_sw128(b_src + k * 32, 16, 1024);
              ptx2::mma_bf16_pair(tmem_d, adesc, bdesc, kIdesc, (kb == 0 && k == 0) ? 0u : 1u);
            }
            if (live) ptx2::mma_commit_pair(empty_bar(s));
            if (kb == k_blocks - 1) ptx2::mma_commit_pair(tmem_full_bar(acc));
          }
          __syncwarp();
        }
      }
    }
  } else {
    // ------------------------------------------------------------------ epilogue warps (both CTAs)
    const int q = warp & 3;  // TMEM lane quarter this warp may read
    const int half = (warp - 2) >> 2;  // which of the two warps of that quarter: even or odd 32-column groups
    uint8_t* stage = smem_al + kPairStages * kPairStage + 256 + (warp - 2) * 4096;  // this warp's transposition buffer
    const uint32_t lead_empty[2] = {ptx2::map_to_cta(tmem_empty_bar(0), 0), ptx2::map_to_cta(tmem_empty_bar(1), 0)};
    const int my_chunk = lane & 7, my_row = lane >> 3;
    int tl = 0;
    for (int tile = pair; tile < total; tile += n_pairs, ++tl) {
      const int m0 = (tile / tiles_n) * 2 * PM + (int)rank * PM;
      const int n0 = (tile % tiles_n) * PN;
      const int acc = tl & 1;
      long long orow[8];  // destination rows of the eight rows this lane stores
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const int grow = m0 + q * 32 + my_row + 4 * j;
        orow[j] = (row_map != nullptr && grow < M) ? (long long)ld_dep(row_map + grow) : (long long)grow;
      }
      // the bias of the tile comes to L1 under the main loop: fetched where it is added, each 64 columns waited for L2
      if (bias != nullptr && lane < PN / 64 && n0 + lane * 64 < N) prefetch_l1(bias + n0 + lane * 64);
      wait(tmem_full_bar(acc), (tl >> 1) & 1);
      if (__any_sync(0xffffffffu, *abort_flag != 0)) break;
      ptx::tc_fence_after_sync();
      // Thread `lane` receives one accumulator row; 64 columns (128 bytes of the output) at a time are turned around in
      // the warp's 4 KB, so that a store instruction covers four whole 128-byte lines.
#pragma unroll 1
      for (int cc = half; cc < PN / 64; cc += 2) {
        if (n0 + cc * 64 >= N) break;  // warp-uniform: columns past the layer's width
        const int gcol = n0 + cc * 64 + my_chunk * 8;
        uint4 old[8];  // what the results are combined with, under the reads of the accumulator
#pragma unroll
        for (int j = 0; j < 8; ++j)
          if (m0 + q * 32 + my_row + 4 * j < M && gcol < N) epi.fetch(out, old[j], orow[j] * ldo + gcol);
        uint32_t r[64];
        const uint32_t at = tmem_base + ((uint32_t)(q * 32) << 16) + acc * PN + cc * 64;
        ptx::tmem_ld_32x32(at, r);
        ptx::tmem_ld_32x32(at + 32, r + 32);
        ptx::tmem_ld_wait();
#pragma unroll
        for (int i = 0; i < 8; ++i) {  // 16-byte chunk i of this row's 128-byte segment
          float v[8];
#pragma unroll
          for (int e = 0; e < 8; ++e) v[e] = __uint_as_float(r[i * 8 + e]);
          const int col = n0 + cc * 64 + i * 8;
          if (bias != nullptr && col < N) {
            float b[8];
            Vec16<__nv_bfloat16>::to_float(__ldg(reinterpret_cast<const uint4*>(bias + col)), b);
#pragma unroll
            for (int e = 0; e < 8; ++e) v[e] += b[e];
          }
          *reinterpret_cast<uint4*>(stage + lane * 128 + ((i ^ (lane & 7)) << 4)) = Vec16<__nv_bfloat16>::from_float(v);
        }
        __syncwarp();
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const int rr = my_row + 4 * j;
          const uint4 v4 = *reinterpret_cast<const uint4*>(stage + rr * 128 + ((my_chunk ^ (rr & 7)) << 4));
          if (m0 + q * 32 + rr < M && gcol < N) epi.finish(out, orow[j] * ldo + gcol, v4, old[j]);
        }
        __syncwarp();
      }
      ptx::tc_fence_before_sync();
      __syncwarp();
      if (lane == 0) ptx2::mbar_arrive_cluster(lead_empty[acc]);  // this warp has drained its quarter of the accumulator
    }
  }
  leave_pair(rank, abort_s, issued_s, full_bar(0), drain_bar);
  if (warp == 1) {
    ptx::tc_fence_after_sync();
    ptx2::tmem_dealloc_pair(tmem_base, 2 * PN);
  }
}

// ------------------------------------------------------------------------------------------------ weight gradient
// dW[n_out][n_in] = dout^T a on CTA pairs: both operands MN-major, K = the device-side packed row count, split over the
// pairs that are resident at once.  The splits are dealt the 64-row blocks of K in turn (split z takes blocks z, z + S,
// ...) and each leaves its fp32 tile in the workspace for the fixed-order reduction.  A pair reads 32 KB per CTA and
// k-block for 256 x 256 x 64 products, half of what two 128 x 128 tiles on an SM need, which were bound by it.
//   Rows past the last packed one: the last k-block of K is loaded on a barrier of each CTA's own, its producer warp
//   zeroes the lines, and only then reports the stage to the leader.
//   Bias gradient: db[m] = sum_k dout[k][m] is the product with a matrix of ones, 16 columns wide, into TMEM columns
//   behind the tile's; the tiles of a row of tiles take the k-blocks of it in turn (every sum of bf16 values is exact
//   up to the fp32 additions, as before).  A column-sum kernel over dout cost 9-11 us where this adds under 1.
// One accumulator: all tiles x splits are resident at once (up to layers of 4.8 M weights), so there is no next tile
// whose main loop an epilogue could run under.
constexpr int kWgSmem = kPairSmem + 1024;  // and the 8 x 64 block of ones

__global__ void __launch_bounds__(kPairThreads)
wgrad_pair_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, float* __restrict__ part,
                  float* __restrict__ part_b, int M, int N, int splits, const int32_t* cu, int n_seg,
                  int capacity, uint32_t wait_limit, int32_t* d_status) {
  constexpr uint32_t kIdesc = ptx::idesc_bf16_f32(2 * PM, PN, true, true);
  constexpr uint32_t kIdescOnes = ptx::idesc_bf16_f32(2 * PM, 16, true, false);
  constexpr int kBars = kPairStages * kPairStage;
  pdl_launch_dependents();

  extern __shared__ uint8_t smem_raw[];
  const uint32_t smem_base = (ptx::smem_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t* smem_al = smem_raw + (smem_base - ptx::smem_u32(smem_raw));
  const uint32_t ones_s = smem_base + kBars, bar_base = ones_s + 1024;
  auto full_bar = [&](int s) { return bar_base + 8u * s; };
  auto empty_bar = [&](int s) { return bar_base + 8u * (kPairStages + s); };
  const uint32_t tmem_full_bar = bar_base + 8u * (2 * kPairStages), tmem_empty_bar = tmem_full_bar + 8, tail_bar = tmem_full_bar + 16;
  const uint32_t drain_bar = tmem_full_bar + 24;
  volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(smem_al + kBars + 1024 + 192);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(smem_al + kBars + 1024 + 196);
  const uint32_t abort_s = bar_base + 196, issued_s = bar_base + 200;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = ptx2::cluster_ctarank();  // 0 = leader
  const int pair = blockIdx.x >> 1, n_pairs = gridDim.x >> 1;
  if (threadIdx.x == 0) {
    ptx::prefetch_tensormap(&tmA);
    ptx::prefetch_tensormap(&tmB);
    for (int s = 0; s < kPairStages; ++s) {
      ptx::mbar_init(full_bar(s), 2);
      ptx::mbar_init(empty_bar(s), 1);
    }
    ptx::mbar_init(tmem_full_bar, 1);
    ptx::mbar_init(tmem_empty_bar, 2 * kPairEpiWarps);
    ptx::mbar_init(tail_bar, 1);
    ptx::mbar_init(drain_bar, 1);
    *abort_flag = 0;
    ptx::fence_mbar_init();
  }
  if (warp == 2) {  // 8 rows of 64 ones: the same under any swizzle
    for (int i = lane; i < 64; i += 32)
      *reinterpret_cast<uint4*>(smem_al + kBars + i * 16) = make_uint4(0x3f803f80u, 0x3f803f80u, 0x3f803f80u, 0x3f803f80u);
    ptx::fence_proxy_async_smem();
  }
  if (warp == 1) ptx2::tmem_alloc_pair(ptx::smem_u32(const_cast<uint32_t*>(tmem_slot)), 2 * PN);
  ptx::tc_fence_before_sync();
  __syncthreads();
  ptx2::cluster_sync();  // both CTAs' barriers exist before either signals the other
  ptx::tc_fence_after_sync();
  const uint32_t tmem = *tmem_slot;

  pdl_wait();  // everything above touched no global memory
  const int K = packed_rows(cu, n_seg, capacity);
  const int tiles_n = (N + PN - 1) / PN, tiles_m = (M + 2 * PM - 1) / (2 * PM);
  const int k_blocks = (K + PK - 1) / PK;
  const int n_splits = k_blocks < splits ? k_blocks : splits;
  const int total = tiles_m * tiles_n * n_splits;
  struct Item { int m0, n0, n_t, z; };  // first row and column of the pair's tile, its column of tiles, its split
  auto item_of = [&](int i) {
    Item c;
    c.n_t = i % tiles_n;
    const int rest = i / tiles_n;
    c.m0 = (rest % tiles_m) * 2 * PM;
    c.z = rest / tiles_m;
    c.n0 = c.n_t * PN;
    return c;
  };
  auto wait_lane = [&](uint32_t bar, uint32_t parity) { return ptx::mbar_wait_or_abort(bar, parity, abort_s, d_status, SPA_ERR_TIMEOUT, wait_limit); };
  auto wait = [&](uint32_t bar, uint32_t parity) { return ptx::mbar_wait_or_abort_warp(bar, parity, abort_s, d_status, SPA_ERR_TIMEOUT, wait_limit); };

  bool tail_open = false;  // copies on tail_bar that were given up on
  uint32_t tail_parity = 0;
  if (warp == 0) {
    // ------------------------------------------------------------------ TMA producer (one per CTA)
    int it = 0, tails = 0;
    bool live = true;  // lane 0: every wait has been satisfied; all lanes: so has every wait for a tail
    for (int i = pair; i < total && !__any_sync(0xffffffffu, !live || *abort_flag != 0); i += n_pairs) {
      const Item c = item_of(i);
      const int m0 = c.m0 + (int)rank * PM, n0 = c.n0 + (int)rank * (PN / 2);
      for (int kb = c.z; kb < k_blocks; kb += n_splits, ++it) {
        const int s = it % kPairStages, k0 = kb * PK;
        const uint32_t a_dst = smem_base + s * kPairStage, b_dst = a_dst + PM * PK * 2;
        const uint32_t lead_full = ptx2::map_to_cta(full_bar(s), 0);
        const bool tail = k0 + PK > K;
        if (lane == 0) {
          live = (it < kPairStages || wait_lane(empty_bar(s), ((it / kPairStages) - 1) & 1)) && live;
          if (!live) {
          } else if (!tail) {
            ptx2::mbar_expect_tx_cluster(lead_full, kPairStage);
#pragma unroll
            for (int j = 0; j < 2; ++j) ptx2::tma_load_2d_pair(a_dst + j * (PK * 128), &tmA, lead_full, m0 + 64 * j, k0);
#pragma unroll
            for (int j = 0; j < 2; ++j) ptx2::tma_load_2d_pair(b_dst + j * (PK * 128), &tmB, lead_full, n0 + 64 * j, k0);
          } else {
            ptx::mbar_expect_tx(tail_bar, kPairStage);
#pragma unroll
            for (int j = 0; j < 2; ++j) ptx::tma_load_2d(a_dst + j * (PK * 128), &tmA, tail_bar, m0 + 64 * j, k0);
#pragma unroll
            for (int j = 0; j < 2; ++j) ptx::tma_load_2d(b_dst + j * (PK * 128), &tmB, tail_bar, n0 + 64 * j, k0);
          }
        }
        if (!__shfl_sync(0xffffffffu, live, 0)) { live = false; break; }
        if (tail) {
          live = __all_sync(0xffffffffu, wait(tail_bar, tails & 1)) != 0;
          if (!live) { tail_open = true; break; }
          ++tails;
          const int first = K - k0;  // lines of the four boxes from here on hold no packed row
          for (int q = lane; q < 4 * (PK - first) * 8; q += 32) {
            const int box = q / ((PK - first) * 8), r = q % ((PK - first) * 8);
            *reinterpret_cast<uint4*>(smem_al + s * kPairStage + box * (PK * 128) + (first + r / 8) * 128 + (r % 8) * 16) = make_uint4(0, 0, 0, 0);
          }
          ptx::fence_proxy_async_smem();
          __syncwarp();
          if (lane == 0) ptx2::mbar_arrive_release_cluster(lead_full);
        }
      }
    }
    if (lane == 0) ptx::sts_s32(issued_s, it);
    tail_parity = tails & 1;
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer: the leader's, for the pair
    if (rank == 0) {
      const uint64_t ones_desc = ptx::smem_desc_sw128(ones_s, 16, 1024);
      int it = 0, tl = 0;
      bool live = true;  // every wait of this lane has been satisfied
      for (int i = pair; i < total && !__any_sync(0xffffffffu, *abort_flag != 0); i += n_pairs, ++tl) {
        const Item c = item_of(i);
        if (tl > 0) live = wait(tmem_empty_bar, (tl - 1) & 1) && live;
        ptx::tc_fence_after_sync();
        bool first = true, first_sum = true;
        for (int kb = c.z; kb < k_blocks; kb += n_splits, ++it) {
          const int s = it % kPairStages;
          live = wait(full_bar(s), (it / kPairStages) & 1) && live;
          ptx::tc_fence_after_sync();
          const uint32_t a_src = smem_base + s * kPairStage, b_src = a_src + PM * PK * 2;
          const bool sum = part_b != nullptr && (kb / n_splits) % tiles_n == c.n_t;
          if (ptx::elect_one()) {
#pragma unroll
            for (int k = 0; k < PK / 16; ++k)
              ptx2::mma_bf16_pair(tmem, ptx::smem_desc_sw128(a_src + k * 2048, PK * 128, 1024),
                                  ptx::smem_desc_sw128(b_src + k * 2048, PK * 128, 1024), kIdesc, (first && k == 0) ? 0u : 1u);
            if (sum) {
#pragma unroll
              for (int k = 0; k < PK / 16; ++k)
                ptx2::mma_bf16_pair(tmem + PN, ptx::smem_desc_sw128(a_src + k * 2048, PK * 128, 1024), ones_desc, kIdescOnes,
                                    (first_sum && k == 0) ? 0u : 1u);
            }
            if (live) ptx2::mma_commit_pair(empty_bar(s));
            if (kb + n_splits >= k_blocks) ptx2::mma_commit_pair(tmem_full_bar);
          }
          first = false;
          first_sum = first_sum && !sum;
          __syncwarp();
        }
      }
    }
  } else {
    // ------------------------------------------------------------------ epilogue warps (both CTAs)
    const int q = warp & 3;            // TMEM lane quarter this warp may read
    const int half = (warp - 2) >> 2;  // which of the two warps of that quarter: even or odd 32-column groups
    uint8_t* stage = smem_al + kBars + 1024 + 256 + (warp - 2) * 4096;  // this warp's transposition buffer
    const uint32_t lead_empty = ptx2::map_to_cta(tmem_empty_bar, 0);
    const int my_chunk = lane & 7, my_row = lane >> 3;
    int tl = 0;
    for (int i = pair; i < total; i += n_pairs, ++tl) {
      const Item c = item_of(i);
      const int m0 = c.m0 + (int)rank * PM + q * 32;
      float* obase = part + (long long)c.z * M * N;
      wait(tmem_full_bar, tl & 1);
      if (__any_sync(0xffffffffu, *abort_flag != 0)) break;
      ptx::tc_fence_after_sync();
      const uint32_t lanes = tmem + ((uint32_t)(q * 32) << 16);
      // Thread `lane` receives one accumulator row; 32 columns (128 bytes) at a time are turned around in the warp's
      // 4 KB, so that a store instruction covers four whole 128-byte lines.
#pragma unroll 1
      for (int cc = half; cc < PN / 32; cc += 2) {
        if (c.n0 + cc * 32 >= N) break;  // warp-uniform: columns past the layer's width
        uint32_t r[32];
        ptx::tmem_ld_32x32(lanes + cc * 32, r);
        ptx::tmem_ld_wait();
#pragma unroll
        for (int e = 0; e < 8; ++e)
          *reinterpret_cast<uint4*>(stage + lane * 128 + ((e ^ (lane & 7)) << 4)) = make_uint4(r[4 * e], r[4 * e + 1], r[4 * e + 2], r[4 * e + 3]);
        __syncwarp();
        const int gcol = c.n0 + cc * 32 + my_chunk * 4;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const int rr = my_row + 4 * j;
          const uint4 v = *reinterpret_cast<const uint4*>(stage + rr * 128 + ((my_chunk ^ (rr & 7)) << 4));
          if (m0 + rr < M && gcol < N) *reinterpret_cast<uint4*>(obase + (long long)(m0 + rr) * N + gcol) = v;
        }
        __syncwarp();
      }
      if (part_b != nullptr && half == 0) {
        uint32_t r[16];
        ptx::tmem_ld_32x16(lanes + PN, r);
        ptx::tmem_ld_wait();
        // k-blocks of this split: z, z + S, ...; the tile has taken those whose turn falls on its column of tiles
        const int mine = (k_blocks - c.z + n_splits - 1) / n_splits;
        if (m0 + lane < M) part_b[((long long)c.z * tiles_n + c.n_t) * M + m0 + lane] = mine > c.n_t ? __uint_as_float(r[0]) : 0.f;
      }
      ptx::tc_fence_before_sync();
      __syncwarp();
      if (lane == 0) ptx2::mbar_arrive_cluster(lead_empty);  // this warp has drained its quarter of the accumulator
    }
  }
  leave_pair(rank, abort_s, issued_s, full_bar(0), drain_bar, tail_open ? tail_bar : 0u, tail_parity);
  if (warp == 1) {
    ptx::tc_fence_after_sync();
    ptx2::tmem_dealloc_pair(tmem, 2 * PN);
  }
}

constexpr int kMaxPairs = kNumSMs / 2;

// `pairs` clusters of two CTAs
template <typename... KArgs, typename... Args>
int launch_clusters(void (*kern)(KArgs...), int pairs, int smem, cudaStream_t st, const char* what, Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(2 * pairs);
  cfg.blockDim = dim3(kPairThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl_enabled() ? 2 : 1;
  cudaError_t e = cudaLaunchKernelEx(&cfg, kern, static_cast<KArgs>(args)...);
  if (e != cudaSuccess) { set_cuda_error(e, what); return SPA_ERR_CUDA; }
  SPA_CUDA_CHECK_LAUNCH(what);
  return SPA_OK;
}

template <bool kBMn, int kKind>
int launch_pair(const CUtensorMap& tmA, const CUtensorMap& tmB, const __nv_bfloat16* bias, __nv_bfloat16* out, long long ldo,
                int N, int K, const int32_t* cu, int n_seg, int capacity, const int32_t* row_map, RowEpilogue<kKind> epi,
                uint32_t wait_limit, int32_t* d_status, cudaStream_t st, const char* what) {
  auto kern = gemm_pair_kernel<kBMn, kKind>;
  static DeviceOnce smem_attr;  // per instantiation and device
  cudaError_t ea = smem_attr.run([&] { return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kPairSmem); });
  if (ea != cudaSuccess) { set_cuda_error(ea, what); return SPA_ERR_CUDA; }
  const long long tiles = (long long)((N + PN - 1) / PN) * ((capacity + 2 * PM - 1) / (2 * PM));
  const int pairs = (int)(tiles < kMaxPairs ? (tiles < 1 ? 1 : tiles) : kMaxPairs);
  return launch_clusters(kern, pairs, kPairSmem, st, what, tmA, tmB, bias, out, ldo, N, K, cu, n_seg, capacity, row_map, epi, wait_limit, d_status);
}

}  // namespace

PairWgradPlan pair_wgrad_plan(int capacity, int n_in, int n_out) {
  PairWgradPlan pl;
  pl.tiles_n = (n_in + PN - 1) / PN;
  pl.tiles = pl.tiles_n * ((n_out + 2 * PM - 1) / (2 * PM));
  // as many splits as keep all tiles x splits resident; at least four k-blocks each when half of the capacity is in
  // use (a split costs a tile of partial sums written and read); 31 leave room for the bias partials in a workspace of
  // 32 splits
  int s = kMaxPairs / pl.tiles;
  const int by_rows = (capacity / 2 + 4 * PK - 1) / (4 * PK);
  if (s > by_rows) s = by_rows;
  if (s > 31) s = 31;
  pl.splits = s < 1 ? 1 : s;
  return pl;
}

int launch_wgrad_pair(const spa_params& p, const void* a, const void* dout, int n_in, int n_out, const int32_t* cu, float* part,
                      float* part_b, const PairWgradPlan& pl, int32_t* d_status, cudaStream_t st) {
  CUtensorMap tmA, tmB;
  if (!make_tmap_bf16_2d(&tmA, dout, n_out, p.capacity, (uint64_t)n_out * 2, 64, PK) ||
      !make_tmap_bf16_2d(&tmB, a, n_in, p.capacity, (uint64_t)n_in * 2, 64, PK))
    return SPA_ERR_UNSUPPORTED;
  static DeviceOnce smem_attr;
  cudaError_t ea = smem_attr.run([&] { return cudaFuncSetAttribute(wgrad_pair_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kWgSmem); });
  if (ea != cudaSuccess) { set_cuda_error(ea, "wgrad_pair_kernel"); return SPA_ERR_CUDA; }
  const int tiles = pl.tiles * pl.splits;
  return launch_clusters(wgrad_pair_kernel, tiles < kMaxPairs ? tiles : kMaxPairs, kWgSmem, st, "wgrad_pair_kernel", tmA, tmB, part,
                         part_b, n_out, n_in, pl.splits, cu, p.B, p.capacity, ptx::wait_limit(p.flags), d_status);
}

// The pair kernels pay off where every pair gets a 256 x 256 tile (half of the allocated rows stands for the packed
// ones): 15 120 rows 256 -> 768 13.7 us against 15.0 on single CTAs, 6 272 rows 384 -> 1 152 11.2 against 12.2; with
// fewer tiles the smaller ones spread better (6 272 rows 384 -> 384: 7.9 against 6.5).  Not where K is short and
// an eighth of the pair's columns or more would be padding that 128-column tiles do not have (34 000 rows allocated, 30 % of
// them there: 384 -> 384 10.6 against 8.2, 288 -> 864 14.0 against 12.0; at half and above even).  With a longer main loop the
// pairs win all the same (576 -> 576 13.1 against 15.1, 512 -> 640 10.7 against 12.3; no padded width lies between 384 and 512
// in what was measured).
bool tc_pair_linear_supported(const spa_params& p, int n_in, int n_out, int n_cols) {
  if (p.flags & SPA_FLAG_NO_CTA_PAIRS) return false;
  const long long tiles = (long long)((p.capacity / 2 + 2 * PM - 1) / (2 * PM)) * ((n_cols + PN - 1) / PN);
  const int blocks = (n_cols + 127) / 128;
  const int k = n_cols == n_out ? n_in : n_out;
  const bool padded = blocks % 2 == 1 && blocks <= 7 && k <= 384;
  return n_in % 8 == 0 && n_out % 8 == 0 && tiles >= kMaxPairs && !padded && tensor_maps_available();
}

int launch_linear_fwd_pair(const spa_params& p, const void* a, const void* W, const void* bias, int n_in, int n_out,
                           const int32_t* cu, void* out, int32_t* d_status, cudaStream_t st, const int32_t* row_map,
                           const LinearEpilogue& epi) {
  CUtensorMap tmA, tmB;
  if (!make_tmap_bf16_2d(&tmA, a, n_in, p.capacity, (uint64_t)n_in * 2, PK, PM) ||
      !make_tmap_bf16_2d(&tmB, W, n_in, n_out, (uint64_t)n_in * 2, PK, PN / 2))
    return SPA_ERR_UNSUPPORTED;
  auto go = [&](auto row_epi) {
    return launch_pair<false>(tmA, tmB, (const __nv_bfloat16*)bias, (__nv_bfloat16*)out, n_out, n_out, n_in, cu, p.B, p.capacity,
                              row_map, row_epi, ptx::wait_limit(p.flags), d_status, st, "gemm_pair_kernel(fwd)");
  };
  if (epi.h != nullptr) return go(RowEpilogue<kEpiGelu>{(__nv_bfloat16*)epi.h});
  if (epi.add != nullptr && epi.add != out) return go(RowEpilogue<kEpiAdd>{(__nv_bfloat16*)const_cast<void*>(epi.add)});
  return go(RowEpilogue<kEpiOwn>{epi.add != nullptr ? (__nv_bfloat16*)out : nullptr});
}

// da[M][n_in] = dout[M][n_out] W[n_out][n_in]
int launch_linear_dgrad_pair(const spa_params& p, const void* W, const void* dout, int n_in, int n_out, const int32_t* cu,
                             void* da, int32_t* d_status, cudaStream_t st, const int32_t* row_map,
                             const LinearEpilogue& epi) {
  CUtensorMap tmA, tmB;
  if (!make_tmap_bf16_2d(&tmA, dout, n_out, p.capacity, (uint64_t)n_out * 2, PK, PM) ||
      !make_tmap_bf16_2d(&tmB, W, n_in, n_out, (uint64_t)n_in * 2, 64, PK))
    return SPA_ERR_UNSUPPORTED;
  auto go = [&](auto row_epi) {
    return launch_pair<true>(tmA, tmB, nullptr, (__nv_bfloat16*)da, n_in, n_in, n_out, cu, p.B, p.capacity, row_map, row_epi,
                             ptx::wait_limit(p.flags), d_status, st, "gemm_pair_kernel(dgrad)");
  };
  return epi.u != nullptr ? go(RowEpilogue<kEpiGeluGrad>{(__nv_bfloat16*)const_cast<void*>(epi.u)})
                          : go(RowEpilogue<kEpiOwn>{epi.add != nullptr ? (__nv_bfloat16*)da : nullptr});
}

}  // namespace spa
