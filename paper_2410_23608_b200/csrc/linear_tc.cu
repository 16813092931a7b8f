// bf16 linear layers on the packed tokens as tcgen05 GEMMs: QKV / output projection (the 3LC^2 and
// NC^2 terms of Eq. 9), their input gradients and their weight gradients.
//
// One kernel, three operand arrangements.  D[128 x BN] tiles accumulate in TMEM (fp32); operands
// are staged by TMA into 128-byte-swizzled shared memory through a ring of kStages buffers; one
// thread issues tcgen05.mma, one thread issues TMA, four warps drain TMEM and store.
//   forward   out = a W^T      A = a    (K-major),  B = W   (K-major),  M = packed rows (device)
//   dgrad     da  = dout W     A = dout (K-major),  B = W   (MN-major), M = packed rows (device)
//   wgrad     dW  = dout^T a   A = dout (MN-major), B = a   (MN-major), K = packed rows (device)
// The packed row count N_p lives on the device: grids are sized for `capacity` rows and CTAs
// beyond N_p exit at once.  wgrad splits K = N_p across CTAs; each split writes an fp32 partial to
// the workspace and a second kernel adds the partials in a fixed order (no float atomics, bitwise
// reproducible).  Rows of the last K block that lie beyond N_p are zeroed in shared memory before
// the MMA reads them, so unspecified rows of the packed buffers never reach a sum.
#include <mutex>
#include <string>
#include <unordered_map>

#include "sm100_ptx.cuh"
#include "spa_tc.cuh"

namespace spa {

// ------------------------------------------------------------------------------ tensor maps
namespace {
using EncodeFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                              const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                              CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeFn encode_fn() {
  static EncodeFn fn = []() -> EncodeFn {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess)
      return nullptr;
    return reinterpret_cast<EncodeFn>(p);
  }();
  return fn;
}

std::mutex g_tm_mutex;
std::unordered_map<std::string, CUtensorMap> g_tm_cache;
}  // namespace

bool tensor_maps_available() { return encode_fn() != nullptr; }

bool make_tmap_bf16_2d(CUtensorMap* out, const void* base, uint64_t inner, uint64_t rows, uint64_t row_stride_bytes,
                       uint32_t box_inner, uint32_t box_rows, int swizzle_bytes) {
  struct Key { const void* b; uint64_t i, r, s; uint32_t bi, br; int sw; int pad; } key{base, inner, rows, row_stride_bytes,
                                                                                     box_inner, box_rows, swizzle_bytes, 0};
  std::string k(reinterpret_cast<const char*>(&key), sizeof(key));
  std::lock_guard<std::mutex> lock(g_tm_mutex);
  auto it = g_tm_cache.find(k);
  if (it != g_tm_cache.end()) { *out = it->second; return true; }
  EncodeFn fn = encode_fn();
  if (fn == nullptr) return false;
  cuuint64_t dims[2] = {inner, rows};
  cuuint64_t strides[1] = {row_stride_bytes};
  cuuint32_t box[2] = {box_inner, box_rows};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = fn(out, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr,
                  CU_TENSOR_MAP_INTERLEAVE_NONE,
                  swizzle_bytes == 64 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_128B,
                  CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return false;
  if (g_tm_cache.size() > 4096) g_tm_cache.clear();
  g_tm_cache.emplace(std::move(k), *out);
  return true;
}

namespace {

constexpr int BM = 128;
constexpr int BK = 64;
constexpr int kStages = 3;
constexpr int kGemmThreads = 192;  // warp 0: TMA, warp 1: MMA + TMEM owner, warps 2-5: epilogue
constexpr int kABytes = BM * BK * 2;

template <int BN> __host__ __device__ constexpr int stage_bytes() { return kABytes + BN * BK * 2; }
// operand ring, alignment slack, barriers, 2 KB per epilogue warp for the output transposition
template <int BN> __host__ __device__ constexpr int gemm_smem_bytes() { return kStages * stage_bytes<BN>() + 1024 + 128 + 4 * 2048; }

// Tile bookkeeping shared by the three roles of the persistent kernel.
struct TileCoord { int m0, n0, z, n_t; };

// dyn_which: 1 = M is the device-side packed row count, 2 = K is.
// Persistent: each CTA walks tiles blockIdx.x, blockIdx.x + gridDim.x, ... of the (m, n, split) space
// that the device-side row count leaves; two accumulator stages in TMEM let the epilogue of one tile
// overlap the main loop of the next, and the TMA ring runs ahead across tile boundaries.
// row_map (optional): output row i goes to row row_map[i] of `out` (the unpack scatter fused into the
// epilogue).  epi: what a bf16 result goes through on its way out (RowEpilogue; split-K partials go as they are).
template <int BN, bool kDyn, bool kAMn, bool kBMn, typename OutT, int kKind>
__global__ void __launch_bounds__(kGemmThreads)
gemm_tc_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
               const __nv_bfloat16* bias, OutT* __restrict__ out, long long ldo,
               long long split_stride, int M, int N, int K, const int32_t* cu, int n_seg, int capacity,
               int dyn_which, int k_per_split, int k_interleave, const int32_t* row_map,
               RowEpilogue<kKind> epi, uint32_t wait_limit, int32_t* d_status) {
  constexpr int kStage = stage_bytes<BN>();
  pdl_launch_dependents();

  extern __shared__ uint8_t smem_raw[];
  const uint32_t smem_base = (ptx::smem_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t* smem_al = smem_raw + (smem_base - ptx::smem_u32(smem_raw));
  const uint32_t bar_base = smem_base + kStages * kStage;
  auto full_bar = [&](int s) { return bar_base + 8u * s; };
  auto empty_bar = [&](int s) { return bar_base + 8u * (kStages + s); };
  auto tmem_full_bar = [&](int a) { return bar_base + 8u * (2 * kStages + a); };
  auto tmem_empty_bar = [&](int a) { return bar_base + 8u * (2 * kStages + 2 + a); };
  const uint32_t drain_bar = bar_base + 8u * (2 * kStages + 4);
  volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(smem_al + kStages * kStage + 96);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(smem_al + kStages * kStage + 100);
  const uint32_t abort_s = bar_base + 100;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    ptx::prefetch_tensormap(&tmA);
    ptx::prefetch_tensormap(&tmB);
    for (int s = 0; s < kStages; ++s) {
      ptx::mbar_init(full_bar(s), 1);
      ptx::mbar_init(empty_bar(s), 1);
    }
    for (int a = 0; a < 2; ++a) { ptx::mbar_init(tmem_full_bar(a), 1); ptx::mbar_init(tmem_empty_bar(a), 4); }
    ptx::mbar_init(drain_bar, 1);
    *abort_flag = 0;
    ptx::fence_mbar_init();
  }
  if (warp == 1) ptx::tmem_alloc(ptx::smem_u32(const_cast<uint32_t*>(tmem_slot)), 2 * BN);
  ptx::tc_fence_before_sync();
  __syncthreads();
  ptx::tc_fence_after_sync();
  const uint32_t tmem_base = *tmem_slot;

  pdl_wait();  // everything above touched no global memory; the predecessor's results are needed from here on
  {
    const int rows = packed_rows(cu, n_seg, capacity);
    if (dyn_which == 1) M = rows; else if (dyn_which == 2) K = rows;
  }
  const int tiles_m = (M + BM - 1) / BM;
  const int bn = kDyn && (long long)tiles_m * ((N + BN - 1) / BN) <= kNumSMs ? BN / 2 : BN;  // see tile_width
  const int tiles_n = (N + bn - 1) / bn;
  const uint32_t idesc = bn == BN ? ptx::idesc_bf16_f32(BM, BN, kAMn, kBMn) : ptx::idesc_bf16_f32(BM, 64, kAMn, kBMn);
  // Split-K: contiguous spans of k_per_split, or (k_interleave > 0) that many splits dealt the BK-blocks of K in
  // turn - split z takes blocks z, z + splits, ... - so that the splits get equal work whatever K turns out to be.
  const int k_blocks = (K + BK - 1) / BK;
  const int n_splits = k_interleave > 0 ? (k_blocks < k_interleave ? k_blocks : k_interleave)
                                        : (K > 0 ? (K + k_per_split - 1) / k_per_split : 0);
  const int total = tiles_m * tiles_n * n_splits;
  auto coord = [&](int tile) {
    TileCoord c;
    c.n_t = tile % tiles_n;
    const int rest = tile / tiles_n;
    c.m0 = (rest % tiles_m) * BM;
    c.z = rest / tiles_m;
    c.n0 = c.n_t * bn;
    return c;
  };
  auto k_range = [&](int z, int& k_begin, int& k_end, int& k_step) {
    if (k_interleave > 0) {
      k_begin = z * BK;
      k_end = K;
      k_step = n_splits * BK;
    } else {
      k_begin = z * k_per_split;
      k_end = k_begin + k_per_split;
      if (k_end > K) k_end = K;
      k_step = BK;
    }
  };

  auto wait_lane = [&](uint32_t bar, uint32_t parity) { return ptx::mbar_wait_or_abort(bar, parity, abort_s, d_status, SPA_ERR_TIMEOUT, wait_limit); };
  auto wait = [&](uint32_t bar, uint32_t parity) { return ptx::mbar_wait_or_abort_warp(bar, parity, abort_s, d_status, SPA_ERR_TIMEOUT, wait_limit); };

  int issued = 0;       // the producer's: k-blocks whose copies have been issued
  bool failed = false;  // a wait of this thread gave up, or it saw that another one's had
  if (warp == 0) {
    // ------------------------------------------------------------------ TMA producer
    if (lane == 0) {
      int it = 0;  // k-block counter over all tiles of this CTA: ring position and phase
      bool live = true;
      for (int tile = blockIdx.x; tile < total && live && !*abort_flag; tile += gridDim.x) {
        const TileCoord c = coord(tile);
        int k_begin, k_end, k_step;
        k_range(c.z, k_begin, k_end, k_step);
        for (int k0 = k_begin; k0 < k_end; k0 += k_step, ++it) {
          const int s = it % kStages;
          if (it >= kStages && !wait_lane(empty_bar(s), ((it / kStages) - 1) & 1)) { live = false; break; }
          const uint32_t a_dst = smem_base + s * kStage, b_dst = a_dst + kABytes;
          ptx::mbar_expect_tx(full_bar(s), kABytes + bn * BK * 2);
          if (!kAMn) {
            ptx::tma_load_2d(a_dst, &tmA, full_bar(s), k0, c.m0);
          } else {
#pragma unroll
            for (int j = 0; j < BM / 64; ++j)
              ptx::tma_load_2d(a_dst + j * (BK * 128), &tmA, full_bar(s), c.m0 + 64 * j, k0);
          }
          if (!kBMn) {
            constexpr int kBox = kDyn ? 64 : BN;  // rows of W per copy
#pragma unroll
            for (int j = 0; j < BN / kBox; ++j)
              if (j * kBox < bn) ptx::tma_load_2d(b_dst + j * (kBox * 128), &tmB, full_bar(s), k0, c.n0 + kBox * j);
          } else {
#pragma unroll
            for (int j = 0; j < BN / 64; ++j)
              if (j * 64 < bn) ptx::tma_load_2d(b_dst + j * (BK * 128), &tmB, full_bar(s), c.n0 + 64 * j, k0);
          }
        }
      }
      issued = it;
      failed = !live;
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer
    int it = 0, tl = 0;  // k-block counter, tile counter of this CTA
    bool live = true;    // every wait of this lane has been satisfied
    for (int tile = blockIdx.x; tile < total && !__any_sync(0xffffffffu, *abort_flag != 0); tile += gridDim.x, ++tl) {
      const TileCoord c = coord(tile);
      int k_begin, k_end, k_step;
      k_range(c.z, k_begin, k_end, k_step);
      const int acc = tl & 1;
      if (tl >= 2) live = wait(tmem_empty_bar(acc), ((tl >> 1) - 1) & 1) && live;
      ptx::tc_fence_after_sync();
      const uint32_t tmem_d = tmem_base + acc * BN;
      bool first = true;
      for (int k0 = k_begin; k0 < k_end; k0 += k_step, ++it) {
        const int s = it % kStages;
        live = wait(full_bar(s), (it / kStages) & 1) && live;
        const uint32_t a_src = smem_base + s * kStage, b_src = a_src + kABytes;
        const int k_valid = k_end - k0;
        if ((kAMn || kBMn) && k_valid < BK) {
          // K rows beyond the end of the reduction: zero them (a K row is one 128-byte line per 64-wide box)
          const int n_lines = BK - k_valid;
          if (kAMn)
            for (int j = 0; j < BM / 64; ++j)
              for (int q = lane; q < n_lines * 8; q += 32)
                *reinterpret_cast<uint4*>(smem_al + s * kStage + j * (BK * 128) + (k_valid + q / 8) * 128 + (q % 8) * 16) =
                    make_uint4(0, 0, 0, 0);
          if (kBMn)
            for (int j = 0; j < bn / 64; ++j)
              for (int q = lane; q < n_lines * 8; q += 32)
                *reinterpret_cast<uint4*>(smem_al + s * kStage + kABytes + j * (BK * 128) + (k_valid + q / 8) * 128 +
                                          (q % 8) * 16) = make_uint4(0, 0, 0, 0);
          ptx::fence_proxy_async_smem();
          __syncwarp();
        }
        ptx::tc_fence_after_sync();
        if (ptx::elect_one()) {  // one lane of the converged warp issues: the descriptors stay in uniform registers
#pragma unroll
          for (int k = 0; k < BK / 16; ++k) {
            const uint64_t adesc = kAMn ? ptx::smem_desc_sw128(a_src + k * 2048, BK * 128, 1024)
                                        : ptx::smem_desc_sw128(a_src + k * 32, 16, 1024);
            const uint64_t bdesc = kBMn ? ptx::smem_desc_sw128(b_src + k * 2048, BK * 128, 1024)
                                        : ptx::smem_desc_sw128(b_src + k * 32, 16, 1024);
            ptx::mma_bf16(tmem_d, adesc, bdesc, idesc, (first && k == 0) ? 0u : 1u);
          }
          if (live) ptx::mma_commit(empty_bar(s));
        }
        first = false;
        __syncwarp();
      }
      if (!first && ptx::elect_one()) ptx::mma_commit(tmem_full_bar(acc));  // the same lane as above: it covers its products
    }
    failed = !live;
  } else {
    // ------------------------------------------------------------------ epilogue warps
    const int q = warp & 3;          // TMEM lane quarter this warp may read
    uint8_t* stage = smem_al + kStages * kStage + 128 + (warp - 2) * 2048;  // this warp's transposition buffer
    int tl = 0;
    for (int tile = blockIdx.x; tile < total; tile += gridDim.x, ++tl) {
      const TileCoord c = coord(tile);
      const int acc = tl & 1;
      // Thread `lane` receives row (q*32 + lane) of the accumulator.  Written straight from there, every
      // store instruction would touch 32 rows with 16 bytes each; instead the warp turns 64-byte row
      // segments around in its private 2 KB of shared memory, so that a store instruction covers 8 rows
      // with 64 contiguous bytes each (whole 32-byte sectors only).
      OutT* obase = out + (long long)c.z * split_stride;
      constexpr int kPasses = sizeof(OutT) == 2 ? 1 : 2;        // 64-byte segments per 32 accumulator columns
      constexpr int kSegCols = 64 / (int)sizeof(OutT);          // output columns per segment
      const int my_chunk = lane & 3, my_row = lane >> 2;        // role of this lane on the store side
      long long orow[4];                                        // destination rows of the four rows this lane stores
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int grow = c.m0 + q * 32 + my_row + 8 * j;
        orow[j] = (row_map != nullptr && grow < M) ? (long long)ld_dep(row_map + grow) : (long long)grow;
      }
      // the bias of the tile comes to L1 under the main loop: fetched where it is added, each 32 columns waited for L2
      if (bias != nullptr && lane < bn / 64 && c.n0 + lane * 64 < N) prefetch_l1(bias + c.n0 + lane * 64);
      wait(tmem_full_bar(acc), (tl >> 1) & 1);
      if (__any_sync(0xffffffffu, *abort_flag != 0)) { failed = true; break; }
      ptx::tc_fence_after_sync();
#pragma unroll 1
      for (int cc = 0; cc < bn / 32; ++cc) {
        uint4 old[4];  // what the results are combined with, under the read of the accumulator
        if constexpr (sizeof(OutT) == 2) {
#pragma unroll
          for (int j = 0; j < 4; ++j)
            if (c.m0 + q * 32 + my_row + 8 * j < M && c.n0 + cc * 32 + my_chunk * 8 < N)
              epi.fetch(obase, old[j], orow[j] * ldo + c.n0 + cc * 32 + my_chunk * 8);
        }
        uint32_t r[32];
        ptx::tmem_ld_32x32(tmem_base + ((uint32_t)(q * 32) << 16) + acc * BN + cc * 32, r);
        ptx::tmem_ld_wait();
#pragma unroll
        for (int ps = 0; ps < kPasses; ++ps) {
#pragma unroll
          for (int i = 0; i < 4; ++i) {  // 16-byte chunk i of this row's segment
            uint4 packed;
            if (sizeof(OutT) == 2) {
              float v[8];
#pragma unroll
              for (int e = 0; e < 8; ++e) v[e] = __uint_as_float(r[i * 8 + e]);
              const int col = c.n0 + cc * 32 + i * 8;
              if (bias != nullptr && col < N) {
                float b[8];
                Vec16<__nv_bfloat16>::to_float(__ldg(reinterpret_cast<const uint4*>(bias + col)), b);
#pragma unroll
                for (int e = 0; e < 8; ++e) v[e] += b[e];
              }
              packed = Vec16<__nv_bfloat16>::from_float(v);
            } else {
              packed = make_uint4(r[ps * 16 + i * 4], r[ps * 16 + i * 4 + 1], r[ps * 16 + i * 4 + 2], r[ps * 16 + i * 4 + 3]);
            }
            *reinterpret_cast<uint4*>(stage + lane * 64 + ((i ^ ((lane >> 1) & 3)) << 4)) = packed;
          }
          __syncwarp();
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const int rr = my_row + 8 * j;
            const uint4 v4 = *reinterpret_cast<const uint4*>(stage + rr * 64 + ((my_chunk ^ ((rr >> 1) & 3)) << 4));
            const int grow = c.m0 + q * 32 + rr;
            const int gcol = c.n0 + cc * 32 + ps * kSegCols + my_chunk * (16 / (int)sizeof(OutT));
            if (grow < M && gcol < N) {
              if constexpr (sizeof(OutT) == 2) epi.finish(obase, orow[j] * ldo + gcol, v4, old[j]);
              else *reinterpret_cast<uint4*>(obase + orow[j] * ldo + gcol) = v4;
            }
          }
          __syncwarp();
        }
      }
      ptx::tc_fence_before_sync();
      __syncwarp();
      if (lane == 0) ptx::mbar_arrive(tmem_empty_bar(acc));  // this warp has drained its quarter of the accumulator
    }
  }
  ptx::tc_fence_before_sync();
  if (__builtin_expect(__syncthreads_or(failed ? 1 : 0), 0)) ptx::drain_cta(issued, kStages, full_bar(0), drain_bar);
  if (warp == 1) {
    ptx::tc_fence_after_sync();
    ptx::tmem_dealloc(tmem_base, 2 * BN);
  }
}

// ---- wgrad helpers --------------------------------------------------------------------------------
// Partial column sums of dout over one chunk of rows: part[chunk][col].  A streaming reduction: CTA (x, y) owns 64
// columns and the rows of chunk y, eight threads across the columns (16 bytes each) and 32 down the rows with four
// loads in flight per thread; the 32 row lanes are added up in shared memory in a fixed order.
constexpr int kColsumChunks = 64;  // row chunks over the allocated rows (rows per chunk: a multiple of 8)
inline int colsum_rows_per_chunk(int capacity) { return (((capacity + kColsumChunks - 1) / kColsumChunks) + 7) & ~7; }

__global__ void __launch_bounds__(256)
colsum_partial_kernel(const __nv_bfloat16* dout, int n_out, const int32_t* cu, int n_seg,
                      int capacity, int rows_per_chunk, float* __restrict__ part) {
  pdl_entry();
  const int rows = packed_rows(cu, n_seg, capacity);
  const int r_begin = blockIdx.y * rows_per_chunk;
  if (r_begin >= rows) return;  // chunks past the valid rows are not read by the reduction
  int r_end = r_begin + rows_per_chunk;
  if (r_end > rows) r_end = rows;
  __shared__ float red[32][65];
  const int cg = threadIdx.x & 7, rl = threadIdx.x >> 3;  // 8 column groups of 8, 32 row lanes
  const int col = blockIdx.x * 64 + cg * 8;
  float acc[8] = {};
  if (col < n_out) {
    for (int i0 = r_begin + rl; i0 < r_end; i0 += 128) {
      uint4 v[4];
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (i0 + 32 * u < r_end) v[u] = ld_stream16(dout + (long long)(i0 + 32 * u) * n_out + col);
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        if (i0 + 32 * u < r_end) {
          float f[8];
          Vec16<__nv_bfloat16>::to_float(v[u], f);
#pragma unroll
          for (int e = 0; e < 8; ++e) acc[e] += f[e];
        }
      }
    }
  }
#pragma unroll
  for (int e = 0; e < 8; ++e) red[rl][cg * 8 + e] = acc[e];
  __syncthreads();
  if (threadIdx.x < 64) {
    const int c = blockIdx.x * 64 + threadIdx.x;
    if (c < n_out) {
      float s = 0.f;
#pragma unroll
      for (int r = 0; r < 32; ++r) s += red[r][threadIdx.x];
      part[(long long)blockIdx.y * n_out + c] = s;
    }
  }
}

// out[e] = sum over the splits that hold rows (in split order) of part[s][e]; zero if there are none.
// Two arrays in one launch: the weight-gradient partials (a few splits: a thread adds them in split order) and,
// optionally, the bias-gradient partials, one per row chunk or (rows_per_chunk2 = 0) tiles_n2 per split - up to hundreds
// of them for a few thousand outputs, so there a warp owns four outputs: lane l adds chunks l, l + 32, ... in order and a fixed shuffle
// tree adds the lanes.  The first ceil(n2 / 32) blocks take the second array.
__device__ __forceinline__ float4 ld_part(const float* part, long long j) {
  const uint4 v = ld_stream16(reinterpret_cast<const float4*>(part) + j);
  return make_float4(__uint_as_float(v.x), __uint_as_float(v.y), __uint_as_float(v.z), __uint_as_float(v.w));
}

__global__ void __launch_bounds__(256)
split_reduce_kernel(const float* part, long long n, const float* part2, long long n2,
                    int splits, int rows_per_chunk2, int tiles_n2, const int32_t* cu, int n_seg, int capacity,
                    float* __restrict__ out, float* __restrict__ out2) {
  pdl_entry();
  const int rows = packed_rows(cu, n_seg, capacity);
  const int k_blocks = (rows + BK - 1) / BK;  // the splits were dealt the BK-blocks of the rows in turn
  const int valid1 = k_blocks < splits ? k_blocks : splits;
  const long long n4 = n >> 2, m4 = n2 >> 2;
  const int nb2 = (int)((m4 + 7) / 8);
  if ((int)blockIdx.x < nb2) {
    const int valid2 = rows_per_chunk2 > 0 ? (rows + rows_per_chunk2 - 1) / rows_per_chunk2 : valid1 * tiles_n2;
    const long long j = (long long)blockIdx.x * 8 + (threadIdx.x >> 5);
    if (j >= m4) return;
    const int lane = threadIdx.x & 31;
    float4 s4 = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int z = lane; z < valid2; z += 32) {
      const float4 v = ld_part(part2 + (long long)z * n2, j);
      s4.x += v.x; s4.y += v.y; s4.z += v.z; s4.w += v.w;
    }
#pragma unroll
    for (int off = 16; off >= 1; off >>= 1) {
      s4.x += __shfl_xor_sync(0xffffffffu, s4.x, off);
      s4.y += __shfl_xor_sync(0xffffffffu, s4.y, off);
      s4.z += __shfl_xor_sync(0xffffffffu, s4.z, off);
      s4.w += __shfl_xor_sync(0xffffffffu, s4.w, off);
    }
    if (lane == 0) reinterpret_cast<float4*>(out2)[j] = s4;
    return;
  }
  const long long first = (long long)(blockIdx.x - nb2) * blockDim.x + threadIdx.x;
  for (long long j = first; j < n4; j += (long long)(gridDim.x - nb2) * blockDim.x) {
    float4 s4 = make_float4(0.f, 0.f, 0.f, 0.f);
    // four splits' loads in flight at a time; the additions stay in split order
    auto add = [&](const float4& v) { s4.x += v.x; s4.y += v.y; s4.z += v.z; s4.w += v.w; };
    auto at = [&](int z) { return ld_part(part + (long long)z * n, j); };
    int z = 0;
    for (; z + 4 <= valid1; z += 4) {
      const float4 v0 = at(z), v1 = at(z + 1), v2 = at(z + 2), v3 = at(z + 3);
      add(v0); add(v1); add(v2); add(v3);
    }
    for (; z < valid1; ++z) add(at(z));
    reinterpret_cast<float4*>(out)[j] = s4;
  }
}

struct SplitPlan { int splits, k_per_split; };

// The BK-blocks of K = packed rows are dealt to the splits in turn, so every split is in use whatever the row count;
// as many splits as keep tiles x splits within the CTAs that are resident at once (a second tile for some of the CTAs
// would double the longest path).
SplitPlan plan_splits(int capacity, int n_in, int n_out) {
  const int tiles = ((n_out + BM - 1) / BM) * ((n_in + 127) / 128);
  int splits = (2 * kNumSMs) / tiles;
  const int max_by_rows = (capacity + BK - 1) / BK;
  if (splits > max_by_rows) splits = max_by_rows;
  if (splits > 31) splits = 31;  // the bias partials fit beside them in a workspace of 32
  if (splits < 1) splits = 1;
  int kps = (capacity + splits - 1) / splits;
  kps = ((kps + BK - 1) / BK) * BK;
  splits = (capacity + kps - 1) / kps;
  return {splits, kps};
}

size_t wgrad_workspace_bytes(int capacity, int n_in, int n_out) {
  const SplitPlan sp = plan_splits(capacity, n_in, n_out);
  const PairWgradPlan pl = pair_wgrad_plan(capacity, n_in, n_out);
  auto bytes = [&](int splits, int sums) {
    return (((size_t)splits * n_out * n_in * sizeof(float) + 255) & ~(size_t)255) + (size_t)sums * n_out * sizeof(float) + 256;
  };
  const size_t one = bytes(sp.splits, kColsumChunks), two = bytes(pl.splits, pl.splits * pl.tiles_n);
  return one > two ? one : two;
}

inline bool wgrad_on_pairs(const spa_params& p) { return !(p.flags & SPA_FLAG_NO_CTA_PAIRS); }

template <int BN, bool kDyn, bool kAMn, bool kBMn, typename OutT, int kKind>
int launch_gemm(const CUtensorMap& tmA, const CUtensorMap& tmB, const __nv_bfloat16* bias, OutT* out, long long ldo,
                long long split_stride, int M, int N, int K, const int32_t* cu, int n_seg, int capacity, int dyn_which,
                int k_per_split, int splits, int k_interleave, const int32_t* row_map, RowEpilogue<kKind> epi,
                uint32_t wait_limit, int32_t* d_status, cudaStream_t st, const char* what) {
  auto kern = gemm_tc_kernel<BN, kDyn, kAMn, kBMn, OutT, kKind>;
  static DeviceOnce attr;  // per instantiation and device
  cudaError_t ea = attr.run([&] { return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, gemm_smem_bytes<BN>()); });
  if (ea != cudaSuccess) { set_cuda_error(ea, what); return SPA_ERR_CUDA; }
  // persistent grid: two CTAs per SM (99 KB of shared memory and 256 TMEM columns each), never more
  // CTAs than there are tiles when every allocated row is in use
  long long tiles = (long long)((N + BN - 1) / BN) * ((M + BM - 1) / BM) * splits * (kDyn ? 2 : 1);
  const int grid = (int)(tiles < 2 * kNumSMs ? (tiles < 1 ? 1 : tiles) : 2 * kNumSMs);
  launch_pdl(kern, grid, kGemmThreads, gemm_smem_bytes<BN>(), st, tmA, tmB, bias, out, ldo, split_stride, M, N, K, cu,
             n_seg, capacity, dyn_which, k_per_split, k_interleave, row_map, epi, wait_limit, d_status);
  SPA_CUDA_CHECK_LAUNCH(what);
  return SPA_OK;
}

// Tiles of 64 columns where that leaves every tile a CTA of its own from the start (two per SM): twice the SMs share the
// operands' way into shared memory, which bounds the main loop, and the epilogue.  98 rows 384 -> 1 152: 5.9 -> 4.8 us; 1 568
// rows 1 536 -> 384: 10.6 -> 9.4; past that line they lose up to 40 % (3 120 rows 2 304 -> 768: 16.3 -> 23.2).  The rows that
// there are decide, the host knows the capacity, of which about half is filled: up to 148 wide tiles for all of it narrow ones,
// up to twice as many the kernel chooses (0.3 us slower with wide tiles than the kernel that has no choice), above wide ones.
enum TileWidth { kNarrow, kByRows, kWide };
inline TileWidth tile_width(int capacity, int n_cols) {
  const long long wide = (long long)((capacity + BM - 1) / BM) * ((n_cols + 127) / 128);
  return wide <= kNumSMs ? kNarrow : (wide <= 2 * kNumSMs ? kByRows : kWide);
}
template <bool kBMn, int kKind>
int launch_width(TileWidth width, const CUtensorMap& tmA, const CUtensorMap& tmB, const __nv_bfloat16* bias, __nv_bfloat16* out,
                 const spa_params& p, int n_cols, int k, const int32_t* cu, const int32_t* row_map, RowEpilogue<kKind> epi,
                 int32_t* d_status, cudaStream_t st, const char* what) {
  auto run = width == kNarrow   ? launch_gemm<64, false, false, kBMn, __nv_bfloat16, kKind>
             : width == kByRows ? launch_gemm<128, true, false, kBMn, __nv_bfloat16, kKind>
                                : launch_gemm<128, false, false, kBMn, __nv_bfloat16, kKind>;
  return run(tmA, tmB, bias, out, n_cols, 0, p.capacity, n_cols, k, cu, p.B, p.capacity, 1, k, 1, 0, row_map, epi,
             ptx::wait_limit(p.flags), d_status, st, what);
}

}  // namespace

bool tc_linear_supported(int n_in, int n_out) {
  return n_in % 8 == 0 && n_out % 8 == 0 && n_in >= 64 && n_out >= 64 && encode_fn() != nullptr;
}

size_t tc_weight_grad_workspace_bytes(const spa_params& p, int n_in, int n_out) {
  return p.dtype == SPA_BF16 && tc_linear_supported(n_in, n_out) ? wgrad_workspace_bytes(p.capacity, n_in, n_out) : 0;
}

size_t tc_linear_workspace_bytes(const spa_params& p) {
  if (p.dtype != SPA_BF16 || !tc_linear_supported(p.C, 3 * p.C)) return 0;
  const size_t a = wgrad_workspace_bytes(p.capacity, p.C, 3 * p.C);
  const size_t b = wgrad_workspace_bytes(p.capacity, p.C, p.C);
  return a > b ? a : b;
}

int launch_linear_fwd_tc(const spa_params& p, const void* a, const void* W, const void* bias, int n_in, int n_out,
                         const int32_t* cu, void* out, int32_t* d_status, cudaStream_t st, const int32_t* row_map,
                         const LinearEpilogue& epi) {
  if (tc_pair_linear_supported(p, n_in, n_out, n_out))
    return launch_linear_fwd_pair(p, a, W, bias, n_in, n_out, cu, out, d_status, st, row_map, epi);
  const TileWidth width = tile_width(p.capacity, n_out);
  CUtensorMap tmA, tmB;
  if (!make_tmap_bf16_2d(&tmA, a, n_in, p.capacity, (uint64_t)n_in * 2, BK, BM) ||
      !make_tmap_bf16_2d(&tmB, W, n_in, n_out, (uint64_t)n_in * 2, BK, width == kWide ? 128 : 64))
    return SPA_ERR_UNSUPPORTED;
  auto go = [&](auto row_epi) {
    return launch_width<false>(width, tmA, tmB, (const __nv_bfloat16*)bias, (__nv_bfloat16*)out, p, n_out, n_in, cu, row_map, row_epi,
                               d_status, st, "gemm_tc_kernel(fwd)");
  };
  if (epi.h != nullptr) return go(RowEpilogue<kEpiGelu>{(__nv_bfloat16*)epi.h});
  if (epi.add != nullptr && epi.add != out) return go(RowEpilogue<kEpiAdd>{(__nv_bfloat16*)const_cast<void*>(epi.add)});
  return go(RowEpilogue<kEpiOwn>{epi.add != nullptr ? (__nv_bfloat16*)out : nullptr});
}

int launch_linear_bwd_tc(const spa_params& p, const void* a, const void* W, const void* dout, int n_in, int n_out,
                         const int32_t* cu, void* da, float* dW, float* db, void* workspace, int32_t* d_status,
                         cudaStream_t st, const int32_t* row_map, const LinearEpilogue& epi) {
  CUtensorMap tmA, tmB, tmA2, tmB2;
  if (da != nullptr && (!make_tmap_bf16_2d(&tmA, dout, n_out, p.capacity, (uint64_t)n_out * 2, BK, BM) ||
                        !make_tmap_bf16_2d(&tmB, W, n_in, n_out, (uint64_t)n_in * 2, 64, BK)))
    return SPA_ERR_UNSUPPORTED;
  if (dW != nullptr && (!make_tmap_bf16_2d(&tmA2, dout, n_out, p.capacity, (uint64_t)n_out * 2, 64, BK) ||
                        !make_tmap_bf16_2d(&tmB2, a, n_in, p.capacity, (uint64_t)n_in * 2, 64, BK)))
    return SPA_ERR_UNSUPPORTED;
  const bool pair_dgrad = da != nullptr && tc_pair_linear_supported(p, n_in, n_out, n_in);
  if (pair_dgrad) {
    int rc = launch_linear_dgrad_pair(p, W, dout, n_in, n_out, cu, da, d_status, st, row_map, epi);
    if (rc != SPA_OK) return rc;
  } else if (da != nullptr) {  // da[M][n_in] = dout[M][n_out] W[n_out][n_in]
    auto go = [&](auto row_epi) {
      return launch_width<true>(tile_width(p.capacity, n_in), tmA, tmB, nullptr, (__nv_bfloat16*)da, p, n_in, n_out, cu, row_map, row_epi,
                                d_status, st, "gemm_tc_kernel(dgrad)");
    };
    int rc = epi.u != nullptr ? go(RowEpilogue<kEpiGeluGrad>{(__nv_bfloat16*)const_cast<void*>(epi.u)})
                              : go(RowEpilogue<kEpiOwn>{epi.add != nullptr ? (__nv_bfloat16*)da : nullptr});
    if (rc != SPA_OK) return rc;
  }
  if (dW == nullptr && db == nullptr) return SPA_OK;
  const PairWgradPlan pl = pair_wgrad_plan(p.capacity, n_in, n_out);
  // CTA pairs where there are enough of their 256 x 256 tiles and enough rows to split between them (768 x 768 over 9 216
  // rows: 18 us on pairs, 30 on clusters; 1 536 x 512 over 3 402: 17 either way; 1 536 x 384 over 1 568: 14 and 12).  The line
  // runs through 768 x 768 and 8 192 allocated rows and is on the safe side: at 6 144, all or half of them there, pairs are
  // ahead too (768 x 768 14.1 against 21.1 and 11.7 against 14.2, 576 x 576 13.7 against 15.3 and 11.4 against 11.7).
  if (dW != nullptr && wgrad_on_pairs(p) && (pl.tiles < 9 || p.capacity < 128 * BK))
    return launch_wgrad_cluster(p, a, dout, n_in, n_out, cu, dW, db, d_status, st);
  const SplitPlan sp = plan_splits(p.capacity, n_in, n_out);
  const bool pair = dW != nullptr && wgrad_on_pairs(p);
  const int splits = pair ? pl.splits : sp.splits;
  float* part_w = reinterpret_cast<float*>(workspace);
  size_t off = ((size_t)splits * n_out * n_in * sizeof(float) + 255) & ~(size_t)255;
  float* part_b = reinterpret_cast<float*>(reinterpret_cast<uint8_t*>(workspace) + off);
  const long long n_w = (long long)n_out * n_in;
  const int rpc = colsum_rows_per_chunk(p.capacity);
  if (db != nullptr && !pair) {  // db[j] = sum_i dout[i][j]: partial sums per row chunk, added up by the reduction below
    dim3 grid((n_out + 63) / 64, (p.capacity + rpc - 1) / rpc);
    launch_pdl(colsum_partial_kernel, grid, 256, 0, st, (const __nv_bfloat16*)dout, n_out, cu, p.B, p.capacity, rpc, part_b);
    SPA_CUDA_CHECK_LAUNCH("colsum_partial_kernel");
  }
  if (dW != nullptr) {  // dW[n_out][n_in] = sum_i dout[i][:]^T a[i][:]
    int rc = pair ? launch_wgrad_pair(p, a, dout, n_in, n_out, cu, part_w, db != nullptr ? part_b : nullptr, pl, d_status, st)
                  : launch_gemm<128, false, true, true, float>(tmA2, tmB2, nullptr, part_w, n_in, n_w, n_out, n_in, p.capacity,
                                                        cu, p.B, p.capacity, 2, sp.k_per_split, sp.splits, sp.splits,
                                                        nullptr, RowEpilogue<kEpiOwn>{nullptr}, ptx::wait_limit(p.flags), d_status, st,
                                                        "gemm_tc_kernel(wgrad)");
    if (rc != SPA_OK) return rc;
    const long long n_b = db != nullptr ? n_out : 0;
    int grid = (int)((n_w / 4 + 255) / 256);
    if (grid > kNumSMs * 8) grid = kNumSMs * 8;
    grid += (int)((n_b / 4 + 7) / 8);  // the blocks of the bias gradient come first
    launch_pdl(split_reduce_kernel, grid, 256, 0, st, part_w, n_w, part_b, n_b, splits, pair ? 0 : rpc, pl.tiles_n, cu, p.B, p.capacity,
               dW, db);
    SPA_CUDA_CHECK_LAUNCH("split_reduce_kernel");
  } else {  // db alone
    launch_pdl(split_reduce_kernel, (n_out / 4 + 7) / 8, 256, 0, st, (const float*)nullptr, 0LL, (const float*)part_b,
               (long long)n_out, 0, rpc, 0, cu, p.B, p.capacity, (float*)nullptr, db);
    SPA_CUDA_CHECK_LAUNCH("split_reduce_kernel(db)");
  }
  return SPA_OK;
}

}  // namespace spa
