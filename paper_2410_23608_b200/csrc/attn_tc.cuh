// What the tensor-core attention kernels share: operand tiles, segments of packed rows, and how the CTAs of a persistent grid
// come by their work items.
#pragma once

#include "sm100_ptx.cuh"
#include "spa_tc.cuh"

namespace spa {
namespace {

template <int D> struct HeadTile {
  static constexpr int kRowBytes = D * 2;          // 128 (d = 64) or 64 (d = 32): also the swizzle span
  static constexpr int kTileBytes = 128 * kRowBytes;
  static constexpr int kSbo = 8 * kRowBytes;
  // Operand descriptor of a tile at `addr`: low word, and high word (the same for all).  A K-major operand (Q or K rows, head
  // dimension contiguous) moves by kStepK per 16 head dimensions, an MN-major one (V: key rows are the K dimension) by kStepMN
  // per 16 keys; addresses of shared memory do not carry out of their field.
  static constexpr uint32_t kDescHi = (uint32_t)(kSbo >> 4) | (1u << 14) | ((D == 64 ? 2u : 4u) << 29);
  static constexpr uint32_t kStepK = 2, kStepMN = kRowBytes;
  __device__ static __forceinline__ uint32_t desc_lo(uint32_t addr) { return (addr >> 4) | (1u << 16); }
  __device__ static __forceinline__ uint64_t desc(uint32_t lo) { return ((uint64_t)kDescHi << 32) | lo; }
  __device__ static __forceinline__ uint64_t kmajor(uint32_t addr, int k) { return desc(desc_lo(addr) + k * kStepK); }
  __device__ static __forceinline__ uint64_t mnmajor(uint32_t addr, int k) { return desc(desc_lo(addr) + k * kStepMN); }
};

// Segment bounds of packed row i (hi clamped to the valid rows) from offsets held in shared memory.
__device__ __forceinline__ RowSeg row_segment_staged(const int32_t* s_off, int n_seg, int Np, int i) {
  RowSeg r{0, 0};
  if (i < Np) {
    int lo = 0, hi = n_seg;  // invariant: s_off[lo] <= i < s_off[hi]
    while (hi - lo > 1) {
      const int mid = (lo + hi) >> 1;
      if (s_off[mid] <= i) lo = mid; else hi = mid;
    }
    r.lo = s_off[lo];
    const int h2 = s_off[lo + 1];
    r.hi = h2 < Np ? h2 : Np;
  }
  return r;
}

constexpr int kShortMax = 128;  // segments of at most this many rows are taken by the one-pass backward kernel

// Rotation of the 16-byte chunks of row r of a [128][D] bf16 tile in shared memory that makes the
// accesses of 8 neighbouring rows to one chunk index fall into different banks.
template <int D> __device__ __forceinline__ int chunk_rot(int r) { return D == 64 ? (r & 7) : ((r >> 1) & 3); }

// Copy a [128][D] bf16 tile that the threads wrote to shared memory (chunk c of row r at position
// c ^ chunk_rot(r)) to rows r0.. of a matrix with `ld` elements per row: a warp covers whole rows, so the
// stores are full 64- or 128-byte lines.  Rows from Np on are not written.
template <int D, int kThreads>
__device__ __forceinline__ void copy_tile_out(const uint8_t* tile, __nv_bfloat16* dst, long long ld, int r0, int Np, int tid,
                                              const volatile uint8_t* row_ok = nullptr) {
  constexpr int kChunks = D * 2 / 16;
#pragma unroll
  for (int i = tid; i < 128 * kChunks; i += kThreads) {
    const int r = i / kChunks, c = i % kChunks;
    if (r0 + r < Np && (row_ok == nullptr || row_ok[r]))
      *reinterpret_cast<uint4*>(dst + (long long)(r0 + r) * ld + c * 8) =
          *reinterpret_cast<const uint4*>(tile + r * (D * 2) + ((c ^ chunk_rot<D>(r)) << 4));
  }
}

// Up to this many segments, a CTA's first item is looked up by one warp straight from the offsets.
constexpr int kEarlySegments = 512;  // sixteen offsets a lane, their loads in flight together (280 segments of 49: 14.5 -> 14.2 us)

// ---- work items -------------------------------------------------------------------------------------------------
// The persistent kernels draw their (row tile, head) items from a counter in global memory, longest rows of key tiles
// first: static strides left the last CTA busy for 1.36 times the mean (detection, 210 to 1 680 rows per segment).
constexpr int kMaxOrder = 512;  // row tiles that are put in order of length; beyond, there are items enough to even out

// Position of the row tiles [first, n_tiles) in that order (ties in ascending order, so that all CTAs agree):
// tile[rank], less first.  By kThreads threads behind named barrier `id`, offsets staged; about 1 000 clocks, which fit under the loads of a CTA's first item.
struct __align__(16) ItemOrder { uint4 cost16[kMaxOrder / 16]; uint16_t tile[kMaxOrder]; };
template <int kThreads>
__device__ __forceinline__ void order_items(ItemOrder* o, const int32_t* s_off, int n_seg, int Np, int first, int n_tiles, int id) {
  uint8_t* cost = reinterpret_cast<uint8_t*>(o->cost16);
  const int n = n_tiles - first;
  for (int i = threadIdx.x; i < ((n + 15) & ~15); i += kThreads) {
    int c = 0;
    if (i < n) {
      const int r0 = (first + i) * 128, last = r0 + 127 < Np - 1 ? r0 + 127 : Np - 1;
      c = (row_segment_staged(s_off, n_seg, Np, last).hi - row_segment_staged(s_off, n_seg, Np, r0).lo + 127) >> 7;
    }
    cost[i] = (uint8_t)(c < 255 ? c : 255);
  }
  ptx::named_barrier(id, kThreads);
  for (int i = threadIdx.x; i < n; i += kThreads) {
    const uint32_t mine = cost[i] * 0x01010101u;
    int rank = 0;
    for (int w = 0; w < (n + 15) / 16; ++w) {
      const uint4 v = o->cost16[w];
      const uint32_t c[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int below = i - 16 * w - 4 * u;  // tiles of this word in front of tile i
        const uint32_t front = below >= 4 ? 0x01010101u : (below > 0 ? 0x01010101u & ((1u << (8 * below)) - 1u) : 0u);
        rank += __popc((__vcmpgtu4(c[u], mine) & 0x01010101u) | (__vcmpeq4(c[u], mine) & front));
      }
    }
    o->tile[rank] = (uint16_t)i;
  }
}

// The next item for this CTA, after its first.  The first `given` items (whole row tiles) go to the CTAs of their number,
// the others are drawn: every CTA draws until it gets a number past the last item, so that a launch takes n_items - given
// + gridDim.x numbers and the counter wraps to zero with the last of them, for the next launch.  Without a
// counter: a static stride.
__device__ __forceinline__ int draw_item(unsigned* counter, int given, int n_items, int& own) {
  own += gridDim.x;
  if (counter == nullptr || n_items <= given) return own;
  return (int)atomicInc(counter, (unsigned)(n_items - given) + gridDim.x - 1u) + given;
}

// Segment of packed row `row` (lane l of a converged warp asks for row0 + l); rows from Np on get an empty range.  A
// 32-way search for the warp's first row, then the offsets behind it, 32 at a time, looked up with shuffles.
template <typename Load>
__device__ __forceinline__ RowSeg warp_row_segment(Load off, int n_seg, int Np, int row0) {
  const int lane = threadIdx.x & 31, row = row0 + lane;
  RowSeg r{0, 0};
  if (row0 >= Np) return r;  // the same for the whole warp
  int lo = 0, n = n_seg;     // off(lo) <= row0, and the segment sought is one of the n from lo on
  while (n > 1) {
    const int step = (n + 31) >> 5, at = lo + lane * step;
    const unsigned le = __ballot_sync(0xffffffffu, lane * step < n && off(at) <= row0);
    const int k = 31 - __clz(le);  // lane 0 always counts
    n = n - k * step < step ? n - k * step : step;
    lo += k * step;
  }
  int seg = -1;
  for (int base = lo;; base += 32) {
    const int at = base + 1 + lane;
    const int end = at <= n_seg ? off(at) : 0x7fffffff;  // end of segment base + lane
    int c = 0;                                           // segments of this group that end at or before the row
#pragma unroll
    for (int s = 16; s >= 1; s >>= 1)
      if (__shfl_sync(0xffffffffu, end, c + s - 1) <= row) c += s;
    const int last_end = __shfl_sync(0xffffffffu, end, 31);
    if (c == 31 && last_end <= row) c = 32;
    const int hi = __shfl_sync(0xffffffffu, end, c & 31);
    int start = __shfl_sync(0xffffffffu, end, (c + 31) & 31);
    if (c == 0) start = off(base);
    if (seg < 0 && c < 32) { seg = base + c; r.lo = start; r.hi = hi; }
    if (__all_sync(0xffffffffu, seg >= 0 || row >= Np)) break;
  }
  if (row >= Np) return RowSeg{0, 0};
  if (r.hi > Np) r.hi = Np;
  return r;
}
}  // namespace

// The counter that a launch which writes `out` draws its items from, or nullptr (then a static stride assigns them).
unsigned* item_counter(const void* out);

// The dK / dV pass by attn_bwd_kv_kernel (attn_bwd_kv.cu), where that is the faster one
bool attention_bwd_kv_applies(const spa_params& p, int n_seg);
int launch_attention_bwd_kv(const spa_params& p, const void* qkv, const float* lse, const float* delta, const void* dao,
                            const int32_t* seg, int n_seg, void* dqkv, bool skip_short, int32_t* d_status, cudaStream_t st);

}  // namespace spa
