// Attention backward on tcgen05 tensor cores, the dK / dV pass of large problems (Sec. 3.2: packed tokens attend only to
// tokens of the same image; gradient of the 2L^2C term of Eq. 9).
#include <math_constants.h>

#include "attn_tc.cuh"

namespace spa {
namespace {

// An item is 128 packed key rows j of one head; per tile of 128 queries i    S^T = K Q^T, dP^T = V dO^T,
// P^T = 2^(S^T - lse_i) and dS^T = P^T (dP^T - D_i) written to TMEM as bf16,    dV += P^T dO,  dK += dS^T Q.
// dV and dK accumulate in TMEM over the item's tiles, so that no sum is split across CTAs.
//
// One CTA per SM with all of TMEM and one continuous pipeline over all its items: phases are counted over the whole run and
// nothing joins the CTA between items.  What has to be hidden is the way from the arithmetic to the tensor core and back
// (announcement, issue, products, announcement: 700 to 1 200 clocks, as long as a tile's arithmetic), so every product is
// issued a phase before its result is needed:
//   S^T   two buffers: that of tile g + 1 is computed under the arithmetic of tile g, whose P^T and dS^T each thread writes
//         over its own columns of S^T of tile g;
//   dP^T  one buffer: issued as soon as the warps hold that of tile g in registers, under the exponentials of tile g + 1.
// Sixteen arithmetic warps: four threads per key row, 32 of the 128 queries each, in two groups of eight that need not be in
// step.  Three warps issue the products (S^T and dP^T | dV | dK): one for all of them was what the tiles waited for, 20 or 24
// products and seven waits in 2 800 clocks a tile.  The last warp draws the items, looks up their rows' segments, issues every
// copy and stages the queries' statistics, up to kStages tiles and an item ahead.  A finished item's accumulators are
// drained behind the exponentials of the next item's first tile, when the wait for its last products is over.
// What bounds it: the exponentials are 1 024 clocks of a tile's 2 500 (16 segments of 210 to 1 680 rows, 8 heads of 32), the
// rest is the chain wait - load - arithmetic - store - announcement of a warp, four of which share a scheduler (96 registers, of
// which 16 to 28 bytes are spilled).  The whole backward with it, against two CTAs per SM on 64-query tiles with a prologue per
// item: that workload 211.5 -> 169.5 us, cut into containers of 49 rows 61.5 -> 54.0; 32 segments of 58 to 518 rows, 12 heads of 64,
// 96.9 -> 84.5.
constexpr int kMathWarps = 16, kMathThreads = 32 * kMathWarps;
// warps behind the arithmetic ones: products S^T and dP^T | dV | dK; items and copies
constexpr int kWarpS = kMathWarps, kWarpV = kMathWarps + 1, kWarpK = kMathWarps + 2, kWarpLoad = kMathWarps + 3;
constexpr int kKvThreads = kMathThreads + 128;
// Up to so many segments, whose offsets are searched in shared memory; its size goes by them.
constexpr int kKvSegStage = 12288;
constexpr uint32_t kColDP = 256, kColDV = 384, kColDK = 448;  // S^T: columns 0 and 128

template <int D> struct KvSmem {
  static constexpr int kTile = HeadTile<D>::kTileBytes;
  static constexpr int kStages = D == 64 ? 3 : 6;             // streamed stages of a Q and a dO tile
  static constexpr int kY = 4 * kTile;                        // behind two items' K and V
  static constexpr int kStat = kY + kStages * 2 * kTile;      // [kStages][2][128]: -lse_i log2e, -D_i of the queries
  static constexpr int kRows = kStat + kStages * 2 * 128 * 4;
  static constexpr int kBar = kRows + 4 * 2 * 128 * 4;        // rows' segments of four items: [lo][hi]
  static constexpr int kOrder = kBar + 512;                   // barriers, item slots
  static constexpr int kSeg = kOrder + (int)sizeof(ItemOrder);
  static constexpr int bytes(int offsets) { return kSeg + offsets * 4 + 1024; }  // and the alignment of the base
  static constexpr int kMaxBytes = bytes(kKvSegStage);
  static_assert(kMaxBytes <= 227 * 1024, "shared memory of a CTA");
};

template <int D>
__global__ void __launch_bounds__(kKvThreads, 1)
attn_bwd_kv_kernel(const __grid_constant__ CUtensorMap tm_qkv, const __grid_constant__ CUtensorMap tm_do, const float* lse,
                   const float* delta, const int32_t* seg, int n_seg, int capacity, int C, int H, float scale,
                   __nv_bfloat16* __restrict__ dqkv, bool skip_short, unsigned* counter, bool even_items, uint32_t wait_limit,
                   int32_t* d_status) {
  using HT = HeadTile<D>;
  using SM = KvSmem<D>;
  constexpr int kTile = SM::kTile, kStages = SM::kStages;
  constexpr float kLog2e = 1.4426950408889634f;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

  extern __shared__ uint8_t smem_raw[];
  const uint32_t smem_base = (ptx::smem_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t* smem_al = smem_raw + (smem_base - ptx::smem_u32(smem_raw));
  auto x_s = [&](int item, int which) { return smem_base + kTile * (2 * (item & 1) + which); };
  auto y_s = [&](int st, int which) { return smem_base + SM::kY + kTile * (2 * st + which); };
  const uint32_t bar = smem_base + SM::kBar;
  auto bar_x = [&](int item) { return bar + 8 * (item & 1); };              // the item's own tiles have landed
  auto bar_item = [&](int item) { return bar + 16 + 8 * (item & 1); };      // the item slot is filled
  auto bar_acc = [&](int item) { return bar + 32 + 8 * (item & 1); };       // the item's last products have completed
  auto bar_drained = [&](int item) { return bar + 48 + 8 * (item & 1); };   // 8: its accumulators are in registers
  auto bar_s = [&](int g) { return bar + 64 + 8 * (g & 1); };
  auto bar_p = [&](int g, int grp) { return bar + 80 + 16 * (g & 1) + 8 * grp; };  // 8: exponentials of tile g done, P^T in TMEM
  const uint32_t bar_dp = bar + 112;
  const uint32_t bar_dpfree = bar + 120;  // 16: every warp holds its dP of tile g in registers
  // 8: dS of tile g is in TMEM.  Two, as of P: dP of tile g + 1 is issued before dS of tile g is waited for, and the second
  // phase of one barrier completing under a wait for the first would look like neither
  auto bar_ds = [&](int g, int grp) { return bar + 128 + 16 * (g & 1) + 8 * grp; };
  const uint32_t bar_order = bar + 176;   // 16: the order of the items is there
  const uint32_t bar_drain = bar + 184;   // 3: the products of an issuing warp have completed, all of them
  auto bar_y = [&](int st) { return bar + 192 + 8 * st; };   // 2: copies of a stage have landed, its statistics are there
  auto bar_free = [&](int st) { return bar + 240 + 8 * st; };  // the products that read a stage have completed
  const uint32_t tmem_slot = bar + 288, abort_any = bar + 292;
  auto item_slot = [&](int item) { return bar + 304 + 16 * (item & 3); };   // {r0, h, first streamed row, tiles * 128 + over}
  auto row_s = [&](int item) { return smem_base + SM::kRows + (item & 3) * 1024; };
  int32_t* seg_s = reinterpret_cast<int32_t*>(smem_al + SM::kSeg);
  ItemOrder* order = reinterpret_cast<ItemOrder*>(smem_al + SM::kOrder);

  // everything up to the wait touches no global memory, so it runs under the previous kernel's tail
  if (tid == 32 * kWarpLoad) {
    ptx::prefetch_tensormap(&tm_qkv);
    ptx::prefetch_tensormap(&tm_do);
    for (int b = 0; b < 2; ++b) {
      ptx::mbar_init(bar_x(b), 1);
      ptx::mbar_init(bar_item(b), 1);
      ptx::mbar_init(bar_acc(b), 2);
      ptx::mbar_init(bar_drained(b), kMathWarps / 2);
      ptx::mbar_init(bar_s(b), 1);
      ptx::mbar_init(bar_p(0, b), kMathWarps / 2);
      ptx::mbar_init(bar_p(1, b), kMathWarps / 2);
      ptx::mbar_init(bar_ds(0, b), kMathWarps / 2);
      ptx::mbar_init(bar_ds(1, b), kMathWarps / 2);
    }
    ptx::mbar_init(bar_dp, 1);
    ptx::mbar_init(bar_dpfree, kMathWarps);
    ptx::mbar_init(bar_order, kMathWarps);
    ptx::mbar_init(bar_drain, 3);
    for (int st = 0; st < kStages; ++st) {
      ptx::mbar_init(bar_y(st), 2);
      ptx::mbar_init(bar_free(st), 2);
    }
    ptx::sts_s32(abort_any, 0);
    ptx::fence_mbar_init();
  }
  pdl_entry();
#pragma unroll 4
  for (int i = tid; i <= n_seg; i += kKvThreads) seg_s[i] = ld_dep(seg + i);
  const int Np = packed_rows(seg, n_seg, capacity);
  const int row_tiles = (Np + 127) / 128, n_items = row_tiles * H;
  if ((int)blockIdx.x >= n_items) return;
  if (warp == kWarpS) ptx::tmem_alloc(tmem_slot, 512);
  // see the forward kernel
  const bool draws = counter != nullptr && n_items > (int)gridDim.x;
  const int given = draws ? (int)gridDim.x / H * H : n_items;
  const bool ordered = !even_items && draws && 2 * n_items >= 3 * (int)gridDim.x && row_tiles - given / H <= kMaxOrder;
  // The loading warp gets the streamed rows of the CTA's first item straight from the offsets, of which a lane takes a few, and
  // starts its copies before the CTA comes together.
  const bool early = warp == kWarpLoad && n_seg < kEarlySegments && !skip_short && !(draws && (int)blockIdx.x >= given);
  int lo = 0, hi = Np;  // the rows of the other side that the loading warp's item visits: the union of its rows' segments
  auto load_own = [&](int n, int r0, int h) {
    if (ptx::elect_one()) {
      ptx::mbar_expect_tx(bar_x(n), 2 * kTile);
      ptx::tma_load_2d(x_s(n, 0), &tm_qkv, bar_x(n), C + h * D, r0);      // K
      ptx::tma_load_2d(x_s(n, 1), &tm_qkv, bar_x(n), 2 * C + h * D, r0);  // V
    }
    __syncwarp();
  };
  auto load_tile = [&](int st, int y0, int h) {
    if (ptx::elect_one()) {
      ptx::mbar_expect_tx(bar_y(st), 2 * kTile);
      ptx::tma_load_2d(y_s(st, 0), &tm_qkv, bar_y(st), h * D, y0);  // Q
      ptx::tma_load_2d(y_s(st, 1), &tm_do, bar_y(st), h * D, y0);   // dO
    }
    __syncwarp();
  };
  if (early) {
    const int r0 = (int)blockIdx.x / H * 128, h = (int)blockIdx.x % H;
    load_own(0, r0, h);
#pragma unroll 4
    for (int i = lane; i <= n_seg; i += 32) {
      const int o = ld_dep(seg + i);
      if (o <= r0 && o > lo) lo = o;
      if (o > r0 + 127 && o < hi) hi = o;
    }
    lo = __reduce_max_sync(0xffffffffu, lo);
    hi = __reduce_min_sync(0xffffffffu, hi);
    load_tile(0, lo, h);
  }
  ptx::tc_fence_before_sync();
  __syncthreads();  // barriers, TMEM address and staged offsets are visible
  ptx::tc_fence_after_sync();
  const uint32_t tmem = (uint32_t)ptx::lds_s32(tmem_slot);
  // Bounded; nobody branches on a wait that gave up inside an item (see mbar_wait_or_abort)
  auto wait = [&](uint32_t b, uint32_t parity) { return ptx::mbar_wait_or_abort_warp(b, parity, abort_any, d_status, SPA_ERR_TIMEOUT, wait_limit); };
  const bool is_math = warp < kMathWarps;
  auto aborted = [&]() { return __any_sync(0xffffffffu, ptx::lds_s32(abort_any) != 0) != 0; };

  int n = 0, filled = 0;  // items whose copies have been issued or looked at, tiles whose copies have been

  if (warp == kWarpLoad) {
    // ---------------------------------------------------------------- items, copies and statistics: one warp
    int own = blockIdx.x, drawn = blockIdx.x;
    if (draws && (int)blockIdx.x >= given && lane == 0) drawn = draw_item(counter, given, n_items, own);
    bool order_ready = false, ok = true;
    int st = 0, use = 0;  // stage of the next tile and how often it has been filled
    int v;
    auto wait_all = [&](uint32_t b, uint32_t parity) { ok = __all_sync(0xffffffffu, wait(b, parity)) != 0 && ok; };
    for (;;) {
      v = __shfl_sync(0xffffffffu, drawn, 0);
      if (v >= n_items) break;
      const int rank = v / H, h = v - rank * H;
      const bool by_order = ordered && v >= given, started = early && n == 0;
      if (by_order && !order_ready) {
        wait_all(bar_order, 0);
        order_ready = true;
      }
      const int r0 = (by_order ? given / H + (int)order->tile[rank - given / H] : rank) * 128;
      // the own tiles' memory and everything older is free when the item before last is through with its products
      if (n >= 2) wait_all(bar_acc(n), ((n - 2) >> 1) & 1);
      if (!ok) break;
      if (!skip_short && !started) load_own(n, r0, h);
      // the segments of its rows, four to a lane, in step
      RowSeg s[4];
      int a[4] = {}, b[4];  // seg_s[a] <= row < seg_s[b]
#pragma unroll
      for (int i = 0; i < 4; ++i) b[i] = n_seg;
      for (int step = 32 - __clz(n_seg - 1 > 0 ? n_seg - 1 : 0); step > 0; --step) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int mid = (a[i] + b[i]) >> 1;  // = a once b = a + 1: no change then
          if (seg_s[mid] <= r0 + 32 * i + lane) a[i] = mid; else b[i] = mid;
        }
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int end = seg_s[a[i] + 1];
        s[i] = r0 + 32 * i + lane < Np ? RowSeg{seg_s[a[i]], end < Np ? end : Np} : RowSeg{0, 0};
      }
      const uint32_t rs = row_s(n) + lane * 4;
      int lo_rows = 0x7fffffff, hi_rows = 0;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        if (skip_short && s[i].hi - s[i].lo <= kShortMax) s[i] = RowSeg{0, 0};  // a row of the one-pass kernel is none of this one
        if (s[i].hi > s[i].lo) {
          lo_rows = s[i].lo < lo_rows ? s[i].lo : lo_rows;
          hi_rows = s[i].hi > hi_rows ? s[i].hi : hi_rows;
        }
        ptx::sts_s32(rs + 128 * i, s[i].lo);
        ptx::sts_s32(rs + 512 + 128 * i, s[i].hi);
      }
      if (!started) {
        lo = __reduce_min_sync(0xffffffffu, lo_rows);
        hi = __reduce_max_sync(0xffffffffu, hi_rows);
      }
      const int n_tiles = hi > lo ? (hi - lo + 127) / 128 : 0;  // none: every row belongs to the one-pass kernel
      // The last tile's `over` queries behind the item's segments are another image's, or no one's, and an infinity or NaN there times the
      // zeros of P^T and dS^T would be NaN in this image's sums.  So the products that sum over queries leave out the groups of
      // 16 that have none of the item's, and the rest of the group that has both is cleared in shared memory.
      // (Whole backward: 16 segments of 210 to 1 680 rows, 8 heads of 32, 174.7 -> 168.6 us, one of 4 200 rows 148.8 -> 135.6, in
      // containers of 49 54.2 -> 53.2: before, only lines behind the last valid row were cleared, all of them.)
      const int over = n_tiles * 128 - (hi - lo);
      if (n_tiles > 0) {
        if (skip_short) load_own(n, r0, h);
        float sl[4], sd[4];  // statistics of the next tile's queries, on their way
        auto fetch_stats = [&](int y0) {
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const int row = y0 + 32 * i + lane;
            sl[i] = sd[i] = 0.f;
            if (row < hi) { sl[i] = lse[(long long)h * capacity + row]; sd[i] = delta[(long long)h * capacity + row]; }
          }
        };
        fetch_stats(lo);
        if (lane == 0) {
          ptx::sts_s32(item_slot(n), r0);
          ptx::sts_s32(item_slot(n) + 4, h);
          ptx::sts_s32(item_slot(n) + 8, lo);
          ptx::sts_s32(item_slot(n) + 12, n_tiles * 128 + over);
        }
        __syncwarp();
        if (lane == 0) ptx::mbar_arrive(bar_item(n));
        for (int t = 0; t < n_tiles; ++t) {
          if (t == n_tiles - 1 && lane == 0) drawn = draw_item(counter, given, n_items, own);  // the next item
          if (use > 0) wait_all(bar_free(st), (use - 1) & 1);
          if (!ok) break;
          if (!(started && t == 0)) load_tile(st, lo + t * 128, h);
          const uint32_t stat = smem_base + SM::kStat + st * 1024 + lane * 4;
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            ptx::sts_s32(stat + 128 * i, __float_as_int(-sl[i] * kLog2e));
            ptx::sts_s32(stat + 512 + 128 * i, __float_as_int(-sd[i]));
          }
          if (t + 1 < n_tiles) fetch_stats(lo + (t + 1) * 128);
          __syncwarp();
          if (lane == 0) ptx::mbar_arrive(bar_y(st));
          ++filled;
          if (++st == kStages) { st = 0; ++use; }
        }
        ++n;
        if (!ok) break;
      } else if (lane == 0) {
        drawn = draw_item(counter, given, n_items, own);
      }
      __syncwarp();
    }
    if (ok) {  // past the last item
      if (n >= 2) wait_all(bar_acc(n), ((n - 2) >> 1) & 1);
      if (ok && lane == 0) {
        ptx::sts_s32(item_slot(n) + 12, 0);
        ptx::mbar_arrive(bar_item(n));
      }
    }
    while (draws && lane == 0 && drawn < n_items) drawn = draw_item(counter, given, n_items, own);  // after a wait that gave up: the numbers have to add up
    __syncwarp();
  } else if (!is_math) {
    // ---------------------------------------------------------------- products: three warps, whose lanes all follow the tiles
    // and take every wait together; one elected lane issues (see ptx::elect_one)
    constexpr uint32_t kIdescS = ptx::idesc_bf16_f32(128, 128, false, false);
    constexpr uint32_t kIdescAcc = ptx::idesc_bf16_f32(128, D, false, true);
    struct Tile { int item, left, over, st; uint32_t use; };  // left: tiles of the item from this one on; 0: past the end
    auto open = [&](Tile& t) {  // the item's slot
      wait(bar_item(t.item), (t.item >> 1) & 1);
      const bool gone = aborted();
      const int tiles = __shfl_sync(0xffffffffu, ptx::lds_s32(item_slot(t.item) + 12), 0);
      t.left = gone ? 0 : tiles >> 7;
      t.over = tiles & 127;
    };
    auto advance = [&](Tile t, bool& first) {
      if (++t.st == kStages) { t.st = 0; t.use ^= 1u; }
      first = --t.left == 0;
      if (first) {
        ++t.item;
        open(t);
      }
      return t;
    };
    const uint32_t y_lo = HT::desc_lo(y_s(0, 0)), x_lo = HT::desc_lo(smem_base);
    constexpr uint32_t kTileLo = kTile / 16;
    Tile c{0, 0, 0, 0, 0};
    bool c_first = true;  // the tile opens an item
    open(c);
    if (warp == kWarpS) {
      auto issue_s = [&](const Tile& t, int g, bool first) {
        if (first) wait(bar_x(t.item), (t.item >> 1) & 1);
        wait(bar_y(t.st), t.use);
        if (t.left == 1 && (t.over & 15) != 0) {
          constexpr int kChunks = HT::kRowBytes / 16;
          const int n_chunks = (t.over & 15) * kChunks, at = SM::kY + 2 * kTile * t.st + (128 - t.over) * HT::kRowBytes;
          for (int i = lane; i < 2 * n_chunks; i += 32)
            *reinterpret_cast<uint4*>(smem_al + at + (i < n_chunks ? i : kTile / 16 + i - n_chunks) * 16) = make_uint4(0, 0, 0, 0);
          ptx::fence_proxy_async_smem();
          __syncwarp();
        }
        ptx::tc_fence_after_sync();
        const uint32_t a = x_lo + 2 * kTileLo * (t.item & 1), b = y_lo + 2 * kTileLo * t.st;
        if (ptx::elect_one()) {
#pragma unroll
          for (int k = 0; k < D / 16; ++k)
            ptx::mma_bf16(tmem + 128 * (g & 1), HT::desc(a + k * HT::kStepK), HT::desc(b + k * HT::kStepK), kIdescS, k != 0 ? 1u : 0u);
          ptx::mma_commit(bar_s(g));
        }
        __syncwarp();
      };
      auto issue_dp = [&](const Tile& t) {
        const uint32_t a = x_lo + 2 * kTileLo * (t.item & 1) + kTileLo, b = y_lo + 2 * kTileLo * t.st + kTileLo;
        if (ptx::elect_one()) {
#pragma unroll
          for (int k = 0; k < D / 16; ++k)
            ptx::mma_bf16(tmem + kColDP, HT::desc(a + k * HT::kStepK), HT::desc(b + k * HT::kStepK), kIdescS, k != 0 ? 1u : 0u);
          ptx::mma_commit(bar_dp);
        }
        __syncwarp();
      };
      // c: tile g, whose S and dP have been issued; d: tile g + 1, whose S has
      Tile d = c;
      bool d_first = false;
      if (c.left > 0) {
        issue_s(c, 0, true);
        issue_dp(c);
        d = advance(c, d_first);
        if (d.left > 0) issue_s(d, 1, d_first);
      }
      for (int g = 0; c.left > 0 && d.left > 0; ++g) {
        wait(bar_dpfree, g & 1);  // under the rest of tile g's dS and the exponentials of tile g + 1
        ptx::tc_fence_after_sync();
        issue_dp(d);
        bool e_first;
        const Tile e = advance(d, e_first);
        wait(bar_free(c.st), c.use);  // P and dS of tile g, whose columns S of tile g + 2 takes, have been read
        if (aborted()) break;
        if (e.left > 0) issue_s(e, g + 2, e_first);
        c = d;
        d = e;
      }
    } else {
      const bool is_v = warp == kWarpV;
      const uint32_t out = tmem + (is_v ? kColDV : kColDK), b_lo = y_lo + (is_v ? kTileLo : 0u);
      for (int g = 0; c.left > 0; ++g) {
        wait(bar_y(c.st), c.use);
        // k-step k (16 queries): columns that the threads of column group k / 2 have written over their S
        const uint32_t a = tmem + 128 * (g & 1) + (is_v ? 0 : 16), b = b_lo + 2 * kTileLo * c.st;
        const uint32_t acc = c_first ? 0u : 1u;
        const int steps = c.left == 1 ? 8 - (c.over >> 4) : 8;
        bool gone = false;
#pragma unroll
        for (int grp = 0; grp < 2; ++grp) {  // dV += P^T dO | dK += dS^T Q: queries 64 grp ..
          wait(is_v ? bar_p(g, grp) : bar_ds(g, grp), (g >> 1) & 1);
          if (grp == 0 && c_first && c.item > 0) wait(bar_drained(c.item - 1), ((c.item - 1) >> 1) & 1);
          ptx::tc_fence_after_sync();
          if (grp == 1) gone = aborted();
          if (!gone && ptx::elect_one()) {
#pragma unroll
            for (int k = 4 * grp; k < 4 * grp + 4; ++k)
              if (k < steps)
                ptx::mma_bf16_ts(out, a + (k >> 1) * 32 + (k & 1) * 8, HT::desc(b + k * HT::kStepMN), kIdescAcc, k == 0 ? acc : 1u);
            if (grp == 1) {
              ptx::mma_commit(bar_free(c.st));
              if (c.left == 1) ptx::mma_commit(bar_acc(c.item));
            }
          }
          __syncwarp();
        }
        if (gone) break;
        c = advance(c, c_first);
      }
    }
    __syncwarp();
    if (ptx::elect_one()) ptx::mma_commit(bar_drain);
    __syncwarp();
  } else {
    // ---------------------------------------------------------------- arithmetic: four threads per key row, two of each group.
    // A warp may touch the quarter of the TMEM lanes of its number modulo four.
    const int quarter = warp & 3, part = warp >> 2, grp = part >> 1, half = part & 1, rl = quarter * 32 + lane, col0 = part * 32;
    const uint32_t lane_base = tmem + ((uint32_t)(quarter * 32) << 16);
    const float scale_log2e = scale * kLog2e;
    const uint64_t scale2 = ptx::pair(scale_log2e, scale_log2e);
    if (ordered) {
      order_items<kMathThreads>(order, seg_s, n_seg, Np, given / H, row_tiles, 1);
      __syncwarp();
      if (lane == 0) ptx::mbar_arrive(bar_order);
    }
    // An item's accumulators out to global memory, by the first group: half the columns of its row per thread, 32-byte sectors
    int out_r0 = 0, out_h = 0;
    bool out_ok = false;  // this row is one of the item's
    auto store_acc = [&](uint32_t acc_col, int which, float mul) {  // which: 1 dK, 2 dV
      constexpr int kDh = D / 2;
      uint32_t r[kDh];
      if (kDh == 32) ptx::tmem_ld_32x32(lane_base + acc_col + half * kDh, r);
      else ptx::tmem_ld_32x16(lane_base + acc_col + half * kDh, r);
      ptx::tmem_ld_wait();
      __nv_bfloat16* dst = dqkv + (long long)(out_r0 + rl) * (3LL * C) + which * C + out_h * D + half * kDh;
#pragma unroll
      for (int c = 0; c < kDh; c += 16) {
        uint4 o[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          float f[8];
#pragma unroll
          for (int e = 0; e < 8; ++e) f[e] = __uint_as_float(r[c + 8 * u + e]) * mul;
          o[u] = Vec16<__nv_bfloat16>::from_float(f);
        }
        if (out_ok) st_global32(dst + c, o[0], o[1], (reinterpret_cast<uintptr_t>(dqkv) & 31u) == 0);  // rows and heads are whole sectors then
      }
    };
    auto drain = [&](int item) {
      wait(bar_acc(item), (item >> 1) & 1);
      ptx::tc_fence_after_sync();
      store_acc(kColDV, 2, 1.f);
      store_acc(kColDK, 1, scale);
      ptx::tc_fence_before_sync();
      __syncwarp();
      if (lane == 0) ptx::mbar_arrive(bar_drained(item));
    };
    int g = 0, st = 0;
    uint32_t use = 0;
    for (;; ++n) {
      wait(bar_item(n), (n >> 1) & 1);
      const bool gone = aborted();
      int left = ptx::lds_s32(item_slot(n) + 12) >> 7;
      if (gone || left == 0) break;
      // the row's segment relative to this thread's first column of the tile; it moves down tile by tile
      int lo = ptx::lds_s32(row_s(n) + rl * 4), hi = ptx::lds_s32(row_s(n) + 512 + rl * 4);
      const bool valid = hi > lo;
      {
        const int y0 = ptx::lds_s32(item_slot(n) + 8) + col0;
        lo -= y0;
        hi -= y0;
      }
      for (bool first = true; left > 0; --left, ++g, lo -= 128, hi -= 128, first = false) {
        const uint32_t s_col = lane_base + 128 * (g & 1) + col0;
        const uint32_t stat = smem_base + SM::kStat + st * 1024 + col0 * 4;
        // ---- P^T = 2^(S^T - lse).  A thread whose 32 queries lie wholly outside its row's segment writes zeros without the
        // arithmetic; the mask costs something only where a boundary crosses.
        wait(bar_s(g), (g >> 1) & 1);
        wait(bar_y(st), use);  // the statistics, which a warp other than the issuing one has staged
        ptx::tc_fence_after_sync();
        uint32_t rs[32], pk[16];
        ptx::tmem_ld_32x32(s_col, rs);
        ptx::tmem_ld_wait();
        const bool some = hi > 0 && lo < 32, partial = some && (lo > 0 || hi < 32);
        const uint32_t in = partial ? (0xffffffffu >> (hi < 32 ? 32 - hi : 0)) & (0xffffffffu << (lo > 0 ? lo : 0)) : 0u;
        if (some) {
          if (partial) {
#pragma unroll
            for (int j = 0; j < 32; ++j)
              if ((in & (1u << j)) == 0) rs[j] = 0xff800000u;  // p = 2^-inf = 0
          }
          // all exponents, then all exponentials, then what uses them: in the formula's order a warp waits out the unit's
          // latency with every pair
#pragma unroll
          for (int j = 0; j < 32; j += 4) {
            uint64_t l2[2];
            ptx::lds_pairs(stat + j * 4, l2[0], l2[1]);
            ptx::unpair(ptx::fma2(ptx::pair(rs[j], rs[j + 1]), scale2, l2[0]), rs[j], rs[j + 1]);
            ptx::unpair(ptx::fma2(ptx::pair(rs[j + 2], rs[j + 3]), scale2, l2[1]), rs[j + 2], rs[j + 3]);
          }
#pragma unroll
          for (int j = 0; j < 32; ++j) rs[j] = __float_as_uint(ptx::ex2_approx(__uint_as_float(rs[j])));
#pragma unroll
          for (int j = 0; j < 32; j += 2) pk[j >> 1] = ptx::bf16_pair(__uint_as_float(rs[j]), __uint_as_float(rs[j + 1]));
        } else {
#pragma unroll
          for (int j = 0; j < 16; ++j) pk[j] = 0u;
        }
        ptx::tmem_st_32x16(s_col, pk);  // over this thread's own columns of S^T
        ptx::tmem_st_wait();
        ptx::tc_fence_before_sync();
        __syncwarp();
        if (lane == 0) ptx::mbar_arrive(bar_p(g, grp));
        if (first) {
          if (grp == 0 && n > 0) drain(n - 1);
          out_r0 = ptx::lds_s32(item_slot(n));
          out_h = ptx::lds_s32(item_slot(n) + 4);
          out_ok = valid;
        }
        // ---- dS^T = P^T (dP^T - D)
        wait(bar_dp, g & 1);
        ptx::tc_fence_after_sync();
        uint32_t rp[32];
        ptx::tmem_ld_32x32(lane_base + kColDP + col0, rp);  // by the whole warp: the load is a collective
        ptx::tmem_ld_wait();
        ptx::tc_fence_before_sync();
        __syncwarp();
        if (lane == 0) ptx::mbar_arrive(bar_dpfree);
        if (some) {
          if (partial) {
#pragma unroll
            for (int j = 0; j < 32; ++j)
              if ((in & (1u << j)) == 0) rp[j] = 0u;
          }
#pragma unroll
          for (int j = 0; j < 32; j += 4) {
            uint64_t d2[2];
            ptx::lds_pairs(stat + 512 + j * 4, d2[0], d2[1]);
#pragma unroll
            for (int u = 0; u < 2; ++u) {
              const int i = j + 2 * u;
              float s0, s1;
              ptx::unpair(ptx::mul2(ptx::pair(rs[i], rs[i + 1]), ptx::add2(ptx::pair(rp[i], rp[i + 1]), d2[u])), s0, s1);
              pk[i >> 1] = ptx::bf16_pair(s0, s1);
            }
          }
        } else {
#pragma unroll
          for (int j = 0; j < 16; ++j) pk[j] = 0u;
        }
        ptx::tmem_st_32x16(s_col + 16, pk);
        ptx::tmem_st_wait();
        ptx::tc_fence_before_sync();
        __syncwarp();
        if (lane == 0) ptx::mbar_arrive(bar_ds(g, grp));
        if (++st == kStages) { st = 0; use ^= 1u; }
      }
    }
    if (grp == 0 && n > 0 && !aborted()) drain(n - 1);
  }
  ptx::tc_fence_before_sync();
  __syncthreads();
  // Products complete before the CTA's memory goes, and so do copies, which have been waited for unless a wait gave up.  Here, because
  // that may have been in a warp whose partners had left their loops in good order.
  if (warp == kWarpLoad && aborted() && lane == 0) {
    for (int i = filled > kStages ? filled - kStages : 0; i < filled; ++i) ptx::mbar_wait(bar_y(i % kStages), (i / kStages) & 1);
    for (int i = n > 2 ? n - 2 : 0; i <= n; ++i) ptx::mbar_wait(bar_x(i), (i >> 1) & 1, 1u << 14);
  }
  if (warp == kWarpS) {
    ptx::mbar_wait(bar_drain, 0);
    ptx::tc_fence_after_sync();
    ptx::tmem_dealloc(tmem, 512);
  }
}

template <int D>
int kv_launch(const spa_params& p, const void* qkv, const float* lse, const float* delta, const void* dao, const int32_t* seg,
              int n_seg, void* dqkv, bool skip_short, int32_t* d_status, cudaStream_t st) {
  CUtensorMap tm_qkv, tm_do;  // boxes of 128 rows of one head
  if (!make_tmap_bf16_2d(&tm_qkv, qkv, 3ull * p.C, p.capacity, 6ull * p.C, D, 128, D * 2) ||
      !make_tmap_bf16_2d(&tm_do, dao, (uint64_t)p.C, p.capacity, 2ull * p.C, D, 128, D * 2))
    return SPA_ERR_UNSUPPORTED;
  auto kern = attn_bwd_kv_kernel<D>;
  static DeviceOnce attr;
  cudaError_t ea = attr.run([&] { return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, KvSmem<D>::kMaxBytes); });
  if (ea != cudaSuccess) { set_cuda_error(ea, "attn_bwd_kv_kernel"); return SPA_ERR_CUDA; }
  const long long items = (long long)p.H * ((p.capacity + 127) / 128);
  const int grid = (int)(items < kNumSMs ? items : kNumSMs);
  const bool even_items = (long long)p.capacity <= 512ll * (n_seg > 0 ? n_seg : 1);  // as in the forward
  const int offsets = n_seg < 2048 ? 2048 : n_seg + 1;
  launch_pdl(kern, grid, kKvThreads, KvSmem<D>::bytes(offsets), st, tm_qkv, tm_do, lse, delta, seg, n_seg, p.capacity, p.C, p.H,
             softmax_scale_of(p), (__nv_bfloat16*)dqkv, skip_short, items > grid ? item_counter(dqkv) : nullptr, even_items,
             ptx::wait_limit(p.flags), d_status);
  SPA_CUDA_CHECK_LAUNCH("attn_bwd_kv_kernel");
  return SPA_OK;
}

}  // namespace

// By the 128 x 128 tiles that the capacity may hold, items times the tiles that one spans (its own 128 rows and what a segment
// adds), per SM: with few of them the start of the pipeline, a copy, a look-up and a cold instruction cache long, is all there
// is.  dQ and dK / dV together, us, the other kernels -> this one, at tiles per SM of
//   5: 32 images of 196 tokens, 6 heads of 64, 20.1 -> 18.9;  10: 64 of them 24.6 -> 26.2, 4 x 4 200 tokens in containers of 49,
//   8 heads of 32, 19.5 -> 20.4;  11: 24 x 315 tokens, 8 heads of 64, 27.8 -> 27.0;  15.6: 32 x 256, 12 heads of 64, 40.0 -> 37.5,
//   but in a transformer block's step, whose weight gradients then wait for whole SMs, 503 -> 506 when the kernel was new;  16: 8 x 576
//   43.0 -> 38.1;  20: 128 x 196, 6 heads of 64, 45.5 -> 43.3 (a transformer block's step then 538 -> 544), of 32 38.9 -> 37.6, 8 x
//   4 200 in containers 35.3 -> 32.4;  the line;  32: 16 x 576 59.4 -> 51.8;  40: 128 x 196, 12 heads, 56.5 -> 51.5;  60: 1 x 4 200,
//   8 heads of 32, 33.9 -> 27.8;  960: 16 x 4 200 211.5 -> 169.5.  Rows are a part of the capacity; with 1 to 3 % of 16 x 4 200 tokens
//   selected 52 -> 34, of 32 x 576 23.4 -> 19.5.
// And by the segments: searched in global memory, their offsets are what the tiles of short segments wait for.  42 images of 2 782 tokens in
// containers of 49 rows (2 394 segments), 8 heads of 32: the other kernels 230, so 257.7, from shared memory 204.3;  14 000 images
// of 49 tokens, whose offsets do not fit there, 691 -> 746.
bool attention_bwd_kv_applies(const spa_params& p, int n_seg) {
  const long long items = (long long)p.H * ((p.capacity + 127) / 128);
  const long long segment = p.capacity / (n_seg > 0 ? n_seg : 1);
  return n_seg < kKvSegStage && items * (128 + segment) >= 24ll * 128 * kNumSMs;
}

int launch_attention_bwd_kv(const spa_params& p, const void* qkv, const float* lse, const float* delta, const void* dao,
                            const int32_t* seg, int n_seg, void* dqkv, bool skip_short, int32_t* d_status, cudaStream_t st) {
  return p.C / p.H == 64 ? kv_launch<64>(p, qkv, lse, delta, dao, seg, n_seg, dqkv, skip_short, d_status, st)
                         : kv_launch<32>(p, qkv, lse, delta, dao, seg, n_seg, dqkv, skip_short, d_status, st);
}

}  // namespace spa
