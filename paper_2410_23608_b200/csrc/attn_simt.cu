// fp32-FMA segment-masked attention, forward and backward, on the packed tokens (Sec. 3.2: packed
// tokens attend only to tokens of the same image; the 2L^2C term of Eq. 9).  The path of the fp32
// workload and the bring-up reference of the tensor-core kernels.
//
// Work split: a CTA owns 32 consecutive packed rows and one head, wherever segment boundaries fall, and walks the
// rows of the other side that the segments of its rows span, in tiles of 64 staged in shared memory as fp32.  Where there are few CTAs, two
// groups of 128 threads take them in turn, each with a stage of its own, and the first joins the two results at the end: one group's copies
// and softmax run under the other's products, and a CTA's chain, which bounds such problems, is half as long.  Else one group takes
// them all, and other CTAs run under its copies (see one_group).
// A group is a grid of 8 x 16 threads: a product tile of 32 x 64 is 4 x 4 values per thread (8
// vector reads of shared memory per 64 multiply-adds), its softmax statistics are shuffles among 16 lanes, and the
// second product gives a thread 4 rows x D / 16 head dimensions.  No padding token is ever computed, nothing is atomically
// accumulated, and every sum runs in a fixed order.  Against one group with two tiles in flight for all, us: one image of
// 4 200 tokens, 8 heads of 32, forward 81.5 -> 46.1, backward 200.5 -> 151.8; 4 of 196 tokens, 3 heads of 32, 7.4 -> 7.2 and
// 15.8 -> 14.4; 16 of 196, 6 heads of 64, 22.6 -> 21.7 and 76.2 -> 73.0; 64 of them 70.4 -> 62.6 and 254 -> 229.  What bounds it
// then is shared memory: a vector read of 16 bytes per eight multiply-adds, 30 of the 75 TFLOP/s of the multiply-adds.
// Errors against fp64: in the backward, and in the forward of one group, a tile's terms are summed by themselves and then added, so that no
// chain is longer than 64 terms and the number of tiles (with one chain, one per group, now: 64 images of 186 rows, 8 heads of 32,
// outputs 3.2e-7, 2.8e-7, 2.6e-7, gradients 3.9e-7, 3.6e-7, 3.4e-7; 4 000 rows of one segment, 2 heads of 64, two groups, outputs
// 1.16e-6, 8.5e-7, 8.5e-7, gradients 1.24e-6, 9.4e-7, 5.2e-7).
#include <math_constants.h>

#include "simt_stage.cuh"
#include "spa_common.cuh"

namespace spa {
namespace {

constexpr int kR = 32;          // packed rows per CTA
constexpr int kT = 64;          // rows of a streamed tile
constexpr int kGroup = 128;     // threads; of kGroups groups, one or two, group q takes the streamed tiles q, q + kGroups, ..
constexpr int kTX = 16, kTY = 8;  // thread (ty, tx) of a group: rows ty + 8 i (i < 4), streamed rows tx + 16 j (j < 4)
constexpr int kLdP = kT + 4;    // leading dimension of the probability tiles
template <int D> constexpr int kLd = D + 4;  // rows 4 banks apart

// Rows [row0, row0 + kRows) of one head's slice (column col0 of a [*, ld] matrix); rows from row_end on become zero.
template <typename T, int D, int kRows, int kBy>
__device__ __forceinline__ void stage_rows(float* dst, const T* src, long long ld, int col0, int row0, int row_end,
                                           int tid) {
  constexpr int E = Vec16<T>::kElems, kPer = D / E;
#pragma unroll
  for (int c = tid; c < kRows * kPer; c += kBy) {
    const int r = c / kPer, cc = (c % kPer) * E;
    stage16<T>(dst + r * kLd<D> + cc, src + (long long)(row0 + r) * ld + col0 + cc, row0 + r < row_end, src);
  }
}

// s[i][j] += a_row(ty + 8 i) . b_row(tx + 16 j) over D
template <int D>
__device__ __forceinline__ void dots(float (*s)[4], const float* a, const float* b, int ty, int tx) {
#pragma unroll
  for (int e = 0; e < D; e += 4) {
    float4 av[4], bv[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) av[i] = *reinterpret_cast<const float4*>(a + (ty + kTY * i) * kLd<D> + e);
#pragma unroll
    for (int j = 0; j < 4; ++j) bv[j] = *reinterpret_cast<const float4*>(b + (tx + kTX * j) * kLd<D> + e);
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        s[i][j] = fmaf(av[i].x, bv[j].x, s[i][j]);
        s[i][j] = fmaf(av[i].y, bv[j].y, s[i][j]);
        s[i][j] = fmaf(av[i].z, bv[j].z, s[i][j]);
        s[i][j] = fmaf(av[i].w, bv[j].w, s[i][j]);
      }
  }
}

template <int W> __device__ __forceinline__ void add_to(float (*sum)[W], const float (*v)[W]) {
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int d = 0; d < W; ++d) sum[i][d] += v[i][d];
}
// o[i][d] += sum over the tile's rows k < n of p[ty + 8 i][k] * v[k][tx * (D / 16) + d]
template <int D>
__device__ __forceinline__ void weighted(float (*o)[D / kTX], const float* p, const float* v, int n, int ty, int tx) {
  constexpr int W = D / kTX;  // 2 or 4
  for (int k = 0; k < n; k += 4) {  // p is zero from row n on
    float4 pv[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) pv[i] = *reinterpret_cast<const float4*>(p + (ty + kTY * i) * kLdP + k);
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      float w[W];
      const float* src = v + (k + u) * kLd<D> + tx * W;
      if (W == 4) {
        const float4 t = *reinterpret_cast<const float4*>(src);
        w[0] = t.x; w[1] = t.y; w[W - 2] = t.z; w[W - 1] = t.w;
      } else {
        const float2 t = *reinterpret_cast<const float2*>(src);
        w[0] = t.x; w[1] = t.y;
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float pi = u == 0 ? pv[i].x : u == 1 ? pv[i].y : u == 2 ? pv[i].z : pv[i].w;
#pragma unroll
        for (int d = 0; d < W; ++d) o[i][d] = fmaf(pi, w[d], o[i][d]);
      }
    }
  }
}

// A zero weight times an infinity or NaN of another segment in the same tile is NaN.  Sums that are not finite, where the
// CTA's rows are of several segments, are therefore formed again from their own segment's rows alone: rare, one value after
// the other from global memory.  (Tiles looked at as they come in, or a second pass over the tiles: 3 us of 69 each.)
template <int W> __device__ __forceinline__ bool finite_sums(const float* o) {
  float s = 0.f;
#pragma unroll
  for (int d = 0; d < W; ++d) s += fabsf(o[d]);
  return s < CUDART_INF_F;
}
template <typename T, int D> __device__ __forceinline__ float row_dot(const T* a, const T* b) {
  float s = 0.f;
#pragma unroll 1
  for (int e = 0; e < D; ++e) s = fmaf(to_f32<T>(a[e]), to_f32<T>(b[e]), s);
  return s;
}

// W consecutive values of one row
template <typename T, int W> __device__ __forceinline__ void store_row(T* dst, const float* v) {
#pragma unroll
  for (int d = 0; d < W; ++d) dst[d] = from_f32<T>(v[d]);
}
template <> __device__ __forceinline__ void store_row<float, 4>(float* dst, const float* v) {
  *reinterpret_cast<float4*>(dst) = make_float4(v[0], v[1], v[2], v[3]);
}
template <> __device__ __forceinline__ void store_row<float, 2>(float* dst, const float* v) {
  *reinterpret_cast<float2*>(dst) = make_float2(v[0], v[1]);
}

__device__ __forceinline__ void group_sync(int q) { asm volatile("bar.sync %0, %1;" ::"r"(q + 1), "n"(kGroup) : "memory"); }

// The CTA's own rows are there, of which every thread has copied a part: kBehind is the number of copy groups that a thread
// with a streamed tile has committed behind its part.  One without a tile has none behind it and waits for all it has:
// counted like the others, its part could still be on its way behind the barrier.
template <int kBehind> __device__ __forceinline__ void own_rows_landed(bool has_tile) {
  if (has_tile) cp_async_wait<kBehind>();
  else cp_async_wait<0>();
  __syncthreads();
}

__device__ __forceinline__ float max16(float v) {
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}
__device__ __forceinline__ float sum16(float v) {
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Segments of the CTA's 32 rows in seg_s[32] (threads 0-31 search one each); returns the range they span together.
__device__ __forceinline__ RowSeg tile_segments(RowSeg* seg_s, const int32_t* seg, int n_seg, int Np, int i0,
                                                int tid) {
  if (tid < kR) seg_s[tid] = row_segment(seg, n_seg, Np, i0 + tid);
  __syncthreads();
  const int last = i0 + kR - 1 < Np - 1 ? kR - 1 : Np - 1 - i0;
  return RowSeg{seg_s[0].lo, seg_s[last].hi};
}

// ------------------------------------------------------------------------------------ forward
template <int D, int kGroups> constexpr int kFwdFloats = (kR + kGroups * 2 * kT) * kLd<D> + kGroups * kR * kLdP;  // Q; per group K and V, P

template <typename T, int D, int kGroups>
__global__ void __launch_bounds__(kGroups * kGroup, 4 / kGroups)
attn_fwd_simt_kernel(const T* qkv, const int32_t* seg, int n_seg, int capacity, int C,
                     float scale, T* __restrict__ ao, float* __restrict__ lse) {
  pdl_entry();
  constexpr int W = D / kTX, kThreads = kGroups * kGroup;
  extern __shared__ __align__(16) float sm[];
  __shared__ RowSeg seg_s[kR];
  constexpr int kTile = kT * kLd<D>;
  const int Np = packed_rows(seg, n_seg, capacity);
  const int i0 = blockIdx.x * kR;
  if (i0 >= Np) return;
  const int grp = threadIdx.x / kGroup, tid = threadIdx.x % kGroup, tx = tid % kTX, ty = tid / kTX, h = blockIdx.y;
  float* Qs = sm;
  float* Ks = sm + kR * kLd<D> + grp * 2 * kTile;  // this group's K, V behind it
  float* Ps = sm + kR * kLd<D> + kGroups * 2 * kTile + grp * kR * kLdP;
  const long long ld = 3LL * C;
  stage_rows<T, D, kR, kThreads>(Qs, qkv, ld, h * D, i0, Np, threadIdx.x);
  cp_async_commit();
  const RowSeg all = tile_segments(seg_s, seg, n_seg, Np, i0, threadIdx.x);
  const int n_tiles = (all.hi - all.lo + kT - 1) / kT;
  const bool several = seg_s[0].hi < all.hi;  // segments that the CTA's rows are of
  auto stage = [&](int t) {
    const int kv0 = all.lo + t * kT;
    stage_rows<T, D, kT, kGroup>(Ks, qkv, ld, C + h * D, kv0, all.hi, tid);
    cp_async_commit();
    stage_rows<T, D, kT, kGroup>(Ks + kTile, qkv, ld, 2 * C + h * D, kv0, all.hi, tid);
    cp_async_commit();
  };
  if (grp < n_tiles) stage(grp);

  float o[4][W] = {}, m[4], l[4] = {};
  RowSeg mine[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) { m[i] = -CUDART_INF_F; mine[i] = seg_s[ty + kTY * i]; }
  own_rows_landed<2>(grp < n_tiles);  // Q; K and V of the first tile may be on their way
  for (int t = grp; t < n_tiles; t += kGroups) {
    cp_async_wait<1>();
    group_sync(grp);  // K; V is waited for behind the first product
    const int kv0 = all.lo + t * kT;
    float s[4][4] = {}, alpha[4];
    dots<D>(s, Qs, Ks, ty, tx);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      float cm = -CUDART_INF_F;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int ja = kv0 + tx + kTX * j;
        s[i][j] = (ja >= mine[i].lo && ja < mine[i].hi) ? s[i][j] * scale : -CUDART_INF_F;
        cm = fmaxf(cm, s[i][j]);
      }
      const float m_new = fmaxf(m[i], max16(cm));
      const float m_use = m_new == -CUDART_INF_F ? 0.f : m_new;  // no key of this row so far
      alpha[i] = expf(m[i] - m_use);
      float rs = 0.f;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float p = expf(s[i][j] - m_use);
        rs += p;
        Ps[(ty + kTY * i) * kLdP + tx + kTX * j] = p;
      }
      l[i] = l[i] * alpha[i] + sum16(rs);
      if constexpr (kGroups > 1) {
#pragma unroll
        for (int d = 0; d < W; ++d) o[i][d] *= alpha[i];
      }
      m[i] = m_new;
    }
    cp_async_wait<0>();
    group_sync(grp);  // V, and the rows of P
    const int n = all.hi - kv0 < kT ? all.hi - kv0 : kT;
    if constexpr (kGroups == 1) {  // a sum of its own: the chain is a tile long and then a term per tile
      float tile[4][W] = {};
      weighted<D>(tile, Ps, Ks + kTile, n, ty, tx);
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int d = 0; d < W; ++d) o[i][d] = fmaf(o[i][d], alpha[i], tile[i][d]);
    } else {  // half the tiles: as short a chain as before, and 1 % faster
      weighted<D>(o, Ps, Ks + kTile, n, ty, tx);
    }
    group_sync(grp);  // the stage is free
    if (t + kGroups < n_tiles) stage(t + kGroups);
  }
  if (kGroups > 1 && n_tiles == 1 && grp == 1) return;
  if (kGroups > 1 && n_tiles > 1) {  // the second group's share of every row, in the memory of its stage
    float* part = sm + kR * kLd<D> + 2 * kTile + tid;  // [4 (W + 2)][kGroup]
    if (grp == 1) {
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        part[(i * (W + 2)) * kGroup] = m[i];
        part[(i * (W + 2) + 1) * kGroup] = l[i];
#pragma unroll
        for (int d = 0; d < W; ++d) part[(i * (W + 2) + 2 + d) * kGroup] = o[i][d];
      }
    }
    __syncthreads();
    if (grp == 1) return;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float m1 = part[(i * (W + 2)) * kGroup], l1 = part[(i * (W + 2) + 1) * kGroup];
      const float m_new = fmaxf(m[i], m1), m_use = m_new == -CUDART_INF_F ? 0.f : m_new;
      const float a0 = expf(m[i] - m_use), a1 = expf(m1 - m_use);
      l[i] = l[i] * a0 + l1 * a1;
#pragma unroll
      for (int d = 0; d < W; ++d) o[i][d] = o[i][d] * a0 + part[(i * (W + 2) + 2 + d) * kGroup] * a1;
      m[i] = m_new;
    }
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int row = i0 + ty + kTY * i;
    if (row >= Np) continue;
    if (several && !finite_sums<W>(o[i])) {
#pragma unroll
      for (int d = 0; d < W; ++d) o[i][d] = 0.f;
#pragma unroll 1
      for (int k = mine[i].lo; k < mine[i].hi; ++k) {
        const T* key = qkv + k * ld + C + h * D;
        const float p = expf(row_dot<T, D>(qkv + row * ld + h * D, key) * scale - m[i]);
#pragma unroll
        for (int d = 0; d < W; ++d) o[i][d] = fmaf(p, to_f32<T>(key[C + tx * W + d]), o[i][d]);
      }
    }
    const float inv_l = 1.f / l[i];
#pragma unroll
    for (int d = 0; d < W; ++d) o[i][d] *= inv_l;
    store_row<T, W>(ao + (long long)row * C + h * D + tx * W, o[i]);
    if (tx == 0) lse[(long long)h * capacity + row] = m[i] + logf(l[i]);
  }
}

// ------------------------------------------------------------------------------------ backward
// One launch for both passes, which need nothing of each other (D_i = dO_i . O_i is taken by either from the rows it
// holds), so that they share the GPU: blockIdx.z = 0: own rows are queries, streamed rows keys,
//   S = Q K^T, dP = dO V^T, dS = P (dP - D), dQ += dS K;
// blockIdx.z = 1: own rows are keys, streamed rows queries, everything transposed: dV += P^T dO, dK += dS^T Q.
template <int D, int kGroups> constexpr int kBwdFloats = (2 * kR + kGroups * 2 * kT) * kLd<D> + kGroups * (kR * kLdP + 2 * kT);

template <typename T, int D, int kGroups>
__global__ void __launch_bounds__(kGroups * kGroup, 4 / kGroups)
attn_bwd_simt_kernel(const T* qkv, const T* ao, const float* lse,
                     const T* dao, const int32_t* seg, int n_seg, int capacity, int C,
                     float scale, T* __restrict__ dqkv) {
  constexpr int kThreads = kGroups * kGroup;
  pdl_entry();
  constexpr int W = D / kTX, E = Vec16<T>::kElems;
  constexpr int kTile = kT * kLd<D>;
  extern __shared__ __align__(16) float sm[];
  __shared__ RowSeg seg_s[kR];
  const int grp = threadIdx.x / kGroup, tid = threadIdx.x % kGroup, tx = tid % kTX, ty = tid / kTX, h = blockIdx.y;
  float* A1 = sm;                       // Q | K of the own rows
  float* A2 = A1 + kR * kLd<D>;         // dO | V
  float* Y1 = A2 + kR * kLd<D> + grp * 2 * kTile;  // this group's K | Q
  float* Y2 = Y1 + kTile;                          // V | dO
  float* Ps = A2 + kR * kLd<D> + kGroups * 2 * kTile + grp * (kR * kLdP + 2 * kT);  // P^T, then dS | dS^T
  float* s2 = Ps + kR * kLdP;           // second pass: lse_i of the streamed rows, D_i behind it
  const bool dq = blockIdx.z == 0;
  const int Np = packed_rows(seg, n_seg, capacity);
  const int i0 = blockIdx.x * kR;
  if (i0 >= Np) return;
  const long long ld = 3LL * C;
  // D of packed row i: eight or sixteen 16-byte loads, all in flight together
  auto row_D = [&](int i) {
    float s = 0.f;
    const T* po = ao + (long long)i * C + h * D;
    const T* pg = dao + (long long)i * C + h * D;
#pragma unroll
    for (int c = 0; c < D / E; ++c) {
      float a[E], b[E];
      Vec16<T>::to_float(*reinterpret_cast<const uint4*>(po + c * E), a);
      Vec16<T>::to_float(*reinterpret_cast<const uint4*>(pg + c * E), b);
#pragma unroll
      for (int e = 0; e < E; ++e) s = fmaf(a[e], b[e], s);
    }
    return s;
  };
  stage_rows<T, D, kR, kThreads>(A1, qkv, ld, (dq ? 0 : C) + h * D, i0, Np, threadIdx.x);
  if (dq) stage_rows<T, D, kR, kThreads>(A2, dao, (long long)C, h * D, i0, Np, threadIdx.x);
  else stage_rows<T, D, kR, kThreads>(A2, qkv, ld, 2 * C + h * D, i0, Np, threadIdx.x);
  cp_async_commit();
  const RowSeg all = tile_segments(seg_s, seg, n_seg, Np, i0, threadIdx.x);
  const int n_tiles = (all.hi - all.lo + kT - 1) / kT;
  const bool several = seg_s[0].hi < all.hi;  // segments that the CTA's rows are of
  auto stage = [&](int t) {
    const int y0 = all.lo + t * kT;
    stage_rows<T, D, kT, kGroup>(Y1, qkv, ld, (dq ? C : 0) + h * D, y0, all.hi, tid);
    if (dq) stage_rows<T, D, kT, kGroup>(Y2, qkv, ld, 2 * C + h * D, y0, all.hi, tid);
    else stage_rows<T, D, kT, kGroup>(Y2, dao, (long long)C, h * D, y0, all.hi, tid);
    cp_async_commit();
    if (!dq && tid < kT) {
      const bool in = y0 + tid < all.hi;
      s2[tid] = in ? lse[(long long)h * capacity + y0 + tid] : 0.f;
      s2[kT + tid] = in ? row_D(y0 + tid) : 0.f;
    }
  };
  if (grp < n_tiles) stage(grp);

  RowSeg mine[4];
  float my_lse[4] = {}, my_D[4] = {};
#pragma unroll
  for (int i = 0; i < 4; ++i) mine[i] = seg_s[ty + kTY * i];
  if (dq) {
    // lane tx < 4 fetches row ty + 8 tx, the others take it from there
    const int r = i0 + ty + kTY * (tx & 3);
    const float dv = r < Np ? row_D(r) : 0.f, lv = r < Np ? lse[(long long)h * capacity + r] : 0.f;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      my_D[i] = __shfl_sync(0xffffffffu, dv, i, kTX);
      my_lse[i] = __shfl_sync(0xffffffffu, lv, i, kTX);
    }
  }
  float acc1[4][W] = {}, acc2[4][W] = {};  // dQ | dK and dV
  own_rows_landed<1>(grp < n_tiles);
  for (int t = grp; t < n_tiles; t += kGroups) {
    cp_async_wait<0>();
    group_sync(grp);
    const int y0 = all.lo + t * kT;
    float s[4][4] = {}, dp[4][4] = {};
    dots<D>(s, A1, Y1, ty, tx);
    dots<D>(dp, A2, Y2, ty, tx);
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int c = tx + kTX * j, ya = y0 + c;
        const float l = dq ? my_lse[i] : s2[c], Dv = dq ? my_D[i] : s2[kT + c];
        const float p = (ya >= mine[i].lo && ya < mine[i].hi) ? expf(s[i][j] * scale - l) : 0.f;
        if (!dq) Ps[(ty + kTY * i) * kLdP + c] = p;
        dp[i][j] = p * (dp[i][j] - Dv);
      }
    const int n = all.hi - y0 < kT ? all.hi - y0 : kT;
    if (!dq) {
      __syncwarp();  // the rows of P and dS that this warp reads are the ones its own lanes wrote
      float tile[4][W] = {};
      weighted<D>(tile, Ps, Y2, n, ty, tx);
      add_to<W>(acc2, tile);
      __syncwarp();
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) Ps[(ty + kTY * i) * kLdP + tx + kTX * j] = dp[i][j];
    __syncwarp();
    float tile[4][W] = {};
    weighted<D>(tile, Ps, Y1, n, ty, tx);
    add_to<W>(acc1, tile);
    group_sync(grp);  // the stage is free
    if (t + kGroups < n_tiles) stage(t + kGroups);
  }
  if (kGroups > 1 && n_tiles == 1 && grp == 1) return;
  if (kGroups > 1 && n_tiles > 1) {  // the second group's share of every sum, in the memory of its stage
    float* part = A2 + kR * kLd<D> + 2 * kTile + tid;  // [8 W][kGroup]
    if (grp == 1) {
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int d = 0; d < W; ++d) {
          part[(i * W + d) * kGroup] = acc1[i][d];
          part[((4 + i) * W + d) * kGroup] = acc2[i][d];
        }
    }
    __syncthreads();
    if (grp == 1) return;
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int d = 0; d < W; ++d) {
        acc1[i][d] += part[(i * W + d) * kGroup];
        acc2[i][d] += part[((4 + i) * W + d) * kGroup];
      }
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int row = i0 + ty + kTY * i;
    if (row >= Np) continue;
    if (several && !(finite_sums<W>(acc1[i]) && finite_sums<W>(acc2[i]))) {
#pragma unroll
      for (int d = 0; d < W; ++d) acc1[i][d] = acc2[i][d] = 0.f;
#pragma unroll 1
      for (int k = mine[i].lo; k < mine[i].hi; ++k) {
        const int q = dq ? row : k, j = dq ? k : row;  // query and key of the pair
        const T *Q = qkv + q * ld + h * D, *K = qkv + j * ld + C + h * D, *dO = dao + (long long)q * C + h * D;
        const float p = expf(row_dot<T, D>(Q, K) * scale - lse[(long long)h * capacity + q]);
        const float ds = p * (row_dot<T, D>(dO, K + C) - row_dot<T, D>(dO, ao + (long long)q * C + h * D));
#pragma unroll
        for (int d = 0; d < W; ++d) {
          acc1[i][d] = fmaf(ds, to_f32<T>((dq ? K : Q)[tx * W + d]), acc1[i][d]);
          if (!dq) acc2[i][d] = fmaf(p, to_f32<T>(dO[tx * W + d]), acc2[i][d]);
        }
      }
    }
    T* dst = dqkv + (long long)row * ld + h * D + tx * W;
#pragma unroll
    for (int d = 0; d < W; ++d) acc1[i][d] *= scale;
    store_row<T, W>(dst + (dq ? 0 : C), acc1[i]);
    if (!dq) store_row<T, W>(dst + 2 * C, acc2[i]);
  }
}

template <typename T, int D, int kGroups>
int fwd_launch(const spa_params& p, const void* qkv, const int32_t* seg, int n_seg, void* ao, float* lse,
               cudaStream_t st) {
  auto kern = attn_fwd_simt_kernel<T, D, kGroups>;
  constexpr int kSmem = kFwdFloats<D, kGroups> * (int)sizeof(float);
  static DeviceOnce attr;
  cudaError_t e = attr.run([&] { return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem); });
  if (e != cudaSuccess) { set_cuda_error(e, "attn_fwd_simt_kernel"); return SPA_ERR_CUDA; }
  launch_pdl(kern, dim3((p.capacity + kR - 1) / kR, p.H), kGroups * kGroup, kSmem, st, (const T*)qkv, seg, n_seg, p.capacity, p.C,
             softmax_scale_of(p), (T*)ao, lse);
  SPA_CUDA_CHECK_LAUNCH("attn_fwd_simt_kernel");
  return SPA_OK;
}

template <typename T, int D, int kGroups>
int bwd_launch(const spa_params& p, const void* qkv, const void* ao, const float* lse, const void* dao,
               const int32_t* seg, int n_seg, void* dqkv, cudaStream_t st) {
  auto kern = attn_bwd_simt_kernel<T, D, kGroups>;
  constexpr int kSmem = kBwdFloats<D, kGroups> * (int)sizeof(float);
  static DeviceOnce attr;
  cudaError_t e = attr.run([&] { return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem); });
  if (e != cudaSuccess) { set_cuda_error(e, "attn_bwd_simt_kernel"); return SPA_ERR_CUDA; }
  launch_pdl(kern, dim3((p.capacity + kR - 1) / kR, p.H, 2), kGroups * kGroup, kSmem, st, (const T*)qkv, (const T*)ao, lse,
             (const T*)dao, seg, n_seg, p.capacity, p.C, softmax_scale_of(p), (T*)dqkv);
  SPA_CUDA_CHECK_LAUNCH("attn_bwd_simt_kernel");
  return SPA_OK;
}

// One group where the CTAs that the capacity may fill are many per SM: four of them run on an SM (three in the backward at
// d = 64) instead of two, and none has a second group that idles over an odd tile.  By the capacity, of which a part is rows: 12
// per SM, 6 where segments have 64 rows or fewer and most CTAs one tile (10 in the forward at d = 64, where few CTAs land unevenly).
// us, two groups -> one, forward and backward: 8 heads of 32, 64 images of 196 tokens, half selected, 55.7 -> 47.9 and 170 -> 151, a
// fifth 19.6 -> 16.2 and 51 -> 42; 4 x 4 200 tokens in containers of 49, two thirds selected, 64 -> 49 and 202 -> 158; 6 heads of 64, 64
// images 68 -> 63 and 245 -> 229.  Below the line: 3 heads of 32, 16 images 13.7 -> 14.9 and 26.9 -> 35.2, 6 of 64 23.3 -> 31.8 and
// 76.5 -> 80.4.  Not with more than 8 tiles, which two groups share evenly: 2 heads of 64, 4 images of 4 039 tokens 129 -> 132 and
// 360 -> 400.
bool one_group(const spa_params& p, int n_seg, bool forward) {
  const long long ctas = (long long)((p.capacity + kR - 1) / kR) * p.H * (forward ? 1 : 2), tile = (long long)kT * n_seg;
  const int per_sm = p.capacity > tile ? 12 : forward && p.C / p.H == 64 ? 10 : 6;
  return p.capacity <= 8 * tile && ctas >= per_sm * kNumSMs;
}

}  // namespace

#define SPA_SIMT_LAUNCH(WHICH, FORWARD, ...)                                                                               \
  const int d = p.C / p.H;                                                                                               \
  if (one_group(p, n_seg, FORWARD)) {                                                                                             \
    if (p.dtype == SPA_F32) return d == 32 ? WHICH<float, 32, 1>(__VA_ARGS__) : WHICH<float, 64, 1>(__VA_ARGS__);        \
    return d == 32 ? WHICH<__nv_bfloat16, 32, 1>(__VA_ARGS__) : WHICH<__nv_bfloat16, 64, 1>(__VA_ARGS__);                \
  }                                                                                                                      \
  if (p.dtype == SPA_F32) return d == 32 ? WHICH<float, 32, 2>(__VA_ARGS__) : WHICH<float, 64, 2>(__VA_ARGS__);          \
  return d == 32 ? WHICH<__nv_bfloat16, 32, 2>(__VA_ARGS__) : WHICH<__nv_bfloat16, 64, 2>(__VA_ARGS__)

int launch_attention_fwd_simt(const spa_params& p, const void* qkv, const int32_t* seg, int n_seg, void* ao,
                              float* lse, cudaStream_t st) {
  SPA_SIMT_LAUNCH(fwd_launch, true, p, qkv, seg, n_seg, ao, lse, st);
}

int launch_attention_bwd_simt(const spa_params& p, const void* qkv, const void* ao, const float* lse,
                              const void* dao, const int32_t* seg, int n_seg, void* dqkv, cudaStream_t st) {
  SPA_SIMT_LAUNCH(bwd_launch, false, p, qkv, ao, lse, dao, seg, n_seg, dqkv, st);
}
#undef SPA_SIMT_LAUNCH

}  // namespace spa
