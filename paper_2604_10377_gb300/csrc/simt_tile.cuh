// Output tiles of FP32 GEMMs on the CUDA cores, 256 threads, 4 x 4 outputs per thread, slabs of 16
// reduction indices through shared memory:
//   32 x 32  four groups of 64 threads take every fourth slab, and their sums are added in order at the
//            end. For batches that do not fill the SMs, where the chain of a tile (a global load, a
//            slab through shared memory, 16 steps of FMAs, a barrier) bounds a launch: it is a quarter
//            as long, and spread over four times the SMs.
//   64 x 64  one group of 256 threads takes every slab: half the loads per product.
#pragma once

#include <stdint.h>

#include "tc_ptx.cuh"

namespace fmap {
namespace simt {

constexpr int kS = 16;         // reduction indices per slab
constexpr int kThreads = 256;

template <int kTile>
struct Tile {
  static_assert(kTile == 32 || kTile == 64, "tile edge");
  static constexpr int kGroup = (kTile / 4) * (kTile / 4);     // threads of a group
  static constexpr int kGroups = kThreads / kGroup;
  static constexpr int kPer = kTile * kS / 4 / kGroup;         // quads of an operand's slab per thread
  static constexpr int kLd = kTile + 4;
  static constexpr int kRows = kTile * kTile / 4 / kThreads;   // quads of the tile per thread at the end
  union Smem {
    float slab[kGroups][2][2][kS][kLd];                        // group, buffer, operand, reduction index, row
    float part[kGroups > 1 ? kGroups : 1][kGroups > 1 ? kTile : 1][kTile];   // group, row, column
  };
};

// Row and first column, within the tile, of quad i of this thread's results.
template <int kTile>
__device__ __forceinline__ int out_row(int i) {
  return kTile == 32 ? threadIdx.x >> 3 : 4 * (threadIdx.x >> 4) + i;
}
template <int kTile>
__device__ __forceinline__ int out_col() {
  return 4 * (threadIdx.x & (kTile / 4 - 1));
}

// An operand: element (r, m) of `rows` x `len` (r an output row or column, m the reduction index)
// at p[m ld + r] (kAcross) or p[r ld + m]. The latter is read in quads of a row, which take few addresses (the
// adjoint's dA_y at d = 512: 4 pairs of k = 100 23 us against 25, 128 of k = 64 71 against 75), or by 16
// lanes along a row, whose loads touch a quarter of the lines (the loss, where both operands are so: 128
// pairs of k = 100 72 -> 62 us in tiles of 32, 58 -> 52 in tiles of 64).
enum Layout { kAcross, kQuads, kLanes };
struct Operand {
  const float* p;
  int64_t ld;
  int rows, len;
};

template <int kTile>
__device__ __forceinline__ void group_sync(int g) {   // constant ids: a variable one reserves all sixteen
  if (Tile<kTile>::kGroups == 1) {
    __syncthreads();
  } else {
#pragma unroll
    for (int u = 0; u < Tile<kTile>::kGroups; ++u)
      if (g == u) tc::named_barrier_sync(1 + u, Tile<kTile>::kGroup);
  }
}

// Row and reduction index, within the slab, of value j of quad u of thread t of a group.
template <int kTile, Layout kL>
__device__ __forceinline__ void slab_at(int t, int u, int j, int& r, int& m) {
  constexpr int kG = Tile<kTile>::kGroup, kQ = kTile / 4;
  if (kL == kAcross) {
    r = 4 * (t & (kQ - 1)) + j;
    m = t / kQ + kG / kQ * u;
  } else if (kL == kQuads) {
    r = (t >> 2) + kG / 4 * u;
    m = 4 * (t & 3) + j;
  } else {
    r = (t >> 4) + kG / 16 * (4 * u + j);
    m = t & 15;
  }
}

template <int kTile, Layout kL>
__device__ __forceinline__ void fetch_slab(const Operand& o, int r0, int m0, int t, float (&v)[Tile<kTile>::kPer][4]) {
#pragma unroll
  for (int u = 0; u < Tile<kTile>::kPer; ++u) {
    int r, m;
    slab_at<kTile, kL>(t, u, 0, r, m);
    r += r0;
    m += m0;
    const float* q = kL == kAcross ? o.p + (int64_t)m * o.ld + r : o.p + (int64_t)r * o.ld + m;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      if (kL == kLanes) {
        slab_at<kTile, kL>(t, u, j, r, m);
        r += r0;
        m += m0;
        v[u][j] = r < o.rows && m < o.len ? __ldg(o.p + (int64_t)r * o.ld + m) : 0.f;
      } else {
        v[u][j] = (kL == kAcross ? m < o.len && r + j < o.rows : r < o.rows && m + j < o.len) ? __ldg(q + j) : 0.f;
      }
    }
  }
}

template <int kTile, Layout kL>
__device__ __forceinline__ void store_slab(float (*s)[Tile<kTile>::kLd], int t, const float (&v)[Tile<kTile>::kPer][4]) {
#pragma unroll
  for (int u = 0; u < Tile<kTile>::kPer; ++u) {
    int r, m;
    if (kL == kAcross) {
      slab_at<kTile, kL>(t, u, 0, r, m);
      *reinterpret_cast<float4*>(&s[m][r]) = make_float4(v[u][0], v[u][1], v[u][2], v[u][3]);
    } else {
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        slab_at<kTile, kL>(t, u, j, r, m);
        s[m][r] = v[u][j];
      }
    }
  }
}

// sum_m X1(i0 + i, m) Y1(j0 + j, m) + sign2 sum_m X2(i0 + i, m) Y2(j0 + j, m) for one tile (the
// second term absent when X2.len is 0): out[q] is the quad at (out_row(q), out_col()).
template <int kTile, Layout kX, Layout kY>
__device__ __forceinline__ void tile_gemm(typename Tile<kTile>::Smem& sm, const Operand& x1, const Operand& y1,
                                          const Operand& x2, const Operand& y2, float sign2, int i0, int j0,
                                          float (&out)[Tile<kTile>::kRows][4]) {
  using T = Tile<kTile>;
  const int tid = threadIdx.x, g = tid / T::kGroup, t = tid & (T::kGroup - 1);
  const int tx = t & (kTile / 4 - 1), ty = t / (kTile / 4);
  float acc[4][4] = {};
  const int n1 = (x1.len + kS - 1) / kS, n = n1 + (x2.len + kS - 1) / kS;
  float rx[T::kPer][4], ry[T::kPer][4];
  auto fetch = [&](int sl) {
    const bool second = sl >= n1;
    const int m0 = (second ? sl - n1 : sl) * kS;
    fetch_slab<kTile, kX>(second ? x2 : x1, i0, m0, t, rx);
    fetch_slab<kTile, kY>(second ? y2 : y1, j0, m0, t, ry);
  };
  if (g < n) fetch(g);
  int buf = 0;
  for (int sl = g; sl < n; sl += T::kGroups, buf ^= 1) {
    float(*sx)[T::kLd] = sm.slab[g][buf][0];
    float(*sy)[T::kLd] = sm.slab[g][buf][1];
    if (sl >= n1) {
#pragma unroll
      for (int u = 0; u < T::kPer; ++u)
#pragma unroll
        for (int j = 0; j < 4; ++j) rx[u][j] *= sign2;
    }
    store_slab<kTile, kX>(sx, t, rx);
    store_slab<kTile, kY>(sy, t, ry);
    group_sync<kTile>(g);   // (the other buffer's readers passed it one slab ago)
    if (sl + T::kGroups < n) fetch(sl + T::kGroups);
#pragma unroll
    for (int c = 0; c < kS; ++c) {
      const float4 xa = *reinterpret_cast<const float4*>(&sx[c][ty * 4]);
      const float4 yb = *reinterpret_cast<const float4*>(&sy[c][tx * 4]);
      const float xv[4] = {xa.x, xa.y, xa.z, xa.w}, yv[4] = {yb.x, yb.y, yb.z, yb.w};
#pragma unroll
      for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) acc[a][b] = fmaf(xv[a], yv[b], acc[a][b]);
    }
  }
  if constexpr (T::kGroups == 1) {
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int b = 0; b < 4; ++b) out[a][b] = acc[a][b];
  } else {
    __syncthreads();   // every group has read its slabs
#pragma unroll
    for (int a = 0; a < 4; ++a)
      *reinterpret_cast<float4*>(&sm.part[g][4 * ty + a][4 * tx]) = make_float4(acc[a][0], acc[a][1], acc[a][2], acc[a][3]);
    __syncthreads();
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int u = 0; u < T::kGroups; ++u) {
      const float4 w = *reinterpret_cast<const float4*>(&sm.part[u][out_row<kTile>(0)][out_col<kTile>()]);
      v.x += w.x; v.y += w.y; v.z += w.z; v.w += w.w;
    }
    out[0][0] = v.x; out[0][1] = v.y; out[0][2] = v.z; out[0][3] = v.w;
  }
}

}  // namespace simt
}  // namespace fmap
