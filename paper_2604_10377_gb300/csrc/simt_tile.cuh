// 32 x 32 output tiles of small FP32 GEMMs on the CUDA cores, 256 threads, 4 x 4 outputs per
// thread: four groups of 64 threads take every fourth slab of 16 reduction indices, and their
// sums are added in order at the end. The batches these serve do not fill the SMs, so the chain
// of a tile (a global load, a slab through shared memory, 16 steps of FMAs, a barrier) bounds a
// launch; the split makes it a quarter as long as one chain per tile, and a tile a quarter of
// 64 x 64 spreads it over four times the SMs.
#pragma once

#include <stdint.h>

#include "tc_ptx.cuh"

namespace fmap {
namespace simt {

constexpr int kT = 32;         // tile edge
constexpr int kS = 16;         // reduction indices per slab
constexpr int kGroups = 4;
constexpr int kThreads = 64 * kGroups;
constexpr int kLd = kT + 4;

union Smem {
  float slab[kGroups][2][2][kS][kLd];   // group, buffer, operand, reduction index, row
  float part[kGroups][kT][kT];          // group, row, column
};

// An operand: element (r, m) of `rows` x `len` (r an output row or column, m the reduction index)
// at p[r ld + m] (kContig) or p[m ld + r].
struct Operand {
  const float* p;
  int64_t ld;
  int rows, len;
};

__device__ __forceinline__ void group_sync(int g) {   // constant ids: a variable one reserves all sixteen
#pragma unroll
  for (int u = 0; u < kGroups; ++u)
    if (g == u) tc::named_barrier_sync(1 + u, 64);
}

// Slab values of thread t (0 .. 63): two quads. kContig: indices m0 + 4 (t & 3) .. + 3 of rows
// r0 + t / 4 and + 16; else rows r0 + 4 (t & 7) .. + 3 of indices m0 + t / 8 and + 8.
template <bool kContig>
__device__ __forceinline__ void fetch_slab(const Operand& o, int r0, int m0, int t, float (&v)[2][4]) {
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    const int r = kContig ? r0 + (t >> 2) + 16 * u : r0 + 4 * (t & 7);
    const int m = kContig ? m0 + 4 * (t & 3) : m0 + (t >> 3) + 8 * u;
    const float* q = kContig ? o.p + (int64_t)r * o.ld + m : o.p + (int64_t)m * o.ld + r;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const bool ok = kContig ? (r < o.rows && m + j < o.len) : (m < o.len && r + j < o.rows);
      v[u][j] = ok ? __ldg(q + j) : 0.f;
    }
  }
}

template <bool kContig>
__device__ __forceinline__ void store_slab(float (*s)[kLd], int t, const float (&v)[2][4]) {
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    if (kContig) {
      const int r = (t >> 2) + 16 * u, m = 4 * (t & 3);
#pragma unroll
      for (int j = 0; j < 4; ++j) s[m + j][r] = v[u][j];
    } else {
      *reinterpret_cast<float4*>(&s[(t >> 3) + 8 * u][4 * (t & 7)]) = make_float4(v[u][0], v[u][1], v[u][2], v[u][3]);
    }
  }
}

// sum_m X1(i0 + i, m) Y1(j0 + j, m) + sign2 sum_m X2(i0 + i, m) Y2(j0 + j, m) for one tile (the
// second term absent when X2.len is 0). Thread t returns columns 4 (t & 7) .. + 3 of row t / 8.
template <bool kXContig, bool kYContig>
__device__ __forceinline__ float4 tile_gemm(Smem& sm, const Operand& x1, const Operand& y1, const Operand& x2,
                                            const Operand& y2, float sign2, int i0, int j0) {
  const int tid = threadIdx.x, g = tid >> 6, t = tid & 63, tx = t & 7, ty = t >> 3;
  float acc[4][4] = {};
  const int n1 = (x1.len + kS - 1) / kS, n = n1 + (x2.len + kS - 1) / kS;
  float rx[2][4], ry[2][4];
  auto fetch = [&](int sl) {
    const bool second = sl >= n1;
    const int m0 = (second ? sl - n1 : sl) * kS;
    fetch_slab<kXContig>(second ? x2 : x1, i0, m0, t, rx);
    fetch_slab<kYContig>(second ? y2 : y1, j0, m0, t, ry);
  };
  if (g < n) fetch(g);
  int buf = 0;
  for (int sl = g; sl < n; sl += kGroups, buf ^= 1) {
    float(*sx)[kLd] = sm.slab[g][buf][0];
    float(*sy)[kLd] = sm.slab[g][buf][1];
    if (sl >= n1) {
#pragma unroll
      for (int u = 0; u < 2; ++u)
#pragma unroll
        for (int j = 0; j < 4; ++j) rx[u][j] *= sign2;
    }
    store_slab<kXContig>(sx, t, rx);
    store_slab<kYContig>(sy, t, ry);
    group_sync(g);   // (the other buffer's readers passed it one slab ago)
    if (sl + kGroups < n) fetch(sl + kGroups);
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
  __syncthreads();   // every group has read its slabs
#pragma unroll
  for (int a = 0; a < 4; ++a)
    *reinterpret_cast<float4*>(&sm.part[g][4 * ty + a][4 * tx]) = make_float4(acc[a][0], acc[a][1], acc[a][2], acc[a][3]);
  __syncthreads();
  float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
  for (int u = 0; u < kGroups; ++u) {
    const float4 w = *reinterpret_cast<const float4*>(&sm.part[u][tid >> 3][4 * (tid & 7)]);
    v.x += w.x; v.y += w.y; v.z += w.z; v.w += w.w;
  }
  return v;
}

}  // namespace simt
}  // namespace fmap
