// Gram matrix and right-hand sides of the row systems (Eq. 4):
//   G = A_x A_x^T (k_X x k_X) and R = A_y A_x^T (k_Y x k_X), per pair.
// 32 x 32 output tiles, 4 x 4 outputs per thread. A block's four or eight groups of 64 threads
// take every fourth or eighth slab of 16 features, and their sums are added in order at the
// end: a tile's chain is a quarter or an eighth of the feature dimension, and one pair of
// k = 200 is 28 + 49 tiles (64 x 64 tiles with one chain each leave most SMs idle on a few
// pairs and compute twice the outputs G has at k = 200). Launch times: one pair of k = 200,
// d = 256 0.073 -> 0.023 ms, four of d = 512 0.128 -> 0.037, the ragged 256-pair batch
// 0.417 -> 0.318; the double-float sums (10 FP32 operations a product) bound the last.
// G is symmetric: only its lower tiles are computed; each is written twice (transposed), and
// once more into a packed copy of the lower rows (each row up to the end of its 8 x 8
// diagonal block) that the row solves load into shared memory with a single bulk copy.
// For pairs flagged hi_gram (large k) G is accumulated in double-float
// arithmetic: every product is split exactly (fma) and summed with an
// error-free transformation, which keeps ~48 significant bits, as an FP64
// accumulation would, on the FP32 pipe (GB300's FP64 rate is a small fraction
// of its FP32 rate). The (hi, lo) pair is kept for the residual of iterative
// refinement, and hi + lo rounded to FP32 feeds the Cholesky factorisation.
#include "fmap_internal.cuh"
#include "tc_ptx.cuh"

namespace fmap {
namespace {

constexpr int kT = 32;         // tile edge
constexpr int kS = 16;         // features per slab
constexpr int kLd = kT + 4;

// (hi, lo) += a * b with an exact product and an error-free sum.
__device__ __forceinline__ void df_fma(float& hi, float& lo, float a, float b) {
  const float p = __fmul_rn(a, b);
  const float pe = fmaf(a, b, -p);
  const float s = __fadd_rn(hi, p);
  const float bb = __fsub_rn(s, hi);
  const float e = __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bb)), __fsub_rn(p, bb));
  hi = s;
  lo = __fadd_rn(lo, __fadd_rn(e, pe));
}

// (hi, lo) += (h2, l2), the sum of the heads kept exactly.
__device__ __forceinline__ void df_add(float& hi, float& lo, float h2, float l2) {
  const float s = __fadd_rn(hi, h2);
  const float bb = __fsub_rn(s, hi);
  const float e = __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bb)), __fsub_rn(h2, bb));
  hi = s;
  lo = __fadd_rn(__fadd_rn(lo, l2), e);
}

// Barrier of one group of 64 threads (constant ids: a variable one reserves all sixteen).
template <int kGroups>
__device__ __forceinline__ void group_sync(int g) {
#pragma unroll
  for (int u = 0; u < kGroups; ++u)
    if (g == u) tc::named_barrier_sync(1 + u, 64);
}

template <int kGroups>
struct GramSmem {
  union {
    float slab[kGroups][2][2][kS][kLd];        // group, buffer, operand, feature, row
    float part[2][kGroups][kT][kT];            // (hi, lo), group, row, column
  };
};

// out[i][j] = sum_f X[i0 + i][f] Y[j0 + j][f] for one tile (X has kx rows, Y ky), left as the
// groups' (hi, lo) sums in sm.part. Ends with a block barrier.
template <bool kDF, int kGroups>
__device__ __forceinline__ void gram_tile(GramSmem<kGroups>& sm, const float* X, const float* Y, int kx, int ky, int d, int i0,
                                          int j0) {
  const int tid = threadIdx.x, g = tid >> 6, t = tid & 63, tx = t & 7, ty = t >> 3;
  float hi[4][4], lo[4][4];
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) { hi[a][b] = 0.f; lo[a][b] = 0.f; }
  // thread t loads features 4 (t & 3) .. + 3 of rows t / 4 and t / 4 + 16 (any d and alignment:
  // the allocation-free solve takes descriptors as they come)
  const int lr = t >> 2, lc = 4 * (t & 3);
  const bool vec = ((reinterpret_cast<uintptr_t>(X) | reinterpret_cast<uintptr_t>(Y)) & 15) == 0 && (d & 3) == 0;
  float4 rx[2], ry[2];
  auto load4 = [&](const float* M, int rows, int r, int f) {
    if (r >= rows || f >= d) return make_float4(0.f, 0.f, 0.f, 0.f);
    const float* q = M + (int64_t)r * d + f;
    if (vec) return __ldg(reinterpret_cast<const float4*>(q));
    return make_float4(__ldg(q), f + 1 < d ? __ldg(q + 1) : 0.f, f + 2 < d ? __ldg(q + 2) : 0.f,
                       f + 3 < d ? __ldg(q + 3) : 0.f);
  };
  auto fetch = [&](int f0) {
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      rx[u] = load4(X, kx, i0 + lr + 16 * u, f0 + lc);
      ry[u] = load4(Y, ky, j0 + lr + 16 * u, f0 + lc);
    }
  };
  const int nslab = (d + kS - 1) / kS;
  if (g < nslab) fetch(g * kS);
  int buf = 0;
  for (int sl = g; sl < nslab; sl += kGroups, buf ^= 1) {
    float(*sx)[kLd] = sm.slab[g][buf][0];
    float(*sy)[kLd] = sm.slab[g][buf][1];
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int r = lr + 16 * u;
      sx[lc][r] = rx[u].x; sx[lc + 1][r] = rx[u].y; sx[lc + 2][r] = rx[u].z; sx[lc + 3][r] = rx[u].w;
      sy[lc][r] = ry[u].x; sy[lc + 1][r] = ry[u].y; sy[lc + 2][r] = ry[u].z; sy[lc + 3][r] = ry[u].w;
    }
    group_sync<kGroups>(g);   // (the other buffer's readers passed it one slab ago)
    if (sl + kGroups < nslab) fetch((sl + kGroups) * kS);
#pragma unroll 4
    for (int c = 0; c < kS; ++c) {
      const float4 xa = *reinterpret_cast<const float4*>(&sx[c][ty * 4]);
      const float4 yb = *reinterpret_cast<const float4*>(&sy[c][tx * 4]);
      const float xv[4] = {xa.x, xa.y, xa.z, xa.w};
      const float yv[4] = {yb.x, yb.y, yb.z, yb.w};
#pragma unroll
      for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) {
          if (kDF)
            df_fma(hi[a][b], lo[a][b], xv[a], yv[b]);
          else
            hi[a][b] = fmaf(xv[a], yv[b], hi[a][b]);
        }
    }
  }
  __syncthreads();   // every group has read its slabs
#pragma unroll
  for (int a = 0; a < 4; ++a) {
    *reinterpret_cast<float4*>(&sm.part[0][g][4 * ty + a][4 * tx]) = make_float4(hi[a][0], hi[a][1], hi[a][2], hi[a][3]);
    if (kDF)
      *reinterpret_cast<float4*>(&sm.part[1][g][4 * ty + a][4 * tx]) = make_float4(lo[a][0], lo[a][1], lo[a][2], lo[a][3]);
  }
  __syncthreads();
}

template <int kGroups>
__global__ void __launch_bounds__(64 * kGroups) gram_kernel(BatchDev b, const float* a, float* ws) {
  extern __shared__ __align__(16) uint8_t gram_smem[];
  GramSmem<kGroups>& sm = *reinterpret_cast<GramSmem<kGroups>*>(gram_smem);
  const PairDev pd = b.pairs[blockIdx.y];
  const int k = pd.k, d = pd.d;
  const int nt = (k + kT - 1) / kT;
  const float* ax = a + b.shapes[pd.x].a_off;
  const float* ay = a + b.shapes[pd.y].a_off;
  // thread t finishes columns 4 (t & 7) .. + 3 of row t / 8 of the tile
  const int row = threadIdx.x >> 3, col = 4 * (threadIdx.x & 7);
  const bool fin = row < kT;
  if (blockIdx.z == 0) {
    // G: lower tiles only (ti >= tj), mirrored on store
    int t = blockIdx.x, ti = 0;
    while (t > ti) { t -= ti + 1; ++ti; }
    const int tj = t;
    if (ti >= nt) return;
    const int i0 = ti * kT, j0 = tj * kT;
    float* g = ws + pd.g_off;
    float* gp = g + gram_packed_off(k);   // the same values in the row solves' packed layout
    const int ldg = gram_ld(k);
    float2* ghl = pd.hi_gram ? reinterpret_cast<float2*>(ws) + pd.g64_off : nullptr;
    if (pd.hi_gram)
      gram_tile<true, kGroups>(sm, ax, ax, k, k, d, i0, j0);
    else
      gram_tile<false, kGroups>(sm, ax, ax, k, k, d, i0, j0);
    float v[4];
#pragma unroll
    for (int q = 0; fin && q < 4; ++q) {
      float hi = sm.part[0][0][row][col + q], lo = ghl ? sm.part[1][0][row][col + q] : 0.f;
#pragma unroll
      for (int u = 1; u < kGroups; ++u) {
        const float h2 = sm.part[0][u][row][col + q];
        if (ghl)
          df_add(hi, lo, h2, sm.part[1][u][row][col + q]);
        else
          hi += h2;
      }
      float e = 0.f;
      v[q] = hi;
      if (ghl) {
        v[q] = __fadd_rn(hi, lo);
        e = __fsub_rn(lo, __fsub_rn(v[q], hi));
      }
      const int i = i0 + row, j = j0 + col + q;
      if (i >= k || j >= k) continue;
      g[(int64_t)i * ldg + j] = v[q];
      if (j <= (i | 7)) gp[rowoff(i) + j] = v[q];
      if (ghl && j <= i) ghl[(int64_t)i * k + j] = make_float2(v[q], e);   // the solves read its lower triangle
    }
    // the transposed half, and the entries right of the diagonal inside the packed rows' blocks
    __syncthreads();
    float(*tr)[kT + 1] = reinterpret_cast<float(*)[kT + 1]>(&sm.part[0][0][0][0]);
#pragma unroll
    for (int q = 0; fin && q < 4; ++q) tr[col + q][row] = v[q];
    __syncthreads();
#pragma unroll
    for (int q = 0; fin && q < 4; ++q) {
      const int j = j0 + row, i = i0 + col + q;      // G_ji = G_ij
      if (i >= k || j >= k) continue;
      g[(int64_t)j * ldg + i] = tr[row][col + q];
      if (i <= (j | 7)) gp[rowoff(j) + i] = tr[row][col + q];
    }
  } else {
    // R = A_y A_x^T (ky x k): every tile
    const int ky = b.shapes[pd.y].k, nty = (ky + kT - 1) / kT;
    if ((int)blockIdx.x >= nty * nt) return;
    const int i0 = (blockIdx.x / nt) * kT, j0 = (blockIdx.x % nt) * kT;
    gram_tile<false, kGroups>(sm, ay, ax, ky, k, d, i0, j0);
    float* r = ws + pd.r_off;
#pragma unroll
    for (int q = 0; fin && q < 4; ++q) {
      const int i = i0 + row, j = j0 + col + q;
      float v = sm.part[0][0][row][col + q];
#pragma unroll
      for (int u = 1; u < kGroups; ++u) v += sm.part[0][u][row][col + q];
      if (i < ky && j < k) r[(int64_t)i * k + j] = v;
    }
  }
}

}  // namespace

cudaError_t gram_set_smem() {
  return cudaFuncSetAttribute(gram_kernel<8>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(GramSmem<8>));
}

cudaError_t launch_gram(const BatchDev& b, int max_k, int max_d, bool hi_gram, const float* a, float* ws,
                        cudaStream_t st, bool with_r) {
  if (b.n_pairs <= 0) return cudaSuccess;
  // Four groups, or eight where a tile's chain bounds the launch: double-float sums while G has at most a
  // tile per SM, FP32 sums of 256 features or more while all tiles together leave a third of the SMs
  // idle. us, four / eight: one, 4, 8 pairs of k = 200, d = 512 37 / 33, 60 / 40, 64 / 68, one, 2, 4 of k = 300
  // 41 / 33, 60 / 41, 64 / 68, 4 of k = 64, d = 384 with double-float sums 30 / 27, 16 of k = 100 47 / 47; FP32
  // sums, d = 512, one, 2, 4 of k = 199 14.2 / 13.4, 18.4 / 18.6, 24 / 27, one and 8 of k = 100 14.1 / 13.1,
  // 18.5 / 20.3, one of k = 100, d = 128 8.2 / 8.6.
  // G first: its double-float tiles are the longest
  const int nt = (max_k + kT - 1) / kT;
  dim3 grid(nt * nt, b.n_pairs, with_r ? 2 : 1);
  const int64_t g_tiles = (int64_t)nt * (nt + 1) / 2 * b.n_pairs, tiles = g_tiles + (with_r ? (int64_t)nt * nt * b.n_pairs : 0);
  if (hi_gram ? g_tiles <= 152 : (tiles <= 100 && max_d >= 256))
    gram_kernel<8><<<grid, 512, sizeof(GramSmem<8>), st>>>(b, a, ws);
  else
    gram_kernel<4><<<grid, 256, sizeof(GramSmem<4>), st>>>(b, a, ws);
  return cudaGetLastError();
}

}  // namespace fmap
