// A pair's map C is k_Y x k_X: k_X = pd.k (shape x, row-system size, columns of C) and
// k_Y = the basis size of shape y (rows of C); the paper's maps are square.
//
// Adjoint of the row-wise solve (given Gamma from the adjoint row solves):
// W = Gamma^T C + C^T Gamma, dA_x = Gamma^T A_y - W A_x, dA_y = Gamma A_x,
// dD = -lambda Gamma o C, dlambda = -sum(D o Gamma o C); the per-shape gather of
// dA contributions; the training loss; the status clear.
#include <math.h>

#include <algorithm>
#include <vector>

#include "fmap_internal.cuh"
#include "simt_tile.cuh"

namespace fmap {
namespace {

__device__ __forceinline__ float mask_entry(const PairDev& pd, const float* evx, const float* evy, int i, int a) {
  if (pd.mask) return pd.mask[(int64_t)i * pd.k + a];
  const float t = evy[i] - evx[a];
  return t * t;
}

// ---------------------------------------------------------------- adjoint GEMMs
// Batches that are too small for launch_adjoint_tc, on simt::tile_gemm. Launch times of the two
// together, 64 x 64 tiles with one chain and one buffer each -> these: one pair of k = 200, d = 256 62 ->
// 23 us, one of k = 300, d = 512 88 -> 38, 4 of k = 200, d = 512 72 -> 48, 8 of k = 100, d = 512 44 -> 31,
// 32 of k = 100 80 -> 71; the two launches of the loss 48 -> 21 at k = 300, 32 pairs of k = 200 97 -> 74.
using simt::Operand;
using simt::out_col;
using simt::out_row;
using simt::Tile;

// W = Gamma^T C + C^T Gamma (k_X x k_X; Gamma and C are k_Y x k_X).
template <int kT>
__global__ void __launch_bounds__(simt::kThreads) adjoint_w_kernel(BatchDev b, const float* c_flat, float* ws) {
  __shared__ __align__(16) typename Tile<kT>::Smem sm;
  const PairDev pd = b.pairs[blockIdx.y];
  const int k = pd.k, ky = b.shapes[pd.y].k;   // Gamma, C: ky x k
  const int nt = (k + kT - 1) / kT;
  if ((int)blockIdx.x >= nt * nt) return;
  const int a0 = (blockIdx.x / nt) * kT, b0 = (blockIdx.x % nt) * kT;
  const Operand gam{ws + pd.gam_off, k, k, ky}, c{c_flat + pd.c_off, k, k, ky};
  float v[Tile<kT>::kRows][4];
  simt::tile_gemm<kT, simt::kAcross, simt::kAcross>(sm, gam, c, c, gam, 1.f, a0, b0, v);
  const int j = b0 + out_col<kT>();
#pragma unroll
  for (int u = 0; u < Tile<kT>::kRows; ++u) {
    const int i = a0 + out_row<kT>(u);
    float* w = ws + pd.w_off + (int64_t)i * k + j;
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (i < k && j + q < k) w[q] = v[u][q];
  }
}

// The mask gradient dD = -lambda_i Gamma o C (when d_mask is given; lambda_i = lambda
// without row weights), dlambda_p = -sum_ij D_ij Gamma_ij C_ij (when d_lambda is given;
// with row weights the sum of the per-row gradients) and, for pairs with row weights and an
// output for them, dlambda_i = -sum_j D_ij Gamma_ij C_ij (one warp per row, lanes in a fixed
// order); over the k_Y x k_X entries, fixed-order block reductions (one block per pair).
__global__ void __launch_bounds__(256) adjoint_dlambda_kernel(BatchDev b, const float* c_flat, float* d_mask,
                                                              float* d_lambda, const float* ws) {
  __shared__ float red[256];
  const int p = blockIdx.x;
  const PairDev pd = b.pairs[p];
  const int k = pd.k, ky = b.shapes[pd.y].k, n = ky * pd.k;   // the ky x k entries
  const float* gam = ws + pd.gam_off;
  const float* cm = c_flat + pd.c_off;
  const float* evx = b.shapes[pd.x].evals;
  const float* evy = b.shapes[pd.y].evals;
  if (d_mask)
    for (int e = threadIdx.x; e < n; e += 256) {
      const float lam = pd.lam_rows ? pd.lam_rows[e / k] : pd.lam;
      d_mask[pd.c_off + e] = -lam * gam[e] * cm[e];
    }
  if (pd.dlam_rows) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int i = warp; i < ky; i += 8) {
      float acc = 0.f;
      for (int j = lane; j < k; j += 32) {
        const int e = i * k + j;
        acc = fmaf(mask_entry(pd, evx, evy, i, j) * gam[e], cm[e], acc);
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
      if (lane == 0) pd.dlam_rows[i] = -acc;
    }
  }
  if (!d_lambda) return;
  float acc = 0.f;
  for (int e = threadIdx.x; e < n; e += 256) {
    const int i = e / k, j = e % k;
    acc = fmaf(mask_entry(pd, evx, evy, i, j) * gam[e], cm[e], acc);
  }
  red[threadIdx.x] = acc;
  __syncthreads();
  for (int s = 128; s > 0; s >>= 1) {
    if ((int)threadIdx.x < s) red[threadIdx.x] += red[threadIdx.x + s];
    __syncthreads();
  }
  if (threadIdx.x == 0) d_lambda[p] = -red[0];
}

// Per-pair contributions (Gamma is k_Y x k_X, W k_X x k_X and symmetric):
//   which 0: dA_x = Gamma^T A_y - W A_x   (k_X x d, into sx_off)
//   which 1: dA_y = Gamma A_x             (k_Y x d, into sy_off)
template <int kT>
__global__ void __launch_bounds__(simt::kThreads) adjoint_da_kernel(BatchDev b, const float* a_flat, float* ws) {
  __shared__ __align__(16) typename Tile<kT>::Smem sm;
  const PairDev pd = b.pairs[blockIdx.y];
  const int k = pd.k, ky = b.shapes[pd.y].k, d = pd.d;
  const int which = blockIdx.z;
  const int rows = which == 0 ? k : ky;                    // rows of the contribution
  const int ntf = (d + kT - 1) / kT, nta = (rows + kT - 1) / kT;
  if ((int)blockIdx.x >= ntf * nta) return;
  const int a0 = (blockIdx.x / ntf) * kT, f0 = (blockIdx.x % ntf) * kT;
  const float* gam = ws + pd.gam_off;
  const Operand ax{a_flat + b.shapes[pd.x].a_off, d, d, k}, ay{a_flat + b.shapes[pd.y].a_off, d, d, ky};
  float v[Tile<kT>::kRows][4];
  if (which == 0)
    simt::tile_gemm<kT, simt::kAcross, simt::kAcross>(sm, Operand{gam, k, k, ky}, ay, Operand{ws + pd.w_off, k, k, k}, ax, -1.f, a0, f0, v);
  else
    simt::tile_gemm<kT, simt::kQuads, simt::kAcross>(sm, Operand{gam, k, ky, k}, ax, Operand{nullptr, 0, 0, 0}, Operand{nullptr, 0, 0, 0},
                                     1.f, a0, f0, v);
  const int f = f0 + out_col<kT>();
  float* out = ws + (which == 0 ? pd.sx_off : pd.sy_off) + f;
#pragma unroll
  for (int u = 0; u < Tile<kT>::kRows; ++u) {
    const int i = a0 + out_row<kT>(u);
    // d is a multiple of 16 and the contributions are 256-byte aligned
    if (i < rows && f < d) *reinterpret_cast<float4*>(out + (int64_t)i * d) = make_float4(v[u][0], v[u][1], v[u][2], v[u][3]);
  }
}

// dA_s = sum of the shape's contributions, in pair order. Each thread sums four
// consecutive entries (one float4 per contribution when the shape's output is 16-byte
// aligned; the contribution slots always are).
__global__ void gather_da_kernel(BatchDev b, float* d_a, const float* ws) {
  const ShapeDev s = b.shapes[blockIdx.y];
  const int64_t kd = (int64_t)s.k * s.d;
  const int64_t e0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) * 4;
  if (e0 >= kd) return;
  float* out = d_a + s.a_off;
  const bool vec = ((kd & 3) == 0) && ((reinterpret_cast<uintptr_t>(out) & 15) == 0);
  if (vec) {
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int q = s.slot_beg; q < s.slot_end; ++q) {
      const float4 u = *reinterpret_cast<const float4*>(ws + b.slot_list[q] + e0);
      acc.x += u.x; acc.y += u.y; acc.z += u.z; acc.w += u.w;
    }
    *reinterpret_cast<float4*>(out + e0) = acc;
  } else {
    for (int j = 0; j < 4 && e0 + j < kd; ++j) {
      float acc = 0.f;
      for (int q = s.slot_beg; q < s.slot_end; ++q) acc += ws[b.slot_list[q] + e0 + j];
      out[e0 + j] = acc;
    }
  }
}

// Training loss ||C C^T - I||^2 + ||C - C_gt||^2 and dL/dC = 4 (C C^T - I) C + 2 (C - C_gt),
// as two tiled passes over (output tile, pair):
//   pass 1: E = C C^T - I (into the workspace) and per-tile partial sums of the loss;
//   pass 2: dC = 4 E C + 2 (C - C_gt); tile 0 of each pair adds the partials in a fixed order.

template <int kT>
__global__ void __launch_bounds__(simt::kThreads) loss_e_kernel(BatchDev b, const float* c_flat, const float* gt_flat,
                                                                float* ws, float* partial) {
  __shared__ __align__(16) typename Tile<kT>::Smem sm;
  __shared__ float red[simt::kThreads];
  const int p = blockIdx.y;
  const PairDev pd = b.pairs[p];
  const int k = pd.k, ky = b.shapes[pd.y].k;   // C is ky x k, E = C C^T - I is ky x ky
  // tiles over ky rows and max(ky, k) columns: E where the column is < ky, the
  // ||C - C_gt||^2 term where it is < k
  const int nta = (ky + kT - 1) / kT, ntb = (max(ky, k) + kT - 1) / kT;
  if ((int)blockIdx.x >= nta * ntb) return;
  const int a0 = (blockIdx.x / ntb) * kT, b0 = (blockIdx.x % ntb) * kT;
  const float* c = c_flat + pd.c_off;
  const float* gt = gt_flat + pd.c_off;
  float* e = ws + pd.e_off;
  const int tid = threadIdx.x;
  const Operand none{nullptr, 0, 0, 0};
  const Operand cr{c, k, ky, b0 < ky ? k : 0};   // no products in the tiles past E's columns
  float v[Tile<kT>::kRows][4];
  simt::tile_gemm<kT, simt::kLanes, simt::kLanes>(sm, cr, cr, none, none, 1.f, a0, b0, v);
  float part = 0.f;
#pragma unroll
  for (int u = 0; u < Tile<kT>::kRows; ++u) {
    const int a = a0 + out_row<kT>(u);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int bb = b0 + out_col<kT>() + j;
      if (a < ky && bb < k) {
        const float r = c[(int64_t)a * k + bb] - gt[(int64_t)a * k + bb];
        part = fmaf(r, r, part);
      }
      if (a < ky && bb < ky) {
        const float x = v[u][j] - (a == bb ? 1.f : 0.f);
        e[(int64_t)a * ky + bb] = x;
        part = fmaf(x, x, part);
      }
    }
  }
  red[tid] = part;
  __syncthreads();
  for (int st = simt::kThreads / 2; st > 0; st >>= 1) {
    if (tid < st) red[tid] += red[tid + st];
    __syncthreads();
  }
  if (tid == 0) partial[(int64_t)p * kMaxLossTiles + blockIdx.x] = red[0];
}

template <int kT>
__global__ void __launch_bounds__(simt::kThreads) loss_grad_kernel(BatchDev b, const float* c_flat, const float* gt_flat,
                                                                   float* loss, float* d_c, const float* ws,
                                                                   const float* partial) {
  __shared__ __align__(16) typename Tile<kT>::Smem sm;
  const int p = blockIdx.y;
  const PairDev pd = b.pairs[p];
  const int k = pd.k, ky = b.shapes[pd.y].k;
  const int nta = (ky + kT - 1) / kT, ntb = (k + kT - 1) / kT;
  if (blockIdx.x == 0 && threadIdx.x < 32 && loss) {
    // the partial sums of loss_e's tiles: a lane's in tile order, then across the lanes
    const int nte = nta * ((max(ky, k) + kT - 1) / kT);
    float total = 0.f;
    for (int t = threadIdx.x; t < nte; t += 32) total += partial[(int64_t)p * kMaxLossTiles + t];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) total += __shfl_xor_sync(0xffffffffu, total, o);
    if (threadIdx.x == 0) loss[p] = total;
  }
  if (d_c == nullptr) return;
  // dC = 4 E C + 2 (C - C_gt): ky x k tiles, reduction over ky
  if ((int)blockIdx.x >= nta * ntb) return;
  const int a0 = (blockIdx.x / ntb) * kT, b0 = (blockIdx.x % ntb) * kT;
  const float* c = c_flat + pd.c_off;
  const float* gt = gt_flat + pd.c_off;
  const Operand none{nullptr, 0, 0, 0};
  float v[Tile<kT>::kRows][4];
  simt::tile_gemm<kT, simt::kLanes, simt::kAcross>(sm, Operand{ws + pd.e_off, ky, ky, ky}, Operand{c, k, k, ky}, none, none, 1.f, a0, b0, v);
#pragma unroll
  for (int u = 0; u < Tile<kT>::kRows; ++u) {
    const int a = a0 + out_row<kT>(u);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int bb = b0 + out_col<kT>() + j;
      if (a >= ky || bb >= k) continue;
      const int64_t idx = (int64_t)a * k + bb;
      d_c[pd.c_off + idx] = 4.f * v[u][j] + 2.f * (c[idx] - gt[idx]);
    }
  }
}

__global__ void status_clear_kernel(int32_t* status, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) status[i] = 0;
}

}  // namespace

namespace {

// Tiles of edge t of an m x n output.
int64_t tiles_of(int m, int n, int t) { return (int64_t)((m + t - 1) / t) * ((n + t - 1) / t); }
int slabs_of(int len) { return (len + simt::kS - 1) / simt::kS; }

}  // namespace

// Which tile, for both: 64 x 64 once the 32 x 32 tiles are more than the SMs hold at a time (six
// blocks each) and at least 3.2 times as many (an edge that 64 pads to much more than 32 does stays
// with 32). Times in us, 32 / 64: the loss of 32, 48, 64, 128 pairs of k = 100 26 / 26, 31 / 34, 38 / 35,
// 62 / 52, of 16 and 32 of k = 250 58 / 56, 103 / 91, of 64 of k = 90 (ratio 2.25) 26 / 32; the adjoint
// (d = 512) of 12, 24, 48 of k = 100 41 / 43, 65 / 60, 121 / 101, of 16 and 32 of k = 128 52 / 56,
// 88 / 82, of 32 and 64 of k = 64 32 / 32, 53 / 47, of 32 of k = 77 (ratio 3) 48 / 51, of 32 and 64 of k = 150
// (ratio 3.3) 133 / 135, 249 / 242. For the adjoint the line is at fifteen tiles of dA per SM (its reductions
// are longer) and a ratio of 3.5.
SimtChoice loss_simt_choice(const std::vector<int3>& shapes) {
  int64_t n32 = 0, n64 = 0, w32 = 0, w64 = 0;   // tiles of E; tiles times slabs of both launches
  for (const int3& q : shapes) {
    const int k = q.x, ky = q.y;
    n32 += tiles_of(ky, std::max(k, ky), 32);
    n64 += tiles_of(ky, std::max(k, ky), 64);
    w32 += tiles_of(ky, ky, 32) * slabs_of(k) + tiles_of(ky, k, 32) * slabs_of(ky);
    w64 += tiles_of(ky, ky, 64) * slabs_of(k) + tiles_of(ky, k, 64) * slabs_of(ky);
  }
  if (n32 > 6 * 152 && 10 * n32 > 32 * n64) return {64, 10.0 + 4.75e-3 * (double)w64};
  return {32, 10.0 + 1.55e-3 * (double)w32};
}

SimtChoice adjoint_simt_choice(const std::vector<int3>& shapes) {
  int64_t n32 = 0, n64 = 0, w32 = 0, w64 = 0;   // tiles of dA; tiles times slabs of both launches
  for (const int3& q : shapes) {
    const int k = q.x, ky = q.y, d = q.z;
    n32 += tiles_of(k, d, 32) + tiles_of(ky, d, 32);
    n64 += tiles_of(k, d, 64) + tiles_of(ky, d, 64);
    const int sw = 2 * slabs_of(ky), sx = slabs_of(ky) + slabs_of(k), sy = slabs_of(k);
    w32 += tiles_of(k, k, 32) * sw + tiles_of(k, d, 32) * sx + tiles_of(ky, d, 32) * sy;
    w64 += tiles_of(k, k, 64) * sw + tiles_of(k, d, 64) * sx + tiles_of(ky, d, 64) * sy;
  }
  if (n32 > 15 * 152 && 10 * n32 > 35 * n64) return {64, 15.0 + 4.7e-3 * (double)w64};
  return {32, 10.0 + 1.5e-3 * (double)w32};
}

cudaError_t launch_adjoint_gemms(const BatchDev& b, int max_k, int max_d, const float* a, const float* c,
                                 float* d_mask, float* d_lambda, bool row_grads, float* ws, int simt_tile,
                                 cudaStream_t st) {
  if (b.n_pairs <= 0) return cudaSuccess;
  auto tiles = [&](int n) { return (n + simt_tile - 1) / simt_tile; };
  cudaError_t e;
  if (simt_tile) {
    const dim3 grid(tiles(max_k) * tiles(max_k), b.n_pairs);
    if (simt_tile == 64)
      adjoint_w_kernel<64><<<grid, simt::kThreads, 0, st>>>(b, c, ws);
    else
      adjoint_w_kernel<32><<<grid, simt::kThreads, 0, st>>>(b, c, ws);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  if (d_lambda || d_mask || row_grads) {
    adjoint_dlambda_kernel<<<b.n_pairs, 256, 0, st>>>(b, c, d_mask, d_lambda, ws);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  if (!simt_tile) return cudaSuccess;
  const dim3 grid(tiles(max_k) * tiles(max_d), b.n_pairs, 2);
  if (simt_tile == 64)
    adjoint_da_kernel<64><<<grid, simt::kThreads, 0, st>>>(b, a, ws);
  else
    adjoint_da_kernel<32><<<grid, simt::kThreads, 0, st>>>(b, a, ws);
  return cudaGetLastError();
}

cudaError_t launch_gather_da(const BatchDev& b, int max_kd, float* d_a, const float* ws, cudaStream_t st) {
  if (b.n_shapes <= 0) return cudaSuccess;
  gather_da_kernel<<<dim3((max_kd + 1023) / 1024, b.n_shapes), 256, 0, st>>>(b, d_a, ws);
  return cudaGetLastError();
}

cudaError_t launch_loss_orth(const BatchDev& b, int max_k, const float* c, const float* c_gt, float* loss,
                             float* d_c, float* ws, float* partial, int simt_tile, cudaStream_t st) {
  if (b.n_pairs <= 0) return cudaSuccess;
  const int nt = (max_k + simt_tile - 1) / simt_tile;
  const dim3 grid(nt * nt, b.n_pairs);
  if (simt_tile == 64)
    loss_e_kernel<64><<<grid, simt::kThreads, 0, st>>>(b, c, c_gt, ws, partial);
  else
    loss_e_kernel<32><<<grid, simt::kThreads, 0, st>>>(b, c, c_gt, ws, partial);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  if (simt_tile == 64)
    loss_grad_kernel<64><<<grid, simt::kThreads, 0, st>>>(b, c, c_gt, loss, d_c, ws, partial);
  else
    loss_grad_kernel<32><<<grid, simt::kThreads, 0, st>>>(b, c, c_gt, loss, d_c, ws, partial);
  return cudaGetLastError();
}

cudaError_t launch_status_clear(int32_t* status, int n, cudaStream_t st) {
  if (n <= 0 || status == nullptr) return cudaSuccess;
  status_clear_kernel<<<(n + 255) / 256, 256, 0, st>>>(status, n);
  return cudaGetLastError();
}

}  // namespace fmap
