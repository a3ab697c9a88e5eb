// Row-wise regularised solve (Eq. 5-9) and the adjoint row solves.
//
// One thread block per row system S_i = G + lambda diag(D_i) (row i of pair p).
// S_i is padded to kp = k rounded up to 8 (identity in the padding) and kept in
// shared memory as packed lower rows (rowoff: row a holds 8 (a/8 + 1) + 4 floats, so a
// row's 8-column tile segment is two aligned float4 and consecutive rows fall on
// different banks). The Gram kernel leaves G in that layout too, so one bulk copy
// loads it; then lambda D_i is added to the diagonal. Two factorisations, chosen per
// class of k at launch_solve, both blocked right-looking Cholesky in FP32 with 8-column
// panels and the right-hand side as a bordered row:
//   chol_solve_kernel  trailing matrix in shared memory, updated in 8x4 or 4x4 register
//                      tiles, S_AB -= L_AJ L_BJ^T, two columns per packed FP32x2 FMA (each
//                      lane of the pair rounds like a scalar fmaf); warp 0 factors the next
//                      diagonal block meanwhile (one panel of lookahead). Two block barriers
//                      per panel, every thread solves one row of the panel.
//   chol_reg_kernel    trailing matrix in registers (factor_registers).
// What bounds them is the chain of the panels (25 at k = 200), not a pipe: a panel is an
// 8-pivot block (about 400 cycles of dependent square roots), a row solve against it and a
// rank-8 update, each behind a barrier and a round trip of shared memory, 2360 cycles alone on
// an SM at k = 200 in the register kernel, and two systems fit an SM.
// The substitutions after the factorisation work on 16-row blocks in a unit block form whose
// steps hold no inverse (scale_blocks): 4.1k cycles per triangular solve at k = 200 against 12k
// with an inverse in every step. `ir_steps` steps of iterative refinement take the residual
// rhs - S x in FP32, for hi_gram pairs with G as the two FP32 halves (hi + lo) of its
// double-float accumulation.
#include <math.h>

#include "fmap_internal.cuh"
#include "tc_ptx.cuh"

namespace fmap {
namespace {

// Rounds of 128 columns that cover a row of G in the refinement residual of chol_solve_kernel.
constexpr int kResRounds = (kSolveBounds[4] + 127) / 128;

// Floats of one factor: the packed rows plus the Q inverse diagonal blocks.
__host__ __device__ __forceinline__ int factor_floats(int Q) { return 32 * Q * (Q + 2) + 64 * Q; }

__device__ __forceinline__ float mask_entry(const PairDev& pd, const float* evx, const float* evy, int i, int a) {
  if (pd.mask) return pd.mask[(int64_t)i * pd.k + a];
  const float t = evy[i] - evx[a];
  return t * t;
}

__device__ __forceinline__ void set_status(int32_t* status, int p, int32_t code) {
  if (status) atomicCAS(status + p, 0, code);
}

// Warp 0: factor the 8 x 8 diagonal block J in place and store its inverse. Lanes
// 0-7 each factor the block in registers (the same arithmetic on every lane, loads
// broadcast), then lane c forms column c of L_JJ^-1 from its own registers. Returns
// false on a bad pivot.
__device__ __forceinline__ bool diag_block(float* S, float* linv, int J, int lane) {
  const int r0 = 8 * J;
  bool bad = false;
  if (lane < 8) {
    float a[8][8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const float4* rp = reinterpret_cast<const float4*>(S + rowoff(r0 + i) + r0);
      const float4 u0 = rp[0], u1 = rp[1];
      a[i][0] = u0.x; a[i][1] = u0.y; a[i][2] = u0.z; a[i][3] = u0.w;
      a[i][4] = u1.x; a[i][5] = u1.y; a[i][6] = u1.z; a[i][7] = u1.w;
    }
    float rinv[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const float piv = a[j][j];
      if (!(piv > 0.f) || !(piv < INFINITY)) bad = true;
      const float r = rsqrtf(piv);     // 1 / L_jj; iterative refinement absorbs its last-bit error
      a[j][j] = piv * r;
      rinv[j] = r;
#pragma unroll
      for (int i = j + 1; i < 8; ++i) a[i][j] *= r;
#pragma unroll
      for (int i = j + 1; i < 8; ++i)
#pragma unroll
        for (int m = j + 1; m <= i; ++m) a[i][m] = fmaf(-a[i][j], a[m][j], a[i][m]);
    }
    // column `lane` of L_JJ^-1: forward substitution on the unit vector
    float x[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      float t = (i == lane) ? 1.f : 0.f;
#pragma unroll
      for (int m = 0; m < i; ++m) t = fmaf(-a[i][m], x[m], t);
      x[i] = (i >= lane) ? t * rinv[i] : 0.f;
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) linv[J * 64 + i * 8 + lane] = x[i];
    if (lane == 0) {
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        float4* rp = reinterpret_cast<float4*>(S + rowoff(r0 + i) + r0);
        rp[0] = make_float4(a[i][0], a[i][1], a[i][2], a[i][3]);
        rp[1] = make_float4(a[i][4], a[i][5], a[i][6], a[i][7]);
      }
    }
  }
  bad = __shfl_sync(0xffffffffu, bad ? 1 : 0, 0) != 0;
  __syncwarp();
  return !bad;
}

// Row index of entry t of a lower triangle enumerated row by row (t = a(a+1)/2 + b).
__device__ __forceinline__ void tri_decode(int t, int& a, int& b) {
  int ai = (int)((sqrtf(8.f * (float)t + 1.f) - 1.f) * 0.5f);
  while ((ai + 1) * (ai + 2) / 2 <= t) ++ai;
  while (ai * (ai + 1) / 2 > t) --ai;
  a = ai;
  b = t - ai * (ai + 1) / 2;
}

__device__ __forceinline__ uint64_t pk2(float x, float y) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y));
  return r;
}
__device__ __forceinline__ void upk2(uint64_t v, float& x, float& y) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(v));
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}

// S[A.., B..] -= L[A.., J] L[B.., J]^T for one R x C tile (R, C in {4, 8}), with the
// panel's 8 columns read from `pan` (column-major, leading dimension kp). Pairs of
// columns are updated with packed FP32x2 FMAs.
template <int R, int C>
__device__ __forceinline__ void trail_tile(float* S, const float* pan, int kp, int A, int B) {
  uint64_t acc[R][C / 2];
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const float4* sr = reinterpret_cast<const float4*>(S + rowoff(A + r) + B);
#pragma unroll
    for (int h = 0; h < C / 4; ++h) {
      const float4 u = sr[h];
      acc[r][2 * h] = pk2(u.x, u.y); acc[r][2 * h + 1] = pk2(u.z, u.w);
    }
  }
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    float la[R];
    uint64_t lb[C / 2];
    const float4* pa = reinterpret_cast<const float4*>(pan + c * kp + A);
    const float4* pb = reinterpret_cast<const float4*>(pan + c * kp + B);
#pragma unroll
    for (int h = 0; h < R / 4; ++h) {
      const float4 u = pa[h];
      la[4 * h] = -u.x; la[4 * h + 1] = -u.y; la[4 * h + 2] = -u.z; la[4 * h + 3] = -u.w;
    }
#pragma unroll
    for (int h = 0; h < C / 4; ++h) {
      const float4 u = pb[h];
      lb[2 * h] = pk2(u.x, u.y); lb[2 * h + 1] = pk2(u.z, u.w);
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const uint64_t l2 = pk2(la[r], la[r]);
#pragma unroll
      for (int q = 0; q < C / 2; ++q) acc[r][q] = fma2(l2, lb[q], acc[r][q]);
    }
  }
#pragma unroll
  for (int r = 0; r < R; ++r) {
    float4* sr = reinterpret_cast<float4*>(S + rowoff(A + r) + B);
#pragma unroll
    for (int h = 0; h < C / 4; ++h) {
      float x0, x1, x2, x3;
      upk2(acc[r][2 * h], x0, x1); upk2(acc[r][2 * h + 1], x2, x3);
      sr[h] = make_float4(x0, x1, x2, x3);
    }
  }
}

// The triangular solves work on 16-row blocks p (rows 16p .. 16p+15; the last block has
// 8 rows when Q is odd). The inverse of a 16-row diagonal block is formed from the two
// 8x8 inverses A^-1, B^-1 and the block below the diagonal L21:
//   [A 0; L21 B]^-1 = [A^-1 0; M B^-1] with M = -B^-1 L21 A^-1,
// and M (64 floats per 16-row block) is computed once per factor: one thread per column j
// of a block forms T = L21 (column j of A^-1), then column j of M = -B^-1 T.
__device__ __forceinline__ void load8(const float* src, float (&d)[8]) {
  const float4 u0 = reinterpret_cast<const float4*>(src)[0], u1 = reinterpret_cast<const float4*>(src)[1];
  d[0] = u0.x; d[1] = u0.y; d[2] = u0.z; d[3] = u0.w;
  d[4] = u1.x; d[5] = u1.y; d[6] = u1.z; d[7] = u1.w;
}

__device__ __forceinline__ void store8(float* dst, const float (&d)[8]) {
  reinterpret_cast<float4*>(dst)[0] = make_float4(d[0], d[1], d[2], d[3]);
  reinterpret_cast<float4*>(dst)[1] = make_float4(d[4], d[5], d[6], d[7]);
}

__device__ __forceinline__ void pair_blocks_prepare(const float* S, const float* linv, float* mo, int Q, int tid,
                                                    int nt) {
  const int np = Q >> 1;   // 16-row blocks with two 8-row halves
  for (int e = tid; e < np * 8; e += nt) {
    const int p = e >> 3, j = e & 7;
    const float* Ai = linv + (2 * p) * 64;        // A^-1, row-major
    const float* Bi = linv + (2 * p + 1) * 64;    // B^-1
    float ac[8];
#pragma unroll
    for (int l = 0; l < 8; ++l) ac[l] = Ai[l * 8 + j];
    float T[8];
#pragma unroll
    for (int m = 0; m < 8; ++m) {
      // (L21 A^-1)[m][j]
      float l21[8];
      load8(S + rowoff(16 * p + 8 + m) + 16 * p, l21);
      float t = 0.f;
#pragma unroll
      for (int l = 0; l < 8; ++l) t = fmaf(l21[l], ac[l], t);
      T[m] = t;
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      float bi[8];
      load8(Bi + i * 8, bi);
      float acc = 0.f;
#pragma unroll
      for (int m = 0; m < 8; ++m) acc = fmaf(bi[m], T[m], acc);
      mo[p * 64 + i * 8 + j] = -acc;
    }
  }
}

// Triangular solves with L = Lt D, D the 16-row diagonal blocks of L and Lt unit block lower:
// the rows below block p are scaled once, Lt_ap = L_ap D_p^-1, and S x = b is then
// Lt z = b, w = D^-T D^-1 z (every block at once), Lt^T x = w. No inverse stands between two
// steps of a solve, and a step is one block barrier, 16 FMAs and a store per row.
//
// Lt_ap in place of L_ap: one lane per row, 32 rows of one block per warp pass.
__device__ __forceinline__ void scale_blocks(float* S, const float* linv, const float* mo, int Q, int warp, int nw,
                                             int lane) {
  const int kp = 8 * Q, nb = (Q + 1) >> 1;
  int t = warp;
  for (int p = 0; p + 1 < nb; ++p) {
    const int rows = kp - 16 * (p + 1), groups = (rows + 31) >> 5;
    for (; t < groups; t += nw) {
      const int a = 16 * (p + 1) + 32 * t + lane;
      if (a >= kp) continue;
      float* row = S + rowoff(a) + 16 * p;
      const float* Ai = linv + 128 * p;
      float x0[8], x1[8], o0[8], o1[8];
      load8(row, x0);
      load8(row + 8, x1);
#pragma unroll
      for (int c = 0; c < 8; ++c) { o0[c] = 0.f; o1[c] = 0.f; }
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        float ar[8], mr[8], br[8];
        load8(Ai + 8 * j, ar);
        load8(mo + 64 * p + 8 * j, mr);
        load8(Ai + 64 + 8 * j, br);
#pragma unroll
        for (int c = 0; c < 8; ++c) {
          if (c <= j) o0[c] = fmaf(x0[j], ar[c], o0[c]);
          o0[c] = fmaf(x1[j], mr[c], o0[c]);
          if (c <= j) o1[c] = fmaf(x1[j], br[c], o1[c]);
        }
      }
      store8(row, o0);
      store8(row + 8, o1);
    }
    t -= groups;
  }
}

// v <- Lt^-1 v (thread t owns row t; NT >= kp). Ends with v complete after the caller's barrier.
__device__ __forceinline__ void unit_fwd(const float* S, float* v, int Q, int tid) {
  const int kp = 8 * Q, nb = (Q + 1) >> 1;
  float t = tid < kp ? v[tid] : 0.f;
  const float* row = S + rowoff(tid < kp ? tid : 0);
  for (int p = 0; p + 1 < nb; ++p) {
    const bool on = tid >= 16 * (p + 1) && tid < kp;
    float l[16];
    if (on) {
      load8(row + 16 * p, *reinterpret_cast<float(*)[8]>(l));
      load8(row + 16 * p + 8, *reinterpret_cast<float(*)[8]>(l + 8));
    }
    __syncthreads();                   // block p of v is final
    if (on) {
      float z[16];
      load8(v + 16 * p, *reinterpret_cast<float(*)[8]>(z));
      load8(v + 16 * p + 8, *reinterpret_cast<float(*)[8]>(z + 8));
      float s[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int q = 0; q < 16; ++q) s[q & 3] = fmaf(l[q], z[q], s[q & 3]);
      t -= (s[0] + s[1]) + (s[2] + s[3]);
      if (tid < 16 * (p + 2)) v[tid] = t;
    }
  }
  __syncthreads();
}

// v <- Lt^-T v, blocks from the last to the first.
__device__ __forceinline__ void unit_bwd(const float* S, float* v, int Q, int tid) {
  const int kp = 8 * Q, nb = (Q + 1) >> 1;
  float t = tid < kp ? v[tid] : 0.f;
  for (int p = nb - 1; p >= 1; --p) {
    const bool on = tid < 16 * p, two = 2 * p + 1 < Q;
    float l[16];
    if (on) {
      const float* c0 = S + rowoff(16 * p) + tid;
      const float* c1 = S + rowoff(16 * p + 8) + tid;
      const int ld = 16 * p + 12;
#pragma unroll
      for (int q = 0; q < 8; ++q) l[q] = c0[q * ld];
#pragma unroll
      for (int q = 0; q < 8; ++q) l[8 + q] = two ? c1[q * (ld + 8)] : 0.f;
    }
    __syncthreads();                   // block p of v is final
    if (on) {
      float z[16];
      load8(v + 16 * p, *reinterpret_cast<float(*)[8]>(z));
      if (two) load8(v + 16 * p + 8, *reinterpret_cast<float(*)[8]>(z + 8));
      float s[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int q = 0; q < 16; ++q) s[q & 3] = fmaf(l[q], (q < 8 || two) ? z[q] : 0.f, s[q & 3]);
      t -= (s[0] + s[1]) + (s[2] + s[3]);
      if (tid >= 16 * (p - 1)) v[tid] = t;
    }
  }
  __syncthreads();
}

// v <- D^-T D^-1 v, or D^-T v alone (both_sides false): thread t, row t; a 16-row block lies in
// one warp. The caller's barrier orders v before and after.
__device__ __forceinline__ void block_diag_solve(const float* linv, const float* mo, float* v, int Q, int tid,
                                                 bool both_sides) {
  const int kp = 8 * Q, p = tid >> 4, i = tid & 15, r0 = 16 * p;
  const bool on = tid < kp, two = 2 * p + 1 < Q, lowr = i >= 8;
  const float* Ai = linv + 128 * p;
  const float* Bi = Ai + 64;
  const float* Mp = mo + 64 * p;
  if (both_sides) {
    float y = 0.f;
    if (on) {
      float a[8], z[8];
      load8((lowr ? Mp : Ai) + 8 * (i & 7), a);
      load8(v + r0, z);
#pragma unroll
      for (int j = 0; j < 8; ++j) y = fmaf(a[j], z[j], y);
      if (lowr) {
        load8(Bi + 8 * (i & 7), a);
        load8(v + r0 + 8, z);
#pragma unroll
        for (int j = 0; j < 8; ++j) y = fmaf(a[j], z[j], y);
      }
    }
    __syncwarp();
    if (on) v[tid] = y;
    __syncwarp();
  }
  float y = 0.f;
  if (on) {
    float z[8];
    if (!lowr) {
      load8(v + r0, z);
#pragma unroll
      for (int j = 0; j < 8; ++j) y = fmaf(Ai[8 * j + i], z[j], y);
    }
    if (two) {
      load8(v + r0 + 8, z);
      const float* m = lowr ? Bi : Mp;
#pragma unroll
      for (int j = 0; j < 8; ++j) y = fmaf(m[8 * j + (i & 7)], z[j], y);
    }
  }
  __syncwarp();
  if (on) v[tid] = y;
}

template <int NT>
__global__ void __launch_bounds__(NT, (NT >= 256 ? 2 : (NT >= 128 ? 4 : 8)))
    chol_solve_kernel(BatchDev b, const int2* systems, int first, int count, int mode, const float* rhs_flat,
                      float* out_flat, float* saved, int32_t* status, float* ws, int gs_ok) {
  constexpr int NW = NT / 32;
  extern __shared__ __align__(16) float smem[];
  __shared__ int s_bad;
  __shared__ __align__(8) uint64_t s_bar;   // bulk copies of the Gram rows
  __shared__ int s_abort;
  if ((int)blockIdx.x >= count) return;
  const int2 sys = systems[first + blockIdx.x];
  const int p = sys.x, i = sys.y;
  const PairDev pd = b.pairs[p];
  const int k = pd.k;
  const int Q = (k + 7) >> 3, kp = 8 * Q;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const float* evx = b.shapes[pd.x].evals;
  const float* evy = b.shapes[pd.y].evals;
  const int ssz = rowoff(kp);
  float* S = smem;                 // packed skewed lower rows
  float* linv = S + ssz;           // inverse diagonal blocks, Q x 64
  float* pan = linv + 64 * Q;      // current panel, column-major: pan[c * kp + a]
  float* v = pan + 8 * kp;         // working vector
  float* xs = v + kp;              // solution
  float* rh = xs + kp;             // right-hand side
  float* dg = rh + kp;             // lambda D_i (the diagonal shift of this row system)
  float* Gs = dg + kp;             // copy of G for the refinement residual (launches with gs_ok)
  const float* G = ws + pd.g_off;
  const int ldg = gram_ld(k);
  const float2* Ghl = pd.g64_off >= 0 ? reinterpret_cast<const float2*>(ws) + pd.g64_off : nullptr;
  const float* rhs = (mode == kSolveForward) ? ws + pd.r_off + (int64_t)i * k : rhs_flat + pd.c_off + (int64_t)i * k;
  float* out = (mode == kSolveForward) ? out_flat + pd.c_off + (int64_t)i * k : ws + pd.gam_off + (int64_t)i * k;
  const int fsz = factor_floats(Q);
  float* fac = (saved != nullptr && pd.fac_off >= 0) ? saved + pd.fac_off + (int64_t)i * fsz : nullptr;
  const float lam = pd.lam_rows ? pd.lam_rows[i] : pd.lam;   // row weight of this system
  const int n_ir = mode == kSolveForward ? b.ir_steps : b.ir_steps_adj;
  // small FP32-Gram systems keep G in shared memory for the refinement residual
  const bool use_gs = gs_ok != 0 && Ghl == nullptr && n_ir > 0;
  const uint32_t gs_bytes = use_gs ? (uint32_t)k * (uint32_t)ldg * 4u : 0u;

  if (tid == 0) {
    s_bad = 0;
    s_abort = 0;
    tc::mbar_init(&s_bar, 1);
    tc::fence_mbar_init();
    // a projection wait that timed out leaves its error in the workspace's first word
    if (i == 0 && reinterpret_cast<const int*>(ws)[0] != 0) set_status(status, p, FMAP_ERR_TIMEOUT);
  }
  for (int a = tid; a < kp; a += NT) {
    rh[a] = a < k ? rhs[a] : 0.f;
    dg[a] = a < k ? lam * mask_entry(pd, evx, evy, i, a) : 0.f;
  }

  if (mode == kSolveAdjoint && fac != nullptr) {
    // the saved factor (packed rows and inverse blocks) and, for refinement, G: bulk copies
    __syncthreads();   // barrier initialised
    if (tid == 0) {
      tc::mbar_arrive_expect_tx(&s_bar, (uint32_t)fsz * 4u + gs_bytes);
      tc::bulk_g2s(S, fac, (uint32_t)fsz * 4u, &s_bar);
      if (use_gs) tc::bulk_g2s(Gs, G, gs_bytes, &s_bar);
    }
    tc::mbar_wait(&s_bar, 0, &s_abort);
    __syncthreads();
    if (s_abort) {
      // a copy that never completed: report, give it a bounded time to land, leave (every
      // thread of the block takes this branch together)
      if (tid == 0) set_status(status, p, FMAP_ERR_TIMEOUT);
      const uint64_t t0 = tc::globaltimer();
      while (!tc::mbar_try_wait(&s_bar, 0) && tc::globaltimer() - t0 < tc::kWaitTimeoutNs) {}
      return;
    }
  } else {
    // S = G + lambda diag(D_i). The Gram kernel left rows 0 .. k-1 of G in this packed
    // layout (each row up to the end of its diagonal block; the entries above the
    // diagonal inside a diagonal block are never read): one bulk copy brings them in
    // (with G itself for the residual when it stays in shared memory). Padding rows are
    // identity rows, written meanwhile.
    __syncthreads();   // barrier initialised
    if (tid == 0) {
      const uint32_t s_bytes = (uint32_t)rowoff(k) * 4u;
      tc::mbar_arrive_expect_tx(&s_bar, s_bytes + gs_bytes);
      tc::bulk_g2s(S, G + gram_packed_off(k), s_bytes, &s_bar);
      if (use_gs) tc::bulk_g2s(Gs, G, gs_bytes, &s_bar);
    }
    for (int a = k + tid; a < kp; a += NT) {
      float* row = S + rowoff(a);
      for (int c = 0; c < (a & ~7) + 8; ++c) row[c] = (c == a) ? 1.f : 0.f;
    }
    tc::mbar_wait(&s_bar, 0, &s_abort);
    __syncthreads();   // every thread's copies are visible
    if (s_abort) {
      if (tid == 0) set_status(status, p, FMAP_ERR_TIMEOUT);
      const uint64_t t0 = tc::globaltimer();
      while (!tc::mbar_try_wait(&s_bar, 0) && tc::globaltimer() - t0 < tc::kWaitTimeoutNs) {}
      return;
    }
    for (int a = tid; a < k; a += NT) S[rowoff(a) + a] += dg[a];
    for (int a = tid; a < kp; a += NT) v[a] = rh[a];   // right-hand side, reduced during the factorisation
    __syncthreads();
    if (warp == 0 && !diag_block(S, linv, 0, lane) && lane == 0) s_bad = 1;
    __syncthreads();
    for (int J = 0; J < Q && !s_bad; ++J) {
      const int r0 = 8 * J;
      const float* li = linv + J * 64;
      // forward substitution, bordered into the factorisation: y_J = L_JJ^-1 v_J, on the
      // last warp when it has no panel rows (off the TRSM's critical path), else warp 0
      const int yw = (r0 + 8 + (NW - 1) * 32 >= kp) ? NW - 1 : 0;
      if (warp == yw) {
        float y = 0.f;
        if (lane < 8)
#pragma unroll
          for (int j = 0; j < 8; ++j) y = fmaf(li[lane * 8 + j], v[r0 + j], y);
        __syncwarp();
        if (lane < 8) v[r0 + lane] = y;
      }
      // TRSM: rows below the diagonal block, x = s L_JJ^-T. Thread t owns row r0 + 8 + t
      // (every launch has NT >= kp threads) here and in (a), which reuses x.
      const int ar = r0 + 8 + tid;
      float x[8];
      if (ar < kp) {
        float4* ra = reinterpret_cast<float4*>(S + rowoff(ar) + r0);
        const float4 s0 = ra[0], s1 = ra[1];
        const float sv[8] = {s0.x, s0.y, s0.z, s0.w, s1.x, s1.y, s1.z, s1.w};
        const float4* l4 = reinterpret_cast<const float4*>(li);
#pragma unroll
        for (int c = 0; c < 8; ++c) {
          const float4 q0 = l4[2 * c];
          float lr[8] = {q0.x, q0.y, q0.z, q0.w, 0.f, 0.f, 0.f, 0.f};
          if (c >= 4) {
            const float4 q1 = l4[2 * c + 1];
            lr[4] = q1.x; lr[5] = q1.y; lr[6] = q1.z; lr[7] = q1.w;
          }
          float t = 0.f;
#pragma unroll
          for (int m = 0; m <= c; ++m) t = fmaf(sv[m], lr[m], t);
          x[c] = t;
        }
        ra[0] = make_float4(x[0], x[1], x[2], x[3]);
        ra[1] = make_float4(x[4], x[5], x[6], x[7]);
#pragma unroll
        for (int c = 0; c < 8; ++c) pan[c * kp + ar] = x[c];
      }
      __syncthreads();
      if (J + 1 == Q) break;
      // (a) the next column block, one row per thread; the row's right-hand side
      // takes the panel's contribution, v_a -= L_aJ y_J
      const int n0 = r0 + 8;
      if (ar < kp) {
        float4* ra = reinterpret_cast<float4*>(S + rowoff(ar) + n0);
        const float4 u0 = ra[0], u1 = ra[1];
        float acc[8] = {u0.x, u0.y, u0.z, u0.w, u1.x, u1.y, u1.z, u1.w};
        const float4 y0 = reinterpret_cast<const float4*>(v + r0)[0], y1 = reinterpret_cast<const float4*>(v + r0)[1];
        const float yv[8] = {y0.x, y0.y, y0.z, y0.w, y1.x, y1.y, y1.z, y1.w};
        float va = v[ar];
#pragma unroll
        for (int c = 0; c < 8; ++c) {
          const float la = x[c];
          va = fmaf(-la, yv[c], va);
          const float4* pb = reinterpret_cast<const float4*>(pan + c * kp + n0);
          const float4 b0 = pb[0], b1 = pb[1];
          acc[0] = fmaf(-la, b0.x, acc[0]); acc[1] = fmaf(-la, b0.y, acc[1]);
          acc[2] = fmaf(-la, b0.z, acc[2]); acc[3] = fmaf(-la, b0.w, acc[3]);
          acc[4] = fmaf(-la, b1.x, acc[4]); acc[5] = fmaf(-la, b1.y, acc[5]);
          acc[6] = fmaf(-la, b1.z, acc[6]); acc[7] = fmaf(-la, b1.w, acc[7]);
        }
        ra[0] = make_float4(acc[0], acc[1], acc[2], acc[3]);
        ra[1] = make_float4(acc[4], acc[5], acc[6], acc[7]);
        v[ar] = va;
      }
      // (a) writes column block J+1 and (b)'s tiles touch only blocks J+2.. (both read the
      // panel), so no block barrier separates them: warp 0 updated the diagonal block's
      // rows itself (threads 0-7) and factors it right away
      __syncwarp();
      // (b) warp 0: next diagonal block; warps 1..: trailing tiles (A, B), J+2 <= B <= A < Q
      if (warp == 0) {
        if (!diag_block(S, linv, J + 1, lane) && lane == 0) s_bad = 1;
      } else {
        // trailing blocks (A, B), J+2 <= B <= A < Q, as 8x4 or 4x4 register tiles: the
        // size whose rounds over the NT - 32 threads cost the fewest instructions (8x8
        // tiles fit the registers only with a partly rolled panel loop and ran slower)
        const int m = Q - J - 2;
        const int nb = NT - 32, t0 = tid - 32, base = 8 * (J + 2);
        const int T84 = m * (m + 1), T44 = m * (2 * m + 1);
        const int c84 = (T84 + nb - 1) / nb * 296, c44 = (T44 + nb - 1) / nb * 152;
        if (c84 <= c44) {
          for (int t = t0; t < T84; t += nb) {
            int ai, bi;
            tri_decode(t >> 1, ai, bi);
            trail_tile<8, 4>(S, pan, kp, base + 8 * ai, base + 8 * bi + 4 * (t & 1));
          }
        } else {
          for (int t = t0; t < T44; t += nb) {
            int ai, bi;
            tri_decode(t, ai, bi);
            trail_tile<4, 4>(S, pan, kp, base + 4 * ai, base + 4 * bi);
          }
        }
      }
      __syncthreads();
    }
    if (s_bad) {
      if (tid == 0) set_status(status, p, FMAP_ERR_NOT_SPD | (i << 8));
      for (int a = tid; a < k; a += NT) out[a] = __int_as_float(0x7fc00000);
      return;
    }
  }

  // inverses of the 16-row diagonal blocks (their off-diagonal parts, in the panel's space)
  float* mo = pan;
  const bool load_factor = mode == kSolveAdjoint && fac != nullptr;
  pair_blocks_prepare(S, linv, mo, Q, tid, NT);
  if (load_factor)
    for (int a = tid; a < kp; a += NT) v[a] = rh[a];
  __syncthreads();
  if (!load_factor) {
    scale_blocks(S, linv, mo, Q, warp, NW, lane);
    if (mode == kSolveForward && fac != nullptr) {
      // the factor (Lt, the diagonal blocks of L and their inverses) leaves with a bulk copy
      tc::fence_proxy_async_smem();
      __syncthreads();
      if (tid == 0) {
        tc::bulk_s2g(fac, S, (uint32_t)fsz * 4u);
        tc::bulk_commit_group();
      }
    }
  }

  // x = S^{-1} rhs: the factorisation already applied L^{-1} to v
  if (load_factor) unit_fwd(S, v, Q, tid);
  block_diag_solve(linv, mo, v, Q, tid, load_factor);
  __syncthreads();
  unit_bwd(S, v, Q, tid);
  float* ycol = pan + 4 * kp;   // past the 16-row inverse blocks (mo holds at most 4 kp floats)
  for (int a = tid; a < kp; a += NT) {
    xs[a] = v[a];
    ycol[a] = 0.f;
  }
  __syncthreads();

  // iterative refinement: x += S^{-1} (rhs - S x). With G in shared memory every thread
  // forms one row's residual (float4 reads, four partial sums); otherwise the warps read
  // the lower triangle of G from global memory, four rows in flight per warp.
  const float* Gres = use_gs ? Gs : G;
  for (int it = 0; it < n_ir; ++it) {
    if (use_gs) {
      for (int a = tid; a < kp; a += NT) {
        float s4[4] = {0.f, 0.f, 0.f, 0.f};
        if (a < k) {
          const float4* gr = reinterpret_cast<const float4*>(Gs + (int64_t)a * ldg);
          const float4* xq = reinterpret_cast<const float4*>(xs);
          const int nq = k >> 2;   // full quads; the columns past k hold no G entries
          for (int q = 0; q < nq; ++q) {
            const float4 g4 = gr[q], x4 = xq[q];
            s4[0] = fmaf(g4.x, x4.x, s4[0]);
            s4[1] = fmaf(g4.y, x4.y, s4[1]);
            s4[2] = fmaf(g4.z, x4.z, s4[2]);
            s4[3] = fmaf(g4.w, x4.w, s4[3]);
          }
          for (int c = 4 * nq; c < k; ++c) s4[c & 3] = fmaf(Gs[(int64_t)a * ldg + c], xs[c], s4[c & 3]);
        }
        v[a] = a < k ? rh[a] - fmaf(dg[a], xs[a], (s4[0] + s4[1]) + (s4[2] + s4[3])) : 0.f;
      }
      __syncthreads();
      unit_fwd(S, v, Q, tid);
      block_diag_solve(linv, mo, v, Q, tid, true);
      __syncthreads();
      unit_bwd(S, v, Q, tid);
      for (int a = tid; a < kp; a += NT) xs[a] += v[a];
      __syncthreads();
      continue;
    }
    // G is symmetric: only its lower triangle is read. Row a's entries c <= a give the row
    // part of (G x)_a (reduced across the warp into v[a]); each entry c < a also gives
    // G_ac x_a to (G x)_c, summed per lane over the warp's rows (column c = lane + 32 j in
    // colacc[j]) and added into ycol warp by warp in a fixed order (reproducible sums).
    float colacc[4 * kResRounds];
#pragma unroll
    for (int j = 0; j < 4 * kResRounds; ++j) colacc[j] = 0.f;
    for (int a0 = warp; a0 < kp; a0 += 4 * NW) {
      float sum[4] = {0.f, 0.f, 0.f, 0.f};
      float xa[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int a = a0 + u * NW;
        xa[u] = a < k ? xs[a] : 0.f;
      }
      const int amax = min(a0 + 3 * NW, k - 1);   // the longest row of the group
#pragma unroll
      for (int r = 0; r < kResRounds; ++r) {       // 128 columns (four per lane) per round
        const int c0 = 128 * r;
        if (c0 > amax) break;
        if (Ghl) {
          float2 g[4][4];
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int a = a0 + u * NW;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              const int c = c0 + lane + 32 * q;
              g[u][q] = (a < k && c <= a) ? Ghl[(int64_t)a * k + c] : make_float2(0.f, 0.f);
            }
          }
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const int c = c0 + lane + 32 * q;
            const float xv = c < k ? xs[c] : 0.f;
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              sum[u] = fmaf(g[u][q].y, xv, fmaf(g[u][q].x, xv, sum[u]));
              const float xo = (c < a0 + u * NW) ? xa[u] : 0.f;   // off-diagonal entries only
              colacc[4 * r + q] = fmaf(g[u][q].y, xo, fmaf(g[u][q].x, xo, colacc[4 * r + q]));
            }
          }
        } else {
          float g[4][4];
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int a = a0 + u * NW;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              const int c = c0 + lane + 32 * q;
              g[u][q] = (a < k && c <= a) ? Gres[(int64_t)a * ldg + c] : 0.f;
            }
          }
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const int c = c0 + lane + 32 * q;
            const float xv = c < k ? xs[c] : 0.f;
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              sum[u] = fmaf(g[u][q], xv, sum[u]);
              const float xo = (c < a0 + u * NW) ? xa[u] : 0.f;
              colacc[4 * r + q] = fmaf(g[u][q], xo, colacc[4 * r + q]);
            }
          }
        }
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) sum[u] += __shfl_xor_sync(0xffffffffu, sum[u], o);
        const int a = a0 + u * NW;
        if (lane == 0 && a < kp) v[a] = sum[u];
      }
    }
    for (int w = 0; w < NW; ++w) {
      if (warp == w) {
#pragma unroll
        for (int j = 0; j < 4 * kResRounds; ++j) {
          const int c = 32 * j + lane;
          if (c < k) ycol[c] += colacc[j];
        }
      }
      __syncthreads();
    }
    for (int a = tid; a < kp; a += NT)
      v[a] = a < k ? rh[a] - fmaf(dg[a], xs[a], v[a] + ycol[a]) : 0.f;
    __syncthreads();
    unit_fwd(S, v, Q, tid);
    block_diag_solve(linv, mo, v, Q, tid, true);
    __syncthreads();
    unit_bwd(S, v, Q, tid);
    for (int a = tid; a < kp; a += NT) {
      xs[a] += v[a];
      ycol[a] = 0.f;
    }
    __syncthreads();
  }

  bool finite = true;
  for (int a = tid; a < k; a += NT) {
    const float xv = xs[a];
    out[a] = xv;
    if (!isfinite(xv)) finite = false;
  }
  if (!finite) set_status(status, p, FMAP_ERR_NONFINITE | (i << 8));
  if (tid == 0) tc::bulk_wait_group_read0();   // the factor has left shared memory
}

// ---- above k = 100 (but 201 .. 208): the trailing matrix in registers ----------------
// Pairs of column halves of a panel in shared memory: entry (row a, column c) of the
// current panel is at c * 2 * half + ((a >> 2) & 1) * half + 4 * (a >> 3) + (a & 3), so
// that consecutive 8-row blocks read consecutive float4 and, with half = 16 mod 32, the
// 32 rows of a warp store to 32 banks. Room for kp rows and the right-hand side.
__host__ __device__ __forceinline__ int pan_half(int Q) { return (4 * (Q + 1) - 16 + 31) / 32 * 32 + 16; }
__host__ __device__ __forceinline__ int pan_idx(int a) { return 4 * (a >> 3) + (a & 3); }

// One row of the panel: s <- s - x L^T for the 8 columns whose rows of L (panel c, rows
// n0 .. n0+7) are in `pan`.
__device__ __forceinline__ void row_update(float (&s)[8], const float (&x)[8], const float* pan, int half, int blk) {
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    const float4 b0 = *reinterpret_cast<const float4*>(pan + c * 2 * half + 4 * blk);
    const float4 b1 = *reinterpret_cast<const float4*>(pan + c * 2 * half + half + 4 * blk);
    s[0] = fmaf(-x[c], b0.x, s[0]); s[1] = fmaf(-x[c], b0.y, s[1]);
    s[2] = fmaf(-x[c], b0.z, s[2]); s[3] = fmaf(-x[c], b0.w, s[3]);
    s[4] = fmaf(-x[c], b1.x, s[4]); s[5] = fmaf(-x[c], b1.y, s[5]);
    s[6] = fmaf(-x[c], b1.z, s[6]); s[7] = fmaf(-x[c], b1.w, s[7]);
  }
}

// Cholesky factor of the 8 x 8 block d (lower part) in registers, r[j] = 1 / L_jj. kSafe:
// reciprocal square roots that also take subnormal pivots, and a check of every pivot.
// Without it the caller tests r: a pivot that is negative, zero, subnormal or not a number spreads
// through the updates and leaves a value that is not finite and positive in r[7]; an infinite one
// leaves its own r[j] = 0 and the columns after it untouched.
template <bool kSafe>
__device__ __forceinline__ bool factor8(float (&d)[8][8], float (&r)[8]) {
  bool ok = true;
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const float piv = d[j][j];
    if (kSafe) {
      ok = ok && piv > 0.f && piv < INFINITY;
      r[j] = rsqrtf(piv);
    } else {
      asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r[j]) : "f"(piv));
    }
    d[j][j] = piv * r[j];
#pragma unroll
    for (int i = j + 1; i < 8; ++i) d[i][j] *= r[j];
#pragma unroll
    for (int i = j + 1; i < 8; ++i)
#pragma unroll
      for (int q = j + 1; q <= i; ++q) d[i][q] = fmaf(-d[i][j], d[q][j], d[i][q]);
  }
  return ok;
}

__device__ __forceinline__ void load_lower8(const float* src, int ld, float (&d)[8][8]) {
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const float4 u0 = *reinterpret_cast<const float4*>(src + ld * i);
    d[i][0] = u0.x; d[i][1] = u0.y; d[i][2] = u0.z; d[i][3] = u0.w;
    if (i >= 4) {
      const float4 u1 = *reinterpret_cast<const float4*>(src + ld * i + 4);
      d[i][4] = u1.x; d[i][5] = u1.y; d[i][6] = u1.z; d[i][7] = u1.w;
    }
  }
}

// Factor S (packed lower rows in shared memory, kp = 8 Q rows) in place, v <- L^-1 v, and
// linv <- the inverses of the 8 x 8 diagonal blocks.
//
// Warp 0 takes the diagonal blocks. OW owner warps hold the 8 x 8 blocks (A, B) of columns
// B >= c0 in registers, one block per thread (-S_AB, 32 packed pairs), in column order. RW
// row warps hold kSlots rows each per thread (rows t, t + 32 RW, ...; row kp is the
// right-hand side). Panel J:
//   warp 0   brings the diagonal block J up to panel J - 1, factors it in registers and
//            stores it; then, while the rows are solved, its inverse;
//   rows     meanwhile bring column J up to panel J - 1 (their entries of that panel are
//            still in registers), then solve against the diagonal block, x = s L_JJ^-T;
//   barrier  the panel's columns are in `pan` (two buffers);
//   owners   -S_AB += L_AJ L_BJ^T for B >= J + 2; column J + 2 is then complete up to panel
//            J and goes back to S, where the rows find it one panel later.
// The chain of a panel is warp 0's block and one solve of the rows; the first c0 columns
// (those that do not fit the owners' registers, at least 2) are updated in S by the rows.
// The trailing update reads 16 floats of shared memory per 64 FMAs and never re-reads or
// re-writes S, which an update of tiles in shared memory does every panel.
template <int OW, int RW, int kSlots>
__device__ __forceinline__ void factor_registers(float* S, float* linv, float* pan, float* v, float* dbuf, int Q,
                                                 int* s_bad) {
  constexpr int NT = 32 * (1 + OW + RW), RT = 32 * RW, TT = RT + 32;
  const int kp = 8 * Q, half = pan_half(Q), pbuf = 16 * half;
  const int tid = threadIdx.x;
  // the owners' triangle: m block columns from c0, m (m + 1) / 2 <= 32 OW
  int m = Q - 2;
  while (m * (m + 1) / 2 > 32 * OW) --m;
  const int c0 = Q - m;
  if (tid >= TT) {
    const int o = tid - TT, nb = m * (m + 1) / 2;
    int A = 0, B = -1;
    if (o < nb) {
      int ai, bi;
      tri_decode(nb - 1 - o, ai, bi);
      B = Q - 1 - ai;
      A = Q - 1 - bi;
    }
    // pairs (r, c) (r+1, c+1) and (r, c+1) (r+1, c): both take the row pair (a_r, a_r+1) as it
    // was loaded, so that only the four swapped column pairs cost moves
    uint64_t acc[4][4][2];
    if (B >= 0) {
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        float u[8], w[8];
        load8(S + rowoff(8 * A + 2 * r) + 8 * B, u);
        load8(S + rowoff(8 * A + 2 * r + 1) + 8 * B, w);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          acc[r][q][0] = pk2(-u[2 * q], -w[2 * q + 1]);
          acc[r][q][1] = pk2(-u[2 * q + 1], -w[2 * q]);
        }
      }
    }
    for (int J = 0; J < Q; ++J) {
      __syncwarp();
      tc::named_barrier_sync(2, NT);   // panel J is in pan
      if (B < J + 2) continue;
      const float* pa = pan + (J & 1) * pbuf + 4 * A;
      const float* pb = pan + (J & 1) * pbuf + 4 * B;
#pragma unroll
      for (int c = 0; c < 8; ++c) {
        const float4 a0 = *reinterpret_cast<const float4*>(pa + c * 2 * half);
        const float4 a1 = *reinterpret_cast<const float4*>(pa + c * 2 * half + half);
        const float4 b0 = *reinterpret_cast<const float4*>(pb + c * 2 * half);
        const float4 b1 = *reinterpret_cast<const float4*>(pb + c * 2 * half + half);
        const uint64_t la[4] = {pk2(a0.x, a0.y), pk2(a0.z, a0.w), pk2(a1.x, a1.y), pk2(a1.z, a1.w)};
        const uint64_t lb[4] = {pk2(b0.x, b0.y), pk2(b0.z, b0.w), pk2(b1.x, b1.y), pk2(b1.z, b1.w)};
        const uint64_t ls[4] = {pk2(b0.y, b0.x), pk2(b0.w, b0.z), pk2(b1.y, b1.x), pk2(b1.w, b1.z)};
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            acc[r][q][0] = fma2(la[r], lb[q], acc[r][q][0]);
            acc[r][q][1] = fma2(la[r], ls[q], acc[r][q][1]);
          }
      }
      if (B == J + 2) {
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          float u[8], w[8];
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            upk2(acc[r][q][0], u[2 * q], w[2 * q + 1]);
            upk2(acc[r][q][1], u[2 * q + 1], w[2 * q]);
          }
#pragma unroll
          for (int q = 0; q < 8; ++q) { u[q] = -u[q]; w[q] = -w[q]; }
          store8(S + rowoff(8 * A + 2 * r) + 8 * B, u);
          store8(S + rowoff(8 * A + 2 * r + 1) + 8 * B, w);
        }
      }
    }
    return;
  }
  if (tid < 32) {
    // ---- diagonal blocks
    const int i = tid >> 2, c = 2 * (tid & 3);
    for (int J = 0; J < Q; ++J) {
      const int n0 = 8 * J;
      float2 e = *reinterpret_cast<const float2*>(S + rowoff(n0 + i) + n0 + c);
      if (J > 0) {
        float li[8], l0[8], l1[8];
        load8(S + rowoff(n0 + i) + n0 - 8, li);
        load8(S + rowoff(n0 + c) + n0 - 8, l0);
        load8(S + rowoff(n0 + c + 1) + n0 - 8, l1);
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          e.x = fmaf(-li[q], l0[q], e.x);
          e.y = fmaf(-li[q], l1[q], e.y);
        }
      }
      *reinterpret_cast<float2*>(dbuf + 8 * i + c) = e;
      __syncwarp();
      float d[8][8], r[8];
      load_lower8(dbuf, 8, d);
      factor8<false>(d, r);
      const float rmin = fminf(fminf(fminf(r[0], r[1]), fminf(r[2], r[3])), fminf(fminf(r[4], r[5]), r[6]));
      if (!(r[7] > 0.f && r[7] < INFINITY && rmin > 0.f)) {
        load_lower8(dbuf, 8, d);
        if (!factor8<true>(d, r)) *s_bad = 1;
      }
      if (tid == 0) {
        float* row = S + rowoff(n0) + n0;
        const int ld = 8 * J + 12;
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          *reinterpret_cast<float4*>(row + ld * q) = make_float4(d[q][0], d[q][1], d[q][2], d[q][3]);
          if (q >= 4) *reinterpret_cast<float4*>(row + ld * q + 4) = make_float4(d[q][4], d[q][5], d[q][6], d[q][7]);
        }
        store8(linv + 64 * J, r);      // until the inverse takes its place
      }
      __syncwarp();
      tc::named_barrier_sync(1, TT);
      // column `tid` of L_JJ^-1: forward substitution on the unit vector
      float w[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        float t = (q == tid) ? 1.f : 0.f;
#pragma unroll
        for (int z = 0; z < q; ++z) t = fmaf(-d[q][z], w[z], t);
        w[q] = (q >= tid) ? t * r[q] : 0.f;
      }
      __syncwarp();
      tc::named_barrier_sync(2, NT);
      if (tid < 8)
#pragma unroll
        for (int q = 0; q < 8; ++q) linv[64 * J + 8 * q + tid] = w[q];
    }
    return;
  }
  // ---- rows
  const int rt = tid - 32, wbase = rt & ~31;
  float x[kSlots][8];                  // rows: entries of the column block in hand, then of L
#pragma unroll
  for (int u = 0; u < kSlots; ++u) {
    const int a = rt + RT * u;
    if (a <= kp) load8(a < kp ? S + rowoff(a) : v, x[u]);
  }
  for (int J = 0; J < Q; ++J) {
    const int n0 = 8 * J, n1 = n0 + 8;
    __syncwarp();
    tc::named_barrier_sync(1, TT);     // the factor of block J is in S
    float d[8][8], r[8];
    load_lower8(S + rowoff(n0) + n0, n0 + 12, d);
    load8(linv + 64 * J, r);
    float* pw = pan + (J & 1) * pbuf;
#pragma unroll
    for (int u = 0; u < kSlots; ++u) {
      const int a = rt + RT * u;
      if (wbase + RT * u + 31 >= n1 && wbase + RT * u <= kp) {
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          x[u][j] *= r[j];
#pragma unroll
          for (int i = j + 1; i < 8; ++i) x[u][i] = fmaf(-x[u][j], d[i][j], x[u][i]);
        }
        if (a >= n1 && a <= kp) {
          float* q = pw + ((a >> 2) & 1) * half + pan_idx(a);
#pragma unroll
          for (int c = 0; c < 8; ++c) q[c * 2 * half] = x[u][c];
          store8((a < kp ? S + rowoff(a) : v) + n0, x[u]);
        }
      }
    }
    __syncwarp();
    tc::named_barrier_sync(2, NT);     // panel J is in pan; column J + 1 in S is complete up to panel J - 1
    if (J + 1 == Q) break;
    float y[8];
    load8(v + n0, y);
#pragma unroll
    for (int u = 0; u < kSlots; ++u) {
      const int a = rt + RT * u;
      if (wbase + RT * u + 31 >= n1 + 8 && wbase + RT * u <= kp) {
        if (a >= n1 + 8 && a <= kp) {
          float* row = a < kp ? S + rowoff(a) : v;
          float t[8];
          load8(row + n1, t);
          row_update(t, x[u], pw, half, J + 1);
          if (a < kp) {
            // the row's right-hand side takes the panel's contribution, v_a -= L_aJ y_J
            float va = v[a];
#pragma unroll
            for (int c = 0; c < 8; ++c) va = fmaf(-x[u][c], y[c], va);
            v[a] = va;
            for (int C = J + 2; C < c0 && 8 * C <= a; ++C) {   // the columns without owners
              float w[8];
              load8(row + 8 * C, w);
              row_update(w, x[u], pw, half, C);
              store8(row + 8 * C, w);
            }
          }
#pragma unroll
          for (int c = 0; c < 8; ++c) x[u][c] = t[c];
        }
      }
    }
  }
}

// One 16-row by 32-column piece of the residual's product: rows a0 .. a0+15, column c0 + lane.
// Returns in lane l the sum of row a0 + (l & 15) over the piece, and adds the column's sum of
// the entries below the diagonal times x_a to `col`.
template <class Load>
__device__ __forceinline__ float residual_piece(const Load& entry, const float* xs, int a0, int c0, int k, int lane,
                                                float& col) {
  const int c = c0 + lane;
  const float xc = c < k ? xs[c] : 0.f;
  float2 g[16];
#pragma unroll
  for (int i = 0; i < 16; ++i) g[i] = (a0 + i < k && c <= a0 + i) ? entry(a0 + i, c) : make_float2(0.f, 0.f);
  float p[16];
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    const float xa = xs[a0 + i];                       // padded with zeros past k
    p[i] = fmaf(g[i].y, xc, g[i].x * xc);
    const float xo = c < a0 + i ? xa : 0.f;            // the diagonal entry counts once
    col = fmaf(g[i].y, xo, fmaf(g[i].x, xo, col));
  }
  // sums over the 32 lanes of 16 rows: halving exchanges, then the two half-warps
#pragma unroll
  for (int o = 8; o > 0; o >>= 1)
#pragma unroll
    for (int i = 0; i < o; ++i) {
      const bool up = (lane & o) != 0;
      const float give = up ? p[i] : p[i + o], keep = up ? p[i + o] : p[i];
      p[i] = keep + __shfl_xor_sync(0xffffffffu, give, o);
    }
  return p[0] + __shfl_xor_sync(0xffffffffu, p[0], 16);
}

// Row systems of those sizes: the factorisation above, then the solves of chol_solve_kernel.
template <int OW, int RW, int kSlots, int kMinBlocks>
__global__ void __launch_bounds__(32 * (1 + OW + RW), kMinBlocks)
    chol_reg_kernel(BatchDev b, const int2* systems, int first, int count, int mode, const float* rhs_flat,
                    float* out_flat, float* saved, int32_t* status, float* ws) {
  constexpr int NW = 1 + OW + RW, NT = 32 * NW;
  extern __shared__ __align__(16) float smem[];
  __shared__ int s_bad;
  __shared__ __align__(8) uint64_t s_bar;
  __shared__ int s_abort;
  if ((int)blockIdx.x >= count) return;
  const int2 sys = systems[first + blockIdx.x];
  const int p = sys.x, i = sys.y;
  const PairDev pd = b.pairs[p];
  const int k = pd.k;
  const int Q = (k + 7) >> 3, kp = 8 * Q;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const float* evx = b.shapes[pd.x].evals;
  const float* evy = b.shapes[pd.y].evals;
  const int pan_floats = 32 * pan_half(Q);
  float* S = smem;                       // packed skewed lower rows
  float* linv = S + rowoff(kp);          // inverse diagonal blocks, Q x 64
  float* pan = linv + 64 * Q;            // two panels of 8 columns (then the solves' scratch)
  float* dbuf = pan + pan_floats;        // the next diagonal block
  float* v = dbuf + 64;                  // working vector
  float* xs = v + kp;                    // solution (zero past k)
  float* rh = xs + kp + 8;               // right-hand side
  float* dg = rh + kp;                   // lambda D_i
  const float* G = ws + pd.g_off;
  const float* rhs = (mode == kSolveForward) ? ws + pd.r_off + (int64_t)i * k : rhs_flat + pd.c_off + (int64_t)i * k;
  float* out = (mode == kSolveForward) ? out_flat + pd.c_off + (int64_t)i * k : ws + pd.gam_off + (int64_t)i * k;
  const int fsz = factor_floats(Q);
  float* fac = (saved != nullptr && pd.fac_off >= 0) ? saved + pd.fac_off + (int64_t)i * fsz : nullptr;
  const bool load_factor = mode == kSolveAdjoint && fac != nullptr;
  const float lam = pd.lam_rows ? pd.lam_rows[i] : pd.lam;
  const int n_ir = mode == kSolveForward ? b.ir_steps : b.ir_steps_adj;

  if (tid == 0) {
    s_bad = 0;
    s_abort = 0;
    tc::mbar_init(&s_bar, 1);
    tc::fence_mbar_init();
    // a projection wait that timed out leaves its error in the workspace's first word
    if (i == 0 && reinterpret_cast<const int*>(ws)[0] != 0) set_status(status, p, FMAP_ERR_TIMEOUT);
    // the saved factor, or rows 0 .. k-1 of G in the packed layout: one bulk copy
    const uint32_t bytes = (load_factor ? (uint32_t)fsz : (uint32_t)rowoff(k)) * 4u;
    tc::mbar_arrive_expect_tx(&s_bar, bytes);
    tc::bulk_g2s(S, load_factor ? fac : G + gram_packed_off(k), bytes, &s_bar);
  }
  for (int a = tid; a < kp; a += NT) {
    const float r = a < k ? rhs[a] : 0.f;
    rh[a] = r;
    v[a] = r;
    dg[a] = a < k ? lam * mask_entry(pd, evx, evy, i, a) : 0.f;
  }
  if (tid < 8) xs[kp + tid] = 0.f;
  if (!load_factor)   // padding rows are identity rows
    for (int a = k + tid; a < kp; a += NT) {
      float* row = S + rowoff(a);
      for (int c = 0; c < (a & ~7) + 8; ++c) row[c] = (c == a) ? 1.f : 0.f;
    }
  __syncthreads();    // barrier initialised
  tc::mbar_wait(&s_bar, 0, &s_abort);
  __syncthreads();
  if (s_abort) {
    // a copy that never completed: report, give it a bounded time to land, leave (every
    // thread of the block takes this branch together)
    if (tid == 0) set_status(status, p, FMAP_ERR_TIMEOUT);
    const uint64_t t0 = tc::globaltimer();
    while (!tc::mbar_try_wait(&s_bar, 0) && tc::globaltimer() - t0 < tc::kWaitTimeoutNs) {}
    return;
  }
  if (!load_factor) {
    for (int a = tid; a < k; a += NT) S[rowoff(a) + a] += dg[a];
    __syncthreads();
    factor_registers<OW, RW, kSlots>(S, linv, pan, v, dbuf, Q, &s_bad);
    __syncthreads();
    if (s_bad) {
      if (tid == 0) set_status(status, p, FMAP_ERR_NOT_SPD | (i << 8));
      for (int a = tid; a < k; a += NT) out[a] = __int_as_float(0x7fc00000);
      return;
    }
  }
  // inverses of the 16-row diagonal blocks (their off-diagonal parts, in the panels' space)
  float* mo = pan;
  pair_blocks_prepare(S, linv, mo, Q, tid, NT);
  __syncthreads();
  if (!load_factor) {
    scale_blocks(S, linv, mo, Q, warp, NW, lane);
    if (mode == kSolveForward && fac != nullptr) {
      // the factor (Lt, the diagonal blocks of L and their inverses) leaves with a bulk copy
      tc::fence_proxy_async_smem();
      __syncthreads();
      if (tid == 0) {
        tc::bulk_s2g(fac, S, (uint32_t)fsz * 4u);
        tc::bulk_commit_group();
      }
    }
  }
  // x = S^{-1} rhs: the factorisation already applied L^{-1} to v
  if (load_factor) unit_fwd(S, v, Q, tid);
  block_diag_solve(linv, mo, v, Q, tid, load_factor);
  __syncthreads();
  unit_bwd(S, v, Q, tid);
  // iterative refinement: x += S^{-1} (rhs - S x), G from global memory (L2), its lower triangle
  // only: each entry below the diagonal serves its row and its column. Every warp sums its
  // pieces into a vector of its own; the vectors are added in a fixed order.
  float* acc = mo + 64 * ((Q + 1) >> 1);
  const int naw = min(NW, (pan_floats - 64 * ((Q + 1) >> 1)) / kp);
  if (tid < kp) xs[tid] = v[tid];
  for (int it = 0; it < n_ir; ++it) {
    for (int e = tid; e < naw * kp; e += NT) acc[e] = 0.f;
    __syncthreads();
    if (warp < naw) {
      float* mine = acc + warp * kp;
      const float2* Ghl = pd.g64_off >= 0 ? reinterpret_cast<const float2*>(ws) + pd.g64_off : nullptr;
      const int ldg = gram_ld(k);
      int u = warp;                       // pieces in order of row groups: group R has R / 2 + 1
      int R = 0, q = 0;
      while (true) {
        while (16 * R < k && u >= R / 2 + 1) { u -= R / 2 + 1; ++R; }
        if (16 * R >= k) break;
        q = u;
        float col = 0.f;
        float row;
        if (Ghl)
          row = residual_piece([&](int a, int c) { return Ghl[(int64_t)a * k + c]; }, xs, 16 * R, 32 * q, k, lane, col);
        else
          row = residual_piece([&](int a, int c) { return make_float2(G[(int64_t)a * ldg + c], 0.f); }, xs, 16 * R,
                               32 * q, k, lane, col);
        if (lane < 16 && 16 * R + lane < kp) mine[16 * R + lane] += row;
        __syncwarp();
        if (32 * q + lane < kp) mine[32 * q + lane] += col;
        __syncwarp();
        u += naw;
      }
    }
    __syncthreads();
    for (int a = tid; a < kp; a += NT) {
      float t = 0.f;
      for (int w = 0; w < naw; ++w) t += acc[w * kp + a];
      v[a] = a < k ? rh[a] - fmaf(dg[a], xs[a], t) : 0.f;
    }
    __syncthreads();
    unit_fwd(S, v, Q, tid);
    block_diag_solve(linv, mo, v, Q, tid, true);
    __syncthreads();
    unit_bwd(S, v, Q, tid);
    if (tid < kp) xs[tid] += v[tid];
    __syncthreads();
  }

  bool finite = true;
  for (int a = tid; a < k; a += NT) {
    const float xv = xs[a];
    out[a] = xv;
    if (!isfinite(xv)) finite = false;
  }
  if (!finite) set_status(status, p, FMAP_ERR_NONFINITE | (i << 8));
  if (tid == 0) tc::bulk_wait_group_read0();   // the factor has left shared memory
}

size_t chol_reg_smem_bytes(int kmax) {
  const int Q = (kmax + 7) / 8, kp = 8 * Q;
  return (size_t)(factor_floats(Q) + 32 * pan_half(Q) + 64 + 4 * kp + 8) * sizeof(float);
}

// Launches for k <= kGsMaxK reserve a copy of G (k x gram_ld(k) floats) after the vectors.
constexpr int kGsMaxK = kSolveBounds[1];

size_t chol_smem_bytes(int kmax, bool g_copy = true) {
  const int Q = (kmax + 7) / 8, kp = 8 * Q;
  const int64_t gs = (g_copy && kmax <= kGsMaxK) ? (int64_t)kmax * gram_ld(kmax) : 0;
  return (size_t)(factor_floats(Q) + 8 * kp + 4 * kp + gs) * sizeof(float);
}

template <typename Kernel>
cudaError_t set_limit(Kernel* kernel, size_t bytes) {
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

}  // namespace

int64_t chol_factor_floats(int k) { return factor_floats((k + 7) / 8); }

cudaError_t solve_set_smem_limits() {
  cudaError_t e;
  if ((e = set_limit(chol_solve_kernel<64>, chol_smem_bytes(64))) != cudaSuccess) return e;
  if ((e = set_limit(chol_solve_kernel<128>, chol_smem_bytes(kSolveBounds[1]))) != cudaSuccess) return e;
  if ((e = set_limit(chol_solve_kernel<256>, chol_smem_bytes(kSolveBounds[4]))) != cudaSuccess) return e;
  if ((e = set_limit(chol_reg_kernel<2, 2, 2, 4>, chol_reg_smem_bytes(120))) != cudaSuccess) return e;
  if ((e = set_limit(chol_reg_kernel<2, 2, 3, 4>, chol_reg_smem_bytes(kSolveBounds[2]))) != cudaSuccess) return e;
  if ((e = set_limit(chol_reg_kernel<5, 4, 2, 2>, chol_reg_smem_bytes(kSolveBounds[3]))) != cudaSuccess) return e;
  if ((e = set_limit(chol_reg_kernel<14, 5, 2, 1>, chol_reg_smem_bytes(kSolveBounds[5]))) != cudaSuccess) return e;
  if ((e = gram_set_smem()) != cudaSuccess) return e;
  return adjoint_tc_set_smem();
}

// One launch per class of kSolveBounds. The trailing matrix stays in shared memory (and with it
// a copy of G for the residual) while three systems fit an SM that way, k <= 100, and for
// 200 < k <= 208, where two fit only without the panels of the register kernel; elsewhere the
// register kernel is faster. ns per row system (solve / adjoint with saved factors, 64 pairs;
// 32 at k = 200), shared memory against registers: k = 77 37.2 / 9.9 against 48.6 / 9.2,
// k = 100 60.0 / 14.3 against 64.9 / 11.0, k = 104 76.5 / 20.0 against 64.5 / 11.0, k = 112
// 81.7 / 19.5 against 71.0 / 11.0, k = 128 98.0 / 20.0 against 99.4 / 11.8, k = 200 252 / 46
// (with an inverse in every step of its solves) against 221 / 27. The adjoint alone would change at
// k = 77; it takes the forward solve's kernel up to 100, a quarter of whose time it is.
cudaError_t launch_solve(const BatchDev& b, const SolveGroup& g, const int2* systems, int mode, const float* rhs_flat,
                         float* out_flat, float* saved, int32_t* status, float* ws, cudaStream_t st) {
  if (g.count <= 0) return cudaSuccess;
  const int k = g.kmax;
  // a slot of a row warp's thread for each of kp rows and the right-hand side
  static_assert(32 * 2 * 2 > 120 && 32 * 2 * 3 > kSolveBounds[2] && 32 * 4 * 2 > kSolveBounds[3] && 32 * 5 * 2 > kSolveBounds[5]);
  auto regs = [&](auto* kernel, int threads) {
    kernel<<<g.count, threads, chol_reg_smem_bytes(k), st>>>(b, systems, g.first, g.count, mode, rhs_flat, out_flat,
                                                             saved, status, ws);
  };
  auto tiles = [&](auto* kernel, int threads) {
    const bool g_copy = g.no_g_copy == 0 && k <= kGsMaxK;
    kernel<<<g.count, threads, chol_smem_bytes(k, g_copy), st>>>(b, systems, g.first, g.count, mode, rhs_flat,
                                                                 out_flat, saved, status, ws, g_copy ? 1 : 0);
  };
  if (k <= kSolveBounds[1]) {
    // one thread per row: the substitutions, the TRSM and the (a) update assume threads >= kp
    if (8 * ((k + 7) / 8) > g.threads) return cudaErrorInvalidValue;
    if (g.threads == 64)
      tiles(chol_solve_kernel<64>, 64);
    else if (g.threads == 128)
      tiles(chol_solve_kernel<128>, 128);
    else
      tiles(chol_solve_kernel<256>, 256);
  } else if (k <= kSolveBounds[2]) {
    if (k <= 120)
      regs(chol_reg_kernel<2, 2, 2, 4>, 160);
    else
      regs(chol_reg_kernel<2, 2, 3, 4>, 160);
  } else if (k <= kSolveBounds[3]) {
    regs(chol_reg_kernel<5, 4, 2, 2>, 320);
  } else if (k <= kSolveBounds[4]) {
    tiles(chol_solve_kernel<256>, 256);
  } else {
    regs(chol_reg_kernel<14, 5, 2, 1>, 640);
  }
  return cudaGetLastError();
}

}  // namespace fmap
