// Spatial gradient features (Sec. "Learned Scaling and Rotation in DiffusionNet"), fused
// in one kernel that writes the features straight into the projection's input layout:
//
//   z_v = sum_u G_vu X_u          (sparse complex gradient operator G, CSR; z = x + i y)
//   [P | Q] = [x | y] W           (W: the 2D x 2D real form of the learned complex A)
//   g_v = x o P + y o Q           (= Re(conj(z) o Az) for variant A)
//
// with P = (Az)_re = A_re x - A_im y and Q = (Az)_im = A_re y + A_im x (variant A) or
// A_re x + A_im y (variant B). One persistent CTA per SM walks 128-vertex tiles:
//   warps 0-15  gather x and y of the tile's vertices, 16 channels of X at a time (8 vertices
//               per warp, 4 lanes each, float4), into a K-major, 128-byte-swizzled FP32 tile in
//               shared memory; K-block j holds x and y of channels 16 j .. 16 j + 15, so a K-block
//               is multiplied while the next channels are gathered. A vertex's CSR entries stay
//               in registers over its channels. Then the epilogue: P and Q from TMEM (one
//               vertex per lane), x and y from the tile, g stored in FP32 or BF16 rows;
//   warp 16     issues tcgen05.mma kind::tf32 (M = 128 vertices, N = 2D, K = 8) into TMEM;
//   warp 17     streams the K-blocks of the W image (built once per call in the workspace,
//               rounded to TF32) through two shared-memory stages.
// A vertex's row of X is read about seven times among its neighbours: 128 vertices times 64 bytes
// keep the rows in hand inside L1, where gathering whole 512-byte rows read every one of them
// from L2 before a tile's products could start (64 shapes, 1.06 M vertices, D = 128: 1.215 ms a
// call, 0.600 this way). What bounds it now is the data pipe of L1 (14.8k wavefronts in the 21.0k
// cycles of a tile: eight rows of X to a load instruction, 32 output rows to a store).
// The x, y tile is the MMA operand and the epilogue's input, so a tile's gather starts
// after the previous tile's epilogue. Waits are bounded; a wait that gives up, or a CSR
// index out of range, sets the caller's status word.
#include "fmap_internal.cuh"
#include "tc_ptx.cuh"

namespace fmap {
namespace {

constexpr int kGfGatherWarps = 16;
constexpr int kGfThreads = 32 * (kGfGatherWarps + 2);
constexpr int kGfTileV = 128;
constexpr int kGfMaxDim = 128;
constexpr int kGfMaxBlocks = kGfMaxDim / 16;             // K-blocks: x and y of 16 channels
constexpr uint32_t kGfABlock = kGfTileV * 128u;          // one K-block of the x, y tile

// Byte offset of the 16-byte chunk ch of row r in a K-block of 128-byte rows with the 128-byte
// swizzle.
__device__ __forceinline__ uint32_t sw_chunk(int r, int ch) {
  return (uint32_t)r * 128u + (uint32_t)((ch ^ (r & 7)) << 4);
}

// W image: K-block kb holds the 2D output columns n (rows of 128 bytes, K-major), value W[k][n]
// rounded to TF32 for the K indices of channels 16 kb .. 16 kb + 15: x (kk < 16), then y. Column
// n < D is P_n, n >= D is Q_{n-D}.
__global__ void gradfeat_w_image_kernel(const float* a_re, const float* a_im, int dim, int variant, float* img) {
  const int n2 = 2 * dim;
  const int total = n2 * n2;
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < total; e += gridDim.x * blockDim.x) {
    const int kb = e / (n2 * 32);
    const int rem = e % (n2 * 32);
    const int n = rem / 32, kk = rem % 32;
    const bool kx = kk < 16, nq = n >= dim;
    const int i = nq ? n - dim : n, j = 16 * kb + (kk & 15);
    const float are = a_re[(int64_t)i * dim + j], aim = a_im[(int64_t)i * dim + j];
    float w;
    if (!nq)
      w = kx ? are : -aim;                                  // P_i = A_re x - A_im y
    else if (variant == 0)
      w = kx ? aim : are;                                   // Q_i = A_re y + A_im x
    else
      w = kx ? are : aim;                                   // Q_i = A_re x + A_im y
    img[(int64_t)(kb * n2 + n) * 32 + (((kk >> 2) ^ (n & 7)) << 2) + (kk & 3)] = tc::tf32_rna(w);
  }
}

struct GfParams {
  int64_t n, n_in, nnz;
  const int64_t* row_ptr;
  const int32_t* col_idx;
  const float2* vals;
  const float* x_in;
  int64_t ld_in;
  int32_t dim;
  void* out;
  int64_t ld_out;
  int32_t out_bf16;
  const float* w_img;
  int32_t* status;
  uint32_t tmem_cols;
};

template <bool kWide>   // rows of X 4 GB apart or more
__global__ void __launch_bounds__(kGfThreads, 1) gradfeat_kernel(GfParams P) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int dim = P.dim, n2 = 2 * dim, nkb = n2 / 32;
  const uint32_t w_stage = (uint32_t)n2 * 128u;                       // one K-block of W
  uint8_t* sA = smem;
  uint8_t* sW = sA + (uint32_t)nkb * kGfABlock;
  uint64_t* w_full = reinterpret_cast<uint64_t*>(sW + 2 * w_stage);
  uint64_t* w_empty = w_full + 2;
  uint64_t* acc_full = w_empty + 2;
  uint64_t* a_full = acc_full + 1;                                    // [kGfMaxBlocks]
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(a_full + kGfMaxBlocks);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  int* bad_index = const_cast<int*>(reinterpret_cast<volatile int*>(tmem_slot + 2));

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (tid == 0) {
    for (int s = 0; s < 2; ++s) {
      tc::mbar_init(&w_full[s], 1);
      tc::mbar_init(&w_empty[s], 1);
    }
    tc::mbar_init(acc_full, 1);
    for (int c = 0; c < kGfMaxBlocks; ++c) tc::mbar_init(&a_full[c], kGfGatherWarps);
    *abort_flag = 0;
    *bad_index = 0;
    tc::fence_mbar_init();
  }
  if (warp == kGfGatherWarps) {
    tc::tmem_alloc(tmem_slot, P.tmem_cols);
    tc::tmem_relinquish();
    tc::tc_fence_before();
  }
  __syncthreads();
  tc::tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  const int64_t ntiles = (P.n + kGfTileV - 1) / kGfTileV;

  if (warp == kGfGatherWarps + 1) {
    // ---------------------------------------------------------------- W
    if (lane == 0) {
      const uint8_t* wsrc = reinterpret_cast<const uint8_t*>(P.w_img);
      int s = 0;
      uint32_t phase = 0;
      for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x)
        for (int kb = 0; kb < nkb; ++kb) {
          if (!tc::mbar_wait(&w_empty[s], phase ^ 1, abort_flag)) goto w_done;
          tc::mbar_arrive_expect_tx(&w_full[s], w_stage);
          for (uint32_t off = 0; off < w_stage; off += 16384u)
            tc::bulk_g2s(sW + (size_t)s * w_stage + off, wsrc + (size_t)kb * w_stage + off,
                         (w_stage - off) < 16384u ? (w_stage - off) : 16384u, &w_full[s]);
          if (++s == 2) { s = 0; phase ^= 1; }
        }
    w_done:
      if (*abort_flag) {
        // let copies already in flight land before the CTA's shared memory goes away
        const uint64_t t0 = tc::globaltimer();
        while (tc::globaltimer() - t0 < 2000000ull) {}
      }
    }
  } else if (warp == kGfGatherWarps) {
    // ---------------------------------------------------------------- MMAs
    if (lane == 0) {
      const uint32_t idesc = tc::idesc_tf32(128, (uint32_t)n2);
      const uint32_t a_base = tc::smem_u32(sA);
      int s = 0;
      uint32_t phase = 0, cphase = 0;
      bool ok = true;
      for (int64_t tile = blockIdx.x; tile < ntiles && ok; tile += gridDim.x) {
        for (int kb = 0; kb < nkb; ++kb) {
          if (!tc::mbar_wait(&w_full[s], phase, abort_flag) || !tc::mbar_wait(&a_full[kb], cphase, abort_flag)) {
            ok = false;
            break;
          }
          tc::tc_fence_after();
          const uint32_t b_base = tc::smem_u32(sW + (size_t)s * w_stage);
#pragma unroll
          for (int ks = 0; ks < 4; ++ks) {
            const uint64_t ad = tc::smem_desc(a_base + (uint32_t)kb * kGfABlock + ks * 32, 16, 1024, tc::kLayoutSW128);
            const uint64_t bd = tc::smem_desc(b_base + ks * 32, 16, 1024, tc::kLayoutSW128);
            tc::mma_tf32(tmem_base, ad, bd, idesc, (kb | ks) != 0 ? 1u : 0u);
          }
          tc::mma_commit(&w_empty[s]);
          if (++s == 2) { s = 0; phase ^= 1; }
        }
        if (!ok) break;
        tc::mma_commit(acc_full);
        cphase ^= 1;
      }
    }
  } else {
    // ---------------------------------------------------------------- gather, epilogue
    const int sub = lane >> 2, cl = lane & 3;            // vertex of the warp's eight, float4 of 16 channels
    const int gr = warp * 8 + sub;                       // its row of the tile
    const char* x_lane = reinterpret_cast<const char*>(P.x_in) + 16 * cl;
    const uint64_t ldb = (uint64_t)P.ld_in * 4u;
    const uint32_t n_cols = (uint32_t)(P.n_in < ((int64_t)1 << 31) ? P.n_in : (int64_t)1 << 31);
    // CSR offsets of the vertex in `tile` (length 0 outside the operator)
    auto meta = [&](int64_t tile, int64_t& e0, int& len) {
      const int64_t v = tile * kGfTileV + gr;
      e0 = 0;
      len = 0;
      if (tile < ntiles && v < P.n) {
        const int64_t a = __ldg(P.row_ptr + v), b = __ldg(P.row_ptr + v + 1);
        if (a < 0 || b < a || b > P.nnz) {
          *bad_index = 1;
        } else {
          e0 = a;
          len = (b - a) < (int64_t)(1 << 30) ? (int)(b - a) : (1 << 30);
        }
      }
    };
    // entries q .. q+7 of a row (column -1: none); a column outside X is reported and skipped
    auto entries = [&](int64_t e0, int len, int q, int32_t (&c)[8], float2 (&g)[8]) {
      bool bad = false;
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        c[u] = -1;
        g[u] = make_float2(0.f, 0.f);
        if (q + u < len) {
          const int32_t cc = __ldg(P.col_idx + e0 + q + u);
          g[u] = __ldg(P.vals + e0 + q + u);
          if ((uint32_t)cc < n_cols)
            c[u] = cc;
          else
            bad = true;
        }
      }
      if (bad) {             // (the values of skipped entries stay out too: they need not be finite)
        *bad_index = 1;
#pragma unroll
        for (int u = 0; u < 8; ++u)
          if (c[u] < 0) g[u] = make_float2(0.f, 0.f);
      }
    };
    // (ax, ay) += the entries' values times four channels of their rows of X, 64 j bytes on
    auto accumulate = [&](const int32_t (&c)[8], const float2 (&g)[8], int j, float4& ax, float4& ay) {
      const char* base = x_lane + 64 * j;
      float4 xr[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const uint64_t off = kWide ? (uint64_t)(uint32_t)c[u] * ldb : (uint64_t)(uint32_t)c[u] * (uint32_t)ldb;
        xr[u] = c[u] >= 0 ? __ldg(reinterpret_cast<const float4*>(base + off)) : make_float4(0.f, 0.f, 0.f, 0.f);
      }
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        ax.x = fmaf(g[u].x, xr[u].x, ax.x); ax.y = fmaf(g[u].x, xr[u].y, ax.y);
        ax.z = fmaf(g[u].x, xr[u].z, ax.z); ax.w = fmaf(g[u].x, xr[u].w, ax.w);
        ay.x = fmaf(g[u].y, xr[u].x, ay.x); ay.y = fmaf(g[u].y, xr[u].y, ay.y);
        ay.z = fmaf(g[u].y, xr[u].z, ay.z); ay.w = fmaf(g[u].y, xr[u].w, ay.w);
      }
    };
    uint32_t aphase = 0;
    int64_t e0;
    int len;
    int32_t c_cur[8];
    float2 g_cur[8];
    meta(blockIdx.x, e0, len);
    entries(e0, len, 0, c_cur, g_cur);
    for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
      int64_t e0n;
      int lenn;
      meta(tile + gridDim.x, e0n, lenn);   // the next tile's offsets
      const int mx = __reduce_max_sync(0xffffffffu, len);
#pragma unroll 1
      for (int j = 0; j < nkb; ++j) {
        float4 ax = make_float4(0.f, 0.f, 0.f, 0.f), ay = ax;
        // rows longer than eight entries: the rest first, eight at a time
#pragma unroll 1
        for (int q = 8; q < mx; q += 8) {
          int32_t c_more[8];
          float2 g_more[8];
          entries(e0, len, q, c_more, g_more);
          accumulate(c_more, g_more, j, ax, ay);
        }
        accumulate(c_cur, g_cur, j, ax, ay);
        // even vertices store x first, odd ones y: eight distinct 16-byte chunks per two vertices
        uint8_t* blk = sA + (uint32_t)j * kGfABlock;
        const bool yf = sub & 1;
        *reinterpret_cast<float4*>(blk + sw_chunk(gr, yf ? 4 + cl : cl)) = yf ? ay : ax;
        *reinterpret_cast<float4*>(blk + sw_chunk(gr, yf ? cl : 4 + cl)) = yf ? ax : ay;
        tc::fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) tc::mbar_arrive(&a_full[j]);
      }
      e0 = e0n;
      len = lenn;
      entries(e0, len, 0, c_cur, g_cur);
      // ------------------------------------------------------------ epilogue
      const int quarter = warp & 3;
      const int r = quarter * 32 + lane;
      const int64_t v = tile * kGfTileV + r;
      const bool ok = tc::warp_wait(acc_full, aphase, abort_flag);
      aphase ^= 1;
      tc::tc_fence_after();
      for (int j = warp >> 2; ok && j < dim / 16; j += kGfGatherWarps / 4) {
        const int c0 = 16 * j;
        float pv[16], qv[16];
        tc::tmem_ld16(tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)c0, pv);
        tc::tmem_ld16(tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(dim + c0), qv);
        const uint8_t* blk = sA + (uint32_t)j * kGfABlock;
        float g[16];
#pragma unroll
        for (int h = 0; h < 4; ++h) {
          const float4 xv = *reinterpret_cast<const float4*>(blk + sw_chunk(r, h));
          const float4 yv = *reinterpret_cast<const float4*>(blk + sw_chunk(r, 4 + h));
          g[4 * h + 0] = fmaf(xv.x, pv[4 * h + 0], yv.x * qv[4 * h + 0]);
          g[4 * h + 1] = fmaf(xv.y, pv[4 * h + 1], yv.y * qv[4 * h + 1]);
          g[4 * h + 2] = fmaf(xv.z, pv[4 * h + 2], yv.z * qv[4 * h + 2]);
          g[4 * h + 3] = fmaf(xv.w, pv[4 * h + 3], yv.w * qv[4 * h + 3]);
        }
        if (v < P.n) {
          if (P.out_bf16) {
            uint32_t w[8];
#pragma unroll
            for (int q = 0; q < 8; ++q)
              w[q] = __bfloat16_as_ushort(__float2bfloat16_rn(g[2 * q])) |
                     ((uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(g[2 * q + 1])) << 16);
            uint4* dst = reinterpret_cast<uint4*>(reinterpret_cast<__nv_bfloat16*>(P.out) + v * P.ld_out + c0);
            dst[0] = make_uint4(w[0], w[1], w[2], w[3]);
            dst[1] = make_uint4(w[4], w[5], w[6], w[7]);
          } else {
            float4* dst = reinterpret_cast<float4*>(reinterpret_cast<float*>(P.out) + v * P.ld_out + c0);
#pragma unroll
            for (int h = 0; h < 4; ++h) dst[h] = make_float4(g[4 * h], g[4 * h + 1], g[4 * h + 2], g[4 * h + 3]);
          }
        }
      }
      tc::tc_fence_before();
      // the tile's epilogue has read sA and TMEM before the next gather and its MMAs
      // (and every warp leaves together if a wait gave up)
      if (tc::named_barrier_or(1, 32 * kGfGatherWarps, !ok)) break;
    }
  }
  __syncthreads();
  if (warp == kGfGatherWarps) tc::tmem_dealloc(tmem_base, P.tmem_cols);
  if (tid == 0 && P.status) {
    if (*abort_flag) atomicCAS(P.status, 0, (int)FMAP_ERR_TIMEOUT);
    if (*bad_index) atomicCAS(P.status, 0, (int)FMAP_ERR_INVALID_ARG);
  }
}

size_t gf_smem_bytes(int dim) {
  return 1024 + (size_t)kGfTileV * 2 * dim * 4 + 2 * (size_t)(2 * dim) * 128 + 192;
}

}  // namespace
}  // namespace fmap

using namespace fmap;

extern "C" FMAP_API size_t fmap_gradient_features_ws_bytes(int32_t dim) {
  if (dim < 16 || dim > kGfMaxDim || dim % 16 != 0) return 0;
  return (size_t)(2 * dim) * (size_t)(2 * dim) * sizeof(float);
}

extern "C" FMAP_API int32_t fmap_gradient_features(int64_t n, const int64_t* row_ptr, const int32_t* col_idx,
                                                   const float* g_vals, int64_t nnz, int64_t n_in, const float* x_in,
                                                   int64_t ld_in, int32_t dim, const float* a_re, const float* a_im,
                                                   int32_t variant, void* out, int64_t ld_out, int32_t out_dtype,
                                                   int32_t* status, void* ws, size_t ws_bytes, void* stream) {
  if (n < 0 || nnz < 0 || n_in < 0) return FMAP_ERR_INVALID_ARG;
  if (variant != 0 && variant != 1) return FMAP_ERR_INVALID_ARG;
  if (out_dtype != FMAP_PREC_FP32 && out_dtype != FMAP_PREC_BF16) return FMAP_ERR_INVALID_ARG;
  if (dim < 16 || dim > kGfMaxDim || dim % 16 != 0) return FMAP_ERR_UNSUPPORTED;
  if (n == 0) return FMAP_OK;
  if (!row_ptr || !out || !a_re || !a_im || !status || (nnz > 0 && (!col_idx || !g_vals)) || (n_in > 0 && !x_in))
    return FMAP_ERR_INVALID_ARG;
  if (ld_in < dim || ld_out < dim) return FMAP_ERR_INVALID_ARG;
  if (ld_in % 4 != 0 || ld_out % 8 != 0) return FMAP_ERR_UNSUPPORTED;
  auto aligned = [](const void* p, uintptr_t a) { return (reinterpret_cast<uintptr_t>(p) % a) == 0; };
  if (!aligned(x_in, 16) || !aligned(out, 16) || !aligned(g_vals, 8) || !aligned(row_ptr, 8) ||
      !aligned(col_idx, 4) || !aligned(a_re, 4) || !aligned(a_im, 4) || !aligned(status, 4))
    return FMAP_ERR_UNSUPPORTED;
  if (!ws || !aligned(ws, 256) || ws_bytes < fmap_gradient_features_ws_bytes(dim)) return FMAP_ERR_WORKSPACE;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return FMAP_ERR_CUDA;
  const size_t smem = gf_smem_bytes(dim);
  auto* kernel = ld_in >= ((int64_t)1 << 30) ? gradfeat_kernel<true> : gradfeat_kernel<false>;
  // the limit belongs to the kernel, which other threads launch too: the same for every D
  if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)gf_smem_bytes(kGfMaxDim)) !=
      cudaSuccess)
    return FMAP_ERR_CUDA;
  if (cudaMemsetAsync(status, 0, sizeof(int32_t), st) != cudaSuccess) return FMAP_ERR_CUDA;
  float* img = static_cast<float*>(ws);
  const int img_elems = (2 * dim) * (2 * dim);
  gradfeat_w_image_kernel<<<std::max(1, std::min((img_elems + 255) / 256, 256)), 256, 0, st>>>(a_re, a_im, dim,
                                                                                                 variant, img);
  GfParams p{};
  p.n = n; p.n_in = n_in; p.nnz = nnz;
  p.row_ptr = row_ptr; p.col_idx = col_idx; p.vals = reinterpret_cast<const float2*>(g_vals);
  p.x_in = x_in; p.ld_in = ld_in; p.dim = dim;
  p.out = out; p.ld_out = ld_out; p.out_bf16 = out_dtype == FMAP_PREC_BF16 ? 1 : 0;
  p.w_img = img; p.status = status;
  uint32_t cols = 32;
  while (cols < (uint32_t)(2 * dim)) cols <<= 1;
  p.tmem_cols = cols;
  const int64_t ntiles = (n + kGfTileV - 1) / kGfTileV;
  const int grid = (int)std::min<int64_t>(ntiles, sms);
  kernel<<<grid, kGfThreads, smem, st>>>(p);
  return cudaGetLastError() == cudaSuccess ? FMAP_OK : FMAP_ERR_CUDA;
}
