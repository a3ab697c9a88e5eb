// Backward spectral projection on the tensor cores for FP32 features (chain rule of
// Eq. 1), by BF16 thirds:
//
//   dF_s (n x d, FP32) = diag(M_s) Phi_s (n x k) . dA_s (k x d)
//
// Same split as the FP32 forward projection: Phi and dA are exact sums of three BF16 numbers
// each, and six of the nine products are accumulated in FP32 (what is left out is at most 2^-24
// of a product).
//
// kind::f16 MMA, M = 128 vertices, N = up to three thirds of one group of <= 64 features, K =
// the basis index, 16 at a time. One persistent CTA per SM walks its list of (shape, vertex
// chunk, feature group) items:
//   warp 0       TMA-loads the Phi tiles (128 vertices x 32 basis functions, FP32, 128-byte
//                swizzle) and, once per item, bulk-copies the group's image of dA^T thirds
//                (built once per backward pass) into shared memory;
//   warps 10-25  split one vertex row per lane and store its thirds to a slot of TMEM (the A
//                operand); a tile's two K-steps and every second tile have warps of their own;
//   warp 1       issues three MMAs per K-step, one per third of Phi on all thirds of dA that it
//                meets, into double-buffered accumulators (three sums per feature);
//   warps 2-9    add the three sums, scale each row (vertex) by its mass, and write dF in FP32
//                through shared memory with TMA stores.
// What bounds it: the writes of dF up to k ~ 64, then the MMAs (six products: 250 TF at k = 200)
// and the hand-over of the slots. 32 shapes of n = 50000, d = 256, against Phi and its remainder in
// shared memory, three TF32 MMAs on 64 features at a time and two images of dA^T, for which groups
// shrank to 32 features above k = 192: k = 30 425 -> 441 us, k = 50 567 -> 508, k = 100 1022 -> 869,
// k = 200 3132 -> 1371 (k = 30 with store boxes of 16 features: 515). One accumulator and six slots: 5 to 14% slower; the groups' items one after
// the other instead of chunk by chunk: up to 3% slower at k <= 64, the same above.
// Waits are bounded like the other tensor-core kernels'.
#include "fmap_internal.cuh"
#include "tc_ptx.cuh"

namespace fmap {
namespace {

constexpr int kEpiWarps = 8;
constexpr int kSlots = 2, kSlotCols = 48;            // TMEM slots of A: three thirds of 32 basis functions
constexpr int kConvWarps = 16;                       // by 32 TMEM lanes, K-step of a tile, tile parity
constexpr int kBufs = 2, kAccCols = 192;             // accumulators: three sums of 64 features
static_assert(kSlots % 2 == 0 && kSlots * kSlotCols + kBufs * kAccCols <= 512, "TMEM columns");
constexpr int kThreads = 32 * (2 + kEpiWarps + kConvWarps);
constexpr int kTileV = 128;                          // vertices per output tile (MMA M)
constexpr uint32_t kAStageBytes = kTileV * 128;      // 128 rows x 32 FP32
constexpr uint32_t kOutWarpBytes = 32 * 128;         // 32 rows x 32 FP32: one TMA store box per epilogue warp

__global__ void __launch_bounds__(kThreads, 1) project_bwd_tc32_kernel(TcBwdParams P) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int S = P.stages;
  uint8_t* sB = smem;                                   // dA^T thirds of the item's feature group
  uint8_t* sA = sB + (size_t)P.b_bytes_max;             // Phi tiles
  uint8_t* sOut = sA + (size_t)S * kAStageBytes;    // FP32 dF staging, kOutWarpBytes per epilogue warp
  uint64_t* bars = reinterpret_cast<uint64_t*>(sOut + (size_t)kEpiWarps * kOutWarpBytes);
  uint64_t* a_full = bars;
  uint64_t* a_empty = bars + S;
  uint64_t* slot_full = bars + 2 * S;         // [kSlots]
  uint64_t* slot_empty = slot_full + kSlots;  // [kSlots]
  uint64_t* b_full = slot_empty + kSlots;
  uint64_t* b_empty = b_full + 1;
  uint64_t* acc_full = b_empty + 1;      // [kBufs]
  uint64_t* acc_empty = acc_full + kBufs;    // [kBufs]
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_empty + kBufs);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int it_beg = P.cta_first[blockIdx.x], it_end = P.cta_first[blockIdx.x + 1];
  if (threadIdx.x == 0) {
    for (int s = 0; s < S; ++s) {
      tc::mbar_init(&a_full[s], 1);
      tc::mbar_init(&a_empty[s], kConvWarps / 2);
    }
    for (int q = 0; q < kSlots; ++q) {
      tc::mbar_init(&slot_full[q], kConvWarps / 2);
      tc::mbar_init(&slot_empty[q], 1);
    }
    tc::mbar_init(b_full, 1);
    tc::mbar_init(b_empty, 1);
    for (int b = 0; b < kBufs; ++b) {
      tc::mbar_init(&acc_full[b], 1);
      tc::mbar_init(&acc_empty[b], kEpiWarps);
    }
    *abort_flag = 0;
    tc::fence_mbar_init();
  }
  if (warp == 1) {
    tc::tmem_alloc(tmem_slot, P.tmem_cols);
    tc::tmem_relinquish();
    tc::tc_fence_before();
  }
  __syncthreads();
  tc::tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  if (warp == 0) {
    // ------------------------------------------------------------ TMA producer
    if (lane == 0) {
      uint32_t stage = 0, phase = 0, bphase = 0;
      for (int it = it_beg; it < it_end; ++it) {
        const TcBwdItem item = P.items[it];
        const CUtensorMap* map = P.phimaps + item.shape;
        tc::prefetch_tmap(map);
        if (!tc::mbar_wait(b_empty, bphase ^ 1, abort_flag)) goto producer_done;
        {
          const uint32_t bbytes = (uint32_t)((item.kb + 1) / 2) * 3u * (uint32_t)item.nf * 128u;
          tc::mbar_arrive_expect_tx(b_full, bbytes);
          const uint8_t* src = reinterpret_cast<const uint8_t*>(P.ws + item.img_off);
          for (uint32_t off = 0; off < bbytes; off += 16384u)
            tc::bulk_g2s(sB + off, src + off, (bbytes - off) < 16384u ? (bbytes - off) : 16384u, b_full);
        }
        bphase ^= 1;
        const int ntiles = (int)((item.v1 - item.v0 + kTileV - 1) / kTileV);
        for (int t = 0; t < ntiles; ++t) {
          const int y = (int)(item.v0 + (int64_t)t * kTileV);
          for (int kb = 0; kb < item.kb; ++kb) {
            if (!tc::mbar_wait(&a_empty[stage], phase ^ 1, abort_flag)) goto producer_done;
            tc::mbar_arrive_expect_tx(&a_full[stage], kAStageBytes);
            uint8_t* dst = sA + (size_t)stage * kAStageBytes;
            tc::tma_load_2d(dst, map, &a_full[stage], kb * 32, y);
            tc::tma_load_2d(dst + kAStageBytes / 2, map, &a_full[stage], kb * 32, y + kTileV / 2);
            if (++stage == (uint32_t)S) { stage = 0; phase ^= 1; }
          }
        }
      }
    producer_done:
      if (*abort_flag) {
        const uint64_t t0 = tc::globaltimer();
        while (tc::globaltimer() - t0 < 2000000ull) {}
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issuer
    const bool lead = lane == 0;
    const uint64_t b0 = tc::smem_desc(tc::smem_u32(sB), 16, 1024, tc::kLayoutSW128);
    uint32_t bphase = 0, slot = 0, slot_phase = 0;
    uint32_t acc_phase[kBufs] = {};
    int buf = 0;
    bool ok = true;
    for (int it = it_beg; it < it_end && ok; ++it) {
      const TcBwdItem item = P.items[it];
      const int steps = (P.shapes[item.shape].k + 15) / 16;
      if (!tc::warp_wait(b_full, bphase, abort_flag)) break;
      bphase ^= 1;
      tc::tc_fence_after();
      const uint32_t nf = (uint32_t)item.nf;
      const uint32_t i1 = tc::idesc_bf16_f32(128, nf, 0, 0), i2 = tc::idesc_bf16_f32(128, 2 * nf, 0, 0);
      const uint32_t i3 = tc::idesc_bf16_f32(128, 3 * nf, 0, 0);
      const int ntiles = (int)((item.v1 - item.v0 + kTileV - 1) / kTileV);
      for (int t = 0; t < ntiles && ok; ++t) {
        if (!tc::warp_wait(&acc_empty[buf], acc_phase[buf] ^ 1, abort_flag)) { ok = false; break; }
        tc::tc_fence_after();
        const uint32_t d = tmem_base + (uint32_t)(buf * kAccCols);
        for (int kb = 0; kb < item.kb; ++kb) {
          const uint64_t b = b0 + (uint64_t)((uint32_t)(kb >> 1) * 3u * nf * 8u + (uint32_t)(kb & 1) * 4u);
          const uint32_t a = tmem_base + (uint32_t)(kBufs * kAccCols) + slot * kSlotCols;
          if (!tc::warp_wait(&slot_full[slot], slot_phase, abort_flag)) { ok = false; break; }
          tc::tc_fence_after();
          if (lead) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              if (2 * kb + h < steps) {    // (thirds side by side: rows [Bh | Bm | Bl] of the image)
                tc::mma_bf16_ta(d, a + 24 * h, b + 2 * h, i3, (kb | h) != 0 ? 1u : 0u);
                tc::mma_bf16_ta(d + nf, a + 24 * h + 8, b + 2 * h, i2, 1u);
                tc::mma_bf16_ta(d + 2 * nf, a + 24 * h + 16, b + 2 * h, i1, 1u);
              }
            }
            tc::mma_commit(&slot_empty[slot]);
          }
          if (++slot == (uint32_t)kSlots) { slot = 0; slot_phase ^= 1; }
        }
        if (!ok) break;
        if (lead) tc::mma_commit(&acc_full[buf]);
        acc_phase[buf] ^= 1;
        buf ^= 1;
      }
      if (!ok) break;
      if (lead) tc::mma_commit(b_empty);
    }
  } else if (warp >= 2 + kEpiWarps) {
    // ------------------------------------------------------------ thirds of Phi
    const int quarter = warp & 3, set = (warp - 2 - kEpiWarps) >> 2;
    const int h = set >> 1;
    const int row = quarter * 32 + lane;
    const uint32_t a0 = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(kBufs * kAccCols) + 24 * h;
    uint32_t block = 0, stage = (uint32_t)set & 1, phase = 0, slot = (uint32_t)set & 1, slot_phase = 0;
    for (int it = it_beg; it < it_end; ++it) {
      const TcBwdItem item = P.items[it];
      const uint32_t end = block + (uint32_t)((item.v1 - item.v0 + kTileV - 1) / kTileV) * (uint32_t)item.kb;
      for (uint32_t g = block + ((block + (uint32_t)set) & 1); g < end; g += 2) {
        const uint32_t a = a0 + slot * kSlotCols;
        if (!tc::warp_wait(&a_full[stage], phase, abort_flag)) goto conv_done;
        const uint8_t* src = sA + (size_t)stage * kAStageBytes + row * 128;
        uint32_t hi[8], mid[8], lo[8];
#pragma unroll
        for (int z = 0; z < 4; ++z) {
          const float4 x = *reinterpret_cast<const float4*>(src + (((4 * h + z) ^ (row & 7)) << 4));
          tc::split3(x.x, x.y, hi[2 * z], mid[2 * z], lo[2 * z]);
          tc::split3(x.z, x.w, hi[2 * z + 1], mid[2 * z + 1], lo[2 * z + 1]);
        }
        if (!tc::warp_wait(&slot_empty[slot], slot_phase ^ 1, abort_flag)) goto conv_done;
        tc::tc_fence_after();
        tc::tmem_st8(a, hi);
        tc::tmem_st8(a + 8, mid);
        tc::tmem_st8(a + 16, lo);
        __syncwarp();
        if (lane == 0) tc::mbar_arrive(&a_empty[stage]);
        tc::tmem_st_wait();
        tc::tc_fence_before();
        __syncwarp();
        if (lane == 0) tc::mbar_arrive(&slot_full[slot]);
        if ((stage += 2) >= (uint32_t)S) { stage -= S; phase ^= 1; }
        if ((slot += 2) >= (uint32_t)kSlots) { slot -= kSlots; slot_phase ^= 1; }
      }
      block = end;
    }
  conv_done:;
  } else {
    // ------------------------------------------------------------ epilogue: TMEM -> M * acc -> FP32 dF
    const int quarter = warp & 3, half = (warp - 2) >> 2;
    uint8_t* stage_out = sOut + (size_t)(warp - 2) * kOutWarpBytes;
    uint32_t acc_phase[kBufs] = {};
    int buf = 0;
    for (int it = it_beg; it < it_end; ++it) {
      const TcBwdItem item = P.items[it];
      const ShapeDev s = P.shapes[item.shape];
      const CUtensorMap* dmap = P.dfmaps + item.shape;
      const int ntiles = (int)((item.v1 - item.v0 + kTileV - 1) / kTileV);
      for (int t = 0; t < ntiles; ++t) {
        const int64_t vrow0 = item.v0 + (int64_t)t * kTileV + quarter * 32;
        const int64_t v = vrow0 + lane;
        const float m = v < item.v1 ? __ldg(s.mass + v) : 0.f;
        if (!tc::warp_wait(&acc_full[buf], acc_phase[buf], abort_flag)) goto epi_done;
        tc::tc_fence_after();
        // 32 features per warp, 128-byte rows with the 128-byte swizzle (conflict-free, and half as
        // many box rows as 16 features would make: a TMA store takes about 6 cycles per row)
        const int c0 = 32 * half, nv = item.nf - c0;
        if (lane == 0) tc::bulk_wait_group_read0();     // the previous box's store has read the buffer
        __syncwarp();
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          float x[16];
          if (16 * q < nv) {
            const uint32_t at = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(buf * kAccCols + c0 + 16 * q);
            tc::tmem_ld16(at, x);
#pragma unroll
            for (int r = 1; r < 3; ++r) {
              float w[16];
              tc::tmem_ld16(at + r * item.nf, w);
#pragma unroll
              for (int e = 0; e < 16; ++e) x[e] += w[e];
            }
#pragma unroll
            for (int z = 0; z < 4; ++z)
              *reinterpret_cast<float4*>(stage_out + lane * 128 + (((4 * q + z) ^ (lane & 7)) << 4)) =
                  make_float4(x[4 * z] * m, x[4 * z + 1] * m, x[4 * z + 2] * m, x[4 * z + 3] * m);
          }
        }
        tc::tc_fence_before();
        __syncwarp();
        if (lane == 0) tc::mbar_arrive(&acc_empty[buf]);
        if (nv > 0 && vrow0 < s.n) {
          tc::fence_proxy_async_smem();
          __syncwarp();
          if (lane == 0) {
            tc::tma_store_2d(dmap, stage_out, item.f0 + c0, (int)vrow0);
            tc::bulk_commit_group();
          }
        }
        acc_phase[buf] ^= 1;
        buf ^= 1;
      }
    }
  epi_done:
    if (lane == 0) tc::bulk_wait_group0();
  }

  __syncthreads();
  if (warp == 1) tc::tmem_dealloc(tmem_base, P.tmem_cols);
  if (threadIdx.x == 0 && *abort_flag) atomicExch(P.err, (int)FMAP_ERR_TIMEOUT);
}

// dA_s^T of one feature group as BF16 thirds, K-major with the 128-byte swizzle: block b (basis 64b ..
// 64b+63) holds nf rows of 128 bytes per third, heads, then middles, then tails; 16-byte chunk c of
// row f at c ^ (f & 7). (3 nf is a multiple of 8, as d is of 16.) Eight basis functions, one chunk of
// each third, per thread.
__global__ void build_dat_image32_kernel(const ShapeDev* shapes, const TcBwdGroup* groups, const float* d_a,
                                         float* ws) {
  const TcBwdGroup g = groups[blockIdx.y];
  const ShapeDev s = shapes[g.shape];
  const int total = (g.kb + 1) / 2 * g.nf * 8;
  uint8_t* img = reinterpret_cast<uint8_t*>(ws + g.img_off);
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < total; e += gridDim.x * blockDim.x) {
    const int f = e % g.nf, p = e / g.nf, b = p >> 3, c = p & 7, n = 8 * p;
    const float* src = d_a + s.a_off + (int64_t)n * s.d + g.f0 + f;
    float x[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) x[i] = n + i < s.k ? src[(int64_t)i * s.d] : 0.f;
    uint4 t[3];
    tc::split3(x[0], x[1], t[0].x, t[1].x, t[2].x);
    tc::split3(x[2], x[3], t[0].y, t[1].y, t[2].y);
    tc::split3(x[4], x[5], t[0].z, t[1].z, t[2].z);
    tc::split3(x[6], x[7], t[0].w, t[1].w, t[2].w);
#pragma unroll
    for (int r = 0; r < 3; ++r) {
      const int row = r * g.nf + f;
      *reinterpret_cast<uint4*>(img + ((int64_t)b * 3 * g.nf + row) * 128 + ((c ^ (row & 7)) << 4)) = t[r];
    }
  }
}

}  // namespace

cudaError_t project_bwd_tc32_set_smem(int bytes) {
  return cudaFuncSetAttribute(project_bwd_tc32_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
}

cudaError_t launch_build_dat_image32(const ShapeDev* shapes, const TcBwdGroup* groups, int n_groups, int max_elems,
                                     const float* d_a, float* ws, cudaStream_t st) {
  if (n_groups <= 0) return cudaSuccess;
  dim3 grid((unsigned)std::max(1, std::min((max_elems + 255) / 256, 1024)), (unsigned)n_groups);
  build_dat_image32_kernel<<<grid, 256, 0, st>>>(shapes, groups, d_a, ws);
  return cudaGetLastError();
}

cudaError_t launch_project_bwd_tc32(const TcBwdParams& p, int grid, int smem_bytes, cudaStream_t st) {
  if (grid <= 0) return cudaSuccess;
  project_bwd_tc32_kernel<<<grid, kThreads, smem_bytes, st>>>(p);
  return cudaGetLastError();
}

}  // namespace fmap
