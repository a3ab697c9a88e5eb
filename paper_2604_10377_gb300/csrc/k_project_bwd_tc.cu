// Backward spectral projection on the tensor cores (chain rule of Eq. 1), BF16 features:
//
//   dF_s (n x d) = diag(M_s) Phi_s (n x k) . dA_s (k x d)
//
// kind::tf32 MMA on CTA pairs (cta_group::2): M = 256 vertices, N = up to 256 features, K = the
// basis index in blocks of 32. A cluster of two CTAs walks the vertex tiles of its items; each
// CTA loads the FP32 Phi rows of its own 128 vertices (TMA, K-major) and holds half of the
// features' dA_s^T, prepared once per backward pass as a K-major swizzled FP32 image in the
// workspace and bulk-copied into shared memory per work item; CTA 0 issues the MMAs for both SMs,
// which read each other's half of the B operand. A Phi tile is so read once per 256 features,
// and a K-step takes 8 KB of an SM's shared memory per 128 x 256 outputs; one CTA per 128
// features takes twice both. 64 shapes of n = 50k, d = 256: k = 30 0.681 -> 0.371 ms (5.5 TB/s),
// k = 100 0.710 -> 0.507 (5.8), k = 200 1.045 -> 0.724 (5.8); 8 of n = 200k, k = 200, d = 512
// 1.015 -> 0.647. HBM bounds it (the copy peak is 6.8 TB/s, writes alone reach 4.0); what it
// took beside the pairs: both CTAs' loads counted on the issuer's barrier (a forwarding arrive
// per stage 1.34 ms on the last), as many Phi stages as an item leaves room for, and no release
// of the stores at the accumulator's arrive (it waits for their acknowledgements: 0.741).
// The mass is a per-row (per-TMEM-lane) scale applied in the epilogue, which
// converts to BF16 and writes dF (and, when the shape asks for it, the same values
// before rounding as an FP32 copy). TF32 keeps ~2^-11 relative accuracy of each
// operand, far inside the BF16 storage of dF. Accumulators are double-buffered in
// TMEM so that the epilogue of one vertex tile overlaps the MMAs of the next.
//
// Waits are bounded like the forward kernel's; a timeout sets the workspace
// control word to FMAP_ERR_TIMEOUT.
#include "fmap_internal.cuh"
#include "tc_ptx.cuh"

namespace fmap {
namespace {

constexpr int kEpiWarps = 8;   // two per TMEM lane quarter, each storing half of the columns
constexpr int kThreads = 32 * (2 + kEpiWarps);
constexpr int kTileV = 128;                       // vertices per CTA and tile (half of the pair's MMA M)
constexpr uint32_t kAStageBytes = kTileV * 128;   // 128 rows x 32 fp32
constexpr uint32_t kOutWarpBytes = 32 * 128;      // 32 rows x 64 BF16 per epilogue warp

constexpr int kBwdMaxStages = 12;

// Phi stages of an item whose half of dA^T takes `bbytes` of the region of operands.
__device__ __forceinline__ int bwd_stages(uint32_t region, uint32_t bbytes) {
  return min(kBwdMaxStages, (int)((region - bbytes) / kAStageBytes));
}

__global__ void __launch_bounds__(kThreads, 1) project_bwd_tc_kernel(TcBwdParams P) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  constexpr int S = kBwdMaxStages;
  // per item: the resident dA^T image of this CTA's half of the features, then Phi tiles in as many
  // stages as fit (about 2 us from a stage's release to its next data: the bytes in flight set
  // the rate)
  uint8_t* sB = smem;
  uint8_t* sOut = sB + P.b_bytes_max;                   // BF16 dF staging, kOutWarpBytes per epilogue warp
  uint64_t* bars = reinterpret_cast<uint64_t*>(sOut + (size_t)kEpiWarps * kOutWarpBytes);
  // (a_full, peer_b and acc_empty are CTA 0's: they also count CTA 1's side)
  uint64_t* a_full = bars;
  uint64_t* a_empty = bars + S;
  uint64_t* b_full = bars + 2 * S;
  uint64_t* b_empty = b_full + 1;
  uint64_t* peer_b = b_empty + 1;
  uint64_t* acc_full = peer_b + 1;       // [2]
  uint64_t* acc_empty = acc_full + 2;    // [2]
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_empty + 2);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = tc::cluster_ctarank();     // 0 or 1: which 128 vertices of a tile, which half of B
  const int cl = blockIdx.x >> 1;                  // CTA pair index
  const int it_beg = P.cta_first[cl], it_end = P.cta_first[cl + 1];
  if (threadIdx.x == 0) {
    for (int s = 0; s < S; ++s) {
      tc::mbar_init(&a_full[s], 1);
      tc::mbar_init(&a_empty[s], 1);     // released by the pair's MMAs
    }
    tc::mbar_init(b_full, 1);
    tc::mbar_init(b_empty, 1);
    tc::mbar_init(peer_b, 1);
    for (int b = 0; b < 2; ++b) {
      tc::mbar_init(&acc_full[b], 1);
      tc::mbar_init(&acc_empty[b], 2 * kEpiWarps);
    }
    *abort_flag = 0;
    tc::fence_mbar_init();
  }
  if (warp == 1) {
    tc::tmem_alloc_pair(tmem_slot, P.tmem_cols);
    tc::tmem_relinquish_pair();
    tc::tc_fence_before();
  }
  __syncthreads();
  tc::cluster_sync();                    // both CTAs' barriers are initialised
  tc::tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  if (warp == 0) {
    // ------------------------------------------------------------ TMA producer
    // This CTA's 128 vertices of every stage, as two boxes of 64 vertices.
    if (lane == 0) {
      uint32_t phases = 0, bphase = 0;     // a bit per stage
      for (int it = it_beg; it < it_end; ++it) {
        const TcBwdItem item = P.items[it];
        const CUtensorMap* map = P.phimaps + item.shape;
        tc::prefetch_tmap(map);
        // every MMA of the previous item has completed
        if (!tc::mbar_wait(b_empty, bphase ^ 1, abort_flag)) goto producer_done;
        const uint32_t bbytes = (uint32_t)item.kb * (uint32_t)(item.nf / 2) * 128u;   // this CTA's half
        const int n_stages = bwd_stages(P.b_bytes_max, bbytes);
        int stage = 0;
        {
          tc::mbar_arrive_expect_tx(b_full, bbytes);
          const uint8_t* src = reinterpret_cast<const uint8_t*>(P.ws + item.img_off) + (size_t)rank * bbytes;
          for (uint32_t off = 0; off < bbytes; off += 16384u)
            tc::bulk_g2s(sB + off, src + off, (bbytes - off) < 16384u ? (bbytes - off) : 16384u, b_full);
        }
        bphase ^= 1;
        const int ntiles = (int)((item.v1 - item.v0 + 2 * kTileV - 1) / (2 * kTileV));
        for (int t = 0; t < ntiles; ++t) {
          // (a box past the last vertex reads zeros)
          const int y = (int)(item.v0 + (int64_t)t * 2 * kTileV) + (int)rank * kTileV;
          for (int kb = 0; kb < item.kb; ++kb) {
            if (!tc::mbar_wait(&a_empty[stage], (phases >> stage & 1) ^ 1, abort_flag)) goto producer_done;
            phases ^= 1u << stage;
            // both CTAs' boxes count on CTA 0's barrier, which its issuer waits for
            if (rank == 0) tc::mbar_arrive_expect_tx(&a_full[stage], 2 * kAStageBytes);
            uint8_t* dst = sB + bbytes + (size_t)stage * kAStageBytes;
            tc::tma_load_2d_pair(dst, map, &a_full[stage], 0, kb * 32, y);
            tc::tma_load_2d_pair(dst + kAStageBytes / 2, map, &a_full[stage], 0, kb * 32, y + kTileV / 2);
            if (++stage == n_stages) stage = 0;
          }
        }
      }
      // no MMA still reads this CTA's shared memory when it leaves
      tc::mbar_wait(b_empty, bphase ^ 1, abort_flag);
    producer_done:
      if (*abort_flag) {
        const uint64_t t0 = tc::globaltimer();
        while (tc::globaltimer() - t0 < 2000000ull) {}
      }
    }
  } else if (warp == 1 && rank == 1) {
    // ------------------------------------------------------------ CTA 1: tells CTA 0 that its half of B is there
    if (lane == 0) {
      uint32_t bphase = 0;
      for (int it = it_beg; it < it_end; ++it) {
        if (!tc::mbar_wait(b_full, bphase, abort_flag)) break;
        bphase ^= 1;
        tc::mbar_arrive_cluster(peer_b, 0);
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------ CTA 0: MMA issuer of the pair
    if (lane == 0) {
      uint32_t phases = 0, bphase = 0;
      uint32_t acc_phase[2] = {0, 0};
      int buf = 0;
      bool ok = true;
      for (int it = it_beg; it < it_end && ok; ++it) {
        const TcBwdItem item = P.items[it];
        if (!tc::mbar_wait(b_full, bphase, abort_flag) || !tc::mbar_wait_cluster(peer_b, bphase, abort_flag)) break;
        bphase ^= 1;
        const uint32_t idesc = tc::idesc_tf32(256, (uint32_t)item.nf);
        const uint32_t b_base = tc::smem_u32(sB);
        const uint32_t bbytes = (uint32_t)item.kb * (uint32_t)(item.nf / 2) * 128u;
        const int n_stages = bwd_stages(P.b_bytes_max, bbytes);
        int stage = 0;
        const int ntiles = (int)((item.v1 - item.v0 + 2 * kTileV - 1) / (2 * kTileV));
        for (int t = 0; t < ntiles && ok; ++t) {
          if (!tc::mbar_wait_cluster(&acc_empty[buf], acc_phase[buf] ^ 1, abort_flag)) { ok = false; break; }
          tc::tc_fence_after();
          const uint32_t d = tmem_base + (uint32_t)(buf * (P.tmem_cols / 2));
          for (int kb = 0; kb < item.kb; ++kb) {
            if (!tc::mbar_wait_cluster(&a_full[stage], phases >> stage & 1, abort_flag)) { ok = false; break; }
            phases ^= 1u << stage;
            tc::tc_fence_after();
            const uint32_t a_base = b_base + bbytes + (uint32_t)stage * kAStageBytes;
#pragma unroll
            for (int ks = 0; ks < 4; ++ks) {
              const uint64_t ad = tc::smem_desc(a_base + ks * 32, 16, 1024, tc::kLayoutSW128);
              const uint64_t bd = tc::smem_desc(b_base + (uint32_t)(kb * (item.nf / 2) * 128) + ks * 32, 16, 1024,
                                                tc::kLayoutSW128);
              tc::mma_tf32_pair(d, ad, bd, idesc, (kb | ks) != 0 ? 1u : 0u);
            }
            tc::mma_commit_pair(&a_empty[stage]);
            if (++stage == n_stages) stage = 0;
          }
          if (!ok) break;
          tc::mma_commit_pair(&acc_full[buf]);
          acc_phase[buf] ^= 1;
          buf ^= 1;
        }
        if (!ok) break;
        tc::mma_commit_pair(b_empty);
      }
    }
  } else {
    // ------------------------------------------------------------ epilogue: TMEM -> M * acc -> BF16 dF
    // Each warp takes 32 rows x 64 features at a time: converted into its own shared memory
    // (128-byte rows, 16-byte chunks swizzled: conflict-free), read back as whole rows and written
    // with 16-byte stores of full lines. (A TMA store from that buffer makes the next box wait
    // until it has been read: 0.823 ms against 0.741 at n = 200k, k = 200, d = 512.)
    const int quarter = warp & 3, half = (warp - 2) >> 2;
    uint8_t* stage_out = sOut + (size_t)(warp - 2) * kOutWarpBytes;
    uint32_t acc_phase[2] = {0, 0};
    int buf = 0;
    for (int it = it_beg; it < it_end; ++it) {
      const TcBwdItem item = P.items[it];
      const ShapeDev s = P.shapes[item.shape];
      const int nv = min(item.nf, s.d - item.f0);      // (the MMA's N, a multiple of 32, may pass d)
      const int ntiles = (int)((item.v1 - item.v0 + 2 * kTileV - 1) / (2 * kTileV));
      const int64_t v_first = item.v0 + (int64_t)rank * kTileV + quarter * 32 + lane;
      float m_next = v_first < item.v1 ? __ldg(s.mass + v_first) : 0.f;
      for (int t = 0; t < ntiles; ++t) {
        const int64_t vrow0 = item.v0 + (int64_t)t * 2 * kTileV + (int64_t)rank * kTileV + quarter * 32;
        const int64_t v = vrow0 + lane;
        // the row's mass, loaded a tile ahead
        const float m = m_next;
        m_next = v + 2 * kTileV < item.v1 ? __ldg(s.mass + v + 2 * kTileV) : 0.f;
        if (!tc::warp_wait(&acc_full[buf], acc_phase[buf], abort_flag)) goto epi_done;
        tc::tc_fence_after();
        const int rows = (int)(item.v1 - vrow0 < 32 ? item.v1 - vrow0 : 32);   // (may be negative)
        __nv_bfloat16* out = reinterpret_cast<__nv_bfloat16*>(s.dfeat) + vrow0 * s.ld_feat + item.f0;
        for (int c0 = 64 * half; c0 < nv && rows > 0; c0 += 128) {
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            if (c0 + 32 * h >= nv) break;
            uint32_t x[32];
            tc::tmem_ld32(tmem_base + ((uint32_t)(quarter * 32) << 16) +
                              (uint32_t)(buf * (P.tmem_cols / 2) + c0 + 32 * h), x);
            tc::tmem_ld_wait(x);
            float y[32];
#pragma unroll
            for (int z = 0; z < 32; ++z) y[z] = __uint_as_float(x[z]) * m;
            if (s.dfeat32 != nullptr && lane < rows) {
              float4* d32 = reinterpret_cast<float4*>(s.dfeat32 + v * s.ld_feat + item.f0 + c0 + 32 * h);
#pragma unroll
              for (int z = 0; z < 8; ++z)
                if (c0 + 32 * h + 4 * z < nv) d32[z] = make_float4(y[4 * z], y[4 * z + 1], y[4 * z + 2], y[4 * z + 3]);
            }
#pragma unroll
            for (int z = 0; z < 4; ++z) {
              uint32_t w[4];
#pragma unroll
              for (int q = 0; q < 4; ++q) {
                const __nv_bfloat162 p2 = __floats2bfloat162_rn(y[8 * z + 2 * q], y[8 * z + 2 * q + 1]);
                w[q] = *reinterpret_cast<const uint32_t*>(&p2);
              }
              *reinterpret_cast<uint4*>(stage_out + lane * 128 + (((4 * h + z) ^ (lane & 7)) << 4)) =
                  make_uint4(w[0], w[1], w[2], w[3]);
            }
          }
          __syncwarp();
          // eight lanes a row, four rows at a time
          const int cc = lane & 7;
          const bool on = c0 + 8 * cc < nv;
#pragma unroll
          for (int z = 0; z < 8; ++z) {
            const int r = 4 * z + (lane >> 3);
            const uint4 u = *reinterpret_cast<const uint4*>(stage_out + r * 128 + ((cc ^ (r & 7)) << 4));
            if (on && r < rows) *reinterpret_cast<uint4*>(out + r * s.ld_feat + c0 + 8 * cc) = u;
          }
          __syncwarp();
        }
        tc::tc_fence_before();
        __syncwarp();
        // (its TMEM reads are what the next MMAs wait for; the stores need no order)
        if (lane == 0) tc::mbar_arrive_cluster_relaxed(&acc_empty[buf], 0);
        acc_phase[buf] ^= 1;
        buf ^= 1;
      }
    }
  epi_done:;
  }

  __syncthreads();
  tc::cluster_sync();                    // neither CTA's shared memory or TMEM is still in use by the other
  if (warp == 1) tc::tmem_dealloc_pair(tmem_base, P.tmem_cols);
  if (threadIdx.x == 0 && *abort_flag) atomicExch(P.err, (int)FMAP_ERR_TIMEOUT);
}

// dA_s^T of one feature group as the K-major, 128-byte-swizzled FP32 image the MMA
// reads, the two CTAs' halves of the features one after the other: block kb (basis
// 32kb..32kb+31) of a half holds nf / 2 rows of 128 bytes (one feature per row), 16-byte
// chunk c of row f stored at chunk c ^ (f & 7). Each value is rounded to
// the nearest TF32 here (the MMA would otherwise drop its low 13 bits), so the only
// truncated operand of the product is Phi.
__global__ void build_dat_image_kernel(const ShapeDev* shapes, const TcBwdGroup* groups, const float* d_a,
                                       float* ws) {
  const TcBwdGroup g = groups[blockIdx.y];
  const ShapeDev s = shapes[g.shape];
  const int nh = g.nf / 2, total = g.kb * nh * 32;
  float* img = ws + g.img_off + (int64_t)blockIdx.z * total;
  const int f0 = g.f0 + (int)blockIdx.z * nh;
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < total; e += gridDim.x * blockDim.x) {
    const int kb = e / (nh * 32);
    const int rem = e % (nh * 32);
    const int f = rem / 32, nl = rem % 32;
    const int n = kb * 32 + nl, fg = f0 + f;
    const float raw = (n < s.k && fg < s.d) ? d_a[s.a_off + (int64_t)n * s.d + fg] : 0.f;
    const int chunk = nl >> 2;
    img[(int64_t)kb * nh * 32 + f * 32 + ((chunk ^ (f & 7)) << 2) + (nl & 3)] = tc::tf32_rna(raw);
  }
}

}  // namespace

cudaError_t project_bwd_tc_set_smem(int bytes) {
  return cudaFuncSetAttribute(project_bwd_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
}

cudaError_t launch_build_dat_image(const ShapeDev* shapes, const TcBwdGroup* groups, int n_groups, int max_elems,
                                   const float* d_a, float* ws, cudaStream_t st) {
  if (n_groups <= 0) return cudaSuccess;
  dim3 grid((unsigned)std::max(1, std::min((max_elems / 2 + 255) / 256, 1024)), (unsigned)n_groups, 2);
  build_dat_image_kernel<<<grid, 256, 0, st>>>(shapes, groups, d_a, ws);
  return cudaGetLastError();
}

cudaError_t launch_project_bwd_tc(const TcBwdParams& p, int grid, int smem_bytes, cudaStream_t st) {
  if (grid <= 0) return cudaSuccess;
  // CTAs 2c and 2c + 1 are a cluster of two
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = (size_t)smem_bytes;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, project_bwd_tc_kernel, p);
}

}  // namespace fmap
