// Spectral projection on the 5th-generation tensor cores (Eq. 1), BF16 features.
//
//   A_s^T (d x k) = F_s^T (d x n) . P_s (n x k),   P_s = diag(M_s) Phi_s
//
// One persistent CTA per SM walks its own contiguous range of the batch's
// (shape, feature group) vertex sequence (stream-K split into equal-cost
// ranges); a range is cut into segments at shape / group boundaries and every
// segment writes one partial A. Per stage of 64 or 32 vertices:
//   warp 0      TMA-loads the F tile (MN-major, 128-byte swizzle), the Phi tile
//               (FP32, 32-column boxes, 128-byte swizzle) and the masses;
//   warps 2-9   read Phi and M from shared memory, form P = M * Phi in FP32 and
//               split it into BF16 hi + lo (P = hi + lo to ~2^-17), written in place
//               over the Phi tile as K-major 128-byte-swizzled B tiles: the mass is
//               fused into the operand load;
//   warp 1      issues tcgen05.mma (M = 128 features, K = 16 vertices) into FP32 accumulators
//               in TMEM: N = k rounded up to 16 for hi and for lo, or, where the columns
//               allow it (tc_merged, stages of 64), one MMA on the rows of hi and lo together,
//               whose two accumulators the epilogue adds.
// What bounds it: the reads of F and Phi (6.1 to 6.6 TB/s for most sizes); at small k the MMAs
// come next, each of which reads the F tile and takes its time to issue. 64 shapes of n = 50000,
// d = 256 at k = 30 / 50 / 100 / 200: 433 / 454 / 500 / 789 us with separate MMAs for hi and lo,
// descriptors built between them, one lane issuing all copies and two stages of 64 vertices at
// k = 200; 380 / 405 / 470 / 771 with one MMA; 335 / 364 / 442 / 642 with descriptors ahead of
// the waits, a lane per copy and stages of 32 where three of 64 do not fit. (With one feature group,
// d <= 128, the conversion of Phi bounds it from k = 176 on: 32 shapes of k = 200, d = 128 277 us.)
// At the end of a segment warps 2-9 read the accumulators back (tcgen05.ld) and
// write the segment's partial A; a second kernel adds the partials of each shape
// in a fixed order. F is exact in BF16, so A carries only the ~2^-17 error of
// the hi/lo split and FP32 accumulation.
//
// Every mbarrier wait is bounded (tc::kWaitTimeoutNs); a wait that gives up
// raises a CTA-wide abort flag, every role stops, TMEM is freed, and the
// workspace error word is set to FMAP_ERR_TIMEOUT (reported per pair by the solve).
#include "fmap_internal.cuh"
#include "tc_ptx.cuh"

namespace fmap {
namespace {

constexpr int kConvWarps = 8;
constexpr int kThreads = 32 * (2 + kConvWarps);
constexpr uint32_t kBoxBytes = 32 * 128;       // one TMA box: 32 vertices x 64 features bf16, or x 32 basis functions fp32

// (a, b) -> BF16 heads RN(a), RN(b) and remainders RN(a - head), RN(b - head), each pair
// packed low = a, high = b (one packed conversion per pair).
__device__ __forceinline__ void split_pair(float a, float b, uint32_t& hi, uint32_t& lo) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
  const float2 hf = __bfloat1622float2(h);
  const __nv_bfloat162 l = __floats2bfloat162_rn(a - hf.x, b - hf.y);
  hi = *reinterpret_cast<const uint32_t*>(&h);
  lo = *reinterpret_cast<const uint32_t*>(&l);
}

// The MMAs of one segment. kV: vertices per stage; kFg: feature groups (0: item.fg); kMerged: tc_merged. The
// time per MMA counts at small k, so the descriptors are computed ahead of the waits. (One thread alone waits
// and issues: with its warp waiting beside it 16 shapes of n = 50000, k = 200, d = 256 take 177 us, not 171.)
template <int kV, int kFg, bool kMerged>
__device__ __forceinline__ bool issue_by_one_thread(const TcProjParams& P, const TcItem& item, int nst, uint32_t tmem_base, uint8_t* sF,
                                      uint8_t* sP, uint64_t* full_f, uint64_t* full_p, uint64_t* empty, uint32_t& stage,
                                      uint32_t& phase, volatile int* abort) {
  const int fg = kFg ? kFg : item.fg;
  const uint32_t npad = (uint32_t)item.npad;
  const uint32_t cols = npad * (kMerged ? 2u : 1u);      // accumulator columns per feature group
  const uint32_t idesc = tc::idesc_bf16_f32(128, cols, 1, 0);
  const uint32_t lo = kV == 64 ? npad * 8 : 4;           // from P hi to P lo, in 16-byte units
  for (int st = 0; st < nst; ++st) {
    const uint64_t ad = tc::smem_desc(tc::smem_u32(sF + (size_t)stage * P.f_stage_bytes), kV * 128, 1024, tc::kLayoutSW128);
    const uint64_t bd = tc::smem_desc(tc::smem_u32(sP + (size_t)stage * P.p_stage_bytes), 16, 1024, tc::kLayoutSW128);
    if (!tc::mbar_wait(&full_f[stage], phase, abort) || !tc::mbar_wait(&full_p[stage], phase, abort)) return false;
    tc::tc_fence_after();
#pragma unroll
    for (int kk = 0; kk < kV / 16; ++kk) {
#pragma unroll
      for (int m = 0; m < (kFg ? kFg : 4); ++m) {
        if (m >= fg) break;
        const uint64_t a = ad + ((m * 2 * kV * 128 + kk * 2048) >> 4), b = bd + ((kk * 32) >> 4);
        const uint32_t d = tmem_base + (uint32_t)m * cols;
        tc::mma_bf16(d, a, b, idesc, (st | kk) != 0 ? 1u : 0u);
        if (!kMerged) tc::mma_bf16(d, a, b + lo, idesc, 1u);
      }
    }
    tc::mma_commit(&empty[stage]);
    if (++stage == (uint32_t)P.stages) { stage = 0; phase ^= 1; }
  }
  return true;
}

template <int kStageV>
__global__ void __launch_bounds__(kThreads, 1) project_tc_kernel(TcProjParams P) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int S = P.stages;
  uint8_t* sF = smem;
  uint8_t* sP = sF + (size_t)S * P.f_stage_bytes;       // Phi tile, converted in place into P hi / lo
  float* sM = reinterpret_cast<float*>(sP + (size_t)S * P.p_stage_bytes);   // kStageV masses per stage
  uint64_t* bars = reinterpret_cast<uint64_t*>(sM + (size_t)S * kStageV);
  uint64_t* full_f = bars;
  uint64_t* full_p = bars + S;
  uint64_t* empty = bars + 2 * S;
  uint64_t* acc_full = bars + 3 * S;
  uint64_t* acc_empty = acc_full + 1;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_empty + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < S; ++s) {
      tc::mbar_init(&full_f[s], 1);
      tc::mbar_init(&full_p[s], kConvWarps);
      tc::mbar_init(&empty[s], 1);
    }
    tc::mbar_init(acc_full, 1);
    tc::mbar_init(acc_empty, kConvWarps);
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
    // each lane issues its own boxes
    {
      uint32_t stage = 0, phase = 0;
      for (int it = P.cta_first[blockIdx.x]; it < P.cta_first[blockIdx.x + 1]; ++it) {
        const TcItem item = P.items[it];
        const CUtensorMap* fmap = P.fmaps + item.shape;
        const CUtensorMap* pmap = P.phimaps + item.shape;
        const CUtensorMap* mmap = P.massmaps + item.shape;
        const int nst = (int)((item.v1 - item.v0 + kStageV - 1) / kStageV);
        const int nf = item.fg * 2, kb = (item.npad + 31) / 32;     // at most 8 + 8 boxes
        const uint32_t bytes = (uint32_t)(nf + kb) * (kStageV * 128) + kStageV * 4;
        if (lane == 0) {
          tc::prefetch_tmap(fmap);
          tc::prefetch_tmap(pmap);
          tc::prefetch_tmap(mmap);
        }
        for (int st = 0; st < nst; ++st) {
          if (!tc::warp_wait(&empty[stage], phase ^ 1, abort_flag)) goto producer_done;
          if (lane == 0) tc::mbar_arrive_expect_tx(&full_f[stage], bytes);
          __syncwarp();
          const int y = (int)(item.v0 + (int64_t)st * kStageV);
#pragma unroll
          for (int h = 0; h < kStageV / 32; ++h) {
            if (lane < nf) {
              tc::tma_load_2d(sF + (size_t)stage * P.f_stage_bytes + lane * (kStageV * 128) + h * kBoxBytes, fmap,
                              &full_f[stage], item.f0 + lane * 64, y + 32 * h);
            } else if (lane < nf + kb) {
              const int b = lane - nf;
              tc::tma_load_2d(sP + (size_t)stage * P.p_stage_bytes + b * (kStageV * 128) + h * kBoxBytes, pmap,
                              &full_f[stage], item.n0 + b * 32, y + 32 * h);
            } else if (lane == 31) {
              tc::tma_load_1d(sM + (size_t)stage * kStageV + 32 * h, mmap, &full_f[stage], y + 32 * h);
            }
          }
          if (++stage == (uint32_t)S) { stage = 0; phase ^= 1; }
        }
      }
    producer_done:
      if (lane == 0 && *abort_flag) {
        // let copies already in flight land before the CTA's shared memory goes away
        const uint64_t t0 = tc::globaltimer();
        while (tc::globaltimer() - t0 < 2000000ull) {}
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issuer
    if (lane == 0) {
      uint32_t stage = 0, phase = 0, acc_phase = 0;
      for (int it = P.cta_first[blockIdx.x]; it < P.cta_first[blockIdx.x + 1]; ++it) {
        const TcItem item = P.items[it];
        if (!tc::mbar_wait(acc_empty, acc_phase ^ 1, abort_flag)) break;
        tc::tc_fence_after();
        const int nst = (int)((item.v1 - item.v0 + kStageV - 1) / kStageV);
        bool ok;
        if constexpr (kStageV == 32) {
          ok = item.fg == 2 ? issue_by_one_thread<32, 2, false>(P, item, nst, tmem_base, sF, sP, full_f, full_p, empty, stage, phase, abort_flag)
                            : issue_by_one_thread<32, 0, false>(P, item, nst, tmem_base, sF, sP, full_f, full_p, empty, stage, phase, abort_flag);
        } else if (tc_merged(item.fg, item.npad)) {
          ok = item.fg == 1   ? issue_by_one_thread<64, 1, true>(P, item, nst, tmem_base, sF, sP, full_f, full_p, empty, stage, phase, abort_flag)
               : item.fg == 2 ? issue_by_one_thread<64, 2, true>(P, item, nst, tmem_base, sF, sP, full_f, full_p, empty, stage, phase, abort_flag)
                              : issue_by_one_thread<64, 0, true>(P, item, nst, tmem_base, sF, sP, full_f, full_p, empty, stage, phase, abort_flag);
        } else {
          ok = issue_by_one_thread<64, 0, false>(P, item, nst, tmem_base, sF, sP, full_f, full_p, empty, stage, phase, abort_flag);
        }
        if (!ok) break;
        tc::mma_commit(acc_full);
        acc_phase ^= 1;
      }
    }
  } else {
    // ------------------------------------------------------------ converters + epilogue
    const int cw = warp - 2;
    const int qs = lane & 7, csub = lane >> 3;
    uint32_t stage = 0, phase = 0, acc_phase = 0;
    // No wait of this thread has given up. The converters meet in a barrier per stage and load TMEM
    // together, so a thread whose wait gave up does not leave: it goes through what remains without
    // waiting (the segment's values are void then, and reported so).
    bool ok = true;
    for (int it = P.cta_first[blockIdx.x]; it < P.cta_first[blockIdx.x + 1]; ++it) {
      const TcItem item = P.items[it];
      const ShapeDev s = P.shapes[item.shape];
      const int nst = (int)((item.v1 - item.v0 + kStageV - 1) / kStageV);
      const int kb = (item.npad + 31) / 32;
      for (int st = 0; st < nst; ++st) {
        if (ok) ok = tc::mbar_wait(&full_f[stage], phase, abort_flag);
        uint8_t* tile = sP + (size_t)stage * P.p_stage_bytes;
        const float* mst = sM + (size_t)stage * kStageV;
        const int64_t vbase = item.v0 + (int64_t)st * kStageV;
        // read phase: unit (box b, row group c = 4 cg + csub, quad qs) = rows 8c..8c+7 x basis 32b+4qs..+3
        float4 x[kStageV / 32][8];
#pragma unroll
        for (int r = 0; r < kStageV / 32; ++r) {
          const int wu = cw + kConvWarps * r;
          if (wu < kStageV / 32 * kb) {
            const int b = kStageV == 64 ? wu >> 1 : wu, c = kStageV == 64 ? 4 * (wu & 1) + csub : csub;
#pragma unroll
            for (int i = 0; i < 8; ++i) {
              const int vl = 8 * c + i;
              x[r][i] = *reinterpret_cast<const float4*>(tile + b * (kStageV * 128) + vl * 128 + ((qs ^ (vl & 7)) << 4));
            }
          }
        }
        tc::named_barrier_sync(1, 32 * kConvWarps);
        // write phase, K-major, 128-byte swizzle: 64 vertices: P hi at [0, npad*128), lo at [npad*128, 2*npad*128);
        // 32: hi in the first half of each row, lo in the second
        uint8_t* th = tile;
        uint8_t* tl = kStageV == 64 ? tile + (size_t)item.npad * 128 : tile;
#pragma unroll
        for (int r = 0; r < kStageV / 32; ++r) {
          const int wu = cw + kConvWarps * r;
          if (wu < kStageV / 32 * kb) {
            const int b = kStageV == 64 ? wu >> 1 : wu, c = kStageV == 64 ? 4 * (wu & 1) + csub : csub;
            float mv[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) mv[i] = (vbase + 8 * c + i < item.v1) ? mst[8 * c + i] : 0.f;
            const int n0 = 32 * b + 4 * qs;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              const int n = n0 + j;
              if (n >= item.npad) continue;
              float pv[8];
#pragma unroll
              for (int i = 0; i < 8; ++i) {
                const float4 q = x[r][i];
                const float xv = j == 0 ? q.x : (j == 1 ? q.y : (j == 2 ? q.z : q.w));
                pv[i] = xv * mv[i];
              }
              uint4 hv, lv;
              split_pair(pv[0], pv[1], hv.x, lv.x);
              split_pair(pv[2], pv[3], hv.y, lv.y);
              split_pair(pv[4], pv[5], hv.z, lv.z);
              split_pair(pv[6], pv[7], hv.w, lv.w);
              const uint32_t off = (uint32_t)n * 128u + ((uint32_t)(c ^ (n & 7)) << 4);
              *reinterpret_cast<uint4*>(th + off) = hv;
              *reinterpret_cast<uint4*>(tl + (kStageV == 64 ? off : off ^ 64u)) = lv;
            }
          }
        }
        tc::fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) tc::mbar_arrive(&full_p[stage]);
        if (++stage == (uint32_t)S) { stage = 0; phase ^= 1; }
      }
      // epilogue: accumulators -> this item's partial A (k x stride, row-major)
      if (ok) ok = tc::mbar_wait(acc_full, acc_phase, abort_flag);
      __syncwarp();
      tc::tc_fence_after();
      {
        const int quarter = warp & 3, half = cw >> 2;
        const int stride = item.fg * 128;
        float* part = P.ws + item.part_off;
        const bool merged = kStageV == 64 && tc_merged(item.fg, item.npad);
        const int cols = item.npad * (merged ? 2 : 1);
        for (int m = 0; m < item.fg; ++m) {
          const int fl = m * 128 + quarter * 32 + lane;
          const bool fok = item.f0 + fl < s.d;
          for (int ch = half; ch < item.npad / 16; ch += 2) {
            float v[16];
            tc::tmem_ld16(tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(m * cols + ch * 16), v);
            if (merged) {
              float w[16];
              tc::tmem_ld16(tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(m * cols + item.npad + ch * 16), w);
#pragma unroll
              for (int t = 0; t < 16; ++t) v[t] += w[t];
            }
            if (fok) {
#pragma unroll
              for (int t = 0; t < 16; ++t) {
                const int n = ch * 16 + t;
                if (n < item.nk) part[(int64_t)n * stride + fl] = v[t];
              }
            }
          }
        }
      }
      tc::tc_fence_before();
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(acc_empty);
      acc_phase ^= 1;
    }
  }

  __syncthreads();
  if (warp == 1) tc::tmem_dealloc(tmem_base, P.tmem_cols);
  if (threadIdx.x == 0 && *abort_flag) atomicExch(P.err, (int)FMAP_ERR_TIMEOUT);
}

// A_s[n0 + n][f0 + f] = sum over the group's partials [n][f], in a fixed order. From 16 partials four
// thread groups take every fourth one, four loads in flight each, and their sums are added in order
// (one thread adding every partial waits for one L2 round trip after another: one pair of n = 5000,
// 76 partials per shape: 17 us against 11); below, a thread takes all of them (40 shapes of n = 1000,
// k = 250, d = 512, 2 partials: 43 us in four groups, 24 so; 64 of n = 4000, k = 200, d = 256, 8: 38, 31).
__global__ void __launch_bounds__(256) project_tc_reduce_kernel(const ShapeDev* shapes, const int64_t* parts,
                                                                const TcRedGroup* groups, float* a_out, const float* ws) {
  __shared__ float4 red[3][64];
  const TcRedGroup g = groups[blockIdx.y];
  // four consecutive features per thread (dspan, f0, d are multiples of 16 and the
  // partials are 256-byte aligned; float4 stores when the output buffer is 16-byte aligned)
  const int q4 = g.dspan >> 2, total = g.nk * q4;
  const int subs = tc_red_subs(g.part_end - g.part_beg), per = 256 / subs;      // thread groups, elements of each
  if ((int)blockIdx.x * per >= total) return;
  const ShapeDev s = shapes[g.shape];
  const bool vec = (reinterpret_cast<uintptr_t>(a_out) & 15) == 0;
  float* out = a_out + s.a_off + (int64_t)g.n0 * s.d + g.f0;
  const int sub = threadIdx.x / per, lane = threadIdx.x - sub * per;
  for (int e0 = blockIdx.x * per; e0 < total; e0 += gridDim.x * per) {
    const int e = e0 + lane;
    const int n = e / q4, f = (e - n * q4) * 4;
    const float* src = ws + (int64_t)n * g.stride + f;
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    if (e < total) {
      for (int i = g.part_beg + sub; i < g.part_end; i += 4 * subs) {
        float4 u[4];
#pragma unroll
        for (int j = 0; j < 4; ++j)
          u[j] = i + subs * j < g.part_end ? *reinterpret_cast<const float4*>(src + __ldg(parts + i + subs * j))
                                           : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int j = 0; j < 4; ++j) { acc.x += u[j].x; acc.y += u[j].y; acc.z += u[j].z; acc.w += u[j].w; }
      }
    }
    if (subs > 1) {
      __syncthreads();                 // (the previous round's sums have been read)
      if (sub > 0) red[sub - 1][lane] = acc;
      __syncthreads();
      if (sub == 0) {
#pragma unroll
        for (int j = 0; j < 3; ++j) {
          const float4 u = red[j][lane];
          acc.x += u.x; acc.y += u.y; acc.z += u.z; acc.w += u.w;
        }
      }
    }
    if (sub == 0 && e < total) {
      float* o = out + (int64_t)n * s.d + f;
      if (vec) {
        *reinterpret_cast<float4*>(o) = acc;
      } else {
        o[0] = acc.x; o[1] = acc.y; o[2] = acc.z; o[3] = acc.w;
      }
    }
  }
}

}  // namespace

cudaError_t project_tc_set_smem(int bytes) {
  const cudaError_t e = cudaFuncSetAttribute(project_tc_kernel<64>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(project_tc_kernel<32>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
}

cudaError_t launch_project_tc(const TcProjParams& p, int grid, int smem_bytes, cudaStream_t st) {
  if (grid <= 0) return cudaSuccess;
  if (p.stage_v == 64) project_tc_kernel<64><<<grid, kThreads, smem_bytes, st>>>(p);
  else project_tc_kernel<32><<<grid, kThreads, smem_bytes, st>>>(p);
  return cudaGetLastError();
}

cudaError_t launch_project_tc_reduce(const ShapeDev* shapes, const int64_t* parts, const TcRedGroup* groups,
                                     int n_groups, int64_t max_blocks, float* a_out, const float* ws, cudaStream_t st) {
  if (n_groups <= 0) return cudaSuccess;
  dim3 grid((unsigned)std::min<int64_t>(max_blocks, 4096), (unsigned)n_groups);
  project_tc_reduce_kernel<<<grid, 256, 0, st>>>(shapes, parts, groups, a_out, ws);
  return cudaGetLastError();
}

}  // namespace fmap
