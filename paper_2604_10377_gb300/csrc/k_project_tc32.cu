// Spectral projection on the tensor cores (Eq. 1) for FP32 features, by BF16 thirds:
//
//   A_s^T (d x k) = F_s^T (d x n) . P_s (n x k),   P_s = diag(M_s) Phi_s
//
// Each FP32 operand is the exact sum of three BF16 numbers (head, middle, tail: 8 bits each,
// rounded to nearest), F = Fh + Fm + Fl and P = Ph + Pm + Pl. Six of the nine products are
// accumulated in FP32,
//   Fh.Ph + (Fh.Pm + Fm.Ph) + (Fh.Pl + Fm.Pm + Fl.Ph),
// which leaves out at most 2^-24 of a product (half an ulp of it; typically 2^-26). Operands below
// about 1e-34 lose their tails, then their middles, to the smallest BF16 (2^-133): 3e-6 of a result at
// 1e-35, 3e-4 at 1e-37.
//
// What bounds it: at small k the reads of F and Phi, and beside them what a stage costs each
// role in turn (issuing its copies and MMAs, splitting, handing over); from k ~ 100 the MMAs and
// the partials. An operand that a converter writes to shared memory costs its write and one read
// per MMA, so the thirds of F go to TMEM (the A operand of the MMA may come from there; a thread
// holds one feature, whose vertices are the K dimension, and no transpose is left), and only the
// thirds of P, the smaller operand, are written to shared memory, in vertex rows as they arrive.
// 32 shapes of n = 50000, d = 256 (3.0 GB at k = 200), against two TF32 parts of each operand in
// shared memory, F transposed, three MMAs: k = 30 646 -> 356 us, k = 50 702 -> 360 us, k = 100
// 809 -> 513 us, k = 200 (two passes over F then, one now) 1718 -> 701 us; error against 64 bits
// at k = 50 3.3e-6 -> 7e-7, at k = 200 3.5e-6 -> 3.2e-6. One lane issuing all copies of a
// stage: 420 us at k = 50; MMA descriptors built between the MMAs: 422 us; twice the converter
// warps: 371 us; three or four slots: no gain; stages of one step: 600 us.
//
// Same schedule as the BF16 kernel (one persistent CTA per SM over a stream-K range of
// (shape, feature group) segments, partials reduced in a fixed order by a second kernel), with
// stages of 32 vertices (two K-steps of 16):
//   warp 0       TMA-loads the F tile (FP32, 32-feature boxes, 128-byte swizzle), the Phi tile
//                (FP32, 32-column boxes) and the masses;
//   warps 2-9    read one feature per lane, split it and store the thirds to a slot of TMEM;
//   warps 10-13  form P = M * Phi, split it and write the thirds to a slot of shared memory
//                (B operand, MN-major, 128-byte swizzle, 64 columns per group);
//   warp 1       issues tcgen05.mma kind::f16 (M = 128 features, N = k rounded up to 16, K = 16
//                vertices): six per feature group and step, or three, one per third of F on all
//                thirds of P that it meets, where three accumulators fit (tc32_accs). With an
//                accumulator of its own the heads' chain has one add per step, and the rounding
//                of the others is 2^-8 smaller.
// Warps 2-9 write a segment's partial at its end. Waits are bounded like the BF16 kernel's.
#include "fmap_internal.cuh"
#include "tc_ptx.cuh"

namespace fmap {
namespace {

constexpr int kFWarps = 8, kPWarps = 4;
constexpr int kThreads = 32 * (2 + kFWarps + kPWarps);
constexpr int kStageV = 32;                       // vertices per pipeline stage
constexpr int kStepV = 16;                        // vertices per K-step (one slot)
constexpr uint32_t kBoxBytes = kStageV * 128;     // one TMA box: 32 vertices x 32 FP32 (features or basis)
constexpr uint32_t kColBytes = kStepV * 128;      // 16 vertices x 64 basis functions of one third

// The MMAs of one segment of kFg feature groups and kAccs accumulators each. One thread issues them,
// and at small k the time it takes per MMA counts: everything but the waits is computed beforehand.
template <int kFg, int kAccs>
__device__ __forceinline__ bool issue(const TcProjParams& P, const TcItem& item, int nst, uint32_t tmem_base, uint8_t* sB,
                                      uint64_t* part_full, uint64_t* part_empty, uint32_t& phase, volatile int* abort) {
  const bool lead = (threadIdx.x & 31) == 0;
  const uint32_t npad = (uint32_t)item.npad;
  const uint32_t i1 = tc::idesc_bf16_f32(128, npad, 0, 1);
  const uint32_t i2 = tc::idesc_bf16_f32(128, 2 * npad, 0, 1), i3 = tc::idesc_bf16_f32(128, 3 * npad, 0, 1);
  const uint64_t third = (uint64_t)(((npad + 63) / 64) * kColBytes) >> 4;      // in descriptor units
  uint64_t bh[kTc32Slots];
#pragma unroll
  for (int q = 0; q < kTc32Slots; ++q)
    bh[q] = tc::smem_desc(tc::smem_u32(sB + (size_t)q * P.part_bytes), kColBytes, 1024, tc::kLayoutSW128);
  for (int st = 0; st < nst; ++st) {
#pragma unroll
    for (int q = 0; q < kTc32Slots; ++q) {
      if (!tc::warp_wait(&part_full[q], phase, abort)) return false;
      tc::tc_fence_after();
      const uint32_t on = st == 0 && q == 0 ? 0u : 1u;
#pragma unroll
      for (int m = 0; m < kFg; ++m) {
        const uint32_t a = tmem_base + (uint32_t)(512 - (q * kFg + m + 1) * kTc32SlotCols);
        const uint32_t d = tmem_base + (uint32_t)(m * kAccs) * npad;
        if (kAccs == 3) {                 // [Ph | Pm | Pl] side by side
          if (lead) tc::mma_bf16_ta(d, a, bh[q], i3, on);
          if (lead) tc::mma_bf16_ta(d + npad, a + 8, bh[q], i2, 1u);
          if (lead) tc::mma_bf16_ta(d + 2 * npad, a + 16, bh[q], i1, 1u);
        } else {
          const uint32_t e = d + (uint32_t)(kAccs - 1) * npad;
          if (lead) tc::mma_bf16_ta(d, a, bh[q], i1, on);
          if (lead) tc::mma_bf16_ta(e, a, bh[q] + third, i1, kAccs == 2 ? on : 1u);
          if (lead) tc::mma_bf16_ta(e, a, bh[q] + 2 * third, i1, 1u);
          if (lead) tc::mma_bf16_ta(e, a + 8, bh[q], i1, 1u);
          if (lead) tc::mma_bf16_ta(e, a + 8, bh[q] + third, i1, 1u);
          if (lead) tc::mma_bf16_ta(e, a + 16, bh[q], i1, 1u);
        }
      }
      if (lead) tc::mma_commit(&part_empty[q]);
    }
    phase ^= 1;
  }
  return true;
}

__global__ void __launch_bounds__(kThreads, 1) project_tc32_kernel(TcProjParams P) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int S = P.stages;
  uint8_t* sF = smem;
  uint8_t* sP = sF + (size_t)S * P.f_stage_bytes;
  uint8_t* sB = sP + (size_t)S * P.p_stage_bytes;                            // kTc32Slots slots
  float* sM = reinterpret_cast<float*>(sB + (size_t)kTc32Slots * P.part_bytes);   // 32 masses per stage
  uint64_t* bars = reinterpret_cast<uint64_t*>(sM + (size_t)S * kStageV);
  uint64_t* full = bars;                // [S] F, Phi and masses have landed
  uint64_t* empty = bars + S;           // [S] every converter has read them
  uint64_t* part_full = bars + 2 * S;   // [kTc32Slots] the thirds are in place
  uint64_t* part_empty = part_full + kTc32Slots;   // the MMAs have read them
  uint64_t* acc_full = part_empty + kTc32Slots;
  uint64_t* acc_empty = acc_full + 1;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_empty + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < S; ++s) {
      tc::mbar_init(&full[s], 1);
      tc::mbar_init(&empty[s], kFWarps + kPWarps);
    }
    for (int q = 0; q < kTc32Slots; ++q) {
      tc::mbar_init(&part_full[q], kFWarps + kPWarps);
      tc::mbar_init(&part_empty[q], 1);
    }
    tc::mbar_init(acc_full, 1);
    tc::mbar_init(acc_empty, kFWarps);
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
    // each lane issues its own boxes: one lane issuing all of a stage's takes longer than the copies
    {
      uint32_t stage = 0, phase = 0;
      for (int it = P.cta_first[blockIdx.x]; it < P.cta_first[blockIdx.x + 1]; ++it) {
        const TcItem item = P.items[it];
        const CUtensorMap* fmap = P.fmaps + item.shape;
        const CUtensorMap* pmap = P.phimaps + item.shape;
        const CUtensorMap* mmap = P.massmaps + item.shape;
        const int nst = (int)((item.v1 - item.v0 + kStageV - 1) / kStageV);
        const int nf = item.fg * 4, kb = (item.npad + 31) / 32;
        const uint32_t bytes = (uint32_t)(nf + kb) * kBoxBytes + kStageV * 4;
        if (lane == 0) {
          tc::prefetch_tmap(fmap);
          tc::prefetch_tmap(pmap);
          tc::prefetch_tmap(mmap);
        }
        for (int st = 0; st < nst; ++st) {
          if (!tc::warp_wait(&empty[stage], phase ^ 1, abort_flag)) goto producer_done;
          if (lane == 0) tc::mbar_arrive_expect_tx(&full[stage], bytes);
          __syncwarp();
          const int y = (int)(item.v0 + (int64_t)st * kStageV);
          if (lane < nf) {
            tc::tma_load_2d(sF + (size_t)stage * P.f_stage_bytes + lane * kBoxBytes, fmap, &full[stage],
                            item.f0 + lane * 32, y);
          } else if (lane < nf + kb) {
            const int b = lane - nf;
            tc::tma_load_2d(sP + (size_t)stage * P.p_stage_bytes + b * kBoxBytes, pmap, &full[stage], item.n0 + b * 32, y);
          } else if (lane == 31) {
            tc::tma_load_1d(sM + (size_t)stage * kStageV, mmap, &full[stage], y);
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
    {
      uint32_t phase = 0, acc_phase = 0;
      for (int it = P.cta_first[blockIdx.x]; it < P.cta_first[blockIdx.x + 1]; ++it) {
        const TcItem item = P.items[it];
        if (!tc::warp_wait(acc_empty, acc_phase ^ 1, abort_flag)) break;
        tc::tc_fence_after();
        const int nst = (int)((item.v1 - item.v0 + kStageV - 1) / kStageV);
        const int accs = tc32_accs(item.fg, item.npad);
        bool ok;
        if (accs == 3) {
          ok = item.fg == 2 ? issue<2, 3>(P, item, nst, tmem_base, sB, part_full, part_empty, phase, abort_flag)
                            : issue<1, 3>(P, item, nst, tmem_base, sB, part_full, part_empty, phase, abort_flag);
        } else if (accs == 2) {
          ok = item.fg == 2 ? issue<2, 2>(P, item, nst, tmem_base, sB, part_full, part_empty, phase, abort_flag)
                            : issue<1, 2>(P, item, nst, tmem_base, sB, part_full, part_empty, phase, abort_flag);
        } else {
          ok = item.fg == 2 ? issue<2, 1>(P, item, nst, tmem_base, sB, part_full, part_empty, phase, abort_flag)
                            : issue<1, 1>(P, item, nst, tmem_base, sB, part_full, part_empty, phase, abort_flag);
        }
        if (!ok) break;
        if (lane == 0) tc::mma_commit(acc_full);
        acc_phase ^= 1;
      }
    }
  } else if (warp < 2 + kFWarps) {
    // ------------------------------------------------------------ thirds of F, epilogue
    const int quarter = warp & 3, set = (warp - 2) >> 2;
    const uint32_t lane_base = tmem_base + ((uint32_t)(quarter * 32) << 16);
    uint32_t off[8];                      // this lane's feature in vertex row i of an 8-row swizzle atom
#pragma unroll
    for (int i = 0; i < 8; ++i) off[i] = (uint32_t)i * 128u + ((uint32_t)((lane >> 2) ^ i) << 4) + (uint32_t)(lane & 3) * 4u;
    uint32_t stage = 0, phase = 0, slot = 0, slot_phase = 0, acc_phase = 0;
    for (int it = P.cta_first[blockIdx.x]; it < P.cta_first[blockIdx.x + 1]; ++it) {
      const TcItem item = P.items[it];
      const ShapeDev s = P.shapes[item.shape];
      const int nst = (int)((item.v1 - item.v0 + kStageV - 1) / kStageV);
      // two feature groups: one each for the two sets of four warps; one group: 8 vertices each
      const bool two = item.fg == 2;
      const int m = two ? set : 0;
      const uint32_t c0 = two ? 0u : (uint32_t)set;
      for (int st = 0; st < nst; ++st) {
        if (!tc::warp_wait(&full[stage], phase, abort_flag)) goto done;
        const uint8_t* tile = sF + (size_t)stage * P.f_stage_bytes + (m * 4 + quarter) * kBoxBytes + c0 * 1024;
#pragma unroll
        for (int step = 0; step < kStageV / kStepV; ++step) {
          float x[16];
#pragma unroll
          for (int i = 0; i < 8; ++i) x[i] = *reinterpret_cast<const float*>(tile + step * 2048 + off[i]);
          if (two) {
#pragma unroll
            for (int i = 0; i < 8; ++i) x[8 + i] = *reinterpret_cast<const float*>(tile + step * 2048 + 1024 + off[i]);
          }
          uint32_t h[4], md[4], l[4];
#pragma unroll
          for (int i = 0; i < 4; ++i) tc::split3(x[2 * i], x[2 * i + 1], h[i], md[i], l[i]);
          if (!tc::warp_wait(&part_empty[slot], slot_phase ^ 1, abort_flag)) goto done;
          tc::tc_fence_after();
          const uint32_t a = lane_base + 512u - (uint32_t)((slot * item.fg + m + 1) * kTc32SlotCols) + c0 * 4;
          tc::tmem_st4(a, h);
          tc::tmem_st4(a + 8, md);
          tc::tmem_st4(a + 16, l);
          if (two) {
#pragma unroll
            for (int i = 0; i < 4; ++i) tc::split3(x[8 + 2 * i], x[9 + 2 * i], h[i], md[i], l[i]);
            tc::tmem_st4(a + 4, h);
            tc::tmem_st4(a + 12, md);
            tc::tmem_st4(a + 20, l);
          }
          if (step == kStageV / kStepV - 1) {
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(&empty[stage]);
          }
          tc::tmem_st_wait();
          tc::tc_fence_before();
          __syncwarp();
          if (lane == 0) tc::mbar_arrive(&part_full[slot]);
          if (++slot == (uint32_t)kTc32Slots) { slot = 0; slot_phase ^= 1; }
        }
        if (++stage == (uint32_t)S) { stage = 0; phase ^= 1; }
      }
      // accumulators -> this item's partial A (nk x stride, row-major)
      if (!tc::warp_wait(acc_full, acc_phase, abort_flag)) goto done;
      tc::tc_fence_after();
      {
        const int accs = tc32_accs(item.fg, item.npad);
        const int stride = item.fg * 128;
        float* part = P.ws + item.part_off;
        for (int g = 0; g < item.fg; ++g) {
          const int fl = g * 128 + quarter * 32 + lane;
          const bool fok = item.f0 + fl < s.d;
          for (int ch = set; ch < item.npad / 16; ch += 2) {
            const uint32_t d = lane_base + (uint32_t)(g * accs * item.npad + ch * 16);
            float v[16];
            tc::tmem_ld16(d, v);
            for (int r = 1; r < accs; ++r) {
              float w[16];
              tc::tmem_ld16(d + r * item.npad, w);
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
  } else {
    // ------------------------------------------------------------ thirds of P
    const int pt = threadIdx.x - 32 * (2 + kFWarps);   // 0 .. 127
    // 8 lanes read 64 columns of one vertex row, 8 each: the two boxes' lanes take their two
    // 16-byte chunks in opposite order, so that each read touches 32 distinct banks
    const int j = pt & 7, v = pt >> 3, swap = j >> 2;
    const uint32_t row = (uint32_t)swap * kBoxBytes + (uint32_t)v * 128u;
    const uint32_t ca = row + ((uint32_t)((2 * (j & 3) + swap) ^ (v & 7)) << 4);
    const uint32_t cb = row + ((uint32_t)((2 * (j & 3) + (swap ^ 1)) ^ (v & 7)) << 4);
    uint32_t stage = 0, phase = 0, slot = 0, slot_phase = 0;
    for (int it = P.cta_first[blockIdx.x]; it < P.cta_first[blockIdx.x + 1]; ++it) {
      const TcItem item = P.items[it];
      const int nst = (int)((item.v1 - item.v0 + kStageV - 1) / kStageV);
      const int ng = (item.npad + 63) / 64;
      // chunk of 8 columns p * stride + j of the slot: the thirds side by side, or 64-column aligned
      const int stride = tc32_accs(item.fg, item.npad) == 3 ? item.npad / 8 : ng * 8;
      uint32_t dst[3];
#pragma unroll
      for (int p = 0; p < 3; ++p) {
        const int ci = p * stride + j;
        dst[p] = (uint32_t)(ci >> 3) * kColBytes + (uint32_t)v * 128u + ((uint32_t)((ci ^ v) & 7) << 4);
      }
      for (int st = 0; st < nst; ++st) {
        if (!tc::warp_wait(&full[stage], phase, abort_flag)) goto done;
#pragma unroll
        for (int step = 0; step < kStageV / kStepV; ++step) {
          const uint8_t* phi = sP + (size_t)stage * P.p_stage_bytes + step * kStepV * 128;
          uint8_t* out = sB + (size_t)slot * P.part_bytes;
          const int vs = step * kStepV + v;
          const float mv = item.v0 + (int64_t)st * kStageV + vs < item.v1 ? sM[(size_t)stage * kStageV + vs] : 0.f;
          // columns 64 g0 .. 64 g0 + 127: both groups' reads first
          for (int g0 = 0; g0 < ng; g0 += 2) {
            float4 x[2], y[2];
            bool on[2];
#pragma unroll
            for (int e = 0; e < 2; ++e) {
              on[e] = (g0 + e) * 64 + j * 8 < item.npad;
              x[e] = y[e] = make_float4(0.f, 0.f, 0.f, 0.f);
              if (on[e]) {
                x[e] = *reinterpret_cast<const float4*>(phi + (g0 + e) * 2 * kBoxBytes + ca);
                y[e] = *reinterpret_cast<const float4*>(phi + (g0 + e) * 2 * kBoxBytes + cb);
              }
            }
#pragma unroll
            for (int e = 0; e < 2; ++e) {
              if (g0 + e >= ng) break;
              const float4 p = swap ? y[e] : x[e], q = swap ? x[e] : y[e];
              uint4 h, md, l;
              tc::split3(p.x * mv, p.y * mv, h.x, md.x, l.x);
              tc::split3(p.z * mv, p.w * mv, h.y, md.y, l.y);
              tc::split3(q.x * mv, q.y * mv, h.z, md.z, l.z);
              tc::split3(q.z * mv, q.w * mv, h.w, md.w, l.w);
              if (g0 + e == 0 && !tc::warp_wait(&part_empty[slot], slot_phase ^ 1, abort_flag)) goto done;
              if (on[e]) {
                *reinterpret_cast<uint4*>(out + (g0 + e) * kColBytes + dst[0]) = h;
                *reinterpret_cast<uint4*>(out + (g0 + e) * kColBytes + dst[1]) = md;
                *reinterpret_cast<uint4*>(out + (g0 + e) * kColBytes + dst[2]) = l;
              }
            }
          }
          tc::fence_proxy_async_smem();
          __syncwarp();
          if (lane == 0) {
            if (step == kStageV / kStepV - 1) tc::mbar_arrive(&empty[stage]);
            tc::mbar_arrive(&part_full[slot]);
          }
          if (++slot == (uint32_t)kTc32Slots) { slot = 0; slot_phase ^= 1; }
        }
        if (++stage == (uint32_t)S) { stage = 0; phase ^= 1; }
      }
    }
  }
done:

  __syncthreads();
  if (warp == 1) tc::tmem_dealloc(tmem_base, P.tmem_cols);
  if (threadIdx.x == 0 && *abort_flag) atomicExch(P.err, (int)FMAP_ERR_TIMEOUT);
}

}  // namespace

cudaError_t project_tc32_set_smem(int bytes) {
  return cudaFuncSetAttribute(project_tc32_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
}

cudaError_t launch_project_tc32(const TcProjParams& p, int grid, int smem_bytes, cudaStream_t st) {
  if (grid <= 0) return cudaSuccess;
  project_tc32_kernel<<<grid, kThreads, smem_bytes, st>>>(p);
  return cudaGetLastError();
}

}  // namespace fmap
