// Overlap-prediction metrics (Sec. "Overlap Prediction Metrics" of the paper): for each
// segment s (the vertices of one shape, or of one pair's overlap region) a vertex is
// predicted overlapping when its score exceeds the threshold (FP32 comparison), and the
// prediction is counted against the binary ground truth:
//   TP = #(pred & label), FP = #(pred & !label), FN = #(!pred & label), TN = the rest.
// From the counts, in FP64: IoU = TP / (TP + FP + FN), accuracy = (TP + TN) / n,
// precision = TP / (TP + FP), recall (sensitivity) = TP / (TP + FN),
// specificity = TN / (TN + FP), F1 = 2 TP / (2 TP + FP + FN) and balanced accuracy =
// (recall + specificity) / 2. A ratio whose denominator is zero is NaN.
//
// The count pass reads each vertex's score (4 bytes) and label (1 byte) once: it is bound
// by HBM bandwidth. The segments are contiguous, so the flat vertex range is cut into equal
// spans, one per warp, whatever the segment lengths (a (chunk, segment) grid leaves most of
// its blocks without work on short segments). 4096 segments, 87 M vertices: 0.088 ms on the
// device = 5.0 TB/s; a call with its upload of the offsets 0.117 ms, 0.181 ms with the grid. A
// warp finds its first segment with a 32-way search over the offsets, reads four scores and four
// labels per lane and load (four such loads in flight), and adds the counts of each segment it
// meets with one integer atomic per count (integer sums: exact and order-independent).
#include <stdint.h>

#include "fmap_internal.cuh"

namespace fmap {
namespace {

constexpr int kOvThreads = 256;
constexpr int kOvWarps = kOvThreads / 32;
constexpr int64_t kOvChunk = 4096;     // a segment is counted up to max_segment_len rounded up to this
constexpr int64_t kOvMinSpan = 1024;   // vertices per warp below which more warps only add searches

// Last index i in [lo, hi) with off[i] <= v (off non-decreasing, off[lo] <= v): the warp probes
// 32 points per round.
__device__ __forceinline__ int warp_find_segment(const int64_t* __restrict__ off, int lo, int hi, int64_t v, int lane) {
  while (hi - lo > 1) {
    const int step = (hi - lo + 31) / 32;
    const int at = lo + lane * step;
    const bool le = at < hi && off[at] <= v;
    const int j = 31 - __clz((int)__ballot_sync(0xffffffffu, le));   // lane 0 always holds off[lo] <= v
    lo += j * step;
    hi = min(hi, lo + step);
  }
  return lo;
}

// One warp's span of vertices: counts per segment met.
__global__ void __launch_bounds__(kOvThreads) overlap_count_kernel(const float* __restrict__ scores,
                                                                   const uint8_t* __restrict__ labels,
                                                                   const int64_t* __restrict__ seg_off, int n_seg,
                                                                   int64_t seg_cap, float thr,
                                                                   unsigned long long* counts) {
  const int lane = threadIdx.x & 31;
  const int64_t warp = (int64_t)blockIdx.x * kOvWarps + (threadIdx.x >> 5);
  const int64_t n_warps = (int64_t)gridDim.x * kOvWarps;
  const int64_t beg = seg_off[0], end = seg_off[n_seg];
  int64_t span = (end - beg + n_warps - 1) / n_warps;
  span = span < kOvMinSpan ? kOvMinSpan : (span + 3) & ~(int64_t)3;
  const int64_t w0 = beg + warp * span;
  if (w0 >= end) return;
  const int64_t w1 = w0 + span < end ? w0 + span : end;
  // vectors of four vertices where scores and labels reach their alignment at the same vertex
  const int mis_s = (int)((reinterpret_cast<uintptr_t>(scores) >> 2) & 3);
  const int mis_l = (int)(reinterpret_cast<uintptr_t>(labels) & 3);
  const bool vec = mis_s == mis_l;
  int s = warp_find_segment(seg_off, 0, n_seg, w0, lane);
  for (int64_t v = w0; v < w1 && s < n_seg; ++s) {
    const int64_t s0 = seg_off[s], s1 = seg_off[s + 1];
    const int64_t lim = s0 + seg_cap < s1 ? s0 + seg_cap : s1;   // counted part of the segment
    const int64_t v1 = lim < w1 ? lim : w1;
    unsigned int tp = 0, np = 0, nl = 0;   // pred & label, pred, label
    auto one = [&](int64_t u) {
      const bool pred = scores[u] > thr, lab = labels[u] != 0;
      tp += pred && lab;
      np += pred;
      nl += lab;
    };
    int64_t b0 = v, b1 = v;                // [b0, b1): whole aligned vectors
    if (vec) {
      b0 = v + ((4 - (int)((v + mis_s) & 3)) & 3);
      b1 = b0 < v1 ? b0 + ((v1 - b0) & ~(int64_t)3) : b0;
      if (b0 > v1) b0 = b1 = v1;
    }
    auto four = [&](const float4 f, uint32_t l) {
      const bool p0 = f.x > thr, p1 = f.y > thr, p2 = f.z > thr, p3 = f.w > thr;
      const uint32_t pm = (p0 ? 1u : 0u) | (p1 ? 0x100u : 0u) | (p2 ? 0x10000u : 0u) | (p3 ? 0x1000000u : 0u);
      const uint32_t lm = __vsetgtu4(l, 0u);   // one per non-zero byte
      np += __popc(pm);
      nl += __popc(lm);
      tp += __popc(pm & lm);
    };
    const float4* s4 = reinterpret_cast<const float4*>(scores + b0);
    const uint32_t* l4 = reinterpret_cast<const uint32_t*>(labels + b0);
    const int64_t n4 = (b1 - b0) >> 2;
    int64_t q = lane;
    for (; q + 96 < n4; q += 128) {
      float4 f[4];
      uint32_t l[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        f[u] = __ldcs(s4 + q + 32 * u);
        l[u] = __ldcs(l4 + q + 32 * u);
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) four(f[u], l[u]);
    }
    for (; q < n4; q += 32) four(__ldcs(s4 + q), __ldcs(l4 + q));
    for (int64_t u = v + lane; u < b0; u += 32) one(u);
    for (int64_t u = b1 + lane; u < v1; u += 32) one(u);
    tp = __reduce_add_sync(0xffffffffu, tp);
    np = __reduce_add_sync(0xffffffffu, np);
    nl = __reduce_add_sync(0xffffffffu, nl);
    if (lane < 3) {
      const unsigned int t = lane == 0 ? tp : (lane == 1 ? np - tp : nl - tp);
      if (t) atomicAdd(&counts[4 * (int64_t)s + lane], (unsigned long long)t);
    }
    v = s1 < w1 ? s1 : w1;
  }
}

// num / den, or a quiet NaN when den is 0 (the ratio is undefined)
__device__ __forceinline__ double ratio(double num, double den) {
  return den > 0.0 ? num / den : __longlong_as_double(0x7ff8000000000000LL);
}

// One thread per segment: TN from the segment length, then the seven metrics.
__global__ void overlap_metrics_kernel(const int64_t* __restrict__ seg_off, int n_seg, unsigned long long* counts,
                                       double* metrics) {
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= n_seg) return;
  const unsigned long long n = (unsigned long long)(seg_off[s + 1] - seg_off[s]);
  const unsigned long long tpi = counts[4 * s], fpi = counts[4 * s + 1], fni = counts[4 * s + 2];
  const unsigned long long tni = n - tpi - fpi - fni;
  counts[4 * s + 3] = tni;
  if (metrics == nullptr) return;
  const double tp = (double)tpi, fp = (double)fpi, fn = (double)fni, tn = (double)tni;
  const double recall = ratio(tp, tp + fn), spec = ratio(tn, tn + fp);
  double* m = metrics + 7 * (int64_t)s;
  m[0] = ratio(tp, tp + fp + fn);             // IoU
  m[1] = (recall + spec) * 0.5;               // balanced accuracy
  m[2] = ratio(tp + tn, (double)n);           // accuracy
  m[3] = ratio(tp, tp + fp);                  // precision
  m[4] = recall;                              // recall (sensitivity)
  m[5] = spec;                                // specificity
  m[6] = ratio(2.0 * tp, 2.0 * tp + fp + fn); // F1
}

}  // namespace

cudaError_t launch_overlap_metrics(const float* scores, const uint8_t* labels, const int64_t* seg_off, int n_seg,
                                   int64_t max_len, float thr, int64_t* counts, double* metrics, cudaStream_t st) {
  if (n_seg <= 0) return cudaSuccess;
  cudaError_t e = cudaMemsetAsync(counts, 0, sizeof(int64_t) * 4 * (size_t)n_seg, st);
  if (e != cudaSuccess) return e;
  auto* cnt = reinterpret_cast<unsigned long long*>(counts);
  if (max_len > 0) {
    max_len = std::min<int64_t>(max_len, (int64_t)1 << 46);   // no overflow below; no array is longer
    // 8 CTAs of 8 warps per SM (one resident wave), fewer where the segments cannot hold that many spans
    const int64_t cap = (max_len + kOvChunk - 1) / kOvChunk * kOvChunk;
    const int64_t need = ((int64_t)n_seg * max_len + kOvWarps * kOvMinSpan - 1) / (kOvWarps * kOvMinSpan);
    const unsigned grid = (unsigned)std::max<int64_t>(1, std::min<int64_t>(need, 152 * 8));
    overlap_count_kernel<<<grid, kOvThreads, 0, st>>>(scores, labels, seg_off, n_seg, cap, thr, cnt);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  overlap_metrics_kernel<<<(n_seg + 127) / 128, 128, 0, st>>>(seg_off, n_seg, cnt, metrics);
  return cudaGetLastError();
}

}  // namespace fmap
