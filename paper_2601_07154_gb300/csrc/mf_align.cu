// Depth alignment across batches (Section 2.2, Fig. 3 "depth alignment"):
// the scale of a batch-local batch is the previous batch's scale times the
// lower median of the single-precision ratios D_prev / D_cur over the
// overlap frames' pixels where both depths are finite and > 0.
//
// The median is found by radix selection on the ratios' bit patterns
// (positive floats order like their bits): three histogram passes over the
// overlap planes (the top 11 bits, the next 11 bits of the ratios whose top
// bits match, the last 10 bits).  The CTA that finishes a pass last finds the
// bin holding the wanted rank.  Everything stays on the device and in the
// stream's order; the counts use integer atomics only, so the result does not
// depend on the order in which pixels are counted.
//
// The planes are a few MB (10 frames of 504x280: 11 MB both), so launches,
// atomics and the selection bound it, not memory: one CTA of 1024 threads per
// SM makes an eighth of the global atomics that eight of 256 made, and the
// selection is a scan across the CTA instead of one thread's walk in a kernel
// of its own.  Two batch-local pushes of 60 frames at 504x280: 146.5 -> 124.8 us a
// pass; with more pixel pairs in flight, runs of equal bins counted in registers
// and the anchoring's chain on two warps (mf_pose_device.cuh) 108.1 -> 105.0.
#include <cfloat>
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "mf_internal.h"

namespace mf {
namespace {

constexpr int kAlignThreads = 1024;
// Pixel pairs a thread has in flight: few round trips of a thread against the
// loads' registers and the pairs past the end of a small overlap.  The choice
// matters only where memory bounds the passes: at 31 M pairs (15 frames of
// 1080p BF16) 4 / 6 / 8 / 10 / 12 / 16 pairs take 215 / 200 / 213 / 200 / 195 /
// 213 us; from 0.15 to 8 M pairs 4 to 12 lie within the 5 us by which two
// processes of one build differ (0.28 M 24 to 27, 8.3 M 62 to 68), and 16 above
// them.
constexpr int kAlignUnroll = 10;
// state words after the three histograms
constexpr int kStRank = 3 * kAlignBins;   // wanted rank among the keys matching the prefix
constexpr int kStPrefix = kStRank + 1;    // key bits selected so far
constexpr int kStEmpty = kStRank + 2;     // 1: no valid pair (the scale stays)
constexpr int kStDone = kStRank + 3;      // CTAs of the pass that are done
static_assert(kStDone < kAlignWorkWords, "work words");

__device__ __forceinline__ float to_float(float v) { return v; }
__device__ __forceinline__ float to_float(__nv_bfloat16 v) { return __bfloat162float(v); }
__device__ __forceinline__ float to_float(__half v) { return __half2float(v); }

// The ratio's bit pattern of a pixel's two depths, if both are finite and > 0.
__device__ __forceinline__ bool ratio_key(float a, float b, unsigned* key) {
  if (!(a > 0.0f && a <= FLT_MAX && b > 0.0f && b <= FLT_MAX)) return false;  // NaN fails too
  *key = __float_as_uint(__fdiv_rn(a, b));  // IEEE single-precision quotient, >= 0
  return true;
}

// The last CTA of a pass: the bin of the pass's histogram g that holds the
// wanted rank (pass 0 first sets it to (n-1)/2 of the n valid pairs, the
// lower median); the prefix grows by that bin, and after the last pass the
// batch scale is multiplied by the selected ratio.  Leaves g and the count
// of finished CTAs at 0 for the next call.
template <int PASS>
__device__ __forceinline__ void select_bin(unsigned* work, double* scale, bool restart) {
  constexpr int kPer = kAlignBins / kAlignThreads;
  __shared__ unsigned warp_sum[kAlignThreads / 32];
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  unsigned* g = work + PASS * kAlignBins;
  // (the state beside the counts: one trip to L2 for both)
  const unsigned was_empty = PASS == 0 ? 0u : __ldcg(work + kStEmpty);
  const unsigned was_rank = PASS == 0 ? 0u : __ldcg(work + kStRank);
  const unsigned prefix = PASS == 0 ? 0u : __ldcg(work + kStPrefix);
  unsigned c[kPer], sum = 0u;
  for (int j = 0; j < kPer; ++j) {
    c[j] = __ldcg(g + t * kPer + j);
    g[t * kPer + j] = 0u;
    sum += c[j];
  }
  unsigned incl = sum;
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned v = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += v;
  }
  if (lane == 31) warp_sum[warp] = incl;
  __syncthreads();
  unsigned before = 0u, n = 0u;
  for (int w = 0; w < kAlignThreads / 32; ++w) {
    before += w < warp ? warp_sum[w] : 0u;
    n += warp_sum[w];
  }
  unsigned acc = before + incl - sum;       // keys in the bins before this thread's
  const bool empty = PASS == 0 ? n == 0u : was_empty != 0u;
  const unsigned rank = PASS == 0 ? (n ? (n - 1u) / 2u : 0u) : was_rank;
  if (t == 0) {
    work[kStDone] = 0u;
    if (PASS == 0) work[kStEmpty] = empty ? 1u : 0u;
    if (PASS == 2 && empty && restart) *scale = 1.0;
  }
  if (empty || rank < acc || rank - acc >= sum) return;
  int bin = t * kPer;                       // this thread's bins hold the rank
  for (int j = 0; j < kPer - 1 && acc + c[j] <= rank; ++j) {
    acc += c[j];
    ++bin;
  }
  work[kStRank] = rank - acc;
  const unsigned pre = PASS == 0 ? (unsigned)bin : (prefix << (PASS == 1 ? 11 : 10)) | (unsigned)bin;
  work[kStPrefix] = pre;
  if (PASS == 2) *scale = (restart ? 1.0 : *scale) * (double)__uint_as_float(pre);
}

// One pass: pass 0 bins the top 11 bits of every key; pass 1 the next 11 bits
// of the keys whose top 11 bits are the selected prefix; pass 2 the last 10
// bits of the keys whose top 22 bits are.
template <typename T, int PASS>
__global__ void __launch_bounds__(kAlignThreads) align_pass_kernel(const T* prev, const T* cur, int64_t count,
                                                                   unsigned* work, double* scale, bool restart) {
  __shared__ unsigned h[kAlignBins];
  __shared__ bool last;
  allow_successor();
  for (int i = threadIdx.x; i < kAlignBins; i += kAlignThreads) h[i] = 0u;
  __syncthreads();
  wait_for_predecessor();
  const bool skip = PASS > 0 && work[kStEmpty] != 0u;
  const unsigned prefix = PASS > 0 ? work[kStPrefix] : 0u;
  // Pass 0 keys nearly all share one or two bins (a bin spans a factor of
  // 2^(1/4)): a thread counts a run of equal bins before it adds them.
  unsigned run_bin = 0u, run = 0u;
  const int64_t stride = (int64_t)gridDim.x * kAlignThreads;
  for (int64_t i0 = (int64_t)blockIdx.x * kAlignThreads + threadIdx.x; i0 < count && !skip;
       i0 += kAlignUnroll * stride) {
    float a[kAlignUnroll], b[kAlignUnroll];
#pragma unroll
    for (int j = 0; j < kAlignUnroll; ++j) {
      const int64_t i = i0 + j * stride;
      a[j] = i < count ? to_float(prev[i]) : 0.0f;   // 0: no pair
      b[j] = i < count ? to_float(cur[i]) : 0.0f;
    }
#pragma unroll
    for (int j = 0; j < kAlignUnroll; ++j) {
      unsigned key;
      if (!ratio_key(a[j], b[j], &key)) continue;
      if (PASS == 0) {
        if (key >> 21 != run_bin) {
          if (run) atomicAdd(&h[run_bin], run);
          run_bin = key >> 21;
          run = 0u;
        }
        ++run;
      } else if (PASS == 1 && (key >> 21) == prefix)
        atomicAdd(&h[(key >> 10) & 0x7ffu], 1u);
      else if (PASS == 2 && (key >> 10) == prefix)
        atomicAdd(&h[key & 0x3ffu], 1u);
    }
  }
  if (PASS == 0 && run) atomicAdd(&h[run_bin], run);
  __syncthreads();
  unsigned* g = work + PASS * kAlignBins;
  for (int i = threadIdx.x; i < kAlignBins; i += kAlignThreads)
    if (h[i]) atomicAdd(&g[i], h[i]);
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(&work[kStDone], 1u) == gridDim.x - 1;
  __syncthreads();
  if (!last) return;
  __threadfence();
  select_bin<PASS>(work, scale, restart);
}

template <typename T>
cudaError_t launch_typed(const AlignParams& p, cudaStream_t st, int64_t* launches) {
  const int64_t want = (p.count + kAlignThreads - 1) / kAlignThreads;
  const int sms = host_kernel_fit(reinterpret_cast<const void*>(align_pass_kernel<T, 0>), kAlignThreads, 0, 0).sms;
  const int blocks = (int)(want < sms ? want : sms);
  const T* prev = static_cast<const T*>(p.prev);
  const T* cur = static_cast<const T*>(p.cur);
  for (auto k : {align_pass_kernel<T, 0>, align_pass_kernel<T, 1>, align_pass_kernel<T, 2>}) {
    const cudaError_t e =
        launch_after(k, blocks, kAlignThreads, 0, st, prev, cur, p.count, p.work, p.scale, p.restart);
    if (e != cudaSuccess) return e;
    ++*launches;
  }
  return cudaSuccess;
}

}  // namespace

cudaError_t launch_depth_align(const AlignParams& p, int depth_dtype, cudaStream_t st, int64_t* launches) {
  if (p.count <= 0) return cudaSuccess;
  switch (depth_dtype) {
    case MF_F32: return launch_typed<float>(p, st, launches);
    case MF_BF16: return launch_typed<__nv_bfloat16>(p, st, launches);
    case MF_F16: return launch_typed<__half>(p, st, launches);
  }
  return cudaErrorInvalidValue;
}

}  // namespace mf
