// Pose-side kernels of one stream (FP64; bodies in mf_pose_device.cuh):
//   pose_kernel      -- Sections 2.2 and 2.3, Eqs. 1-6, one CTA per frame;
//   finalize_kernel  -- per-frame result records (and motion points);
//   ring_copy_kernel -- carries the pose history over when it grows.
#include "mf_pose_device.cuh"

namespace mf {

namespace {
__device__ __forceinline__ void pose_body(const PoseParams& p, const double* in) {
  __shared__ PoseScratch S;
  allow_successor();
  wait_for_predecessor();
  const int64_t g = p.g0 + blockIdx.x;
  PushView pv;
  pv.in = in;
  pv.first = p.first;
  pv.anchor = p.anchor;
  pv.ring = p.ring;
  pv.ring_bad = p.ring_bad;
  pv.ring_mask = p.ring_mask;
  pv.e0 = p.e0;
  pv.scale = p.scale;
  FrameParams fp;
  fp.window = p.window;
  fp.smooth_len = p.smooth_len;
  fp.width = p.width;
  fp.height = p.height;
  fp.sigma_rel = p.sigma_rel;
  fp.s_lo = p.s_lo;
  fp.s_hi = p.s_hi;
  fp.d0 = p.d0;
  pose_frame(pv, g, fp, p.K, p.w, p.recs + (g & p.rec_mask), S);
}
}  // namespace

__global__ void __launch_bounds__(kPoseThreads) pose_kernel(const __grid_constant__ PoseParams p) {
  pose_body(p, p.in);
}

__global__ void __launch_bounds__(kPoseThreads)
    pose_block_kernel(const __grid_constant__ PoseParams p, const __grid_constant__ PoseBlock b) {
  pose_body(p, b.p);
}

__global__ void finalize_kernel(FinalizeParams p) {
  allow_successor();
  wait_for_predecessor();
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (p.info && t < p.n_frames)
    finalize_frame(p.recs + ((p.f0 + t) & p.rec_mask), p.width, p.info + t, p.normalize);
  if (p.points) {
    const int total = p.n_frames * p.window;
    for (int e = t; e < total; e += gridDim.x * blockDim.x) {
      const int f = e / p.window, sl = e - f * p.window;
      motion_point(p.recs + ((p.f0 + f) & p.rec_mask), sl, p.points + e);
    }
  }
}

__global__ void ring_copy_kernel(const double* src, const int32_t* src_bad, int64_t src_mask,
                                 double* dst, int32_t* dst_bad, int64_t dst_mask, int64_t first,
                                 int count) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= count) return;
  const int64_t j = first + k;
  const double* s = src + (j & src_mask) * 12;
  double* t = dst + (j & dst_mask) * 12;
  for (int e = 0; e < 12; ++e) t[e] = s[e];
  dst_bad[j & dst_mask] = src_bad[j & src_mask];
}

// ------------------------------------------------------------ launchers --
cudaError_t launch_pose(const PoseParams& p, cudaStream_t st, int64_t* launches) {
  if (p.n_frames <= 0) return cudaSuccess;
  ++*launches;
  if (p.block) return launch_after(pose_block_kernel, p.n_frames, kPoseThreads, 0, st, p, *p.block);
  return launch_after(pose_kernel, p.n_frames, kPoseThreads, 0, st, p);
}

cudaError_t launch_finalize(const FinalizeParams& p, cudaStream_t st, int64_t* launches) {
  if (p.n_frames <= 0 || (!p.info && !p.points)) return cudaSuccess;
  const int total = p.points ? p.n_frames * p.window : p.n_frames;
  int blocks = (total + 255) / 256;
  if (blocks > 4096) blocks = 4096;
  if (blocks < (p.n_frames + 255) / 256) blocks = (p.n_frames + 255) / 256;
  ++*launches;
  return launch_after(finalize_kernel, blocks, 256, 0, st, p);
}

cudaError_t launch_ring_copy(const double* src, const int32_t* src_bad, int64_t src_mask,
                             double* dst, int32_t* dst_bad, int64_t dst_mask, int64_t first,
                             int count, cudaStream_t st, int64_t* launches) {
  if (count <= 0) return cudaSuccess;
  ring_copy_kernel<<<(count + 127) / 128, 128, 0, st>>>(src, src_bad, src_mask, dst, dst_bad,
                                                         dst_mask, first, count);
  ++*launches;
  return cudaGetLastError();
}

}  // namespace mf
