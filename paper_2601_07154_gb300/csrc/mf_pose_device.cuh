// Per-frame pose-side device code shared by the per-stream kernels
// (mf_pose_kernels.cu) and the batched engine kernels (mf_engine_kernels.cu),
// FP64 throughout:
//   pose_frame     -- one CTA builds a frame's record: Section 2.2 for the
//                     pushed poses its window needs (rigidity check,
//                     gravity-locked incremental anchoring of a batch-local
//                     pose, append of its own pose to the history), then
//                     Section 2.3, Eqs. 1-6 (N motion points and the focus);
//   finalize_frame -- per-frame result record.
// FP64 stays here because the pose differences are ill-conditioned near zero
// translation.  What bounds it is the FP64 pipe: on GB300 each of an SM's
// four schedulers issues one FP64 instruction every 64 cycles, however many
// lanes are active (a square root takes 680 cycles, a division 570, fmax
// 275), so a frame's cost is the longest chain of FP64 instructions that one
// warp runs.
#pragma once

#include <math.h>

#include "mf_internal.h"

namespace mf {

// Bits of a non-negative FP64 value order like the value (infinity and NaN
// above every finite one), so maxima are taken on integers.
__device__ __forceinline__ unsigned long long abs_bits(double v) {
  return (unsigned long long)__double_as_longlong(v) & 0x7fffffffffffffffull;
}

// Every entry of a pose finite.
__device__ __forceinline__ bool pose_is_finite(const double* P) {
  unsigned long long top = 0ull;
  for (int k = 0; k < 12; ++k) {
    const unsigned long long b = abs_bits(P[k]);
    top = b > top ? b : top;
  }
  return top < 0x7ff0000000000000ull;
}

// |R R^T - I| <= kRigidTol at the entry of rotation rows A and B (a NaN's bits
// lie above the tolerance's).
__device__ __forceinline__ bool rows_are_rigid(const double* A, const double* B, bool same) {
  const double dot = A[0] * B[0] + A[1] * B[1] + A[2] * B[2];
  return abs_bits(dot - (same ? 1.0 : 0.0)) <= abs_bits(kRigidTol);
}

// Every entry finite and |R R^T - I| <= kRigidTol, over the six distinct dot
// products (the other three are the same products).
__device__ __forceinline__ bool pose_is_rigid(const double* P) {
  bool ok = pose_is_finite(P);
  for (int a = 0; a < 3; ++a)
    for (int b = a; b < 3; ++b) ok &= rows_are_rigid(P + 4 * a, P + 4 * b, a == b);
  return ok;
}

// Camera centre of a world-to-camera pose [R | t]: c = -R^T t (Eq. 1 for a
// rigid transform).
__device__ __forceinline__ void pose_centre(const double* P, double c[3]) {
  for (int j = 0; j < 3; ++j)
    c[j] = -(P[0 * 4 + j] * P[3] + P[1 * 4 + j] * P[7] + P[2 * 4 + j] * P[11]);
}

// Largest of the lanes' non-negative FP64 bit patterns.
__device__ __forceinline__ unsigned long long warp_max_bits(unsigned long long v) {
  const unsigned hi = __reduce_max_sync(0xffffffffu, (unsigned)(v >> 32));
  const unsigned lo = __reduce_max_sync(0xffffffffu, (unsigned)(v >> 32) == hi ? (unsigned)v : 0u);
  return ((unsigned long long)hi << 32) | lo;
}

__device__ __forceinline__ double warp_sum(double v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Splits a pixel coordinate u into float hi + lo with hi a multiple of 2^-8
// when |u| < 2^15, so that (integer pixel) - hi is exact in FP32.
__device__ __forceinline__ void split_coord(double u, float& hi, float& lo) {
  const double h = fabs(u) < 32768.0 ? rint(u * 256.0) * (1.0 / 256.0) : u;
  hi = (float)h;
  lo = (float)(u - (double)hi);
}

// One push as pose_frame sees it.
struct PushView {
  const double* in;        // the push's poses, 12 doubles each
  int first;               // first emitted push frame (= overlap or 0)
  int anchor;              // 1: gravity-locked anchoring against the history
  double* ring;            // world-pose history (NULL: none kept, e0 = 0)
  int32_t* ring_bad;
  int64_t ring_mask;
  int64_t e0;              // emitted index of push frame `first`
  const double* scale;     // the push's depth scale (depth alignment; NULL: 1)
};

// Inputs of pose_frame that describe the stream.
struct FrameParams {
  int window, smooth_len;
  int width, height;
  double sigma_rel, s_lo, s_hi;
  double d0;               // reference depth of G (m)
};

// A CTA of pose_frame: one frame, four warps.
constexpr int kPoseThreads = 128;

// Shared scratch of pose_frame.
struct PoseScratch {
  double c[3][kMaxHist];   // centres of the window's poses, by component
  double q[3][kMaxHist];   // Eq. 4 positions of the window's poses, by component
  double d[3][32];         // motion vectors, by component
  double u[32], v[32];
  double Rg[9];            // rotation of the frame's own pose
  double cs, sn;           // anchoring rotation
  double cw[3], cl[3];     // the transition frame's centre in the world and in the push
  unsigned long long rho2, pm2;
  double rho_min;          // smallest |d| of a valid point
  unsigned bad[2];         // poses not usable, by window entry
  unsigned skew[2][2];     // poses whose rotation is none, by checking warp and window entry
  unsigned mask;           // valid points
  int anchor_bad, moving;
};

// Section 2.2, the push's local-to-world transform.  The push is batch-local
// and its frame first-1 is the same camera as the history's last frame e0-1
// (the transition frame): H = T_a^{-1} L_a is reduced to the rotation about
// the world y (gravity) axis closest to it, psi = atan2(R02 - R20, R00 + R22)
// (pitch and roll are not propagated), with the translation that puts the
// anchor's camera centre on its world position; T = L H^{-1}.  Two warps share
// the chain: one has the rotation, the other the centres and the check.
__device__ __forceinline__ void anchor_push(const PushView& pv, PoseScratch& S, bool rotation) {
  double La[12];
  const int64_t aslot = (pv.e0 - 1) & pv.ring_mask;
  const double* Ta = pv.ring + aslot * 12;
  for (int e = 0; e < 12; ++e) La[e] = pv.in[(size_t)(pv.first - 1) * 12 + e];
  if (!rotation) {
    if (pv.scale)
      for (int r = 0; r < 3; ++r) La[4 * r + 3] *= *pv.scale;
    S.anchor_bad = pv.ring_bad[aslot] || !pose_is_rigid(La);
    pose_centre(Ta, S.cw);
    pose_centre(La, S.cl);
    return;
  }
  double rh[3][3];
  for (int r = 0; r < 3; ++r)
    for (int c = 0; c < 3; ++c)
      rh[r][c] = Ta[0 * 4 + r] * La[0 * 4 + c] + Ta[1 * 4 + r] * La[1 * 4 + c] + Ta[2 * 4 + r] * La[2 * 4 + c];
  const double ca = rh[0][0] + rh[2][2], sa = rh[0][2] - rh[2][0];
  const double rr = hypot(ca, sa);
  const double cs = rr > 0.0 ? ca / rr : 1.0;
  const double sn = rr > 0.0 ? sa / rr : 0.0;
  S.cs = cs;
  S.sn = sn;
}

// The record of emitted frame g of a push (its pose is push frame
// first + g - e0), by a CTA of kPoseThreads threads; every thread calls it.
//
// Poses before e0 come from the history, the push's own poses are brought to
// the world frame here, by every frame that needs them, so frames of one
// push do not wait for one another; each frame appends its own pose (the
// slots written, e0 and up, are distinct from the slots read).
//
// The four warps split the FP64 chains: warps 0 and 1 take the window's
// poses, one per lane, while warps 2 and 3 check the rotations of the pushed
// ones, three entries of R R^T each (with anchoring they find that, and
// warps 0 and 1 check their poses); warps 0 to 2 fit one component of the
// motion vectors each, and warp 3 has the distances; then warp 0 has the
// spreads, warps 1 and 2 the projections, warp 3 the frame's scalars.  The
// roles rotate with the CTA so that the CTAs of an SM load its schedulers
// alike.
// Against two kernels (ingest, thread per frame, then points, warp per
// frame): a camera loop at 320x240, window 8, 40.7 -> 34.3 us a frame; two
// batch-local pushes of 60 frames at 504x280 179.8 -> 156.6 us.  The checks
// and the distances beside the centres and positions, not before them:
// camera loop 13.8 -> 12.3 us, 1080p 18.7 -> 17.7 us.
__device__ __forceinline__ void pose_frame(const PushView& pv, int64_t g, const FrameParams& fp,
                                           const double* K, const double* w, FrameRec* rec,
                                           PoseScratch& S) {
  const int lane = threadIdx.x & 31;
  const int role = ((threadIdx.x >> 5) + blockIdx.x) & 3;
  const int W = fp.window, Ks = fp.smooth_len, R = W + Ks - 1;  // R <= kMaxHist = 64
  const int64_t j0 = g - (R - 1);

  // Section 2.2 and Eq. 1: the window's world poses and their centres.
  const int r = 32 * role + lane;
  const int64_t j = j0 + r;
  const bool mine = role < 2 && r < R && j >= 0;
  const bool pushed = mine && j >= pv.e0;
  double P[12];
  bool bad = true;
  if (mine) {
    const double* src = pushed ? pv.in + (size_t)(pv.first + (j - pv.e0)) * 12 : pv.ring + (j & pv.ring_mask) * 12;
    for (int e = 0; e < 12; ++e) P[e] = src[e];
    if (pushed) {
      if (pv.scale)
        for (int a = 0; a < 3; ++a) P[4 * a + 3] *= *pv.scale;
      bad = pv.anchor ? !pose_is_rigid(P) : !pose_is_finite(P);
    } else {
      bad = pv.ring_bad[j & pv.ring_mask] != 0;
    }
  }
  if (role >= 2) {
    for (int h = 0; h < 2; ++h) {
      const int e = 32 * h + lane;
      bool ok = true;
      if (!pv.anchor && e < R && j0 + e >= pv.e0) {
        const double* A = pv.in + (size_t)(pv.first + (j0 + e - pv.e0)) * 12;
        ok = role == 2 ? rows_are_rigid(A, A, true) & rows_are_rigid(A, A + 4, false) & rows_are_rigid(A, A + 8, false)
                       : rows_are_rigid(A + 4, A + 4, true) & rows_are_rigid(A + 4, A + 8, false) &
                             rows_are_rigid(A + 8, A + 8, true);
      }
      const unsigned skew = __ballot_sync(0xffffffffu, !ok);
      if (lane == 0) S.skew[role - 2][h] = skew;
      if (R <= 32) {
        if (lane == 0) S.skew[role - 2][1] = 0u;
        break;
      }
    }
  }
  if (pv.anchor) {
    if (role >= 2) anchor_push(pv, S, role == 3);
    __syncthreads();
    if (pushed) {
      if (S.anchor_bad) {
        bad = true;
      } else {
        const double cs = S.cs, sn = S.sn;
        const double tH[3] = {S.cw[0] - (cs * S.cl[0] + sn * S.cl[2]), S.cw[1] - S.cl[1],
                              S.cw[2] - (-sn * S.cl[0] + cs * S.cl[2])};
        for (int a = 0; a < 3; ++a) {
          const double l0 = P[4 * a + 0], l1 = P[4 * a + 1], l2 = P[4 * a + 2];
          const double r0 = l0 * cs + l2 * sn;
          const double r2 = -l0 * sn + l2 * cs;
          P[4 * a + 0] = r0;
          P[4 * a + 2] = r2;
          P[4 * a + 3] = P[4 * a + 3] - (r0 * tH[0] + l1 * tH[1] + r2 * tH[2]);
        }
      }
    }
  }
  if (role < 2) {
    const unsigned b = __ballot_sync(0xffffffffu, bad);
    if (lane == 0) S.bad[role] = b;
    if (mine) {
      double pc[3];
      pose_centre(P, pc);
      for (int a = 0; a < 3; ++a) S.c[a][r] = pc[a];
      if (r == R - 1) {
        for (int a = 0; a < 3; ++a)
          for (int c = 0; c < 3; ++c) S.Rg[3 * a + c] = P[4 * a + c];
        if (pv.ring)
          for (int e = 0; e < 12; ++e) pv.ring[(g & pv.ring_mask) * 12 + e] = P[e];
      }
    }
  }
  __syncthreads();
  const unsigned long long bads = ((unsigned long long)(S.bad[1] | S.skew[0][1] | S.skew[1][1]) << 32) |
                                  (S.bad[0] | S.skew[0][0] | S.skew[1][0]);
  const bool frame_bad = ((bads >> (R - 1)) & 1ull) != 0;
  if (pv.ring && threadIdx.x == 0) pv.ring_bad[g & pv.ring_mask] = frame_bad ? 1 : 0;

  // Eq. 4 applied to relative positions: q_j = R_n (p_j - p_n), a component
  // per warp, and the largest distances.
  {
    const double gx = S.c[0][R - 1], gy = S.c[1][R - 1], gz = S.c[2][R - 1];
    unsigned long long rho2 = 0ull, pm2 = 0ull;
    for (int e = lane; e < R; e += 32) {
      if ((bads >> e) & 1ull) continue;
      const double cx = S.c[0][e], cy = S.c[1][e], cz = S.c[2][e];
      const double dx = cx - gx, dy = cy - gy, dz = cz - gz;
      if (role < 3) {
        S.q[role][e] = S.Rg[3 * role + 0] * dx + S.Rg[3 * role + 1] * dy + S.Rg[3 * role + 2] * dz;
      } else {
        const unsigned long long r2 = abs_bits(dx * dx + dy * dy + dz * dz);
        const unsigned long long p2 = abs_bits(cx * cx + cy * cy + cz * cz);
        rho2 = r2 > rho2 ? r2 : rho2;
        pm2 = p2 > pm2 ? p2 : pm2;
      }
    }
    if (role == 3) {
      rho2 = warp_max_bits(rho2);
      pm2 = warp_max_bits(pm2);
      if (lane == 0) {
        S.rho2 = rho2;
        S.pm2 = pm2;
      }
    }
  }
  __syncwarp();  // a warp's fit reads its own component
  // Eqs. 2-3: motion vector of point i = g - W + 1 + lane by the K-sample
  // least-squares weights over window entries lane .. lane + K - 1.
  if (role < 3) {
    if (lane < W) {
      const double* q = S.q[role] + lane + Ks - 1;
      double d = 0.0;
      for (int k = 0; k < Ks; ++k) d = fma(w[k], q[-k], d);
      S.d[role][lane] = d;
    }
  } else {
    // largest distances (the square root of the largest square), both at once
    const double x = sqrt(__longlong_as_double((long long)((lane & 1) ? S.pm2 : S.rho2)));
    const double rho = __shfl_sync(0xffffffffu, x, 0), pmax = __shfl_sync(0xffffffffu, x, 1);
    if (lane == 0) {
      S.moving = !frame_bad && rho > 0.0 && rho > kStaticRel * pmax;
      S.rho_min = kValidRelNorm * rho;
    }
  }
  __syncthreads();

  const double fx = K[0];
  bool valid = false;
  double nd = 0.0;
  if (role == 0) {
    const unsigned long long fit = ~0ull >> (64 - Ks);  // 2 <= Ks <= 64
    const bool ok = lane < W && S.moving && ((bads >> lane) & fit) == 0ull;
    if (ok) {
      const double d0 = S.d[0][lane], d1 = S.d[1][lane], d2 = S.d[2][lane];
      nd = sqrt(d0 * d0 + d1 * d1 + d2 * d2);
      valid = nd > S.rho_min && fabs(d2) > kValidRelZ * nd;
    }
    const unsigned m = __ballot_sync(0xffffffffu, valid);
    if (lane == 0) S.mask = m;
  } else if (role == 1) {  // Eq. 6
    if (lane < W) S.u[lane] = K[2] + fx * S.d[0][lane] / S.d[2][lane];
  } else if (role == 2) {
    if (lane < W) S.v[lane] = K[3] + K[1] * S.d[1][lane] / S.d[2][lane];
  }
  __syncthreads();
  const unsigned mask = S.mask;
  const int nv = __popc(mask);
  const bool has = ((mask >> lane) & 1u) != 0;
  const int pos = __popc(mask & ((1u << lane) - 1u));
  if (role == 0) {
    // magnitude s_i and spread sigma_i (Eq. 7)
    const double sum = warp_sum(valid ? nd : 0.0);
    double sig = 0.0, sc = 0.0;
    if (valid) {
      const double mean = sum / nv;
      sc = nd / mean;
      sc = sc > fp.s_lo ? sc : fp.s_lo;
      sc = sc < fp.s_hi ? sc : fp.s_hi;
      sig = fp.sigma_rel * fx * sc;
      // log2(e) / (2 sigma^2): the map kernels evaluate the Gaussian as a
      // power of 2
      double c = 1.4426950408889634 / (2.0 * sig * sig);
      c = c < 1e30 ? c : 1e30;
      const float chi = (float)c;
      rec->c_hi[pos] = chi;
      rec->c_lo[pos] = (float)(c - (double)chi);
    }
    rec->sigma[lane] = sig;
    rec->s[lane] = sc;
    rec->valid[lane] = valid ? 1 : 0;
  } else if (role == 1) {
    const double u = has ? S.u[lane] : 0.0;
    rec->u[lane] = u;
    if (has) {
      float hi, lo;
      split_coord(u, hi, lo);
      rec->ux_hi[pos] = hi;
      rec->ux_lo[pos] = lo;
    }
  } else if (role == 2) {
    const double v = has ? S.v[lane] : 0.0;
    rec->v[lane] = v;
    if (has) {
      float hi, lo;
      split_coord(v, hi, lo);
      rec->vy_hi[pos] = hi;
      rec->vy_lo[pos] = lo;
    }
  } else if (lane == 0) {
    const bool focus = ((mask >> (W - 1)) & 1u) != 0;
    int px = -1, py = -1;
    double u = 0.0, v = 0.0;
    if (focus) {
      u = S.u[W - 1];
      v = S.v[W - 1];
      const double xr = rint(u), yr = rint(v);
      if (xr >= 0.0 && xr < (double)fp.width && yr >= 0.0 && yr < (double)fp.height) {
        px = (int)xr;
        py = (int)yr;
      }
    }
    rec->focus_valid = focus ? 1 : 0;
    rec->focus_u = u;
    rec->focus_v = v;
    rec->focus_px_x = px;
    rec->focus_px_y = py;
    rec->n_valid = nv;
    rec->inv_n = nv ? 1.0f / (float)nv : 0.0f;
    rec->valid_mask = mask;
    rec->status = frame_bad ? MF_FRAME_BAD_POSE : (nv ? MF_FRAME_OK : MF_FRAME_EMPTY);
    rec->frame_index = g;
    rec->argmax_key = 0ull;
    rec->units_done = 0u;
    // G's reference depth in the frame's depth scale: min(1, d0 / (s D)) =
    // min(1, (d0 / s) / D)
    rec->d0 = (float)(pv.scale ? fp.d0 / *pv.scale : fp.d0);
    rec->depth_scale = (float)(pv.scale ? *pv.scale : 1.0);
  }
}

// Divisor of a frame's maps under MF_NORM_MAX: the map maximum found by the
// fused argmax when it is at least kNormFloor, else 1 (a frame whose motion
// points all lie far outside the image keeps its near-zero count-normalised
// maps).  Dividing, rather than multiplying by a reciprocal, maps the
// maximum to exactly 1.
__device__ __forceinline__ float norm_divisor(const FrameRec* rec) {
  const unsigned long long key = rec->argmax_key;
  if (rec->n_valid <= 0 || key == 0ull) return 1.0f;
  const float mx = __uint_as_float((unsigned)(key >> 32));
  return mx >= kNormFloor ? mx : 1.0f;
}

__device__ __forceinline__ void finalize_frame(const FrameRec* rec, int width, mf_frame_info* out,
                                               int normalize = MF_NORM_COUNT) {
  mf_frame_info o;
  o.frame_index = rec->frame_index;
  o.status = rec->status;
  o.n_valid = rec->n_valid;
  o.valid_mask = rec->valid_mask;
  o.focus_valid = rec->focus_valid;
  o.focus_u = rec->focus_u;
  o.focus_v = rec->focus_v;
  o.focus_px_x = rec->focus_px_x;
  o.focus_px_y = rec->focus_px_y;
  const unsigned long long key = __ldcg(&rec->argmax_key);  // other SMs' atomics: from L2
  if (rec->n_valid > 0 && key != 0ull) {
    const unsigned idx = 0xffffffffu - (unsigned)(key & 0xffffffffull);
    o.argmax_x = (int)(idx % (unsigned)width);
    o.argmax_y = (int)(idx / (unsigned)width);
    o.map_max = __uint_as_float((unsigned)(key >> 32));
    if (normalize == MF_NORM_MAX && o.map_max >= kNormFloor) o.map_max = 1.0f;
  } else {
    o.argmax_x = -1;
    o.argmax_y = -1;
    o.map_max = 0.0f;
  }
  o.depth_scale = rec->depth_scale;
  *out = o;
}

__device__ __forceinline__ void motion_point(const FrameRec* rec, int slot, mf_motion_point* out) {
  mf_motion_point q;
  q.u = rec->u[slot];
  q.v = rec->v[slot];
  q.sigma = rec->sigma[slot];
  q.s = rec->s[slot];
  q.valid = rec->valid[slot];
  q.reserved = 0;
  *out = q;
}

}  // namespace mf
