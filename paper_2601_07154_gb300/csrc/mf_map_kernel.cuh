// Per-pixel kernels of the motion-focus path (templates; instantiated by
// mf_map_n8.cu, mf_map_n16.cu and mf_map_n32.cu, one window bucket each, so
// that the build compiles them in parallel): the motion-focus map of Eq. 7
// and the motion-guided depth (Fig. 1(iii), Fig. 5), fused, with the
// per-frame argmax of the map.
//
// The map is a sum of N isotropic Gaussians, so each term factors into a
// column factor and a row factor:
//     exp(-((x-u)^2 + (y-v)^2) c) = exp(-(x-u)^2 c) * exp(-(y-v)^2 c),
// c = 1 / (2 sigma_i^2).  A CTA owns a 128-column x tile_h-row tile of one
// frame: it evaluates the N x 128 column factors and tile_h x N row factors
// (with 1/Z folded into the row factors) in shared memory, then every pixel
// costs N FP32 FMAs, issued two pixels at a time with fma.rn.f32x2, summed in
// fixed point order so results do not depend on the tiling.  Depth is read
// and both maps are written with 128-bit (FP32) or 64-bit (16-bit storage)
// streaming accesses, 4 pixels per thread per row; each warp covers 128
// contiguous pixels of a row (512 B of FP32), so every access is coalesced.
//
// Accuracy: the exponent is formed from an exact FP32 coordinate difference
// (u is split into a hi part on a 2^-8 grid plus a lo part) and a float pair
// for c, so its relative error stays near one FP32 rounding; the hardware's
// base-2 exponential then costs a few ulp per factor.
#pragma once

#include <algorithm>
#include <type_traits>

#include "mf_map_unit.cuh"
#include "mf_pose_device.cuh"

namespace mf {


namespace {

// Storage types: 4 consecutive pixels per access.
template <typename T>
struct Px;

template <>
struct Px<float> {
  static __device__ __forceinline__ float4 load4(const void* b, size_t i) {
    return __ldcs(reinterpret_cast<const float4*>(static_cast<const float*>(b) + i));
  }
  static __device__ __forceinline__ float load1(const void* b, size_t i) {
    return __ldcs(static_cast<const float*>(b) + i);
  }
  static __device__ __forceinline__ void store4(void* b, size_t i, float4 v) {
    __stcs(reinterpret_cast<float4*>(static_cast<float*>(b) + i), v);
  }
  static __device__ __forceinline__ void store1(void* b, size_t i, float v) {
    __stcs(static_cast<float*>(b) + i, v);
  }
};

template <>
struct Px<__nv_bfloat16> {
  static __device__ __forceinline__ float4 load4(const void* b, size_t i) {
    uint2 r = __ldcs(reinterpret_cast<const uint2*>(static_cast<const __nv_bfloat16*>(b) + i));
    const float2 a = __bfloat1622float2(*reinterpret_cast<__nv_bfloat162*>(&r.x));
    const float2 c = __bfloat1622float2(*reinterpret_cast<__nv_bfloat162*>(&r.y));
    return make_float4(a.x, a.y, c.x, c.y);
  }
  static __device__ __forceinline__ float load1(const void* b, size_t i) {
    return __bfloat162float(static_cast<const __nv_bfloat16*>(b)[i]);
  }
  static __device__ __forceinline__ void store4(void* b, size_t i, float4 v) {
    __nv_bfloat162 lo = __floats2bfloat162_rn(v.x, v.y);
    __nv_bfloat162 hi = __floats2bfloat162_rn(v.z, v.w);
    uint2 r;
    r.x = *reinterpret_cast<unsigned*>(&lo);
    r.y = *reinterpret_cast<unsigned*>(&hi);
    __stcs(reinterpret_cast<uint2*>(static_cast<__nv_bfloat16*>(b) + i), r);
  }
  static __device__ __forceinline__ void store1(void* b, size_t i, float v) {
    static_cast<__nv_bfloat16*>(b)[i] = __float2bfloat16_rn(v);
  }
};

template <>
struct Px<__half> {
  static __device__ __forceinline__ float4 load4(const void* b, size_t i) {
    uint2 r = __ldcs(reinterpret_cast<const uint2*>(static_cast<const __half*>(b) + i));
    const float2 a = __half22float2(*reinterpret_cast<__half2*>(&r.x));
    const float2 c = __half22float2(*reinterpret_cast<__half2*>(&r.y));
    return make_float4(a.x, a.y, c.x, c.y);
  }
  static __device__ __forceinline__ float load1(const void* b, size_t i) {
    return __half2float(static_cast<const __half*>(b)[i]);
  }
  static __device__ __forceinline__ void store4(void* b, size_t i, float4 v) {
    __half2 lo = __floats2half2_rn(v.x, v.y);
    __half2 hi = __floats2half2_rn(v.z, v.w);
    uint2 r;
    r.x = *reinterpret_cast<unsigned*>(&lo);
    r.y = *reinterpret_cast<unsigned*>(&hi);
    __stcs(reinterpret_cast<uint2*>(static_cast<__half*>(b) + i), r);
  }
  static __device__ __forceinline__ void store1(void* b, size_t i, float v) {
    static_cast<__half*>(b)[i] = __float2half_rn(v);
  }
};

template <typename TIn, bool VEC>
__device__ __forceinline__ float4 load_depth(const void* base, size_t idx, int xc, int width) {
  if (VEC) return Px<TIn>::load4(base, idx);
  float4 d;
  d.x = (xc + 0 < width) ? Px<TIn>::load1(base, idx + 0) : 0.0f;
  d.y = (xc + 1 < width) ? Px<TIn>::load1(base, idx + 1) : 0.0f;
  d.z = (xc + 2 < width) ? Px<TIn>::load1(base, idx + 2) : 0.0f;
  d.w = (xc + 3 < width) ? Px<TIn>::load1(base, idx + 3) : 0.0f;
  return d;
}

template <typename TOut, bool VEC>
__device__ __forceinline__ void store_px(void* base, size_t idx, float4 v, int xc, int width) {
  if (VEC) {
    Px<TOut>::store4(base, idx, v);
    return;
  }
  if (xc + 0 < width) Px<TOut>::store1(base, idx + 0, v.x);
  if (xc + 1 < width) Px<TOut>::store1(base, idx + 1, v.y);
  if (xc + 2 < width) Px<TOut>::store1(base, idx + 2, v.z);
  if (xc + 3 < width) Px<TOut>::store1(base, idx + 3, v.w);
}

}  // namespace

template <int NMAX, typename TIn, typename TOut, bool VEC>
__global__ void __launch_bounds__(kMapThreads) map_kernel(MapParams p) {
  extern __shared__ float4 smem4[];
  float* Ex = reinterpret_cast<float*>(smem4);   // [NMAX][kTileW]
  float* Ey = Ex + NMAX * kTileW;                // [tile_h][NMAX]
  __shared__ PointsSmem<NMAX> P;
  __shared__ float s_least[NMAX];  // odd widths: the least column factor that a point keeps
  __shared__ unsigned long long s_key[kMapThreads / 32];

  allow_successor();
  wait_for_predecessor();
  const int tpf = p.tiles_x * p.tiles_y;
  const int f = blockIdx.x / tpf;
  const int rem = blockIdx.x - f * tpf;
  const int ty = rem / p.tiles_x;
  const int tx = rem - ty * p.tiles_x;
  FrameRec* rec = const_cast<FrameRec*>(p.recs) + ((p.f0 + f) & p.rec_mask);
  const int n = rec->n_valid;                       // block-uniform
  const int nc = min(NMAX, (n + 3) & ~3);           // padded to a multiple of 4
  const float inv_n = rec->inv_n;
  // Odd widths: points are dropped by the rule of the row-phase units, and
  // tiles lie within its bands.  64 frames of 853x479, window 12, FP32, planes
  // off the boundary: 123 -> 126 us a pass.
  const bool odd = p.band_h > 0;
  int by0 = 0, brows = p.height, x0 = tx * kTileW, y0 = ty * p.tile_h;
  if (odd) {
    const int per_band = (p.band_h + p.tile_h - 1) / p.tile_h;
    by0 = ty / per_band * p.band_h;
    brows = min(p.band_h, p.height - by0);
    y0 = by0 + ty % per_band * p.tile_h;
  }
  const int rows = min(p.tile_h, by0 + brows - y0);
  const int tid = threadIdx.x;

  if (tid < 32) {
    float uh = 0.f, ul = 0.f, vh = 0.f, vl = 0.f, ch = 0.f, cl = 0.f;
    if (tid < n) {
      P.uhi[tid] = uh = rec->ux_hi[tid];
      P.ulo[tid] = ul = rec->ux_lo[tid];
      P.vhi[tid] = vh = rec->vy_hi[tid];
      P.vlo[tid] = vl = rec->vy_lo[tid];
      P.chi[tid] = ch = rec->c_hi[tid];
      P.clo[tid] = cl = rec->c_lo[tid];
    }
    if (odd) {
      const float threshold = odd_threshold(n, p.width, p.height, inv_n, uh, ul, vh, vl, ch, cl);
      if (tid < n) s_least[tid] = least_column(band_row_factor(by0, brows, vh, vl, ch, cl), inv_n, threshold);
    }
  }
  __syncthreads();
  // Column factors Ex[i][c] and row factors Ey[r][i] (1/Z folded in); zero
  // for the padding points n <= i < nc.
  for (int e = tid; e < nc * kTileW; e += kMapThreads) {
    const int i = e >> 7, c = e & (kTileW - 1);
    float f = i < n ? gauss_factor((float)(x0 + c), P.uhi[i], P.ulo[i], P.chi[i], P.clo[i]) : 0.0f;
    if (odd && i < n && f < s_least[i]) f = 0.0f;
    Ex[e] = f;
  }
  for (int r = tid >> 5; r < rows; r += kMapThreads / 32) {
    for (int i = tid & 31; i < nc; i += 32) {
      Ey[r * NMAX + i] =
          i < n ? gauss_factor((float)(y0 + r), P.vhi[i], P.vlo[i], P.chi[i], P.clo[i]) * inv_n
                : 0.0f;
    }
  }
  __syncthreads();

  const int lane = tid & 31, warp = tid >> 5;
  const int xc = x0 + lane * 4;
  const bool col_ok = xc < p.width;
  float2 ex01[NMAX], ex23[NMAX];
#pragma unroll
  for (int i = 0; i < NMAX; ++i) {
    if (i < nc) {
      const float4 e = *reinterpret_cast<const float4*>(Ex + i * kTileW + lane * 4);
      ex01[i] = make_float2(e.x, e.y);
      ex23[i] = make_float2(e.z, e.w);
    }
  }

  const size_t plane = (size_t)p.width * (size_t)p.height;
  const size_t fbase = (size_t)f * plane;
  const void* dep = p.depth;
  float best = -1.0f;
  unsigned bidx = 0;
  const bool has_depth = dep != nullptr;
  float mx = 1.0f, inv = 1.0f;
  const bool scaled = odd && p.normalize == MF_NORM_MAX;  // by the maximum that the first pass found
  if (scaled) {
    mx = norm_divisor(rec);
    inv = 1.0f / mx;
  }
  float4 dnext = make_float4(0.f, 0.f, 0.f, 0.f);
  int r = warp;
  if (has_depth && col_ok && r < rows)
    dnext = load_depth<TIn, VEC>(dep, fbase + (size_t)(y0 + r) * p.width + xc, xc, p.width);
  for (; r < rows; r += kMapThreads / 32) {
    const float4 dv = dnext;
    const int rn = r + kMapThreads / 32;
    const size_t idx = fbase + (size_t)(y0 + r) * p.width + xc;
    if (has_depth && col_ok && rn < rows)
      dnext = load_depth<TIn, VEC>(dep, idx + (size_t)(kMapThreads / 32) * p.width, xc, p.width);
    float2 a01 = make_float2(0.f, 0.f), a23 = make_float2(0.f, 0.f);
    const float4* ey4 = reinterpret_cast<const float4*>(Ey + r * NMAX);
#pragma unroll
    for (int i = 0; i < NMAX; i += 4) {
      if (i >= nc) break;
      const float4 e = ey4[i >> 2];
      a01 = ffma2(ex01[i + 0], e.x, a01);
      a23 = ffma2(ex23[i + 0], e.x, a23);
      a01 = ffma2(ex01[i + 1], e.y, a01);
      a23 = ffma2(ex23[i + 1], e.y, a23);
      a01 = ffma2(ex01[i + 2], e.z, a01);
      a23 = ffma2(ex23[i + 2], e.z, a23);
      a01 = ffma2(ex01[i + 3], e.w, a01);
      a23 = ffma2(ex23[i + 3], e.w, a23);
    }
    if (!col_ok) continue;
    float4 m = make_float4(a01.x, a01.y, a23.x, a23.y);
    if (scaled && mx != 1.0f) {
      m.x = corrected_quotient(m.x, mx, inv);
      m.y = corrected_quotient(m.y, mx, inv);
      m.z = corrected_quotient(m.z, mx, inv);
      m.w = corrected_quotient(m.w, mx, inv);
    }
    if (p.M) store_px<TOut, VEC>(p.M, idx, m, xc, p.width);
    if (p.G) {
      float4 g;
      if (has_depth) {
        g.x = m.x * depth_weight(dv.x, rec->d0);
        g.y = m.y * depth_weight(dv.y, rec->d0);
        g.z = m.z * depth_weight(dv.z, rec->d0);
        g.w = m.w * depth_weight(dv.w, rec->d0);
      } else {
        g = make_float4(0.f, 0.f, 0.f, 0.f);
      }
      store_px<TOut, VEC>(p.G, idx, g, xc, p.width);
    }
    const unsigned pix = (unsigned)((y0 + r) * p.width + xc);
    if (m.x > best) { best = m.x; bidx = pix; }
    if (m.y > best && (VEC || xc + 1 < p.width)) { best = m.y; bidx = pix + 1; }
    if (m.z > best && (VEC || xc + 2 < p.width)) { best = m.z; bidx = pix + 2; }
    if (m.w > best && (VEC || xc + 3 < p.width)) { best = m.w; bidx = pix + 3; }
  }

  // Per-frame argmax: largest M, ties to the lowest linear index.
  unsigned long long key =
      best >= 0.0f ? ((unsigned long long)__float_as_uint(best) << 32) | (0xffffffffu - bidx) : 0ull;
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long k2 = __shfl_xor_sync(0xffffffffu, key, o);
    key = k2 > key ? k2 : key;
  }
  if (lane == 0) s_key[warp] = key;
  __syncthreads();
  if (tid == 0 && n > 0 && !scaled) {
    unsigned long long k = s_key[0];
    for (int w = 1; w < kMapThreads / 32; ++w) k = s_key[w] > k ? s_key[w] : k;
    if (k) atomicMax(&rec->argmax_key, k);
  }
}

// ---------------------------------------------------------------------------
// Streaming kernel for frames whose planes start on CPT-pixel boundaries (the
// common case): persistent CTAs of 8 warps take the frames' units (band of
// up to 256 rows x group of 8 strips) in frame order from the dynamic
// schedule; map_unit does the work.  PH: an odd width, where a band's units are
// its row phases (mf_map_unit.cuh).
template <int NMAX, int CPT, typename TIn, typename TOut, int MODE, bool PH>
__global__ void __launch_bounds__(kUnitThreads, unit_ctas_per_sm(NMAX, CPT))
    map_stream_kernel(MapParams p, int band_h, int sub_h) {
  extern __shared__ float4 smem4[];
  float* Ey = reinterpret_cast<float*>(smem4);                          // [sub_h][NMAX]
  uint4* ring = reinterpret_cast<uint4*>(Ey + (size_t)sub_h * NMAX);    // [8][stages][32]
  __shared__ PointsSmem<kMaxPts> P[kGroupStrips];
  __shared__ uint4 zeros[kZeroBytes / 16];
  allow_successor();
  init_zero_source(zeros);
  wait_for_predecessor();
  constexpr int kGroupW = kGroupStrips * 32 * CPT;
  const int groups_x = (p.width + (PH ? CPT - 1 : 0) + kGroupW - 1) / kGroupW;
  const int bands = (p.height + band_h - 1) / band_h;
  constexpr int phases = PH ? CPT : 1;
  const int cuts = (band_h + phases * sub_h - 1) / (phases * sub_h);
  const int subs = cuts * phases;  // units per band and strip group
  const long long units = (long long)p.n_frames * bands * subs * groups_x;
  const size_t plane = (size_t)p.width * (size_t)p.height;
  // this warp's ring: S rows of 32 lanes x CPT depth elements (uint4 units)
  uint4* my_ring = ring + (size_t)(threadIdx.x >> 5) * ring_stages(CPT, (int)sizeof(TIn), NMAX) * 2 * CPT *
                             (int)sizeof(TIn);
  __shared__ long long s_next[2];
  long long u = blockIdx.x;
  for (int k = 0; u < units; ++k) {
    // p.info and p.points are set where the frames' last units write the
    // result records
    const unsigned claim = claim_unit(p.sched);
    const int per_frame = bands * subs * groups_x;
    const int f = (int)(u / per_frame);
    const int rem = (int)(u - (long long)f * per_frame);
    const int sb = rem / groups_x, g = rem - sb * groups_x;
    const int b = sb / subs;
    UnitGeom ug;
    ug.rec = const_cast<FrameRec*>(p.recs) + ((p.f0 + f) & p.rec_mask);
    ug.depth = p.depth ? static_cast<const char*>(p.depth) + (size_t)f * plane * sizeof(TIn) : nullptr;
    ug.M = p.M ? static_cast<char*>(p.M) + (size_t)f * plane * sizeof(TOut) : nullptr;
    ug.G = p.G ? static_cast<char*>(p.G) + (size_t)f * plane * sizeof(TOut) : nullptr;
    ug.width = p.width;
    ug.fault = p.fault;
    ug.height = p.height;
    ug.by0 = b * band_h;
    ug.brows = min(band_h, p.height - ug.by0);
    const int sub = sb - b * subs;
    if (PH) {
      const int cut = sub / phases;
      ug.y0 = ug.by0 + cut * phases * sub_h + (sub - cut * phases);
      ug.rows = min(sub_h, (ug.by0 + ug.brows - ug.y0 + phases - 1) / phases);
      // distance of pixel (y0, 0) from the CPT-element boundary before it
      ug.shift = (int)((f * plane + (size_t)ug.y0 * p.width) & (CPT - 1));
    } else {
      ug.y0 = ug.by0 + sub * sub_h;
      ug.rows = min(sub_h, ug.by0 + ug.brows - ug.y0);
      ug.shift = 0;
    }
    ug.gx0 = g * kGroupW;
    ug.d0 = ug.rec->d0;
    if (p.points && rem == 0 && threadIdx.x < p.window)
      motion_point(ug.rec, threadIdx.x, p.points + (size_t)f * p.window + threadIdx.x);
    if (ug.rows > 0) map_unit<NMAX, CPT, TIn, TOut, MODE, PH>(ug, Ey, my_ring, P, zeros);
    u = next_unit(p.sched, claim, units, s_next, k);  // after every warp's argmax candidate
    if (p.info && threadIdx.x == 0) {
      __threadfence();
      if (atomicAdd(&ug.rec->units_done, 1u) == (unsigned)per_frame - 1u) {
        __threadfence();
        finalize_frame(ug.rec, p.width, p.info + f, p.normalize);
        ug.rec->units_done = 0u;  // the frame may be rendered again (a retry, a replayed graph)
      }
    }
  }
  bulk_wait_all();
}

namespace mapk {

template <typename T>
constexpr int out_dtype_of() {
  return std::is_same<T, float>::value ? MF_F32 : std::is_same<T, __half>::value ? MF_F16 : MF_BF16;
}

// Parameters of the in-place MF_NORM_MAX pass over p's planes
// (mf_map_kernel.cu).
NormalizeParams normalize_params(const MapParams& p);

// Launches the persistent kernel k over `units` units: one CTA per unit up
// to the CTAs the device holds at the band's largest shared memory.
template <typename K>
cudaError_t launch_persistent(K k, size_t smem_max, long long units, size_t smem, const MapParams& p,
                              int band_h, int sub_h, cudaStream_t st, int64_t* nl) {
  const KernelFit f = host_kernel_fit(reinterpret_cast<const void*>(k), kUnitThreads, smem_max, smem_max);
  const long long grid = std::min<long long>(units, (long long)f.sms * f.per_sm);
  const cudaError_t e = launch_after(k, (unsigned)grid, kUnitThreads, smem, st, p, band_h, sub_h);
  if (e == cudaSuccess) ++*nl;
  return e;
}

// How a launch is cut into units: bands of band_h rows, units of sub_h rows
// of a band (with PH of one of its row phases).
struct UnitPlan {
  int band_h, sub_h;
  long long units;
};

// Rows per band.  Bands of at most 128 rows at up to 16 points skip depth
// and factors at a finer grain (1080p x 304 frames, window 16, against 256
// rows: ACCEL FP32 1.20 -> 1.24 of measured HBM, HEADING unchanged; 64 rows
// reach 1.27 but lose 4 % on HEADING).  At 32 points the Ey table per row
// is twice as costly and 256 rows stay faster.
// Row phases share a band's rows, so their bands are higher.
template <int NMAX, bool PH>
constexpr int band_max() {
  return NMAX <= 16 && !PH ? 128 : kBandMax;
}
inline int band_height(int height, int most) {
  const int bands = (height + most - 1) / most;
  return (height + bands - 1) / bands;
}

template <int NMAX, int CPT, bool PH>
UnitPlan plan_units(const MapParams& p, const KernelFit& fit) {
  UnitPlan u;
  u.band_h = band_height(p.height, band_max<NMAX, PH>());
  const int bands = (p.height + u.band_h - 1) / u.band_h;
  constexpr int kGroupW = kGroupStrips * 32 * CPT;
  constexpr int phases = PH ? CPT : 1;
  const int unit_h = (u.band_h + phases - 1) / phases;  // rows of a band's unit
  const long long per_sub =
      (long long)p.n_frames * bands * phases * ((p.width + (PH ? CPT - 1 : 0) + kGroupW - 1) / kGroupW);
  // Rows per unit of a small launch: a band is cut while the units still fit
  // one wave of resident CTAs, down to kMinRows (below that a unit's factors
  // cost more than its rows).  Whole bands, one CTA each, left most SMs idle:
  // one 320x240 frame 2 units, one 1080p frame 36.  Per pass, whole bands ->
  // cut: 320x240 34.5 -> 29.0 us, 1080p 40.8 -> 32.4, 16 frames of 640x480
  // FP16 36.3 -> 28.7; cutting into two waves instead of one: 16 frames 32.8,
  // two batches of 60 frames at 504x280 unchanged.
  constexpr int kMinRows = 16;
  const long long split = std::max<long long>(
      1, std::min<long long>((long long)fit.sms * fit.per_sm / per_sub, unit_h / kMinRows));
  u.sub_h = (int)((unit_h + split - 1) / split);
  if (split > 1) u.sub_h += u.sub_h & 1;
  u.units = per_sub * ((u.band_h + phases * u.sub_h - 1) / (phases * u.sub_h));
  return u;
}

// The first pass of MF_NORM_MAX: every frame's maximum.  One kernel serves
// every storage type; it reads no depth, so it has no ring and its shared
// memory is the row factors alone.
template <int NMAX, int CPT, bool PH>
cudaError_t launch_max_pass(const MapParams& p, const UnitPlan& u, cudaStream_t st, int64_t* nl) {
  MapParams m = p;
  m.info = nullptr;
  m.points = nullptr;
  return launch_persistent(map_stream_kernel<NMAX, CPT, float, float, kUnitMaxOnly, PH>,
                           row_factor_bytes(NMAX, band_max<NMAX, PH>() / (PH ? CPT : 1)), u.units,
                           row_factor_bytes(NMAX, u.sub_h), m, u.band_h, u.sub_h, st, nl);
}

// The persistent unit kernel with CPT columns per lane over p's frames (one
// launch, or for MF_NORM_MAX a max-only pass then a scaled pass over the same
// units with the same sums); *nl receives the launch count, *recorded whether
// the launch writes the result records.
template <int NMAX, int CPT, typename TIn, typename TOut, bool PH = false>
cudaError_t launch_units(const MapParams& p, cudaStream_t st, int64_t* nl, bool* recorded) {
  const size_t smem_max = unit_smem_bytes(NMAX, band_max<NMAX, PH>() / (PH ? CPT : 1), CPT, (int)sizeof(TIn));
  const KernelFit fit = host_kernel_fit(
      reinterpret_cast<const void*>(map_stream_kernel<NMAX, CPT, TIn, TOut, kUnitFull, PH>), kUnitThreads, smem_max,
      smem_max);
  const UnitPlan u = plan_units<NMAX, CPT, PH>(p, fit);
  const size_t smem = unit_smem_bytes(NMAX, u.sub_h, CPT, (int)sizeof(TIn));
  // Result records.  In a launch of few units the frame's last unit writes
  // its record, which saves a launch where launching is most of the time; a
  // larger one leaves them to the caller's kernel, because each unit's count
  // waits behind a fence for the unit's rows to be written.  Per pass, own
  // kernel -> last unit: camera loop 320x240 (14 units) 15.1 -> 13.8 us, 1080p
  // (432 units) 18.7 -> 19.2, 16 frames of 640x480 (256 units) 20.2 -> 20.9.
  // The launch is worth 1 to 2 us while the host is what a call waits for, the
  // fences cost 0.2 to 0.6 us once it is the GPU; the line lies where one or two
  // frames end: 2 frames of 320x240 at 32 points (30 units) 11.8 -> 10.0 us, 4
  // (60 units) 13.4 -> 13.6, one of 720p (84 units) 11.2 -> 10.6, 8 of 320x240
  // (112 units) 12.3 -> 12.9, 4 of 720p (336 units) 11.6 -> 12.9.
  constexpr long long kFusedUnits = 64;
  MapParams q = p;
  *recorded = u.units <= kFusedUnits;
  if (!*recorded) {
    q.info = nullptr;
    q.points = nullptr;
  }
  cudaError_t e;
  if (p.normalize != MF_NORM_MAX) {
    e = launch_persistent(map_stream_kernel<NMAX, CPT, TIn, TOut, kUnitFull, PH>, smem_max, u.units, smem, q,
                          u.band_h, u.sub_h, st, nl);
  } else {
    e = launch_max_pass<NMAX, CPT, PH>(q, u, st, nl);
    if (e == cudaSuccess)
      e = launch_persistent(map_stream_kernel<NMAX, CPT, TIn, TOut, kUnitScaled, PH>, smem_max, u.units, smem, q,
                            u.band_h, u.sub_h, st, nl);
  }
  return e;
}

template <int NMAX, typename TIn, typename TOut>
cudaError_t launch_typed(const MapParams& p, cudaStream_t st, int64_t* nl, bool* recorded) {
  const long long tiles = (long long)p.n_frames * p.tiles_x * p.tiles_y;
  if (tiles <= 0) return cudaSuccess;
  if (tiles > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
  // Pixels per lane.  FP32 maps: 2, so that windows of up to 16 points fit
  // three CTAs (24 warps) per SM, whose extra loads in flight beat the wider
  // rows (1080p ACCEL, window 16: 1.20 vs 1.16 of measured HBM).  16-bit maps:
  // 4 (8-byte stores; 2 pixels lose 20 % at up to 16 points), also above 16
  // points, where the column factors alone take 128 registers and one CTA
  // fits per SM (HEADING BF16 window 32: 0.49 -> 0.52 against 2 pixels per
  // lane); even widths or planes that do not allow 4 take 2.  Odd widths take
  // the same kernel by row phases, and planes that start elsewhere than on a
  // boundary of as many elements the tiled kernel, which gives the same bits
  // there.  Tiled -> row phases, 120 frames of 853x480, window 12, FP32: 207 ->
  // 134 us a pass.
  constexpr int kWide = sizeof(TOut) == 2 ? 4 : 2;
  auto aligned = [](const void* q, size_t a) { return q == nullptr || ((uintptr_t)q % a) == 0; };
  auto starts = [&](int cpt) {
    return aligned(p.depth, cpt * sizeof(TIn)) && aligned(p.M, cpt * sizeof(TOut)) && aligned(p.G, cpt * sizeof(TOut));
  };
  if ((p.width & 1) && starts(kWide)) {
    return launch_units<NMAX, kWide, TIn, TOut, true>(p, st, nl, recorded);
  } else if (p.width % kWide == 0 && starts(kWide)) {
    return launch_units<NMAX, kWide, TIn, TOut>(p, st, nl, recorded);
  } else if (p.width % 2 == 0 && starts(2)) {
    return launch_units<NMAX, 2, TIn, TOut>(p, st, nl, recorded);
  } else {
    MapParams q = p;
    const bool odd = (p.width & 1) != 0;
    cudaError_t e = cudaSuccess;
    if (odd) {  // the row phases' bands and passes, so that both kernels give the same bits
      q.band_h = band_height(p.height, band_max<NMAX, true>());
      q.tiles_y = (p.height + q.band_h - 1) / q.band_h * ((q.band_h + p.tile_h - 1) / p.tile_h);
      if (p.normalize == MF_NORM_MAX) {
        const size_t smem = row_factor_bytes(NMAX, band_max<NMAX, true>() / kWide);
        const KernelFit fit = host_kernel_fit(
            reinterpret_cast<const void*>(map_stream_kernel<NMAX, kWide, float, float, kUnitMaxOnly, true>),
            kUnitThreads, smem, smem);
        e = launch_max_pass<NMAX, kWide, true>(p, plan_units<NMAX, kWide, true>(p, fit), st, nl);
      }
    }
    const long long all = (long long)p.n_frames * q.tiles_x * q.tiles_y;
    if (e == cudaSuccess && all > 0x7fffffffLL) e = cudaErrorInvalidConfiguration;
    const size_t smem = (size_t)NMAX * kTileW * 4 + (size_t)p.tile_h * NMAX * 4;
    auto k = map_kernel<NMAX, TIn, TOut, false>;
    if (smem > 48 * 1024) host_kernel_fit(reinterpret_cast<const void*>(k), kMapThreads, smem, smem);
    if (e == cudaSuccess) e = launch_after(k, (unsigned)all, kMapThreads, smem, st, q);
    if (e != cudaSuccess) return e;
    *nl += 1;
    if (p.normalize == MF_NORM_MAX && !odd)
      e = launch_normalize(normalize_params(p), out_dtype_of<TOut>(), st, nl);
    return e;
  }
}

template <int NMAX>
cudaError_t launch_n(const MapParams& p, int in_dtype, int out_dtype, cudaStream_t st,
                     int64_t* nl, bool* recorded) {
  switch (in_dtype * 3 + out_dtype) {
    case MF_F32 * 3 + MF_F32: return launch_typed<NMAX, float, float>(p, st, nl, recorded);
    case MF_F32 * 3 + MF_BF16: return launch_typed<NMAX, float, __nv_bfloat16>(p, st, nl, recorded);
    case MF_F32 * 3 + MF_F16: return launch_typed<NMAX, float, __half>(p, st, nl, recorded);
    case MF_BF16 * 3 + MF_F32: return launch_typed<NMAX, __nv_bfloat16, float>(p, st, nl, recorded);
    case MF_BF16 * 3 + MF_BF16: return launch_typed<NMAX, __nv_bfloat16, __nv_bfloat16>(p, st, nl, recorded);
    case MF_BF16 * 3 + MF_F16: return launch_typed<NMAX, __nv_bfloat16, __half>(p, st, nl, recorded);
    case MF_F16 * 3 + MF_F32: return launch_typed<NMAX, __half, float>(p, st, nl, recorded);
    case MF_F16 * 3 + MF_BF16: return launch_typed<NMAX, __half, __nv_bfloat16>(p, st, nl, recorded);
    case MF_F16 * 3 + MF_F16: return launch_typed<NMAX, __half, __half>(p, st, nl, recorded);
  }
  return cudaErrorInvalidValue;
}

}  // namespace mapk
}  // namespace mf
