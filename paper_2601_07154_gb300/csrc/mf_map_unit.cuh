// Device code shared by the per-stream and the batched map kernels: the
// motion-focus map of Eq. 7 and the motion-guided depth over one "unit" (a
// band of up to 256 rows of one frame, across a group of 8 adjacent strips of
// 32*CPT columns), with the frame's argmax.  Both launch paths run exactly
// this code, so a frame's maps do not depend on which path, batch or tile
// schedule produced them.
//
// Per unit:
//   * every warp keeps only the points whose Gaussian can reach the unit: a
//     point whose largest column factor over the unit times its largest row
//     factor over the unit's band (times 1/Z) is below 2^-40 contributes less
//     than 2^-40 to every pixel of it, far inside the 1e-10 absolute floor of
//     the map tolerance; kept points keep their order.  A small launch cuts a
//     band into several units, and all of them keep the band's points, so a
//     frame's maps do not depend on how many frames were launched with it
//     (odd widths: by a rule per column, at odd_threshold below);
//   * each warp applies the same rule to its own strip: a strip that no
//     kept point reaches reads no depth and writes zeros (at most 32 points
//     are dropped from any pixel, each below 2^-40, together below 2^-35);
//   * the CTA evaluates the band's row factors once in shared memory;
//   * each warp owns one strip: every lane holds its CPT columns' factors for
//     the kept points in registers and streams the unit's rows two at a time
//     (four above 16 points on 16-bit maps; CPT/2 independent FMA chains a
//     row), depth arriving through the warp's
//     ring of cp.async stages, maps leaving through streaming stores.
// The map is a sum of N isotropic Gaussians, so each term factors as
//     exp(-((x-u)^2 + (y-v)^2) c) = exp(-(x-u)^2 c) * exp(-(y-v)^2 c),
// c = 1/(2 sigma_i^2); every pixel then costs one FP32 FMA per kept point,
// issued two pixels at a time (fma.rn.f32x2), in point order.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <math.h>

#include <type_traits>

#include "mf_internal.h"

namespace mf {

constexpr float kCullBelow = 9.094947017729282e-13f;  // 2^-40

// Resident warps per SM the persistent map kernels are compiled for: 24
// where 2 pixels per lane and at most 16 points keep the unit within 85
// registers; 8 for 4 pixels per lane above 16 points (the column factors
// alone take 128 registers); else 16 (the 128-register unit).  CTAs per SM:
// that over the warps of a CTA.
__host__ __device__ constexpr int unit_warps_per_sm(int nmax, int cpt) {
  return cpt == 2 && nmax <= 16 ? 24 : (cpt == 4 && nmax > 16 ? 8 : 16);
}
__host__ __device__ constexpr int unit_ctas_per_sm(int nmax, int cpt) {
  return unit_warps_per_sm(nmax, cpt) / kGroupStrips;
}

// Depth rows in flight per warp; the ring packs a row at CPT x in_bytes
// bytes per lane.  Rows of 16 bytes per lane: kStages.  Narrower rows: 2 KB
// per warp where 24 warps share an SM, 4 KB where 16 or 8 do (1080p frames:
// the 4 KB ring gains 2-6 % at 16 warps per SM and loses about 1 % at
// 24).
__host__ __device__ constexpr int ring_stages(int cpt, int in_bytes, int nmax) {
  return cpt * in_bytes >= 16 ? kStages
                              : (unit_warps_per_sm(nmax, cpt) == 24 ? 2048 : 4096) / (32 * cpt * in_bytes);
}

// Whether a unit's row loop takes four rows a step: where the column factors
// leave one CTA per SM and the ring holds at least eight rows.
__host__ __device__ constexpr bool four_rows(int cpt, int in_bytes, int nmax) {
  return cpt == 4 && nmax > 16 && ring_stages(cpt, in_bytes, nmax) >= 8;
}

// A lane's depth bytes of ring row slot `slot` (rows packed at BYTES per lane).
template <int BYTES>
__device__ __forceinline__ uint4 ring_row(const uint4* ring, int slot) {
  const char* q = reinterpret_cast<const char*>(ring) + slot * BYTES;
  uint4 v = make_uint4(0u, 0u, 0u, 0u);
  if (BYTES == 16) {
    v = *reinterpret_cast<const uint4*>(q);
  } else if (BYTES == 8) {
    const uint2 t = *reinterpret_cast<const uint2*>(q);
    v.x = t.x;
    v.y = t.y;
  } else {
    v.x = *reinterpret_cast<const unsigned*>(q);
  }
  return v;
}

template <int NMAX>
struct PointsSmem {
  float uhi[NMAX], ulo[NMAX], vhi[NMAX], vlo[NMAX], chi[NMAX], clo[NMAX];
  int kept;      // entries in use (the map unit's lists)
  float min_peak;  // smallest contribution that keeps a point
};

// 2^x by the hardware base-2 exponential (PTX ex2.approx.ftz: relative
// error of a few ulp; results below 2^-126 flush to 0).
__device__ __forceinline__ float exp2_hw(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// exp(-(q - hi - lo)^2 / (2 sigma^2)) = 2^-((q - hi - lo)^2 (chi + clo)) for an
// integer-valued q, with chi + clo = log2(e) / (2 sigma^2) as a float pair.
// hi lies on a 2^-8 grid with |hi| < 2^15, so q - hi is exact; the square is
// carried as a compensated pair, which keeps the exponent's relative error
// near one FP32 rounding before the base-2 exponential.
__device__ __forceinline__ float gauss_factor(float q, float hi, float lo, float chi, float clo) {
  const float dh = q - hi;
  const float p2 = dh * dh;
  const float e2 = fmaf(dh, dh, -p2);   // dh^2 = p2 + e2 exactly
  float qq = fmaf(-2.0f * dh, lo, e2);  // (dh - lo)^2 = p2 + qq
  qq = fmaf(lo, lo, qq);
  const float t1 = fmaf(clo, p2, chi * qq);
  const float a = fmaf(chi, p2, t1);
  return exp2_hw(-a);
}


__device__ __forceinline__ float2 ffma2(float2 a, float b, float2 c) {
  float2 d;
  asm("{\n\t.reg .b64 ra, rb, rc, rd;\n\t"
      "mov.b64 ra, {%2, %3};\n\t"
      "mov.b64 rb, {%4, %4};\n\t"
      "mov.b64 rc, {%5, %6};\n\t"
      "fma.rn.f32x2 rd, ra, rb, rc;\n\t"
      "mov.b64 {%0, %1}, rd;\n\t}"
      : "=f"(d.x), "=f"(d.y)
      : "f"(a.x), "f"(a.y), "f"(b), "f"(c.x), "f"(c.y));
  return d;
}

// a * b on both lanes of a (the first term of a sum: a product rounds
// exactly as a fused multiply-add onto +0 does when the product is >= +0).
__device__ __forceinline__ float2 fmul2(float2 a, float b) {
  float2 d;
  asm("{\n\t.reg .b64 ra, rb, rd;\n\t"
      "mov.b64 ra, {%2, %3};\n\t"
      "mov.b64 rb, {%4, %4};\n\t"
      "mul.rn.f32x2 rd, ra, rb;\n\t"
      "mov.b64 {%0, %1}, rd;\n\t}"
      : "=f"(d.x), "=f"(d.y)
      : "f"(a.x), "f"(a.y), "f"(b));
  return d;
}

// Lane-wise a + b, a * b and fma(a, b, c) on f32x2 pairs (IEEE round to
// nearest on each lane: the values of the scalar operations).
__device__ __forceinline__ float2 fadd2v(float2 a, float2 b) {
  float2 d;
  asm("{\n\t.reg .b64 ra, rb, rd;\n\tmov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %5};\n\t"
      "add.rn.f32x2 rd, ra, rb;\n\tmov.b64 {%0, %1}, rd;\n\t}"
      : "=f"(d.x), "=f"(d.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return d;
}
__device__ __forceinline__ float2 fmul2v(float2 a, float2 b) {
  float2 d;
  asm("{\n\t.reg .b64 ra, rb, rd;\n\tmov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %5};\n\t"
      "mul.rn.f32x2 rd, ra, rb;\n\tmov.b64 {%0, %1}, rd;\n\t}"
      : "=f"(d.x), "=f"(d.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return d;
}
__device__ __forceinline__ float2 ffma2v(float2 a, float2 b, float2 c) {
  float2 d;
  asm("{\n\t.reg .b64 ra, rb, rc, rd;\n\tmov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %5};\n\t"
      "mov.b64 rc, {%6, %7};\n\tfma.rn.f32x2 rd, ra, rb, rc;\n\tmov.b64 {%0, %1}, rd;\n\t}"
      : "=f"(d.x), "=f"(d.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
  return d;
}

// gauss_factor at q0 and q1 (integer-valued), the exponent's steps on f32x2
// pairs: the same operations in the same order on each lane, with the signs
// carried through exact negations, so the same values.
__device__ __forceinline__ float2 gauss_pair(float q0, float q1, float hi, float lo, float chi, float clo) {
  const float2 dh = fadd2v(make_float2(q0, q1), make_float2(-hi, -hi));           // exact
  const float2 p2 = fmul2v(dh, dh);
  const float2 e2 = ffma2v(dh, dh, fmul2v(p2, make_float2(-1.0f, -1.0f)));        // dh^2 - p2
  float2 qq = ffma2v(fmul2v(dh, make_float2(-2.0f, -2.0f)), make_float2(lo, lo), e2);
  qq = ffma2v(make_float2(lo, lo), make_float2(lo, lo), qq);
  const float2 nt1 = ffma2v(make_float2(-clo, -clo), p2, fmul2v(make_float2(-chi, -chi), qq));
  const float2 na = ffma2v(make_float2(-chi, -chi), p2, nt1);                      // -a
  return make_float2(exp2_hw(na.x), exp2_hw(na.y));
}

// max(a, b, c) in one instruction (three-input max.f32 of sm_100 and later).
__device__ __forceinline__ float fmax3(float a, float b, float c) {
  float d;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}

// Largest of one lane's CPT pixels of rows a and b (b only when `two`).
template <int CPT>
__device__ __forceinline__ float lane_max(const float2 (&a)[CPT / 2], const float2 (&b)[CPT / 2], bool two) {
  float m = fmax3(a[0].x, a[0].y, two ? fmaxf(b[0].x, b[0].y) : a[0].x);
#pragma unroll
  for (int c = 1; c < CPT / 2; ++c) m = fmax3(m, fmaxf(a[c].x, a[c].y), two ? fmaxf(b[c].x, b[c].y) : m);
  return m;
}

// min(1, d0 / x) for x = D - 2^-149, as one approximate reciprocal (PTX
// rcp.approx.ftz, within about an ulp) and one saturating product, with no
// compare or select.  Subtracting the smallest denormal leaves every normal
// D unchanged and moves D = +0 and -0 below zero; the flush to zero of the
// reciprocal's input then gives:
//   normal D > 0        -> min(1, d0 / D);
//   positive denormal D -> 1/x = +inf -> 1 (the clamp of a huge quotient);
//   D = +-0, D < 0      -> 1/x <= -0 -> 0 ("no depth");
//   D = NaN             -> NaN, which the saturation turns into 0;
//   D = +inf            -> 0;  D = -inf -> -0 -> 0.
__device__ __forceinline__ float weight_of(float x, float d0) {
  float r, w;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  asm("mul.rn.sat.f32 %0, %1, %2;" : "=f"(w) : "f"(d0), "f"(r));
  return w;
}
__device__ __forceinline__ float depth_weight(float D, float d0) { return weight_of(D - 0x1p-149f, d0); }

// G = M min(1, d0 / D) for one lane's CPT pixels.
template <int CPT>
__device__ __forceinline__ void guided(const float (&m)[CPT], const float (&D)[CPT], float d0, float (&g)[CPT]) {
#pragma unroll
  for (int c = 0; c < CPT; c += 2) {
    float x0, x1;
    asm("{\n\t.reg .b64 ra, rb, rd;\n\tmov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %4};\n\t"
        "add.rn.f32x2 rd, ra, rb;\n\tmov.b64 {%0, %1}, rd;\n\t}"
        : "=f"(x0), "=f"(x1) : "f"(D[c]), "f"(D[c + 1]), "f"(-0x1p-149f));
    const float w0 = weight_of(x0, d0), w1 = weight_of(x1, d0);
    asm("{\n\t.reg .b64 ra, rb, rd;\n\tmov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %5};\n\t"
        "mul.rn.f32x2 rd, ra, rb;\n\tmov.b64 {%0, %1}, rd;\n\t}"
        : "=f"(g[c]), "=f"(g[c + 1]) : "f"(m[c]), "f"(m[c + 1]), "f"(w0), "f"(w1));
  }
}

__device__ __forceinline__ unsigned smem_u32(const void* p) {
  return static_cast<unsigned>(__cvta_generic_to_shared(p));
}

// A copy of the first `valid` of BYTES bytes; the others arrive as zeros and
// are not read.
template <int BYTES>
__device__ __forceinline__ void cp_async_part(void* dst, const void* src, int valid) {
  if (BYTES == 16)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(smem_u32(dst)), "l"(src), "r"(valid));
  else if (BYTES == 8)
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;\n" ::"r"(smem_u32(dst)), "l"(src), "r"(valid));
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;\n" ::"r"(smem_u32(dst)), "l"(src), "r"(valid));
}

template <int BYTES>
__device__ __forceinline__ void cp_async(void* dst, const void* src) {
  if (BYTES == 16)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(smem_u32(dst)), "l"(src));
  else if (BYTES == 8)
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(smem_u32(dst)), "l"(src));
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(smem_u32(dst)), "l"(src));
}

__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::); }

// Zero rows through the bulk-copy engine: a shared-memory source of zeros,
// at least one unit row wide (kGroupStrips strips x 32 lanes x 4 columns x
// 4 bytes).
constexpr int kZeroBytes = kGroupStrips * 32 * 4 * 4;
__device__ __forceinline__ void bulk_copy_s2g(void* dst, const void* src_smem, uint32_t bytes) {
  asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst),
               "r"((uint32_t)__cvta_generic_to_shared(src_smem)), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
// Every bulk copy this thread issued has written global memory.
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }

// Fills a kernel's zero source (every thread of the CTA calls this once,
// before its first unit) and makes it visible to the bulk-copy engine.
__device__ __forceinline__ void init_zero_source(uint4* zeros) {
  for (int i = threadIdx.x; i < kZeroBytes / 16; i += blockDim.x) zeros[i] = make_uint4(0u, 0u, 0u, 0u);
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  __syncthreads();
}

template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;\n" ::"n"(N));
}

// CPT consecutive storage elements <-> floats.
template <typename T, int CPT>
struct Vec;

template <int CPT>
struct Vec<float, CPT> {
  static __device__ __forceinline__ void unpack(const uint4& r, float (&d)[CPT]) {
    d[0] = __uint_as_float(r.x);
    d[1] = __uint_as_float(r.y);
    if (CPT == 4) {
      d[CPT > 2 ? 2 : 0] = __uint_as_float(r.z);
      d[CPT > 3 ? 3 : 0] = __uint_as_float(r.w);
    }
  }
  static __device__ __forceinline__ void store(void* plane, size_t i, const float (&v)[CPT]) {
    float* q = static_cast<float*>(plane) + i;
    if (CPT == 4)
      __stcs(reinterpret_cast<float4*>(q), make_float4(v[0], v[1], v[CPT > 2 ? 2 : 0], v[CPT > 3 ? 3 : 0]));
    else
      __stcs(reinterpret_cast<float2*>(q), make_float2(v[0], v[1]));
  }
};

template <typename H>
struct Half2Of;
template <>
struct Half2Of<__nv_bfloat16> {
  static __device__ __forceinline__ float2 to_f2(unsigned w) {
    return __bfloat1622float2(*reinterpret_cast<__nv_bfloat162*>(&w));
  }
  static __device__ __forceinline__ unsigned from_f2(float a, float b) {
    __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<unsigned*>(&h);
  }
};
template <>
struct Half2Of<__half> {
  static __device__ __forceinline__ float2 to_f2(unsigned w) {
    return __half22float2(*reinterpret_cast<__half2*>(&w));
  }
  static __device__ __forceinline__ unsigned from_f2(float a, float b) {
    __half2 h = __floats2half2_rn(a, b);
    return *reinterpret_cast<unsigned*>(&h);
  }
};

template <typename H, int CPT>
struct Vec16 {
  static __device__ __forceinline__ void unpack(const uint4& r, float (&d)[CPT]) {
    const float2 a = Half2Of<H>::to_f2(r.x);
    d[0] = a.x;
    d[1] = a.y;
    if (CPT == 4) {
      const float2 c = Half2Of<H>::to_f2(r.y);
      d[CPT > 2 ? 2 : 0] = c.x;
      d[CPT > 3 ? 3 : 0] = c.y;
    }
  }
  static __device__ __forceinline__ void store(void* plane, size_t i, const float (&v)[CPT]) {
    H* q = static_cast<H*>(plane) + i;
    if (CPT == 4) {
      uint2 w;
      w.x = Half2Of<H>::from_f2(v[0], v[1]);
      w.y = Half2Of<H>::from_f2(v[CPT > 2 ? 2 : 0], v[CPT > 3 ? 3 : 0]);
      __stcs(reinterpret_cast<uint2*>(q), w);
    } else {
      __stcs(reinterpret_cast<unsigned*>(q), Half2Of<H>::from_f2(v[0], v[1]));
    }
  }
};
__device__ __forceinline__ float to_f32(float v) { return v; }
__device__ __forceinline__ float to_f32(__nv_bfloat16 v) { return __bfloat162float(v); }
__device__ __forceinline__ float to_f32(__half v) { return __half2float(v); }

// One storage element from a float, with the rounding of Vec::store.
__device__ __forceinline__ void store_one(float* q, float v) { __stcs(q, v); }
__device__ __forceinline__ void store_one(__nv_bfloat16* q, float v) { *q = __float2bfloat16_rn(v); }
__device__ __forceinline__ void store_one(__half* q, float v) { *q = __float2half_rn(v); }

template <int CPT>
struct Vec<__nv_bfloat16, CPT> : Vec16<__nv_bfloat16, CPT> {};
template <int CPT>
struct Vec<__half, CPT> : Vec16<__half, CPT> {};

// Two rows' sums for one lane's CPT columns, points 0..nc-1 in order.  NC > 0
// fixes the trip count at compile time (all NMAX points kept).  INIT: the
// sums start with the first point's product (nc >= 1; no zeroed
// accumulators), else they add onto a and b as given.  Both give the same
// bits: every term is >= +0.
template <int NMAX, int CPT, int NC, bool INIT = false>
__device__ __forceinline__ void accum_two_rows(const float2 (&ex)[NMAX][CPT / 2], const float* ey0,
                                               const float* ey1, int nc, float2 (&a)[CPT / 2],
                                               float2 (&b)[CPT / 2]) {
  const float4* e0p = reinterpret_cast<const float4*>(ey0);
  const float4* e1p = reinterpret_cast<const float4*>(ey1);
#pragma unroll
  for (int i = 0; i < (NC ? NC : NMAX); i += 4) {
    if (NC == 0 && i >= nc) break;
    const float4 e = e0p[i >> 2];
    const float4 f = e1p[i >> 2];
    const float es[4] = {e.x, e.y, e.z, e.w};
    const float fs[4] = {f.x, f.y, f.z, f.w};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
#pragma unroll
      for (int c = 0; c < CPT / 2; ++c) {
        if (INIT && i == 0 && k == 0) {
          a[c] = fmul2(ex[0][c], es[0]);
          b[c] = fmul2(ex[0][c], fs[0]);
        } else {
          a[c] = ffma2(ex[i + k][c], es[k], a[c]);
          b[c] = ffma2(ex[i + k][c], fs[k], b[c]);
        }
      }
    }
  }
}

// Sums of four rows for one lane's CPT columns over NC points (NC > 0): row
// q's operations and their order are accum_two_rows' INIT form, so each sum
// has the same bits.
template <int NMAX, int CPT, int NC>
__device__ __forceinline__ void accum_four_rows(const float2 (&ex)[NMAX][CPT / 2], const float* ey,
                                                float2 (&a)[4][CPT / 2]) {
#pragma unroll
  for (int i = 0; i < NC; i += 4) {
    float es[4][4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const float4 e = reinterpret_cast<const float4*>(ey + q * NMAX)[i >> 2];
      es[q][0] = e.x;
      es[q][1] = e.y;
      es[q][2] = e.z;
      es[q][3] = e.w;
    }
#pragma unroll
    for (int k = 0; k < 4; ++k)
#pragma unroll
      for (int c = 0; c < CPT / 2; ++c)
#pragma unroll
        for (int q = 0; q < 4; ++q)
          a[q][c] = i + k == 0 ? fmul2(ex[0][c], es[q][0]) : ffma2(ex[i + k][c], es[q][k], a[q][c]);
  }
}

// Warp-wide maximum of the lanes' argmax keys, published to the frame's
// record by lane 0 (frames without valid points keep key 0).
__device__ __forceinline__ void publish_key(FrameRec* rec, unsigned long long key, bool any_points) {
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long k2 = __shfl_xor_sync(0xffffffffu, key, o);
    key = k2 > key ? k2 : key;
  }
  if ((threadIdx.x & 31) == 0 && any_points && key) atomicMax(&rec->argmax_key, key);
}

// Trip count of the fast row loop for q groups of 4 kept points (1 <= q):
// 4 q, except that above 16 points counts up to 16 take 8 or 16 (fewer
// compiled copies of the loop where they are rare).
__host__ __device__ constexpr int padded_count(int nmax, int q) {
  return 4 * q >= nmax ? nmax : (nmax > 16 && q <= 4 ? (q <= 2 ? 8 : 16) : 4 * q);
}

// Odd widths.  The rows of a frame start at every offset from an alignment
// boundary, and so do the frames of a clip, so the lanes, strips and groups
// that a pixel falls to, and even the kernel that renders it, depend on where
// a launch's planes begin.  What is dropped must not: at an odd width a point
// is dropped from a column of a band (rows of launch_units' bands, which
// depend on the frame's height alone) when its factor in that column is below
// the frame's threshold over its largest row factor in the band, times 1/Z --
// a rule of the pixel, which every kernel applies to the same FP32 values.
// Lists of points and empty strips only leave out what the rule drops
// (kCullMargin), so maps are the same bits however a clip is cut into
// launches and wherever its planes lie.  The quotient is taken once per point
// and the columns compare against it: 64 frames of 853x479, window 12, BF16 in
// 66 us a pass, with products for every column 72.
//
// The threshold is 2^-40 of the largest single contribution to any pixel of
// the frame, which no map maximum lies below: frames whose points all lie far
// outside keep their tiny maxima and argmax pixels.  Below a contribution of
// 2^-80 nothing is dropped (the compared products stay clear of the
// exponential's flush to zero).  Called by a whole warp; lane i < n holds
// point i.
__device__ __forceinline__ float odd_threshold(int n, int width, int height, float inv_n, float uh, float ul, float vh,
                                               float vl, float ch, float cl) {
  float top = 0.0f;
  if ((int)(threadIdx.x & 31) < n) {
    const float xn = fminf(fmaxf(rintf(uh + ul), 0.0f), (float)(width - 1));
    const float yn = fminf(fmaxf(rintf(vh + vl), 0.0f), (float)(height - 1));
    top = gauss_factor(xn, uh, ul, ch, cl) * gauss_factor(yn, vh, vl, ch, cl) * inv_n;
  }
  top = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(top)));
  return top < 0x1p-80f ? 0.0f : kCullBelow * top;
}
// The point's largest row factor in a band of rows by0 .. by0 + brows - 1.
__device__ __forceinline__ float band_row_factor(int by0, int brows, float vh, float vl, float ch, float cl) {
  return gauss_factor(fminf(fmaxf(rintf(vh + vl), (float)by0), (float)(by0 + brows - 1)), vh, vl, ch, cl);
}
// The rule: the least column factor that a point keeps in a band.
__device__ __forceinline__ float least_column(float band_row, float inv_n, float threshold) {
  return threshold > 0.0f ? __fdiv_rn(threshold, band_row * inv_n) : 0.0f;
}
// A list keeps a point whose largest contribution to its columns reaches this
// share of the threshold: the largest factor is taken at the column nearest to
// the point, and the computed ones of other columns exceed it by their
// rounding at most (below 2^-13 for exponents above -121).
constexpr float kCullMargin = 0.5f;

// m divided by the frame's maximum mx, with inv = 1 / mx: the quotient
// corrected by its residual, which with a correctly rounded reciprocal rounds
// it as an IEEE division does (Markstein 1990).  The maximum maps to 1.
__device__ __forceinline__ float corrected_quotient(float m, float mx, float inv) {
  const float q = m * inv;
  return m == mx ? 1.0f : fmaf(fmaf(-q, mx, m), inv, q);
}

// One unit of one frame.  planes point at the frame's first pixel; the
// caller guarantees that element (y0, gx0 - shift) of every plane lies on a
// CPT-element boundary, and so does that column in all the unit's rows.
// Every thread of the CTA must call this (it holds barriers).
//
// Row phases (PH).  At an odd width the rows of a frame start at different
// offsets from a CPT-element boundary, but rows CPT apart start at the same
// one.  A unit then holds every CPT-th row of its band, with its columns
// moved `shift` to the left so that every lane's CPT pixels are aligned again
// and the accesses keep their width; only the lanes across the frame's left
// and right edge work element by element.
struct UnitGeom {
  FrameRec* rec;
  const char* depth;  // frame plane or NULL
  char* M;            // frame plane or NULL
  char* G;            // frame plane or NULL
  int width, height;
  int y0, rows;       // rows of the unit (with PH every CPT-th from y0), within
  int by0, brows;     // the band whose points it keeps
  int gx0;            // first column of the strip group
  int shift;          // row phases: columns start at gx0 - shift (0 <= shift < CPT)
  float d0;
  unsigned int* fault;  // checked builds: reports an access outside the planes (may be NULL)
};

// Checked builds: rows y of columns x .. x + n - 1 lie in the unit's
// planes (else the fault word is set and the caller skips the access).
// Release builds: always true, and the test compiles away.
__device__ __forceinline__ bool in_plane(const UnitGeom& ug, int y, int x, int n) {
  if (!kChecked) return true;
  const bool ok = y >= 0 && y < ug.height && x >= 0 && n >= 0 && x + n <= ug.width;
  if (!ok && ug.fault) atomicExch_system(ug.fault, kFaultOutOfRange);
  return ok;
}

// What a pass over a unit produces.  Full: M, G and the frame's argmax.
// MaxOnly: the argmax alone (no memory traffic), the first pass of
// MF_NORM_MAX.  Scaled: M and G of the map divided by the frame's maximum
// from that first pass -- the same FP32 sums, so the pixel holding the
// maximum becomes exactly 1.
constexpr int kUnitFull = 0;
constexpr int kUnitMaxOnly = 1;
constexpr int kUnitScaled = 2;

template <int NMAX, int CPT, typename TIn, typename TOut, int MODE = kUnitFull, bool PH = false>
__device__ __forceinline__ void map_unit(const UnitGeom& ug, float* Ey, uint4* my_ring,
                                         PointsSmem<kMaxPts>* Pw, const uint4* zeros) {
  constexpr int kInBytes = CPT * (int)sizeof(TIn);
  constexpr int kStrip = 32 * CPT;
  constexpr int S = ring_stages(CPT, (int)sizeof(TIn), NMAX);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int rows = ug.rows, y0 = ug.y0;
  constexpr int step = PH ? CPT : 1;  // rows of the frame per row of the unit
  const int x0 = ug.gx0 - (PH ? ug.shift : 0) + warp * kStrip;
  const int xc = x0 + lane * CPT;
  const bool col_ok = xc < ug.width;
  const bool full = PH ? xc >= 0 && xc + CPT <= ug.width : col_ok;  // all the lane's pixels lie in the frame
  // The lane's pixels inside the frame: columns xc + px0 .. xc + px1 - 1.
  const int px0 = PH ? max(0, -xc) : 0;
  const int px1 = PH ? min(CPT, ug.width - xc) : CPT;
  // Columns in which a point may reach the unit; with row phases those of
  // every shift.
  const int gcull = PH ? max(0, ug.gx0 - (CPT - 1)) : ug.gx0;
  const int gx1 = min(ug.width, ug.gx0 + kGroupStrips * kStrip) - 1;
  const int64_t row0 = (int64_t)y0 * ug.width + xc;
  const char* dsrc = (MODE != kUnitMaxOnly && ug.depth) ? ug.depth + row0 * (int)sizeof(TIn) : nullptr;
  const size_t dstride = (size_t)ug.width * step * sizeof(TIn);
  static_assert((S & (S - 1)) == 0, "ring stages must be a power of two");
  // Depth rows are requested in order, one group per row: rq is the next
  // row to request and dq its source (a running pointer, no per-row
  // multiply).  FAST steps know that dsrc is set; they read the rows of all
  // lanes (kAll) or of full ones only (kFull).
  int rq = 0;
  uintptr_t dq = reinterpret_cast<uintptr_t>(dsrc);
  enum { kAny, kAll, kFull };
  auto issue = [&](int who) {
    if (rq < rows && (who == kAll || (who == kFull ? full : (col_ok && dsrc))) && in_plane(ug, y0 + rq * step, xc + px0, px1 - px0)) {
      char* slot = reinterpret_cast<char*>(my_ring) + ((rq & (S - 1)) * 32 + lane) * kInBytes;
      // Across the left edge the copy starts in the row above (a first row
      // that starts its buffer is aligned, so the bytes are the buffer's);
      // across the right edge it ends with the row.
      if (PH && who == kAny)
        cp_async_part<kInBytes>(slot, reinterpret_cast<const char*>(dq), px1 * (int)sizeof(TIn));
      else
        cp_async<kInBytes>(slot, reinterpret_cast<const char*>(dq));
    }
    cp_async_commit();
    ++rq;
    dq += dstride;
  };
  // The ring is this warp's own and the previous unit drained it.  Every
  // warp culls the points itself into its own copy of the kept list (the
  // same list in every warp), so no warp waits for another before the row
  // factors; the caller's barrier between units (next_unit) ordered every
  // warp's last use of the previous unit's tables before the writes below.
  // The one-CTA-per-SM unit (4 columns per lane above 16 points) keeps one
  // list, culled by warp 0 between two barriers: its register-bound code
  // measured 5 % slower with per-warp lists (HEADING BF16, window 32),
  // where the others gained up to 2 %.
  constexpr bool kOwnList = !(CPT == 4 && NMAX > 16);
  if (!kOwnList) __syncthreads();  // the previous unit is done with P and Ey

  FrameRec* rec = ug.rec;
  const int n = rec->n_valid;
  const float inv_n = rec->inv_n;
  // The lane's pixels of one row: one access, or across a frame edge each
  // pixel inside.
  auto store_lane = [&](char* q, const float (&v)[CPT]) {
    if (!PH || full) {
      Vec<TOut, CPT>::store(q, 0, v);
    } else {
#pragma unroll
      for (int c = 0; c < CPT; ++c)
        if (c >= px0 && c < px1) store_one(reinterpret_cast<TOut*>(q) + c, v[c]);
    }
  };
  // This warp's strip as zeros: its rows (when write_rows; plain CPT-element
  // stores, or with bulk one bulk copy per row and map, which needs 16-byte
  // aligned rows) and its argmax candidate, the strip's first pixel (0).
  auto zero_strip = [&](bool write_rows, bool bulk) {
    if (write_rows && MODE != kUnitMaxOnly) {
      if (bulk) {
        const uint32_t bytes = (uint32_t)(min(kStrip, ug.width - x0) * (int)sizeof(TOut));
        const size_t first = (size_t)y0 * ug.width + x0;
        for (int r = lane; r < rows; r += 32) {
          const size_t at = (first + (size_t)r * ug.width) * sizeof(TOut);
          if (!in_plane(ug, y0 + r, x0, (int)(bytes / sizeof(TOut)))) continue;
          if (ug.M) bulk_copy_s2g(ug.M + at, zeros, bytes);
          if (ug.G) bulk_copy_s2g(ug.G + at, zeros, bytes);
        }
        bulk_commit();
      } else if (col_ok) {
        const float z[CPT] = {};
        const size_t ostride = (size_t)ug.width * step * sizeof(TOut);
        char* qm = ug.M ? ug.M + row0 * (int)sizeof(TOut) : nullptr;
        char* qg = ug.G ? ug.G + row0 * (int)sizeof(TOut) : nullptr;
        int ry = y0;
        for (size_t off = 0, end = (size_t)rows * ostride; off < end; off += ostride, ry += step) {
          if (!in_plane(ug, ry, xc + px0, px1 - px0)) continue;
          if (qm) store_lane(qm + off, z);
          if (qg) store_lane(qg + off, z);
        }
      }
    }
    if (MODE != kUnitScaled)
      publish_key(rec, col_ok ? (unsigned long long)(0xffffffffu - (unsigned)(y0 * ug.width + xc + px0)) : 0ull,
                  n > 0);
  };
  // The max-only pass looks for the frame's maximum and skips strips that
  // cannot hold it.  A lower bound of it: the largest sum of the points'
  // contributions at any point's own pixel (lane i: point i's, moved into
  // the frame).  What bounds the pass is the FP32 pipe, so n^2 factors per
  // warp are cheap against the strip's n x 64 x rows sums.  120 frames of
  // 1280x720, window 16, MF_NORM_MAX: 290 -> 250 us a pass.
  float least = 0.0f;
  if (MODE == kUnitMaxOnly) {
    float ci = 0.f, cj = 0.f, px = 0.f, py = 0.f;
    float uh = 0.f, ul = 0.f, vh = 0.f, vl = 0.f;
    if (lane < n) {
      uh = rec->ux_hi[lane];
      ul = rec->ux_lo[lane];
      vh = rec->vy_hi[lane];
      vl = rec->vy_lo[lane];
      ci = rec->c_hi[lane];
      cj = rec->c_lo[lane];
      px = fminf(fmaxf(rintf(uh + ul), 0.0f), (float)(ug.width - 1));
      py = fminf(fmaxf(rintf(vh + vl), 0.0f), (float)(ug.height - 1));
    }
    for (int k = 0; k < n; ++k) {
      const float kc = __shfl_sync(0xffffffffu, ci, k), kd = __shfl_sync(0xffffffffu, cj, k);
      least += gauss_factor(px, __shfl_sync(0xffffffffu, uh, k), __shfl_sync(0xffffffffu, ul, k), kc, kd) *
               gauss_factor(py, __shfl_sync(0xffffffffu, vh, k), __shfl_sync(0xffffffffu, vl, k), kc, kd);
    }
    least = lane < n ? least * inv_n : 0.0f;
    least = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(least)));
  }
  PointsSmem<kMaxPts>& P = Pw[kOwnList ? warp : 0];
  int nk;  // <= NMAX: n never exceeds the window's bucket
  float min_peak = kCullBelow;
  if (kOwnList || warp == 0) {
    bool keep = false;
    // loaded with the count, not after it: one trip to L2 less on the way to
    // the unit's first row (entries past the count are not used)
    const float uh = rec->ux_hi[lane], ul = rec->ux_lo[lane], vh = rec->vy_hi[lane], vl = rec->vy_lo[lane],
                ch = rec->c_hi[lane], cl = rec->c_lo[lane];
    float peak = 0.f;
    if (lane < n) {
      // the factors peak at the band's pixel nearest (u, v) in these columns
      const float xn = fminf(fmaxf(rintf(uh + ul), (float)gcull), (float)gx1);
      const float yn = fminf(fmaxf(rintf(vh + vl), (float)ug.by0), (float)(ug.by0 + ug.brows - 1));
      peak = gauss_factor(xn, uh, ul, ch, cl) * gauss_factor(yn, vh, vl, ch, cl) * inv_n;
    }
    if (PH) min_peak = odd_threshold(n, ug.width, ug.height, inv_n, uh, ul, vh, vl, ch, cl);
    keep = lane < n && peak >= (PH ? kCullMargin * min_peak : min_peak);
    const unsigned mask = __ballot_sync(0xffffffffu, keep);
    if (keep) {
      const int pos = __popc(mask & ((1u << lane) - 1u));
      P.uhi[pos] = uh;
      P.ulo[pos] = ul;
      P.vhi[pos] = vh;
      P.vlo[pos] = vl;
      P.chi[pos] = ch;
      P.clo[pos] = cl;
    }
    nk = __popc(mask);
    if (!kOwnList && lane == 0) {
      P.kept = nk;
      P.min_peak = min_peak;
    }
    __syncwarp();
  }
  if (!kOwnList) {
    __syncthreads();  // warp 0's list is complete
    nk = P.kept;
    if (PH) min_peak = P.min_peak;
  }
  // Zero rows by bulk copy need 16-byte aligned rows in both map planes.
  const bool bulk = !PH && zeros != nullptr && ((size_t)ug.width * sizeof(TOut)) % 16 == 0 &&
                    ((uintptr_t)ug.M % 16) == 0 && ((uintptr_t)ug.G % 16) == 0;
  if (nk == 0 && (bulk || PH || sizeof(TOut) == 2)) {
    // No point reaches the unit: M = 0 and G = M min(1, d0/D) = 0 on every
    // pixel, whatever the depth holds, and each lane's maximum is that 0 at
    // its first pixel.  The zero rows leave through the bulk-copy engine
    // (one copy per row and map, issued across the CTA), or with 16-bit
    // maps and unaligned rows through plain stores: no depth copies, factor
    // tables or per-row bookkeeping.  (Measured on 1080p ACCEL frames: FP32
    // maps with plain zero stores lose about 1 % against the general loop,
    // so FP32 without bulk copies keeps that loop.)
    if (bulk && MODE != kUnitMaxOnly) {
      const int cols = min(kGroupStrips * kStrip, ug.width - ug.gx0);
      const uint32_t bytes = (uint32_t)(cols * (int)sizeof(TOut));
      const size_t first = (size_t)y0 * ug.width + ug.gx0;
      for (int r = tid; r < rows; r += kUnitThreads) {
        const size_t at = (first + (size_t)r * ug.width) * sizeof(TOut);
        if (!in_plane(ug, y0 + r, ug.gx0, cols)) continue;
        if (ug.M) bulk_copy_s2g(ug.M + at, zeros, bytes);
        if (ug.G) bulk_copy_s2g(ug.G + at, zeros, bytes);
      }
      bulk_commit();
    }
    if (x0 >= ug.width) return;  // warp-uniform: this strip lies past the frame
    zero_strip(!bulk, false);  // with bulk the CTA's copies above wrote the rows
    return;
  }
  // Depth only scales G: with no G output, or no point kept (M = 0, so G = 0
  // whatever D holds), its rows are not read.
  if (nk == 0 || !ug.G) dsrc = nullptr;
  // A warp whose strip none of the kept points reaches (the same 2^-40 rule
  // over the strip's columns and the band's rows) has M = 0 and G = 0 there:
  // it reads no depth and writes zeros.
  bool strip_zero = false, skip_key = false;
  float least_ex = 0.0f;  // row phases, lane i: the least column factor that kept point i keeps
  {
    const int sx0 = PH ? max(0, ug.gx0 + warp * kStrip - (CPT - 1)) : x0;
    const int sx1 = min(ug.width, (PH ? ug.gx0 + warp * kStrip : x0) + kStrip) - 1;
    bool reach = false;
    float most = 0.0f;  // this point's largest contribution to the strip
    if (lane < nk && sx0 <= sx1) {
      const float xn = fminf(fmaxf(rintf(P.uhi[lane] + P.ulo[lane]), (float)sx0), (float)sx1);
      const float band_row = band_row_factor(ug.by0, ug.brows, P.vhi[lane], P.vlo[lane], P.chi[lane], P.clo[lane]);
      const float peak = gauss_factor(xn, P.uhi[lane], P.ulo[lane], P.chi[lane], P.clo[lane]) * band_row;
      most = peak * inv_n;
      if (PH) least_ex = least_column(band_row, inv_n, min_peak);
      reach = most >= (PH ? kCullMargin * min_peak : min_peak);
    }
    strip_zero = __ballot_sync(0xffffffffu, reach) == 0u;
    if (MODE == kUnitMaxOnly) {
      // The strip's sums lie below the sum of its points' largest terms.
      // The margin of 10^-4 covers the roundings of both bounds and of the
      // sums (a few ulp a factor, 32 terms).  The points this unit dropped
      // add below 2^-35 to the lower bound, which also counts them.
      for (int o = 16; o > 0; o >>= 1) most += __shfl_xor_sync(0xffffffffu, most, o);
      const bool skip = x0 >= ug.width || most * 1.0001f < least - 0x1p-34f;
      // no strip left: no barrier to come either (all warps decide alike)
      if (!__syncthreads_or(!skip)) return;
      if (skip) strip_zero = true;
      skip_key = skip;
    }
  }
  if (strip_zero) dsrc = nullptr;
  // the first depth rows are in flight while the factors are computed
  dq = reinterpret_cast<uintptr_t>(dsrc);  // after the strip test (dsrc may have been dropped)
  constexpr int kStep = four_rows(CPT, (int)sizeof(TIn), NMAX) ? 4 : 2;  // rows per step of the row loop
#pragma unroll
  for (int s = 0; s < S - kStep; ++s) issue(kAny);
  const int nc = min(NMAX, (nk + 3) & ~3);
  // Row factors times 1/Z, two rows per entry and NMAX entries per row
  // pair, so that every lane has work also below 32 points: entry k is point
  // k % NMAX of rows 2 (k / NMAX) and 2 (k / NMAX) + 1.
  for (int k = tid; k < ((rows + 1) >> 1) * NMAX; k += kUnitThreads) {
    const int i = k & (NMAX - 1), r = 2 * (k / NMAX);
    float2 g = make_float2(0.0f, 0.0f);  // zeros past the kept points (padded trip counts)
    if (i < nk) {
      const float q0 = (float)(y0 + r * step);
      g = gauss_pair(q0, q0 + (float)step, P.vhi[i], P.vlo[i], P.chi[i], P.clo[i]);
      g.x *= inv_n;
      g.y *= inv_n;
    }
    Ey[r * NMAX + i] = g.x;
    if (r + 1 < rows) Ey[(r + 1) * NMAX + i] = g.y;
  }
  float2 ex[NMAX][CPT / 2];
#pragma unroll
  for (int i = 0; i < NMAX; ++i) {
    const float least_i = PH ? __shfl_sync(0xffffffffu, least_ex, i) : 0.0f;
#pragma unroll
    for (int c = 0; c < CPT / 2; ++c) {
      ex[i][c] = i < nk && col_ok && !strip_zero
                     ? gauss_pair((float)(xc + 2 * c), (float)(xc + 2 * c + 1), P.uhi[i], P.ulo[i], P.chi[i], P.clo[i])
                     : make_float2(0.f, 0.f);
      if (PH) {
        if (ex[i][c].x < least_i) ex[i][c].x = 0.0f;
        if (ex[i][c].y < least_i) ex[i][c].y = 0.0f;
      }
    }
  }
  __syncthreads();  // Ey complete
  if (x0 >= ug.width) return;  // warp-uniform: this strip lies past the frame (no copies issued)
  if (skip_key) return;
  if (strip_zero) {
    zero_strip(true, bulk);
    return;
  }

  // The lane's running maximum and the first row pair that holds it; the
  // pixel is found once per unit after the rows (ties: lower row, then
  // lower column, i.e. the lowest linear index).
  float best = -1.0f;
  int brow = -1;
  char* mrow = (MODE != kUnitMaxOnly && ug.M) ? ug.M + row0 * (int)sizeof(TOut) : nullptr;
  char* grow = (MODE != kUnitMaxOnly && ug.G) ? ug.G + row0 * (int)sizeof(TOut) : nullptr;
  // Scaled pass: divide by the maximum the first pass found (IEEE reciprocal
  // once per unit, then a product; the maximum itself maps to exactly 1)
  float mx = 0.0f, inv = 1.0f;
  bool scale = false;
  if (MODE == kUnitScaled) {
    const unsigned long long key = rec->argmax_key;
    mx = __uint_as_float((unsigned)(key >> 32));
    scale = n > 0 && key != 0ull && mx >= kNormFloor;
    inv = scale ? 1.0f / mx : 1.0f;
  }
  // The quotient by the maximum (the maximum itself becomes exactly 1).
  auto scaled = [&](float m) {
    if (PH) return corrected_quotient(m, mx, inv);
    return m == mx ? 1.0f : m * inv;
  };
  const size_t ostride = (size_t)ug.width * step * sizeof(TOut);
  // Sums of rows r and r+1 (r alone when !two): they start with the first
  // point's product; no kept point (nc = 0) gives zeros.
  auto sums = [&](int r, bool two, float2 (&a)[CPT / 2], float2 (&b)[CPT / 2]) {
    const float* ey0 = Ey + r * NMAX;
    const float* ey1 = Ey + (two ? r + 1 : r) * NMAX;
    if (nc == NMAX) {
      accum_two_rows<NMAX, CPT, NMAX, true>(ex, ey0, ey1, nc, a, b);
    } else if (nc > 0) {
      accum_two_rows<NMAX, CPT, 0, true>(ex, ey0, ey1, nc, a, b);
    } else {
#pragma unroll
      for (int c = 0; c < CPT / 2; ++c) a[c] = b[c] = make_float2(0.f, 0.f);
    }
  };
  // Row phases: pixels outside the frame never hold the maximum.
  auto outside = [&](float2 (&v)[CPT / 2]) {
#pragma unroll
    for (int c = 0; c < CPT; ++c) {
      float& e = (c & 1) ? v[c / 2].y : v[c / 2].x;
      if (c < px0 || c >= px1) e = -1.0f;
    }
  };
  // Rows r and r+1 per step: the ring slots of rows r-2 and r-1 were
  // consumed by the previous step, so rows r+S-2 and r+S-1 can be requested
  // before rows r, r+1 are read.  FAST: depth, M and G all present and an even
  // number of rows (the common case), so a step carries no null or last-row
  // checks; with EDGE it loads and stores for full lanes only, else every
  // lane is full (the test in every access costs a window of 32 3 %).  Other
  // steps do the lanes that are `on`.
  auto rows_loop = [&](auto fast_tag, auto edge_tag, auto nc_tag, int first, int end, bool on) {
    constexpr bool FAST = decltype(fast_tag)::value;
    constexpr bool EDGE = decltype(edge_tag)::value;
    constexpr int NCF = decltype(nc_tag)::value;  // > 0: the sums' trip count (padded)
    size_t off = (size_t)first * ostride;  // output rows advance by a stride: no per-row 64-bit multiply
    for (int r = first; r < end; r += 2, off += 2 * ostride) {
      const bool TWO = FAST || r + 1 < end;
      issue(FAST ? (EDGE ? kFull : kAll) : kAny);
      issue(FAST ? (EDGE ? kFull : kAll) : kAny);
      cp_async_wait<S - kStep>();
      float d0v[CPT], d1v[CPT];
#pragma unroll
      for (int c = 0; c < CPT; ++c) d0v[c] = d1v[c] = 0.0f;
      if (FAST || dsrc) {
        Vec<TIn, CPT>::unpack(ring_row<kInBytes>(my_ring, (r & (S - 1)) * 32 + lane), d0v);
        if (TWO) Vec<TIn, CPT>::unpack(ring_row<kInBytes>(my_ring, ((r + 1) & (S - 1)) * 32 + lane), d1v);
      }
      float2 a[CPT / 2], b[CPT / 2];
      if constexpr (NCF > 0)
        accum_two_rows<NMAX, CPT, NCF, true>(ex, Ey + r * NMAX, Ey + (TWO ? r + 1 : r) * NMAX, NCF, a, b);
      else
        sums(r, TWO, a, b);
      if (!FAST && !on) continue;
      if (MODE != kUnitMaxOnly) {
        const size_t o = off;
        auto emit = [&](const float2 (&acc)[CPT / 2], const float (&dv)[CPT], size_t oo, int ry) {
          float m[CPT];
#pragma unroll
          for (int c = 0; c < CPT / 2; ++c) {
            m[2 * c] = acc[c].x;
            m[2 * c + 1] = acc[c].y;
          }
          if (MODE == kUnitScaled && scale) {
#pragma unroll
            for (int c = 0; c < CPT; ++c) m[c] = scaled(m[c]);
          }
          if (FAST && EDGE && !full) return;
          if (!in_plane(ug, ry, xc + px0, px1 - px0)) return;
          if (FAST)
            Vec<TOut, CPT>::store(mrow + oo, 0, m);
          else if (mrow)
            store_lane(mrow + oo, m);
          if (FAST || grow) {
            float gv[CPT];
            guided<CPT>(m, dv, ug.d0, gv);
            if (FAST)
              Vec<TOut, CPT>::store(grow + oo, 0, gv);
            else
              store_lane(grow + oo, gv);
          }
        };
        emit(a, d0v, o, y0 + r * step);
        if (TWO) emit(b, d1v, o + ostride, y0 + (r + 1) * step);
      }
      if (PH && !FAST) {
        outside(a);
        outside(b);
      }
      if (MODE != kUnitScaled) {
        const float mm = lane_max<CPT>(a, b, TWO);
        if (mm > best) {
          best = mm;
          brow = r;
        }
      }
    }
  };
  // Four rows per step, under FAST's conditions: where two warps share a
  // scheduler (one CTA per SM), a step's depth loads, reciprocals and stores
  // leave the FP32 pipe idle, and four rows have twice the independent sums
  // to fill it and half the steps.  150 frames of 1080p HEADING, window 32,
  // BF16: 515 -> 495 us a pass.
  auto quads_loop = [&](auto edge_tag, auto nc_tag, int end) {
    constexpr bool EDGE = decltype(edge_tag)::value;
    constexpr int NCF = decltype(nc_tag)::value;
    size_t off = 0;
    for (int r = 0; r < end; r += 4, off += 4 * ostride) {
#pragma unroll
      for (int q = 0; q < 4; ++q) issue(EDGE ? kFull : kAll);
      cp_async_wait<S - 4>();
      uint4 raw[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) raw[q] = ring_row<kInBytes>(my_ring, ((r + q) & (S - 1)) * 32 + lane);
      float2 a[4][CPT / 2];
      accum_four_rows<NMAX, CPT, NCF>(ex, Ey + r * NMAX, a);
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        float m[CPT], dv[CPT], gv[CPT];
#pragma unroll
        for (int c = 0; c < CPT / 2; ++c) {
          m[2 * c] = a[q][c].x;
          m[2 * c + 1] = a[q][c].y;
        }
        if (MODE == kUnitScaled && scale) {
#pragma unroll
          for (int c = 0; c < CPT; ++c) m[c] = scaled(m[c]);
        }
        if ((EDGE && !full) || !in_plane(ug, y0 + (r + q) * step, xc, CPT)) continue;
        Vec<TOut, CPT>::store(mrow + off + q * ostride, 0, m);
        Vec<TIn, CPT>::unpack(raw[q], dv);
        guided<CPT>(m, dv, ug.d0, gv);
        Vec<TOut, CPT>::store(grow + off + q * ostride, 0, gv);
      }
      if (MODE != kUnitScaled) {
#pragma unroll
        for (int q = 0; q < 4; q += 2) {
          const float mm = lane_max<CPT>(a[q], a[q + 1], true);
          if (mm > best) {
            best = mm;
            brow = r + q;
          }
        }
      }
    }
  };
  // Row phases, with FAST steps: the pixels of the lanes across the frame's
  // left and right edge, a lane per row; the same sums in the same order.
  // Returns the largest argmax key.  General steps for all of an edge strip's
  // lanes held up its seven neighbours: 120 frames of 853x480, window 12, FP32
  // 145 -> 134 us a pass, BF16 130 -> 92; of 854x480, window 28, FP32 (the
  // last strip's absent lanes) 184 -> 163.
  auto edge_pixels = [&]() {
    unsigned long long top = 0ull;
    const int wide = ug.width - x0;
    for (int side = 0; side < 2; ++side) {
      const int L = side == 0 ? 0 : wide / CPT;                  // the lane, and its pixels first .. last - 1
      const int first = side == 0 && x0 < 0 ? -x0 : 0;
      const int last = side == 0 ? (x0 < 0 ? min(CPT, wide) : 0) : (wide < kStrip && (L > 0 || x0 >= 0) ? wide % CPT : 0);
#pragma unroll
      for (int c = 0; c < CPT; ++c) {
        if (c < first || c >= last) continue;                    // warp-uniform
        const int x = x0 + L * CPT + c;
        for (int r0 = 0; r0 < rows; r0 += 32) {
          const int r = min(r0 + lane, rows - 1);
          const int y = y0 + r * step;
          const bool mine = r0 + lane < rows && in_plane(ug, y, x, 1);
          const int64_t at = (int64_t)y * ug.width + x;
          const float D = mine ? to_f32(reinterpret_cast<const TIn*>(ug.depth)[at]) : 0.0f;
          float m = 0.0f;
#pragma unroll
          for (int i = 0; i < NMAX; ++i) {
            const float e = __shfl_sync(0xffffffffu, (c & 1) ? ex[i][c / 2].y : ex[i][c / 2].x, L);
            m = i == 0 ? e * Ey[r * NMAX] : fmaf(e, Ey[r * NMAX + i], m);
          }
          if (!mine) continue;
          const unsigned long long key =
              ((unsigned long long)__float_as_uint(m) << 32) | (0xffffffffu - (unsigned)(y * ug.width + x));
          top = key > top ? key : top;
          if (MODE == kUnitScaled && scale) m = scaled(m);
          store_one(reinterpret_cast<TOut*>(ug.M) + at, m);
          store_one(reinterpret_cast<TOut*>(ug.G) + at, m * depth_weight(D, ug.d0));
        }
      }
    }
    return top;
  };
  unsigned long long edge_key = 0ull;
  // FAST steps run the sums with a trip count fixed at compile time: the kept
  // count rounded up to a multiple of 4, and above 16 points of 8 when at
  // most 16 are kept.  The table and column factors past the kept points
  // are zeros, and a zero term leaves a sum of non-negative terms unchanged,
  // so the padded sums have the same bits.
  // (the rows left over by steps of four, and the odd last row that half of
  // the row phases' units have, follow the FAST steps, which read the depth of
  // full lanes only; other units take one loop for all rows)
  const int even = kStep == 4 ? rows & ~3 : (PH ? rows & ~1 : rows);
  if (dsrc && mrow && grow && (even & 1) == 0 && nc > 0) {
    auto fast = [&](auto edge_tag, auto nc_tag) {
      if constexpr (kStep == 4)
        quads_loop(edge_tag, nc_tag, even);
      else
        rows_loop(std::true_type{}, edge_tag, nc_tag, 0, even, full);
    };
    using std::integral_constant;
    const bool inside = (!PH || x0 >= 0) && x0 + kStrip <= ug.width;  // warp-uniform: every lane is full
    if (!inside) {  // one or two strips of a frame: fewer copies of the loop
      if (2 * nc <= NMAX)
        fast(std::true_type{}, integral_constant<int, NMAX / 2>{});
      else
        fast(std::true_type{}, integral_constant<int, NMAX>{});
    } else {
      const std::false_type all{};
      switch (nc >> 2) {  // 1 .. NMAX / 4
        case 1: fast(all, integral_constant<int, padded_count(NMAX, 1)>{}); break;
        case 2: fast(all, integral_constant<int, padded_count(NMAX, 2)>{}); break;
        case 3: fast(all, integral_constant<int, padded_count(NMAX, 3)>{}); break;
        case 4: fast(all, integral_constant<int, padded_count(NMAX, 4)>{}); break;
        case 5: fast(all, integral_constant<int, padded_count(NMAX, 5)>{}); break;
        case 6: fast(all, integral_constant<int, padded_count(NMAX, 6)>{}); break;
        case 7: fast(all, integral_constant<int, padded_count(NMAX, 7)>{}); break;
        default: fast(all, integral_constant<int, NMAX>{}); break;
      }
    }
    if (!inside && !full) best = -1.0f;  // its sums are of pixels outside the frame, or edge_pixels' to count
    if (PH && !inside) edge_key = edge_pixels();
    if ((PH || kStep == 4) && even < rows)
      rows_loop(std::false_type{}, std::false_type{}, std::integral_constant<int, 0>{}, even, rows, full);
  } else {
    rows_loop(std::false_type{}, std::false_type{}, std::integral_constant<int, 0>{}, 0, rows, col_ok);
  }
  cp_async_wait<0>();
  if (MODE != kUnitScaled) {
    unsigned long long key = 0ull;
    if (best >= 0.0f) {
      // the winning row pair again, with the same sums in the same order
      const bool two = brow + 1 < rows;
      float2 a[CPT / 2], b[CPT / 2];
      sums(brow, two, a, b);
      if (PH) {
        outside(a);
        outside(b);
      }
      float ma = fmaxf(a[0].x, a[0].y);
#pragma unroll
      for (int c = 1; c < CPT / 2; ++c) ma = fmax3(ma, a[c].x, a[c].y);
      const bool first = ma == best;
      float m[CPT];
#pragma unroll
      for (int c = 0; c < CPT / 2; ++c) {
        m[2 * c] = first ? a[c].x : b[c].x;
        m[2 * c + 1] = first ? a[c].y : b[c].y;
      }
      unsigned off = CPT - 1;
#pragma unroll
      for (int c = CPT - 2; c >= 0; --c)
        if (m[c] == best) off = c;
      const unsigned bidx = (unsigned)((y0 + (brow + (first ? 0 : 1)) * step) * ug.width + xc) + off;
      key = ((unsigned long long)__float_as_uint(best) << 32) | (0xffffffffu - bidx);
    }
    if (PH) key = key > edge_key ? key : edge_key;
    publish_key(rec, key, n > 0);
  }
}

// Dynamic shared memory of a CTA running units of bucket NMAX with CPT
// pixels per lane and in_bytes-byte depth: the band's row factors, then
// every warp's depth ring.
__host__ __device__ constexpr size_t row_factor_bytes(int nmax, int band_h) { return (size_t)band_h * nmax * 4; }
__host__ __device__ constexpr size_t unit_smem_bytes(int nmax, int band_h, int cpt, int in_bytes) {
  return row_factor_bytes(nmax, band_h) +
         (size_t)kGroupStrips * ring_stages(cpt, in_bytes, nmax) * 32 * cpt * in_bytes;
}

// Dynamic unit schedule of the persistent map kernels.  CTA c starts on
// unit c.  While the CTA works on a unit, its thread 0 holds a claim on the
// next one from a launch-wide counter (claims at or past the last unit end
// the CTA's loop), so CTAs that draw cheap units -- ones no point reaches --
// take more of them instead of idling at the end of the launch.  Every unit
// processed makes one claim, so a launch makes exactly `units` of them and
// the claim that returns units - 1 is its last: that thread puts the counter
// back to 0 for the next launch.  The counter must be 0 at launch, and no
// two launches in flight may share it; a launch holds fewer than 2^32 units.
__device__ __forceinline__ unsigned claim_unit(unsigned* ctr) {
  return threadIdx.x == 0 ? atomicAdd(ctr, 1u) : 0u;
}

// Called by every thread after the CTA's k-th unit with thread 0's claim:
// the CTA's next unit.  s_next is two shared slots, so a slow thread
// still reading slot k & 1 never sees the write of claim k + 1.
__device__ __forceinline__ long long next_unit(unsigned* ctr, unsigned claim, long long units,
                                               long long* s_next, int k) {
  if (threadIdx.x == 0) {
    s_next[k & 1] = (long long)gridDim.x + (long long)claim;
    if ((long long)claim == units - 1) *ctr = 0u;  // the launch's last claim
  }
  __syncthreads();
  return s_next[k & 1];
}

}  // namespace mf
