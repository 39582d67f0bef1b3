// Device helpers shared by the kernels: gradient element traits, 128-bit loads/stores and the
// parameter update of Algorithm 1 line 9.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "adapm_internal.h"

namespace adapm {

__device__ __forceinline__ float bf16_bits_to_float(uint32_t b) { return __uint_as_float(b << 16); }

// bf16 gradients: 8 elements = one 16-byte load, kept packed in registers
struct GradBF16 {
  using elem = uint16_t;
  using raw8 = uint4;
  static __device__ __forceinline__ raw8 load8(const elem* p) { return __ldg(reinterpret_cast<const uint4*>(p)); }
  static __device__ __forceinline__ raw8 load8_guarded(const elem* p, int n) {
    uint32_t h[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) h[i] = (i < n) ? (uint32_t)p[i] : 0u;
    return make_uint4(h[0] | (h[1] << 16), h[2] | (h[3] << 16), h[4] | (h[5] << 16), h[6] | (h[7] << 16));
  }
  static __device__ __forceinline__ void unpack(const raw8& r, float* f) {
    f[0] = __uint_as_float(r.x << 16); f[1] = __uint_as_float(r.x & 0xffff0000u);
    f[2] = __uint_as_float(r.y << 16); f[3] = __uint_as_float(r.y & 0xffff0000u);
    f[4] = __uint_as_float(r.z << 16); f[5] = __uint_as_float(r.z & 0xffff0000u);
    f[6] = __uint_as_float(r.w << 16); f[7] = __uint_as_float(r.w & 0xffff0000u);
  }
  static __device__ __forceinline__ float load1(const elem* p) { return bf16_bits_to_float(*p); }
};

struct F32x8 { float4 a, b; };

struct GradF32 {
  using elem = float;
  using raw8 = F32x8;
  static __device__ __forceinline__ raw8 load8(const elem* p) {
    raw8 r;
    r.a = __ldg(reinterpret_cast<const float4*>(p));
    r.b = __ldg(reinterpret_cast<const float4*>(p) + 1);
    return r;
  }
  static __device__ __forceinline__ raw8 load8_guarded(const elem* p, int n) {
    float h[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) h[i] = (i < n) ? p[i] : 0.f;
    raw8 r;
    r.a = make_float4(h[0], h[1], h[2], h[3]);
    r.b = make_float4(h[4], h[5], h[6], h[7]);
    return r;
  }
  static __device__ __forceinline__ void unpack(const raw8& r, float* f) {
    f[0] = r.a.x; f[1] = r.a.y; f[2] = r.a.z; f[3] = r.a.w;
    f[4] = r.b.x; f[5] = r.b.y; f[6] = r.b.z; f[7] = r.b.w;
  }
  static __device__ __forceinline__ float load1(const elem* p) { return *p; }
};

__device__ __forceinline__ void load8f(const float* p, float* f) {
  const float4 a = *reinterpret_cast<const float4*>(p);
  const float4 b = *(reinterpret_cast<const float4*>(p) + 1);
  f[0] = a.x; f[1] = a.y; f[2] = a.z; f[3] = a.w;
  f[4] = b.x; f[5] = b.y; f[6] = b.z; f[7] = b.w;
}

__device__ __forceinline__ void store8f(float* p, const float* f) {
  *reinterpret_cast<float4*>(p) = make_float4(f[0], f[1], f[2], f[3]);
  *(reinterpret_cast<float4*>(p) + 1) = make_float4(f[4], f[5], f[6], f[7]);
}

// two floats -> packed bf16 pair, round to nearest even (x0 in the low half)
__device__ __forceinline__ uint32_t pack_bf16x2(float x0, float x1) {
  uint32_t d;
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(x1), "f"(x0));
  return d;
}

// Algorithm 1 line 9: W - lr s_b ( clamp(m^c / (sqrt(v) + eps)) + lambda_b W ).
// Comparisons (not fminf/fmaxf) so that a NaN ratio stays NaN.
__device__ __forceinline__ float adapm_param_update(float w, float mc, float v, const StepScalars& sc, float lr_s,
                                                    float wd) {
  const float den = sqrtf(v * sc.inv_bc2) + sc.eps;
  float ratio = (mc * sc.inv_bc1) / den;
  ratio = ratio > sc.clip ? sc.clip : (ratio < -sc.clip ? -sc.clip : ratio);
  return w - lr_s * (ratio + wd * w);
}

// x limited to [-c, c]; a NaN stays NaN.
__device__ __forceinline__ float clamp_keep_nan(float x, float c) {
  float y;
  asm("{\n.reg .f32 t;\nmin.NaN.f32 t, %1, %2;\nmax.NaN.f32 %0, t, %3;\n}" : "=f"(y) : "f"(x), "f"(c), "f"(-c));
  return y;
}

// The same with the values it needs by themselves, for the rare elements of the function below (out of line: its root and
// quotient would be unrolled with that one's loops, and a loop of its own would keep the values in local memory).
static __device__ __noinline__ float adapm_param_update_rare(float w, float mc, float v, float inv_bc1, float inv_bc2, float eps,
                                                             float clip, float lr_s, float wd) {
  float ratio = (mc * inv_bc1) / (sqrtf(v * inv_bc2) + eps);
  ratio = ratio > clip ? clip : (ratio < -clip ? -clip : ratio);
  return w - lr_s * (ratio + wd * w);
}

// The update of N elements with a second moment of their own.  The root and the quotient start from the hardware's
// approximations (an ulp or two off) and take one step of Newton's iteration each, with the residual in a fused
// multiply-add (Markstein, IBM J. Res. Dev. 34, 1990): s += (v - s^2) y / 2 with y ~ 1/sqrt(v), q += (m - q d) r with
// r ~ 1/d.  Half the instructions of sqrtf and the division and no branch per element: the step of the 1.5B shapes with a
// per-element v takes 15.6 ms with it and 16.3 with the functions, the 350M set at rank 128 4.8 and 5.0 ms.
// Compared with sqrtf and / on 2^26 pairs each of v in [1e-14, 1e-3] and in [1e-28, 1e28]: the same largest and the same
// rms error against 64 bits, the root the nearest float every time.
// What lies outside the range where the iteration holds takes the functions themselves: zero and near-zero v, NaN, and
// what could overflow on the way.  With |m^c| <= 1e14, a bias correction of at most 1e6 and d >= 1e-15 neither q nor
// q d - m leaves the range of a float, and only quotients below 1e-20 lose bits of the residual to underflow.
template <int N>
__device__ __forceinline__ void adapm_param_update_n(float* w, const float* mc, const float* v, const StepScalars& sc,
                                                     float lr_s, float wd) {
  float vs[N], lo = 1.f, hi = 1.f;
#pragma unroll
  for (int e = 0; e < N; ++e) {
    vs[e] = v[e] * sc.inv_bc2;
    lo = fminf(lo, vs[e]);
    hi = fmaxf(hi, vs[e]);
  }
  bool usual = lo >= 1e-30f && hi <= 1e30f && sc.eps <= 1e30f && sc.inv_bc1 <= 1e6f;
#pragma unroll
  for (int e = 0; e < N; ++e) usual = usual && fabsf(mc[e]) <= 1e14f && vs[e] == vs[e];      // (false for a NaN)
  if (usual) {
#pragma unroll
    for (int e = 0; e < N; ++e) {
      const float y = rsqrtf(vs[e]);
      float s = vs[e] * y;
      s = fmaf(fmaf(-s, s, vs[e]), 0.5f * y, s);
      const float d = s + sc.eps, r = __fdividef(1.f, d), m = mc[e] * sc.inv_bc1;
      float q = m * r;
      q = fmaf(fmaf(-q, d, m), r, q);
      w[e] = w[e] - lr_s * (clamp_keep_nan(q, sc.clip) + wd * w[e]);
    }
  } else {
#pragma unroll
    for (int e = 0; e < N; ++e)
      w[e] = adapm_param_update_rare(w[e], mc[e], v[e], sc.inv_bc1, sc.inv_bc2, sc.eps, sc.clip, lr_s, wd);
  }
}

}  // namespace adapm
