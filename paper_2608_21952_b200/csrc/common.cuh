// Shared device helpers of the SSDi8 kernels: the binary32 building blocks that
// decide integer codes (never contracted, never approximated) and small utilities.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/ssdi8.h"

namespace ssdi8 {

typedef long long i64;

// round half to even, saturate to [-127, 127] (Eq. 1: 2^(b-1)-1 levels per side)
__device__ __forceinline__ int rne_clamp(float v) {
  float r = rintf(v);
  r = fmaxf(r, -127.0f);  // fmaxf(NaN, a) = a
  r = fminf(r, 127.0f);
  return __float2int_rn(r);
}

// binary32 exponential with a fixed operation sequence (see ssdi8.h): Cody-Waite
// reduction by ln 2, degree-7 Taylor polynomial (Horner, fmaf), scaling by 2^n
// through the exponent field.  0 below -80, argument clamped at +80.
// (The zero below -80 is a selection at the end: the arithmetic in front of it is harmless there.)
__device__ __forceinline__ float exp32(float x0) {
  const float x = fminf(x0, 80.0f);
  const float LOG2E = __uint_as_float(0x3FB8AA3Bu);
  const float LN2_HI = __uint_as_float(0x3F317200u);
  const float LN2_LO = __uint_as_float(0x35BFBE8Eu);
  // n = rint(fmul(x, LOG2E)): |x LOG2E| < 2^22, so adding and subtracting 1.5 * 2^23 rounds to the nearest
  // integer, ties to even, exactly as rint does, and leaves n in the low mantissa bits of the sum (both
  // conversions stay off the conversion pipe)
  const float nm = __fadd_rn(__fmul_rn(x, LOG2E), 12582912.0f);
  const float n = __fadd_rn(nm, -12582912.0f);
  float r = __fmaf_rn(n, -LN2_HI, x);
  r = __fmaf_rn(n, -LN2_LO, r);
  float p = __uint_as_float(0x39500D01u);                 // 1/5040
  p = __fmaf_rn(p, r, __uint_as_float(0x3AB60B61u));      // 1/720
  p = __fmaf_rn(p, r, __uint_as_float(0x3C088889u));      // 1/120
  p = __fmaf_rn(p, r, __uint_as_float(0x3D2AAAABu));      // 1/24
  p = __fmaf_rn(p, r, __uint_as_float(0x3E2AAAABu));      // 1/6
  p = __fmaf_rn(p, r, 0.5f);
  p = __fmaf_rn(p, r, 1.0f);
  p = __fmaf_rn(p, r, 1.0f);
  const float e = __uint_as_float(__float_as_uint(p) + (__float_as_uint(nm) << 23));   // bits(nm) = 0x4B400000 + n: the shift keeps n
  return x0 >= -80.0f ? e : 0.0f;
}
// two at once, the same operations in packed form
__device__ __forceinline__ float2 exp32x2(float x0, float x1) {
  auto both = [](uint32_t bits) { return make_float2(__uint_as_float(bits), __uint_as_float(bits)); };
  const float2 x = make_float2(fminf(x0, 80.0f), fminf(x1, 80.0f));
  // (a multiply and an add that stay two operations: the packed pair would be contracted into one)
  const float2 nm = make_float2(__fadd_rn(__fmul_rn(x.x, __uint_as_float(0x3FB8AA3Bu)), 12582912.0f),
                                __fadd_rn(__fmul_rn(x.y, __uint_as_float(0x3FB8AA3Bu)), 12582912.0f));
  const float2 n = __fadd2_rn(nm, make_float2(-12582912.0f, -12582912.0f));
  float2 r = __ffma2_rn(n, both(0xBF317200u), x);
  r = __ffma2_rn(n, both(0xB5BFBE8Eu), r);
  float2 p = both(0x39500D01u);
  p = __ffma2_rn(p, r, both(0x3AB60B61u));
  p = __ffma2_rn(p, r, both(0x3C088889u));
  p = __ffma2_rn(p, r, both(0x3D2AAAABu));
  p = __ffma2_rn(p, r, both(0x3E2AAAABu));
  p = __ffma2_rn(p, r, make_float2(0.5f, 0.5f));
  p = __ffma2_rn(p, r, make_float2(1.0f, 1.0f));
  p = __ffma2_rn(p, r, make_float2(1.0f, 1.0f));
  const float e0 = __uint_as_float(__float_as_uint(p.x) + (__float_as_uint(nm.x) << 23));
  const float e1 = __uint_as_float(__float_as_uint(p.y) + (__float_as_uint(nm.y) << 23));
  return make_float2(x0 >= -80.0f ? e0 : 0.0f, x1 >= -80.0f ? e1 : 0.0f);
}

// ---- conversions that stay off the quarter-rate conversion pipe (all exact)
constexpr float kMagicIn = 12583040.0f;   // 1.5 * 2^23 + 128
constexpr float kMagicOut = 12582912.0f;  // 1.5 * 2^23
// int8 byte k of w_xor (= word ^ 0x80808080) as a float: the byte + 128 is placed in the mantissa
// of 1.5 * 2^23 and the offset subtracted
__device__ __forceinline__ float s8_to_f32(uint32_t w_xor, int k) {
  return __fadd_rn(__uint_as_float(__byte_perm(w_xor, 0x4B400000u, 0x7650u + k)), -kMagicIn);
}
// int32 with |v| < 2^22 as a float
__device__ __forceinline__ float i22_to_f32(int v) {
  return __fadd_rn(__int_as_float(v + 0x4B400000), -kMagicOut);
}
// bits whose low byte is the int8 code rne(v) saturated to [-127, 127]: clamping before rounding
// equals rounding before clamping, and (v + 1.5 * 2^23) rounds to nearest even.  The clamp is one
// instruction: min(|v|, 127) with the sign of v put back.  (Used on products of finite factors; a NaN
// would give +-127.)
__device__ __forceinline__ uint32_t rne_clamp_bits(float v) {
  float c;
  asm("min.xorsign.abs.f32 %0, %1, %2;" : "=f"(c) : "f"(v), "f"(127.0f));
  return __float_as_uint(__fadd_rn(c, kMagicOut));
}
// the same for a pair (the magic addition as one packed instruction)
__device__ __forceinline__ uint2 rne_clamp_bits2(float2 v) {
  float2 c;
  asm("min.xorsign.abs.f32 %0, %1, %2;" : "=f"(c.x) : "f"(v.x), "f"(127.0f));
  asm("min.xorsign.abs.f32 %0, %1, %2;" : "=f"(c.y) : "f"(v.y), "f"(127.0f));
  const float2 r = __fadd2_rn(c, make_float2(kMagicOut, kMagicOut));
  return make_uint2(__float_as_uint(r.x), __float_as_uint(r.y));
}
__device__ __forceinline__ uint32_t pack4_bits(uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
  return __byte_perm(__byte_perm(a, b, 0x0040u), __byte_perm(c, d, 0x0040u), 0x5410u);
}

// Eq. 1 codes, rne(fdiv_rn(v, alpha)) saturated, four as one word, without a division and without a branch: with y =
// frcp_rn(alpha), q = fmul(v, y) is within two units in the last place of v / alpha, its residual fmaf(-q, alpha, v) is
// exact, and fmaf(residual, y, q) is the quotient up to 2^-22 unit before it is rounded (Markstein's scheme, IBM J. Res.
// Dev. 34, 1990).  It can differ from fdiv_rn only where v / alpha lies that close to the midpoint of two binary32
// numbers, and the code then only where one of the two is k + 1/2: an equation M A - V 2^s = j with M that midpoint's
// 25 bits, A and V the significands and |j| < 8, which has one A for each (k, j, s).  All its solutions up to |j| =
// 200 round as the division does (35 696 pairs; the nearest are in the tests).  |v| is limited to 127.25 alpha first,
// so the code saturates by itself and nothing overflows; quotients below 1/2, whose residuals may underflow, round to 0
// either way.  Step sizes outside [1e-30, 1e30] (`usable` false) take the divisions.
// (Products with y and a division where one came close to a rounding boundary cost 56 instructions per 128 codes, and
// 16-bit inputs under a step size of absmax / 127 are ties in one code of 500, so that a quarter of the warps divided.
// Entry quantiser, bf16, 8960 x 5376: 33.5 -> 22.0 us (6.6 TB/s); 16384 x 5376: 58.9 -> 45.0 us.  A second correction
// step, which needs no such enumeration, with a loop that waited for `usable`: 35.3 and 64.5 us.)
struct Step4 {
  float2 y01, y23, n01, n23;   // reciprocals and negatives of four step sizes
  float4 lim;                  // 127.25 of them
  bool usable;
};
__device__ __forceinline__ Step4 step4(const float4& a) {
  auto normal = [](float x) { return x >= 1e-30f && x <= 1e30f; };
  Step4 s;
  s.y01 = make_float2(__frcp_rn(a.x), __frcp_rn(a.y));
  s.y23 = make_float2(__frcp_rn(a.z), __frcp_rn(a.w));
  s.n01 = make_float2(-a.x, -a.y);
  s.n23 = make_float2(-a.z, -a.w);
  s.lim = make_float4(__fmul_rn(a.x, 127.25f), __fmul_rn(a.y, 127.25f), __fmul_rn(a.z, 127.25f), __fmul_rn(a.w, 127.25f));
  s.usable = normal(a.x) && normal(a.y) && normal(a.z) && normal(a.w);
  return s;
}
__device__ __forceinline__ uint32_t code4(const float4& v, const Step4& s) {
  // v - 0 is v, and a NaN of either sign becomes the positive one that a division gives: its code is +127.  (The zero as a
  // product that the compiler cannot know: the step size might not be finite.)
  const float2 z = make_float2(0.f, 0.f);
  float2 v01 = __ffma2_rn(s.n01, z, make_float2(v.x, v.y)), v23 = __ffma2_rn(s.n23, z, make_float2(v.z, v.w));
  // min(|v|, lim) with the sign of v
  asm("min.xorsign.abs.f32 %0, %1, %2;" : "=f"(v01.x) : "f"(v01.x), "f"(s.lim.x));
  asm("min.xorsign.abs.f32 %0, %1, %2;" : "=f"(v01.y) : "f"(v01.y), "f"(s.lim.y));
  asm("min.xorsign.abs.f32 %0, %1, %2;" : "=f"(v23.x) : "f"(v23.x), "f"(s.lim.z));
  asm("min.xorsign.abs.f32 %0, %1, %2;" : "=f"(v23.y) : "f"(v23.y), "f"(s.lim.w));
  float2 q01 = __fmul2_rn(v01, s.y01), q23 = __fmul2_rn(v23, s.y23);
  q01 = __ffma2_rn(__ffma2_rn(q01, s.n01, v01), s.y01, q01);
  q23 = __ffma2_rn(__ffma2_rn(q23, s.n23, v23), s.y23, q23);
  const float2 mg = make_float2(kMagicOut, kMagicOut);
  const float2 m01 = __fadd2_rn(q01, mg), m23 = __fadd2_rn(q23, mg);
  return pack4_bits(__float_as_uint(m01.x), __float_as_uint(m01.y), __float_as_uint(m23.x), __float_as_uint(m23.y));
}
__device__ __forceinline__ uint32_t code4_by_division(const float4& v, const float4& a) {
  return pack4_bits(rne_clamp_bits(__fdiv_rn(v.x, a.x)), rne_clamp_bits(__fdiv_rn(v.y, a.y)),
                    rne_clamp_bits(__fdiv_rn(v.z, a.z)), rne_clamp_bits(__fdiv_rn(v.w, a.w)));
}

__device__ __forceinline__ uint32_t pack4(int a, int b, int c, int d) {
  return (uint32_t)(a & 0xff) | ((uint32_t)(b & 0xff) << 8) | ((uint32_t)(c & 0xff) << 16) |
         ((uint32_t)(d & 0xff) << 24);
}

__device__ __forceinline__ int sx8(uint32_t w, int k) { return (int)(int8_t)((w >> (8 * k)) & 0xff); }

// softplus of the raw time step (Algorithm 2 module 1) in binary64, every operation a single correctly
// rounded add, multiply, divide or fused multiply-add in the order written in ssdi8.h, so that the
// binary32 result is defined bit for bit: v = (double)fadd(dt_raw, bias); u = exp(-|v|) by Cody-Waite
// reduction and a degree-13 Taylor polynomial; log(1 + u) = 2 atanh(u / (2 + u)) by its odd series up
// to the 27th power; dt = (float)(max(v, 0) + log(1 + u)).
// W values side by side, step by step: each binary64 operation waits for the one before it, and a coefficient is two moves (one
// value after the other takes 120 instructions each, 43 of them binary64; prefill of 256 tokens x 24 heads 23.85 us, two side by
// side 23.25, four 22.7, all eight of a lane 22.55; 5 x 1792 x 80 122.9 and 121.7).
template <int W>
__device__ __forceinline__ void softplus_dt(const float* dt_raw, float bias, float* dt) {
  const double LOG2E = 0x1.71547652b82fep+0, LN2_HI = 0x1.62e42fee00000p-1, LN2_LO = 0x1.a39ef35793c76p-33;
  const double kExp[14] = {1.0 / 6227020800.0, 1.0 / 479001600.0, 1.0 / 39916800.0, 1.0 / 3628800.0, 1.0 / 362880.0,
                           1.0 / 40320.0,      1.0 / 5040.0,      1.0 / 720.0,      1.0 / 120.0,     1.0 / 24.0,
                           1.0 / 6.0,          0.5,               1.0,              1.0};
  double v[W], r[W], p[W], s[W];
  int n[W];
#pragma unroll
  for (int i = 0; i < W; ++i) {
    v[i] = (double)__fadd_rn(dt_raw[i], bias);
    const double a = fabs(v[i]) <= 700.0 ? fabs(v[i]) : 0.0;   // (beyond, u is 0: below)
    const double nd = rint(__dmul_rn(-a, LOG2E));
    n[i] = __double2int_rn(nd);
    r[i] = __fma_rn(nd, -LN2_HI, -a);
    r[i] = __fma_rn(nd, -LN2_LO, r[i]);
    p[i] = kExp[0];
  }
#pragma unroll
  for (int k = 1; k < 14; ++k) {
#pragma unroll
    for (int i = 0; i < W; ++i) p[i] = __fma_rn(p[i], r[i], kExp[k]);
  }
#pragma unroll
  for (int i = 0; i < W; ++i) {
    const double e = __longlong_as_double(__double_as_longlong(p[i]) + ((long long)n[i] << 52));
    const double u = fabs(v[i]) <= 700.0 ? e : 0.0;
    s[i] = __ddiv_rn(u, __dadd_rn(2.0, u));
    r[i] = __dmul_rn(s[i], s[i]);
    p[i] = 1.0 / 27.0;
  }
#pragma unroll
  for (int k = 12; k >= 0; --k) {
#pragma unroll
    for (int i = 0; i < W; ++i) p[i] = __fma_rn(p[i], r[i], 1.0 / (double)(2 * k + 1));
  }
#pragma unroll
  for (int i = 0; i < W; ++i) {
    const double lp = __dmul_rn(__dmul_rn(2.0, s[i]), p[i]);
    dt[i] = (float)__dadd_rn(v[i] > 0.0 ? v[i] : 0.0, lp);
  }
}
__device__ __forceinline__ float softplus_dt(float dt_raw, float bias) {
  float dt;
  softplus_dt<1>(&dt_raw, bias, &dt);
  return dt;
}

// step size of a channel from the bits of its largest magnitude (Eq. 1; an all-zero channel gets 1)
__device__ __forceinline__ float step_of_max(uint32_t bits) { return bits == 0u ? 1.0f : __fdiv_rn(__uint_as_float(bits), 127.0f); }

// Programmatic dependent launch.  Every kernel of the layer lets its successor in the stream be
// scheduled early (launch_dependents at its start) and itself waits for its predecessor's completion
// and memory flush (pdl_wait) before its first access to global memory, so only work that touches no
// global memory (barrier and tensor-memory set-up, descriptor prefetch) runs under the predecessor's
// tail.  Both are no-ops in a kernel that was launched without the attribute.
// A store whose line is to stay in L2 ahead of ordinary ones (for data a later kernel of the same layer reads
// after other kernels have streamed more than an L2 of traffic in between).
__device__ __forceinline__ uint64_t l2_policy_evict_last() {
  uint64_t pol;
  asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(pol));
  return pol;
}
__device__ __forceinline__ void st_global_hint(float* a, float2 v, uint64_t pol) {
  asm volatile("st.global.L2::cache_hint.v2.f32 [%0], {%1, %2}, %3;" ::"l"(a), "f"(v.x), "f"(v.y), "l"(pol) : "memory");
}
__device__ __forceinline__ void st_global_hint(float* a, float4 v, uint64_t pol) {
  asm volatile("st.global.L2::cache_hint.v4.f32 [%0], {%1, %2, %3, %4}, %5;"
               ::"l"(a), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w), "l"(pol)
               : "memory");
}

__device__ __forceinline__ void pdl_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Barrier of a cluster's CTAs in two halves.  Not the .aligned form, which needs a warp whose lanes are together: the loops and the branches
// on the lane ahead of it do not promise that.  All threads of all CTAs arrive, also where a wait has given up; no bound of its own.
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait;" ::: "memory"); }
__device__ __forceinline__ void cluster_sync() {
  cluster_arrive();
  cluster_wait();
}

struct Dims {
  int b, L, H, P, N, G, Q, c;
};

inline Dims make_dims(const ssdi8_dims_t* d) {
  Dims r;
  r.b = d->batch; r.L = d->seqlen; r.H = d->nheads; r.P = d->headdim; r.N = d->dstate;
  r.G = d->ngroups; r.Q = d->chunk; r.c = d->chunk > 0 ? d->seqlen / d->chunk : 0;
  return r;
}

#define SSDI8_CUDA_CHECK(expr)                         \
  do {                                                 \
    cudaError_t e__ = (expr);                          \
    if (e__ != cudaSuccess) return SSDI8_ERR_CUDA;     \
  } while (0)

#define SSDI8_LAUNCH_CHECK()                                       \
  do {                                                             \
    if (cudaPeekAtLastError() != cudaSuccess) {                    \
      (void)cudaGetLastError();                                    \
      return SSDI8_ERR_CUDA;                                       \
    }                                                              \
  } while (0)

}  // namespace ssdi8
