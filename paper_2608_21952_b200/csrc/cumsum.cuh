// The work of a block of ChunkCumsum (see cumsum.cu, which describes it): the rows of the scalar pack of one chunk for as many
// neighbouring heads as the block has warps.
#pragma once
#include "kernels.h"

namespace ssdi8 {
namespace cumsum {

constexpr int kTieWindow = 512;   // binary64 units around a binary32 rounding boundary (see cumsum.cu)

template <int TPL>
__device__ __forceinline__ void st_row(float* p, const float (&v)[TPL], uint64_t pol) {
  if constexpr (TPL == 2) {
    st_global_hint(p, make_float2(v[0], v[1]), pol);
  } else {
#pragma unroll
    for (int j = 0; j < TPL; j += 4) st_global_hint(p + j, make_float4(v[j], v[j + 1], v[j + 2], v[j + 3]), pol);
  }
}

struct Args {
  const float* dt; const float* A; float* pack; float* gamma; float* tap_cs; const float* dt_bias; int32_t* status;
  Dims d;
};

// TPL: tokens per lane, Q / 32; hpb: heads (warps) of the block, a power of two, from h0 on; dts: hpb (Q + 4) floats of shared memory
template <int TPL, bool SOFTPLUS>
__device__ __forceinline__ void chunk_of_heads(float* dts, const int hpb, const int h0, const int k, const int b, const Args& a) {
  constexpr int Q = 32 * TPL, LD = Q + 4;
  const Dims& d = a.d;
  const int lh = 31 - __clz(hpb);
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int h = h0 + w;
  const bool live = h < d.H;
  const float Ah = live ? __ldg(a.A + h) : 0.f;
  {
    const i64 t0 = (i64)b * d.L + (i64)k * Q;
    const int hh = tid & (hpb - 1), t = tid >> lh;   // 32 tokens per round of the block
    const bool ok = h0 + hh < d.H;
    const float* src = a.dt + (t0 + t) * d.H + h0 + hh;
    float v[TPL];
#pragma unroll
    for (int u = 0; u < TPL; ++u) v[u] = ok ? __ldg(src + (i64)(32 * u) * d.H) : 0.f;
    const float bias = (SOFTPLUS && a.dt_bias && ok) ? __ldg(a.dt_bias + h0 + hh) : 0.f;
    if (SOFTPLUS) softplus_dt<TPL>(v, bias, v);
#pragma unroll
    for (int u = 0; u < TPL; ++u) dts[hh * LD + 32 * u + t] = v[u];
  }
  __syncthreads();
  if (!live) return;   // whole warps

  constexpr uint32_t kAll = 0xffffffffu;
  float dv[TPL], cs[TPL];
#pragma unroll
  for (int j = 0; j < TPL; j += 2) {
    const float2 p = *reinterpret_cast<const float2*>(dts + w * LD + lane * TPL + j);
    dv[j] = p.x;
    dv[j + 1] = p.y;
  }
  const double ad = (double)Ah;
  bool redo = false, up = false, down = false;
  {
    double loc[TPL];
    double acc = 0.0;
#pragma unroll
    for (int j = 0; j < TPL; ++j) {
      const double inc = (double)dv[j] * ad;   // exact: the product of two binary32 numbers
      up |= inc > 0.0;
      down |= inc < 0.0;
      acc += inc;
      loc[j] = acc;
    }
    double incl = acc;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const double y = __shfl_up_sync(kAll, incl, o);
      if (lane >= o) incl += y;
    }
    double off = __shfl_up_sync(kAll, incl, 1);
    if (lane == 0) off = 0.0;
#pragma unroll
    for (int j = 0; j < TPL; ++j) {
      const double s = off + loc[j];
      cs[j] = (float)s;
      // the 29 bits that the rounding to binary32 drops; half of their range is the midpoint
      const int lo = __double2loint(s), hi = __double2hiint(s) & 0x7fffffff;
      redo |= abs((lo & 0x1fffffff) - 0x10000000) <= kTieWindow;
      redo |= hi < ((1023 - 100) << 20) ? (hi | lo) != 0 : hi >= 0x7ff00000;
    }
  }
  up = __any_sync(kAll, up);
  down = __any_sync(kAll, down);
  if (__any_sync(kAll, redo) || (up && down)) {
    double carry = 0.0;
#pragma unroll 1
    for (int l = 0; l < 32; ++l) {
      double s = carry;
#pragma unroll
      for (int j = 0; j < TPL; ++j) {
        s += (double)dv[j] * ad;
        if (lane == l) cs[j] = (float)s;
      }
      carry = __shfl_sync(kAll, s, l);
    }
  }
  const bool mono = !up;   // every increment <= 0: cs does not increase over the chunk

  constexpr int LPS = 16 / TPL;        // lanes per 16-token sub-block
  constexpr int NSB = Q / 16, NTRI = NSB * (NSB - 1) / 2;
  const float mine = cs[TPL - 1];      // the lane's last token
  const float cend = __shfl_sync(kAll, mine, lane | (LPS - 1)), clast = __shfl_sync(kAll, mine, 31);
  const float cprev = __shfl_up_sync(kAll, mine, 1);
  const i64 un = ((i64)b * d.H + h) * d.c + k;
  float* const p = a.pack + un * (kPackRows * Q) + lane * TPL;
  // (the pack is read by the state kernel and by ChunkScan after the quantisers and the state kernel have
  // streamed several times the size of L2: its lines are kept ahead of theirs)
  const uint64_t pol = l2_policy_evict_last();
  st_row<TPL>(p + PACK_CS * Q, cs, pol);
  st_row<TPL>(p + PACK_DT * Q, dv, pol);
  if (a.tap_cs) {
#pragma unroll
    for (int j = 0; j < TPL; ++j) a.tap_cs[un * Q + lane * TPL + j] = cs[j];
  }
  float v[TPL];
  float wm = 0.f;
#pragma unroll
  for (int j = 0; j < TPL; j += 2) {
    const float2 e = exp32x2(__fsub_rn(cend, cs[j]), __fsub_rn(cend, cs[j + 1]));
    v[j] = __fmul_rn(dv[j], e.x);
    v[j + 1] = __fmul_rn(dv[j + 1], e.y);
    wm = fmaxf(fmaxf(wm, fabsf(v[j])), fabsf(v[j + 1]));
  }
  st_row<TPL>(p + PACK_WOFF * Q, v, pol);
#pragma unroll
  for (int j = 0; j < TPL; j += 2) {
    const float2 e = exp32x2(__fsub_rn(cs[j], j ? cs[j > 0 ? j - 1 : 0] : cprev), __fsub_rn(cs[j + 1], cs[j]));
    v[j] = e.x;
    v[j + 1] = e.y;
  }
  if (lane == 0) v[0] = 1.0f;
  st_row<TPL>(p + PACK_ATOK * Q, v, pol);
#pragma unroll
  for (int j = 0; j < TPL; j += 2) {
    const float2 e = exp32x2(__fsub_rn(clast, cs[j]), __fsub_rn(clast, cs[j + 1]));
    v[j] = __fmul_rn(dv[j], e.x);
    v[j + 1] = __fmul_rn(dv[j + 1], e.y);
  }
  st_row<TPL>(p + PACK_LUT * Q, v, pol);

  // the bounds row: 127 wmax of sub-block c in lane c; in lane 16 whether cs increases (the lanes beyond fill the sector)
  float* const bounds = a.pack + un * (kPackRows * Q) + PACK_WMAX * Q;
#pragma unroll
  for (int o = 1; o < LPS; o <<= 1) wm = fmaxf(wm, __shfl_xor_sync(kAll, wm, o));
  const int c16 = lane & 15;
  float m = __shfl_sync(kAll, wm, (c16 * LPS) & 31);
  m = c16 < NSB ? __fmul_rn(127.0f, m) : 0.f;
  bounds[lane] = lane >= 16 && !mono ? __int_as_float(0x7f800000) : m;
  // block-to-block decays G[I][c], c < I (triangular: 120 entries for 16 sub-blocks)
#pragma unroll
  for (int r = 0; r < (NTRI + 31) / 32; ++r) {
    const int idx = min(lane + 32 * r, NTRI - 1);
    // I (I - 1) / 2 <= idx < (I + 1) I / 2; 1 + 8 idx is (2 I - 1)^2 at the lower end, so the root is exact there
    const int I = (int)((1.0f + sqrtf((float)(1 + 8 * idx))) * 0.5f);
    const int c = idx - I * (I - 1) / 2;
    const float x = __fsub_rn(__shfl_sync(kAll, mine, LPS * I - 1), __shfl_sync(kAll, mine, LPS * c + LPS - 1));
    if (lane + 32 * r < NTRI) bounds[32 + idx] = exp32(x);
  }
  if (lane == 0) a.gamma[un] = exp32(clast);
}

}  // namespace cumsum
}  // namespace ssdi8
