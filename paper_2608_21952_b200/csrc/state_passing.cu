// StatePassing (Eq. 5-6; Algorithm 2 module 3) on fp32 states:
//   S_k = fmaf(Gamma_k, S_{k-1}, loc_k);  prev[k] = S_{k-1};  hq[k] = rne(fmul(S_{k-1}, 1/s_h))
// The only sequential loop of the layer (over chunks); everything else is parallel over
// (b, h, p, n).  HBM-bound: each thread owns 4 consecutive n (16-byte loads of loc, 4-byte
// packed stores of hq) and keeps several chunk loads in flight.
#include "kernels.h"

namespace ssdi8 {
namespace {

constexpr int SP_T = 256;

// PREV: the entering states are written (they may go over loc, so a chunk's load cannot be moved ahead of the store
// of the one before); without them the loads of eight chunks are in flight at once.
template <bool PREV>
__global__ void __launch_bounds__(SP_T) state_passing_kernel(
    const float4* loc /* may alias prev: no __restrict__ */, const float* __restrict__ gamma, const float4* __restrict__ init,
    const float* __restrict__ s_h, float4* prev, float4* __restrict__ final_state,
    uint32_t* __restrict__ hq, Dims d) {
  pdl_launch_dependents();
  pdl_wait();
  const int N4 = d.N / 4;
  const i64 per_b = (i64)d.H * d.P * N4;               // float4 per (b) slice of one chunk
  const i64 idx = (i64)blockIdx.x * SP_T + threadIdx.x;  // over b * H * P * N4
  if (idx >= per_b * d.b) return;
  const int b = (int)(idx / per_b);
  const i64 r = idx % per_b;                             // (h, p, n4)
  const int hp = (int)(r / N4);                          // h * P + p
  const int h = hp / d.P;
  float inv_h = 0.f;
  if (hq) inv_h = __fdiv_rn(1.0f, s_h[hp]);
  float4 S = init ? init[idx] : make_float4(0.f, 0.f, 0.f, 0.f);
  const float* gm = gamma + ((i64)b * d.H + h) * d.c;
  const i64 stride = per_b;                              // chunk stride in float4
  i64 o = (i64)b * d.c * per_b + r;
  auto step = [&](const float4& l, float g) {
    if (hq)
      hq[o] = pack4(rne_clamp(__fmul_rn(S.x, inv_h)), rne_clamp(__fmul_rn(S.y, inv_h)),
                    rne_clamp(__fmul_rn(S.z, inv_h)), rne_clamp(__fmul_rn(S.w, inv_h)));
    if (PREV) prev[o] = S;
    S.x = __fmaf_rn(g, S.x, l.x);
    S.y = __fmaf_rn(g, S.y, l.y);
    S.z = __fmaf_rn(g, S.z, l.z);
    S.w = __fmaf_rn(g, S.w, l.w);
    o += stride;
  };
  constexpr int K = PREV ? 1 : 8;
  int k = 0;
  for (; k + K <= d.c; k += K) {
    float4 l[K];
    float g[K];
#pragma unroll
    for (int j = 0; j < K; ++j) {
      l[j] = loc[o + j * stride];  // (read before prev[o] is written: prev may alias loc)
      g[j] = gm[k + j];
    }
#pragma unroll
    for (int j = 0; j < K; ++j) step(l[j], g[j]);
  }
  for (; k < d.c; ++k) step(loc[o], gm[k]);
  if (final_state) final_state[idx] = S;
}

}  // namespace

ssdi8_status_t launch_state_passing(const Dims& d, const float* loc, const float* gamma,
                                    const float* init, const float* s_h, float* prev,
                                    float* final_state, int8_t* hq, cudaStream_t st) {
  const i64 n = (i64)d.b * d.H * d.P * (d.N / 4);
  unsigned grid = (unsigned)((n + SP_T - 1) / SP_T);
  return launch_configured(prev ? state_passing_kernel<true> : state_passing_kernel<false>, dim3(grid), dim3(SP_T), 0, -1, false, st,
                           reinterpret_cast<const float4*>(loc), gamma, reinterpret_cast<const float4*>(init), s_h,
                           reinterpret_cast<float4*>(prev), reinterpret_cast<float4*>(final_state),
                           reinterpret_cast<uint32_t*>(hq), d);
}

}  // namespace ssdi8
