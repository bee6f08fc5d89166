// StatePassing (Eq. 5-6; Algorithm 2 module 3) on fp32 states:
//   S_k = fmaf(Gamma_k, S_{k-1}, loc_k);  prev[k] = S_{k-1};  hq[k] = rne(fmul(S_{k-1}, 1/s_h))
// The only sequential loop of the layer (over chunks); everything else is parallel over
// (b, h, p, n).  HBM-bound: each thread owns 4 consecutive n (16-byte loads of loc, 4-byte
// packed stores of hq) and keeps several chunk loads in flight.
#include <type_traits>

#include "kernels.h"

namespace ssdi8 {
namespace {

// K chunks' loads are in flight at once; AHEAD: the next K too, requested before the present ones are used.  PREV: the entering
// states are written; prev may be loc (or start before it): a chunk's load is ahead of the store that goes over it either way.
// FORWARD: inside a forward pass, in place of the fused state kernel, whose codes of a NaN (+127; -127 here) it takes over.
template <bool FORWARD, bool PREV, int K, bool AHEAD, int THREADS>
__global__ void __launch_bounds__(THREADS) state_passing_kernel(
    const float4* loc /* may alias prev: no __restrict__ */, const float* __restrict__ gamma, const float4* __restrict__ init,
    const float* __restrict__ s_h, float4* prev, float4* __restrict__ final_state,
    uint32_t* __restrict__ hq, Dims d) {
  pdl_launch_dependents();
  pdl_wait();
  const int N4 = d.N / 4;
  const i64 per_b = (i64)d.H * d.P * N4;               // float4 per (b) slice of one chunk
  const i64 idx = (i64)blockIdx.x * THREADS + threadIdx.x;  // over b * H * P * N4
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
  struct Batch {
    float4 l[K];
    float g[K];
  };
  auto fetch = [&](Batch& v, i64 at, int k) {
#pragma unroll
    for (int j = 0; j < K; ++j) {
      v.l[j] = loc[at + j * stride];
      v.g[j] = gm[k + j];
    }
  };
  auto step = [&](const float4& l, float g) {
    if (hq) {
      const float4 v = make_float4(__fmul_rn(S.x, inv_h), __fmul_rn(S.y, inv_h), __fmul_rn(S.z, inv_h), __fmul_rn(S.w, inv_h));
      hq[o] = FORWARD ? pack4_bits(rne_clamp_bits(v.x), rne_clamp_bits(v.y), rne_clamp_bits(v.z), rne_clamp_bits(v.w))
                      : pack4(rne_clamp(v.x), rne_clamp(v.y), rne_clamp(v.z), rne_clamp(v.w));
    }
    if (PREV) prev[o] = S;
    S.x = __fmaf_rn(g, S.x, l.x);
    S.y = __fmaf_rn(g, S.y, l.y);
    S.z = __fmaf_rn(g, S.z, l.z);
    S.w = __fmaf_rn(g, S.w, l.w);
    o += stride;
  };
  auto steps = [&](const Batch& v) {
#pragma unroll
    for (int j = 0; j < K; ++j) step(v.l[j], v.g[j]);
  };
  int k = 0;
  if (AHEAD) {
    Batch v0, v1;
    if (K <= d.c) fetch(v0, o, 0);
    for (; k + K <= d.c; k += 2 * K) {
      const bool second = k + 2 * K <= d.c;
      if (second) fetch(v1, o + K * stride, k + K);
      steps(v0);
      if (!second) {
        k += K;
        break;
      }
      if (k + 3 * K <= d.c) fetch(v0, o + K * stride, k + 2 * K);
      steps(v1);
    }
  } else {
    for (; k + K <= d.c; k += K) {
      Batch v;
      fetch(v, o, k);
      steps(v);
    }
  }
  for (; k < d.c; ++k) {
    const float4 l = loc[o];   // (a copy: prev[o] may be the same place)
    step(l, gm[k]);
  }
  if (final_state) final_state[idx] = S;
}

}  // namespace

ssdi8_status_t launch_state_passing(const Dims& d, const float* loc, const float* gamma,
                                    const float* init, const float* s_h, float* prev,
                                    float* final_state, int8_t* hq, cudaStream_t st, bool forward) {
  const i64 n = (i64)d.b * d.H * d.P * (d.N / 4);
  auto launch = [&](auto kernel, int threads) -> ssdi8_status_t {
    return launch_configured(kernel, dim3((unsigned)((n + threads - 1) / threads)), dim3(threads), 0, -1, false, st,
                             reinterpret_cast<const float4*>(loc), gamma, reinterpret_cast<const float4*>(init), s_h,
                             reinterpret_cast<float4*>(prev), reinterpret_cast<float4*>(final_state),
                             reinterpret_cast<uint32_t*>(hq), d);
  };
  // Loads in flight per thread against how many threads the registers leave room for.  With eight chunks and more, eight at a
  // time; from sixteen on, where few threads are all there is, the next eight ahead as well.  us, one batch of eight / the
  // next ahead: 8192 tokens x 24 heads 9.2 / 7.2, 32768 x 4 (chunks of 64) 54 / 36, but 8192 x 80 16.9 / 20.3.  Where prev is
  // written, one at a time / four / eight and the next ahead: 64 sequences of one chunk x 80 heads 89 / 118 / -, 2048 x 80 8.8 /
  // 6.8 / 7.0, 8192 x 80 38 / 36 / 33, 8192 x 24 9.1 / 11.6 / 8.5.
  auto pick = [&](auto fwd) -> ssdi8_status_t {
    constexpr bool F = decltype(fwd)::value;
    if (prev) {
      if (d.c < 4) return launch(state_passing_kernel<F, true, 1, false, 256>, 256);
      if (d.c < 16) return launch(state_passing_kernel<F, true, 4, false, 256>, 256);
      return launch(state_passing_kernel<F, true, 8, true, 128>, 128);
    }
    if (d.c < 8) return launch(state_passing_kernel<F, false, 4, false, 256>, 256);
    if (d.c < 16 || n > 96 * 1024) return launch(state_passing_kernel<F, false, 8, false, 256>, 256);
    return launch(state_passing_kernel<F, false, 8, true, 128>, 128);
  };
  return forward ? pick(std::true_type{}) : pick(std::false_type{});
}

}  // namespace ssdi8
