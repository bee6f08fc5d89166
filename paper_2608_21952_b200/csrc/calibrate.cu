// Kernels of the static calibration (ssdi8_calibrate) that the forward pass does not have: the largest |X_scaled| per
// channel, and the step sizes from the maxima.
#include "kernels.h"

namespace ssdi8 {
namespace {

// absmax_xs[h,p] = max over tokens of |fmul(fmul(float(xq), s_x), LUT_state)| (Eq. 3), as binary32 bits.  A block takes a
// chunk, or 64 tokens of one, of 8 neighbouring heads (512 contiguous bytes of a token), 32 tokens at a time from the last one on; a thread owns
// 16 channels of four of the tokens and keeps their maxima in registers, and after a round that had anything to do the
// token rows of the block meet in shared memory.  LUT_state decays towards the start of a chunk, so a few rounds decide the
// maxima: a token whose 16 products cannot exceed them, |LUT_state| <= min over the channels of max / (128 |s_x|) (fmul is
// monotone, 128 s_x is exact; a slack of 1e-5 covers the quotient), is neither loaded nor multiplied.  One atomic per channel
// and block leaves it, if it raises what is there.  (Every token multiplied, 64 to a block,
// calibration calls: 2 x 2048 x 80 heads 80.5 -> 78.6 us, 4 x 1024 x 128 (G 8) 125.1 -> 117.9, 12 x 512 x 64 91.1 -> 87.8, 16384 x 32 153.8 -> 145.3;
// blocks of 512 threads 79.1, 120.1, 91.5, 151.2.)
constexpr int kXsHeads = 8, kXsThreads = 256, kXsRows = kXsThreads / 32, kXsTokens = 4 * kXsRows;
__global__ void __launch_bounds__(kXsThreads) absmax_xs_kernel(const int8_t* __restrict__ xq, const float* __restrict__ s_x, const float* pack,
                                                        uint32_t* absmax, Dims d, int parts) {
  extern __shared__ __align__(16) float lut[];    // [kXsHeads][Q]
  __shared__ __align__(16) float sxs[kXsHeads * 64];
  __shared__ uint32_t best[16][32];               // channel e of (head, 16 channels) = lane
  pdl_wait();
  pdl_launch_dependents();   // (after the wait: ChunkBMM, launched next, does not wait for this kernel)
  const int tid = threadIdx.x, lane = tid & 31;
  // (head blocks and chunks in one grid dimension: a sequence of more than 4 M tokens has more than 65535 of the latter)
  const int nhb = (d.H + kXsHeads - 1) / kXsHeads, kp = blockIdx.x / nhb, k = kp / parts, b = blockIdx.z;
  const int h0 = (blockIdx.x - kp * nhb) * kXsHeads;
  const int span = d.Q / parts, first = (kp - k * parts) * span;   // tokens of the chunk that the block takes, a power of two
  const int hh = (tid >> 2) & 7, c = tid & 3, row = tid >> 5;   // head, 16 channels, token row of the thread
  const int h = h0 + hh;
  const bool live = h < d.H;
  const uint4* src = reinterpret_cast<const uint4*>(xq + (((i64)b * d.L + (i64)k * d.Q + first + row) * d.H + h) * 64) + c;
  const i64 stride = (i64)kXsRows * d.H * 4;   // kXsRows tokens, in 16-byte words
  uint4 w[4];                                  // (the first round's before LUT_state is there)
#pragma unroll
  for (int u = 0; u < 4; ++u) w[u] = live ? __ldg(src + ((span - kXsTokens) / kXsRows + u) * stride) : make_uint4(0u, 0u, 0u, 0u);
  const int lq = 31 - __clz(span) - 2;          // LUT_state, 16 bytes at a time
  for (int e = tid; e < (kXsHeads << lq); e += kXsThreads) {
    const int hl = e >> lq, i = (e - (hl << lq)) * 4;
    if (h0 + hl < d.H)
      *reinterpret_cast<float4*>(lut + hl * span + i) =
          *reinterpret_cast<const float4*>(pack + ((((i64)b * d.H + h0 + hl) * d.c + k) * kPackRows + PACK_LUT) * d.Q + first + i);
  }
  // (by way of shared memory: ssdi8_calibrate asks for no alignment of s_x beyond a float's, and sixteen loads of one float per
  // thread were 4 us slower)
  for (int e = tid; e < kXsHeads * 64; e += kXsThreads) {
    sxs[e] = h0 + (e >> 6) < d.H ? __ldg(s_x + h0 * 64 + e) : 0.f;
    best[e >> 5][e & 31] = 0u;
  }
  float mx[16];
#pragma unroll
  for (int e = 0; e < 16; ++e) mx[e] = 0.f;
  __syncthreads();
  float2 sx[8];
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const float4 v = *(reinterpret_cast<const float4*>(&sxs[hh * 64 + c * 16]) + e);
    sx[2 * e] = make_float2(v.x, v.y);
    sx[2 * e + 1] = make_float2(v.z, v.w);
  }
  float least = 0.f;                     // |LUT_state| up to here changes nothing
#pragma unroll 1
  for (int i0 = span - kXsTokens; i0 >= 0; i0 -= kXsTokens) {
    float l[4];
    bool any = false;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      l[u] = live ? lut[hh * span + i0 + kXsRows * u + row] : 0.f;
      if (!(fabsf(l[u]) <= least)) {
        if (i0 != span - kXsTokens) w[u] = __ldg(src + (i0 / kXsRows + u) * stride);
        any = true;
      }
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      if (fabsf(l[u]) <= least) continue;
      const float2 l2 = make_float2(l[u], l[u]);
      const uint32_t ww[4] = {w[u].x ^ 0x80808080u, w[u].y ^ 0x80808080u, w[u].z ^ 0x80808080u, w[u].w ^ 0x80808080u};
#pragma unroll
      for (int e = 0; e < 16; e += 2) {
        const float2 xf = make_float2(s8_to_f32(ww[e >> 2], e & 3), s8_to_f32(ww[e >> 2], (e & 3) + 1));
        const float2 v = __fmul2_rn(__fmul2_rn(xf, sx[e >> 1]), l2);
        mx[e] = fmaxf(mx[e], fabsf(v.x));
        mx[e + 1] = fmaxf(mx[e + 1], fabsf(v.y));
      }
    }
    if (any) {
#pragma unroll
      for (int e = 0; e < 16; ++e) atomicMax(&best[e][lane], __float_as_uint(mx[e]));
    }
    if (__syncthreads_or(any) && i0 > 0) {
      least = __int_as_float(0x7f800000);
#pragma unroll
      for (int e = 0; e < 16; ++e) {
        mx[e] = __uint_as_float(*reinterpret_cast<volatile uint32_t*>(&best[e][lane]));
        const float s = fabsf(e & 1 ? sx[e >> 1].y : sx[e >> 1].x);
        const float top = 128.0f * s;
        least = fminf(least, top >= 0x1p-126f ? __fdividef(mx[e], top) : 0.f);   // (below, the quotient's error has no bound: skip nothing)
      }
      least = least < 1e-30f ? 0.f : least * 0.99999f;
    }
  }
  for (int e = tid; e < kXsHeads * 64; e += kXsThreads) {
    const int hc = e & 31, ch = (hc >> 2) * 64 + (hc & 3) * 16 + (e >> 5);   // of best[e >> 5][hc]
    const uint32_t m = best[e >> 5][hc];
    if (h0 + (hc >> 2) < d.H && m > *reinterpret_cast<volatile uint32_t*>(absmax + h0 * 64 + ch)) atomicMax(absmax + h0 * 64 + ch, m);
  }
}

__global__ void clear_words(uint32_t* a, int n) {
  pdl_launch_dependents();
  pdl_wait();
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e < n) a[e] = 0u;
}

// step sizes from maxima: s_h = fdiv(max_h, 127), s_cb = fdiv(fmul(float(max_cb), fmul(s_C, s_B)), 127), 1 where the
// maximum is 0
__global__ void finalize_scales(const uint32_t* max_h, float* s_h, int n, const uint32_t* max_cb, float* s_cb, int nq,
                                const float* s_C, const float* s_B) {
  pdl_launch_dependents();
  pdl_wait();
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k < n) s_h[k] = step_of_max(max_h[k]);
  if (k < nq) {
    const int v = (int)max_cb[k];
    s_cb[k] = v == 0 ? 1.0f : __fdiv_rn(__fmul_rn((float)v, __fmul_rn(s_C[k], s_B[k])), 127.0f);
  }
}

}  // namespace

ssdi8_status_t launch_absmax_xs(const Dims& d, const int8_t* xq, const float* s_x, const float* pack, uint32_t* absmax,
                                cudaStream_t st) {
  const i64 chunks = (i64)((d.H + kXsHeads - 1) / kXsHeads) * d.c;
  const int sms = sm_count();
  if (sms == 0) return SSDI8_ERR_CUDA;
  // Few chunks go 64 tokens to a block, whose rounds are a chain of loads and barriers each; with more of them ChunkBMM, which works beside this kernel,
  // wants the room.  Calibration calls, us, whole chunks / 64 tokens: 512 tokens x 8 heads 30.6 / 28.2, 1280 x 24 43.1 / 40.7, 2048 x 32 48.6 / 46.1, but
  // 4096 x 4 46.5 / 49.6, 8192 x 16 75.3 / 81.0.
  const int parts = d.Q > 64 && (i64)d.b * d.c < 12 && chunks * d.b * (d.Q / 64) <= 2 * sms ? d.Q / 64 : 1;
  const i64 blocks = chunks * parts;
  if (blocks > 0x7fffffff) return SSDI8_ERR_SHAPE;
  const dim3 grid((unsigned)blocks, 1, d.b);
  return launch_sized(absmax_xs_kernel, grid, dim3(kXsThreads), sizeof(float) * kXsHeads * d.Q, sizeof(float) * kXsHeads * 256, kStreamCarveout,
                      false, st, xq, s_x, pack, absmax, d, parts);
}

ssdi8_status_t launch_clear_words(void* a, i64 n, cudaStream_t st) {
  return launch_configured(clear_words, dim3((unsigned)((n + 255) / 256)), dim3(256), 0, -1, false, st,
                           static_cast<uint32_t*>(a), (int)n);
}

ssdi8_status_t launch_finalize_scales(const uint32_t* max_h, float* s_h, i64 n, const uint32_t* max_cb, float* s_cb, i64 nq,
                                      const float* s_C, const float* s_B, cudaStream_t st) {
  const i64 m = n > nq ? n : nq;
  return launch_configured(finalize_scales, dim3((unsigned)((m + 255) / 256)), dim3(256), 0, -1, false, st, max_h, s_h, (int)n,
                           max_cb, s_cb, (int)nq, s_C, s_B);
}

}  // namespace ssdi8
