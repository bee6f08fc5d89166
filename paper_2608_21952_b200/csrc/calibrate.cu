// Kernels of the static calibration (ssdi8_calibrate) that the forward pass does not have: the largest |X_scaled| per
// channel, and the step sizes from the maxima.
#include "kernels.h"

namespace ssdi8 {
namespace {

// absmax_xs[h,p] = max over tokens of |fmul(fmul(float(xq), s_x), LUT_state)| (Eq. 3), as binary32 bits.  Streaming
// over xq: a block takes 8 neighbouring heads (512 contiguous bytes of a token) and 64 tokens; a
// thread owns 16 channels and keeps their maxima in registers, the 8 token rows of the block meet in shared
// memory, and one atomic per channel and block leaves it.  (The ChunkState kernel did this with 16 atomics per
// thread, all CTAs of a head on its 64 channels: 103 us at batch 2 x 2048 x 80 heads against 10.  64 tokens per
// block instead of half a chunk: 2 us more.)
constexpr int kXsHeads = 8, kXsTokens = 64;
__global__ void __launch_bounds__(256) absmax_xs_kernel(const int8_t* __restrict__ xq, const float* __restrict__ s_x,
                                                        const float* __restrict__ pack, uint32_t* __restrict__ absmax, Dims d) {
  __shared__ __align__(16) float lut[kXsHeads][kXsTokens];
  __shared__ __align__(16) float sxs[kXsHeads * 64];
  __shared__ uint32_t best[8][kXsHeads * 64];
  pdl_wait();
  pdl_launch_dependents();   // (after the wait: ChunkBMM, launched next, does not wait for this kernel)
  const int tid = threadIdx.x;
  // (head blocks and token blocks in one grid dimension: a sequence of more than 4 M tokens has more than 65535 of the latter)
  const int nhb = (d.H + kXsHeads - 1) / kXsHeads, tb = blockIdx.x / nhb, b = blockIdx.z;
  const int h0 = (blockIdx.x - tb * nhb) * kXsHeads, k = tb / (d.Q / kXsTokens);
  constexpr int nt = kXsTokens;
  const int i0 = (tb % (d.Q / kXsTokens)) * nt;   // tokens of this block
  for (int e = tid; e < kXsHeads * nt; e += 256) {
    const int hh = e / nt, i = e % nt;
    if (h0 + hh < d.H) lut[hh][i] = __ldg(pack + ((((i64)b * d.H + h0 + hh) * d.c + k) * kPackRows + PACK_LUT) * d.Q + i0 + i);
  }
  // (by way of shared memory: ssdi8_calibrate asks for no alignment of s_x beyond a float's, and sixteen loads of one float per
  // thread were 4 us slower)
  for (int e = tid; e < kXsHeads * 64; e += 256)
    if (h0 + (e >> 6) < d.H) sxs[e] = __ldg(s_x + h0 * 64 + e);
  const int hh = (tid >> 2) & 7, c = tid & 3, row = tid >> 5;   // head, 16 channels, token row of the thread
  const int h = h0 + hh;
  float mx[16];
#pragma unroll
  for (int e = 0; e < 16; ++e) mx[e] = 0.f;
  __syncthreads();
  if (h < d.H) {
    float2 sx[8];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const float4 v = *(reinterpret_cast<const float4*>(&sxs[hh * 64 + c * 16]) + e);
      sx[2 * e] = make_float2(v.x, v.y);
      sx[2 * e + 1] = make_float2(v.z, v.w);
    }
    const uint4* src = reinterpret_cast<const uint4*>(xq + (((i64)b * d.L + (i64)k * d.Q + i0 + row) * d.H + h) * 64) + c;
    const i64 stride = (i64)8 * d.H * 4;   // 8 tokens, in 16-byte words
#pragma unroll 1
    for (int i = 0; i < nt; i += 32) {     // (four tokens per round and thread)
      uint4 w[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) w[u] = __ldg(src + (i / 8 + u) * stride);
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const float l = lut[hh][i + 8 * u + row];
        const float2 l2 = make_float2(l, l);
        const uint32_t ww[4] = {w[u].x ^ 0x80808080u, w[u].y ^ 0x80808080u, w[u].z ^ 0x80808080u, w[u].w ^ 0x80808080u};
#pragma unroll
        for (int e = 0; e < 16; e += 2) {
          const float2 xf = make_float2(s8_to_f32(ww[e >> 2], e & 3), s8_to_f32(ww[e >> 2], (e & 3) + 1));
          const float2 v = __fmul2_rn(__fmul2_rn(xf, sx[e >> 1]), l2);
          mx[e] = fmaxf(mx[e], fabsf(v.x));
          mx[e + 1] = fmaxf(mx[e + 1], fabsf(v.y));
        }
      }
    }
  }
#pragma unroll
  for (int e = 0; e < 16; ++e) best[row][hh * 64 + c * 16 + e] = __float_as_uint(mx[e]);
  __syncthreads();
  for (int e = tid; e < kXsHeads * 64; e += 256) {
    if (h0 + (e >> 6) >= d.H) break;
    uint32_t m = 0u;
#pragma unroll
    for (int r = 0; r < 8; ++r) m = max(m, best[r][e]);
    atomicMax(absmax + h0 * 64 + e, m);
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
  const i64 blocks = (i64)((d.H + kXsHeads - 1) / kXsHeads) * d.c * (d.Q / kXsTokens);
  if (blocks > 0x7fffffff) return SSDI8_ERR_SHAPE;
  const dim3 grid((unsigned)blocks, 1, d.b);
  return launch_configured(absmax_xs_kernel, grid, dim3(256), 0, kStreamCarveout, false, st, xq, s_x, pack, absmax, d);
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
