// ChunkCumsum (Algorithm 2, module 1) and the per-token scalars every later module derives
// from it.  For each (batch, head, chunk) it writes one contiguous pack of 6 rows of Q floats:
//   row 0  cs[i]    = (float) sum_{i'<=i} (double)dt (double)A_h, in token order   (dA_cs)
//   row 1  dt[i]
//   row 2  woff[i]  = fmul(dt_i, exp32(fsub(cs_ie, cs_i))), ie = last token of i's 16-token sub-block
//   row 3  atok[i]  = exp32(fsub(cs_i, cs_{i-1}))  (1 for i = 0): the per-token decay
//   row 4  bounds that let the scan kernels skip sub-blocks that cannot matter (they decide no
//          output bit): [c] = fmul(127, wmax_c), wmax_c the maximum of |woff| over the 16-token
//          sub-block c; [16] = +inf when cs is not non-increasing over the chunk (some dt A > 0),
//          which has the int8 scan visit every sub-block, else [0]; [32 + I (I - 1) / 2 + c], c < I: the decay
//          between the ends of sub-blocks c and I - 1, exp32(fsub(cs[16 I - 1], cs[16 c + 15])), which
//          the scan kernels multiply by a row's own decay to the end of sub-block I - 1; the rest of
//          the row is not written
//   row 5  lut[i]   = fmul(dt_i, exp32(fsub(cs_last, cs_i)))                       (LUT_state)
// and Gamma[b,h,k] = exp32(cs[Q-1]) (Decay_pass, Eq. 5).  Later kernels fetch a pack with one bulk copy
// and need no exponentials per token.
//
// A warp takes one (batch, head, chunk): lane l owns the Q / 32 consecutive tokens from l Q / 32 on, so the
// rows leave as 16-byte stores and everything after the load stays in registers and shuffles.  A block's
// warps take neighbouring heads of one chunk, because the [b,L,H] input has a token's heads together.
//
// The order of the sum is part of the definition (it decides the binary32 rounding of cs), but the sum is
// formed by a warp scan in binary64: for increments of one sign the two orders differ by less than
// 275 units of the binary64 result (255 additions in token order and at most 14 in the scan, each within
// half a unit in the last place, times 2 across a binade), so they round to the same binary32 number unless
// the result lies that close to the midpoint of two such numbers.  A chunk with such a token (one chunk of
// 256 tokens in 2000 at the limit of 512 units used here), with increments of both signs, or with a result
// outside the normal range is summed again in token order, lane after lane.
// Measured against the sequential scan per block that this replaces (8 lanes at work, the other 248 threads
// waiting): 5.4 against 12.5 us at 1024 x 80 heads, 5 against 13 us with the softplus on one chunk of 24
// heads (the shortest a block can take), 17 against 32 us with it at batch 8 x 2048 x 80 heads.
#include "cumsum.cuh"

#include <type_traits>

namespace ssdi8 {
namespace {

// TPL: tokens per lane, Q / 32.  SOFTPLUS: dt holds the raw time step and dt = softplus(dt + dt_bias[h])
// (dt_bias may be NULL) is applied as the values are staged (Algorithm 2 module 1 starts there).
// CLEAR: nclear words are set to 0 as well (calibration).
// status: the caller's status word, cleared here (this is the first kernel of a forward pass), or NULL.
// FEW: a grid of four heads per block for up to half of the SMs, which may take the registers that the shortest chain wants (102 for eight
// tokens a lane).  A larger grid takes eight or four heads per block and few registers, because the quantisers of a layer work
// beside it, but with the softplus three blocks per SM: left to itself the compiler takes 60 registers for it, and the prefill of
// 5 x 1792 tokens x 80 heads 126.2 us (four blocks per SM) instead of 123.8 (80 registers); with two blocks 126.9.  Layer calls, us, 62
// registers / 102: 1024 tokens x 48 heads 29.9 / 28.4, 2048 x 24 32.4 / 32.0, 6 x 1024 x 24 (144 blocks) 47.4 / 48.2, 11 x 1536 x 13
// (264) 64.7 / 66.3.
template <int TPL, bool SOFTPLUS, bool CLEAR, bool FEW>
__global__ void __launch_bounds__(FEW ? 128 : 256, FEW ? 1 : SOFTPLUS ? 3 : 0) cumsum_kernel(const cumsum::Args a, uint32_t* clear,
                                                                                          int nclear) {
  constexpr int kHeads = FEW ? 4 : 8;   // (8 heads of a token are one 32-byte sector of dt)
  __shared__ __align__(16) float dts[kHeads * (32 * TPL + 4)];
  // The wait comes first: a successor that needs nothing of this kernel (the layer step's quantiser of x, B
  // and C) is launched without a wait of its own at its start, so by the time it may be scheduled everything
  // that precedes this kernel in the stream must have completed.
  pdl_wait();
  if (CLEAR) {   // (words that kernels behind the next one use, not all of which wait for this one: cleared ahead of the trigger)
    const int nb = (int)(gridDim.x * gridDim.y * gridDim.z), blk = (int)((blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x);
    for (int i = blk * (int)blockDim.x + (int)threadIdx.x; i < nclear; i += nb * (int)blockDim.x) clear[i] = 0u;
    __threadfence();
    __syncthreads();
  }
  pdl_launch_dependents();
  if (a.status && threadIdx.x == 0 && (blockIdx.x | blockIdx.y | blockIdx.z) == 0) *a.status = 0;
  const int hpb = FEW ? 4 : (int)(blockDim.x >> 5);
  cumsum::chunk_of_heads<TPL, SOFTPLUS>(dts, hpb, (int)blockIdx.x * hpb, (int)blockIdx.y, (int)blockIdx.z, a);
}

// dt = softplus(dt_raw + dt_bias[h]) alone (for callers that calibrate on the positive time step)
__global__ void softplus_dt_kernel(const float* __restrict__ dt_raw, const float* __restrict__ dt_bias,
                                   float* __restrict__ out, i64 n, int H) {
  pdl_launch_dependents();
  pdl_wait();
  const i64 e = (i64)blockIdx.x * blockDim.x + threadIdx.x;
  if (e < n) out[e] = softplus_dt(dt_raw[e], dt_bias ? __ldg(dt_bias + (int)(e % H)) : 0.f);
}

}  // namespace

ssdi8_status_t launch_softplus_dt(const float* dt_raw, const float* dt_bias, float* out, i64 rows, int H,
                                  cudaStream_t st) {
  const i64 n = rows * H;
  if (n == 0) return SSDI8_OK;
  if (launch_pdl(softplus_dt_kernel, dim3((unsigned)((n + 255) / 256)), 0, dim3(256), 0, st, dt_raw, dt_bias, out, n, H) !=
      cudaSuccess)
    return SSDI8_ERR_CUDA;
  SSDI8_LAUNCH_CHECK();
  return SSDI8_OK;
}

ssdi8_status_t launch_cumsum(const Dims& d, const float* dt, const float* A, float* pack, float* gamma, float* tap_cs,
                             cudaStream_t st, const float* dt_bias, bool softplus, int32_t* clear_status,
                             uint32_t* clear, int nclear) {
  const int sms = sm_count();
  if (sms == 0) return SSDI8_ERR_CUDA;
  // a grid that leaves SMs empty takes half the heads per block: one warp per scheduler, twice the SMs
  int hpb = 8;
  if ((i64)((d.H + hpb - 1) / hpb) * d.c * d.b <= sms) hpb /= 2;
  const dim3 grid((d.H + hpb - 1) / hpb, d.c, d.b);
  const bool few = hpb == 4 && (i64)grid.x * d.c * d.b * 2 <= sms;
  auto launch = [&](auto kernel) -> ssdi8_status_t {
    return launch_configured(kernel, grid, dim3(32 * hpb), 0, kStreamCarveout, false, st,
                             cumsum::Args{dt, A, pack, gamma, tap_cs, dt_bias, clear_status, d}, clear, nclear);
  };
  if (nclear && softplus) return SSDI8_ERR_UNSUPPORTED;   // (calibration takes the positive time step)
  auto pick = [&](auto tpl) -> ssdi8_status_t {
    constexpr int T = decltype(tpl)::value;
    if (softplus) return few ? launch(cumsum_kernel<T, true, false, true>) : launch(cumsum_kernel<T, true, false, false>);
    if (nclear) return few ? launch(cumsum_kernel<T, false, true, true>) : launch(cumsum_kernel<T, false, true, false>);
    return few ? launch(cumsum_kernel<T, false, false, true>) : launch(cumsum_kernel<T, false, false, false>);
  };
  const ssdi8_status_t ls = d.Q == 256   ? pick(std::integral_constant<int, 8>{})
                            : d.Q == 128 ? pick(std::integral_constant<int, 4>{})
                                         : pick(std::integral_constant<int, 2>{});
  if (ls != SSDI8_OK) return ls;
  SSDI8_LAUNCH_CHECK();
  return SSDI8_OK;
}

}  // namespace ssdi8
