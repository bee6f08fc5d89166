// ChunkCumsum (Algorithm 2, module 1) and the per-token scalars every later module derives
// from it.  For each (batch, head, chunk) it writes one contiguous pack of 6 rows of Q floats:
//   row 0  cs[i]    = (float) sum_{i'<=i} (double)dt (double)A_h, in token order   (dA_cs)
//   row 1  dt[i]
//   row 2  woff[i]  = fmul(dt_i, exp32(fsub(cs_ie, cs_i))), ie = last token of i's 16-token sub-block
//   row 3  atok[i]  = exp32(fsub(cs_i, cs_{i-1}))  (1 for i = 0): the per-token decay
//   row 4  bounds that let the scan kernel skip sub-blocks that cannot matter (they decide no
//          output bit): [c] = fmul(127, wmax_c), wmax_c the maximum of |woff| over the 16-token
//          sub-block c; [16 + c] = the maximum of the former over sub-blocks 0..c, times
//          1.00001, or +inf when cs is not non-increasing over the chunk (some dt A > 0), which
//          switches the early exits of the scan kernel off; [32 + I (I - 1) / 2 + c], c < I: the decay
//          between the ends of sub-blocks c and I - 1, exp32(fsub(cs[16 I - 1], cs[16 c + 15])), which
//          the scan kernel multiplies by a row's own decay to the end of sub-block I - 1; the rest of
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
#include "kernels.h"

namespace ssdi8 {
namespace {

constexpr int kMaxHeads = 8;      // heads (warps) per block: 8 heads of a token are one 32-byte sector of dt
constexpr int kTieWindow = 512;   // binary64 units around a binary32 rounding boundary (see above)

template <int TPL>
__device__ __forceinline__ void st_row(float* p, const float (&v)[TPL], uint64_t pol) {
  if constexpr (TPL == 2) {
    st_global_hint(p, make_float2(v[0], v[1]), pol);
  } else {
#pragma unroll
    for (int j = 0; j < TPL; j += 4) st_global_hint(p + j, make_float4(v[j], v[j + 1], v[j + 2], v[j + 3]), pol);
  }
}

// TPL: tokens per lane, Q / 32.  SOFTPLUS: dt holds the raw time step and dt = softplus(dt + dt_bias[h])
// (dt_bias may be NULL) is applied as the values are staged (Algorithm 2 module 1 starts there).
// CLEAR: nclear words are set to 0 as well (calibration).
// status: the caller's status word, cleared here (this is the first kernel of a forward pass), or NULL.
template <int TPL, bool SOFTPLUS, bool CLEAR>
__global__ void __launch_bounds__(32 * kMaxHeads) cumsum_kernel(const float* __restrict__ dt, const float* __restrict__ A,
                                                                float* __restrict__ pack, float* __restrict__ gamma,
                                                                float* __restrict__ tap_cs, Dims d,
                                                                const float* __restrict__ dt_bias, int32_t* status,
                                                                uint32_t* clear, int nclear) {
  constexpr int Q = 32 * TPL, LD = Q + 4;
  __shared__ __align__(16) float dts[kMaxHeads * LD];
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
  const int hpb = (int)(blockDim.x >> 5), lh = 31 - __clz(hpb);   // heads of this block (a power of two)
  const int h0 = blockIdx.x * hpb, k = blockIdx.y, b = blockIdx.z;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  if (status && tid == 0 && (blockIdx.x | blockIdx.y | blockIdx.z) == 0) *status = 0;
  const int h = h0 + w;
  const bool live = h < d.H;
  const float Ah = live ? __ldg(A + h) : 0.f;
  {
    const i64 t0 = (i64)b * d.L + (i64)k * Q;
    const int hh = tid & (hpb - 1), t = tid >> lh;   // 32 tokens per round of the block
    const bool ok = h0 + hh < d.H;
    const float* src = dt + (t0 + t) * d.H + h0 + hh;
    float v[TPL];
#pragma unroll
    for (int u = 0; u < TPL; ++u) v[u] = ok ? __ldg(src + (i64)(32 * u) * d.H) : 0.f;
    const float bias = (SOFTPLUS && dt_bias && ok) ? __ldg(dt_bias + h0 + hh) : 0.f;
#pragma unroll
    for (int u = 0; u < TPL; ++u) dts[hh * LD + 32 * u + t] = SOFTPLUS ? softplus_dt(v[u], bias) : v[u];
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
  const double a = (double)Ah;
  bool redo = false, up = false, down = false;
  {
    double loc[TPL];
    double acc = 0.0;
#pragma unroll
    for (int j = 0; j < TPL; ++j) {
      const double inc = (double)dv[j] * a;   // exact: the product of two binary32 numbers
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
        s += (double)dv[j] * a;
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
  float* const p = pack + un * (kPackRows * Q) + lane * TPL;
  // (the pack is read by the state kernel and by ChunkScan after the quantisers and the state kernel have
  // streamed several times the size of L2: its lines are kept ahead of theirs)
  const uint64_t pol = l2_policy_evict_last();
  st_row<TPL>(p + PACK_CS * Q, cs, pol);
  st_row<TPL>(p + PACK_DT * Q, dv, pol);
  if (tap_cs) {
#pragma unroll
    for (int j = 0; j < TPL; ++j) tap_cs[un * Q + lane * TPL + j] = cs[j];
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

  // the bounds row: 127 wmax of sub-block c in lane c and in lane 16 + c, their running maximum by a scan over
  // each half of the warp
  float* const bounds = pack + un * (kPackRows * Q) + PACK_WMAX * Q;
#pragma unroll
  for (int o = 1; o < LPS; o <<= 1) wm = fmaxf(wm, __shfl_xor_sync(kAll, wm, o));
  const int c16 = lane & 15;
  float m = __shfl_sync(kAll, wm, (c16 * LPS) & 31);
  m = c16 < NSB ? __fmul_rn(127.0f, m) : 0.f;
  float pm = m;
#pragma unroll
  for (int o = 1; o < 16; o <<= 1) {
    const float y = __shfl_up_sync(kAll, pm, o, 16);
    if (c16 >= o) pm = fmaxf(pm, y);
  }
  pm = mono ? __fmul_rn(pm, 1.00001f) : __int_as_float(0x7f800000);
  bounds[lane] = lane < 16 ? m : c16 < NSB ? pm : 0.f;
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
  if (lane == 0) gamma[un] = exp32(clast);
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
  if (launch_pdl(softplus_dt_kernel, dim3((unsigned)((n + 255) / 256)), dim3(256), 0, st, dt_raw, dt_bias, out, n, H) !=
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
  int hpb = kMaxHeads;
  if ((i64)((d.H + hpb - 1) / hpb) * d.c * d.b <= sms) hpb /= 2;
  const dim3 grid((d.H + hpb - 1) / hpb, d.c, d.b);
  auto launch = [&](auto kernel) -> ssdi8_status_t {
    return launch_configured(kernel, grid, dim3(32 * hpb), 0, kStreamCarveout, false, st, dt, A, pack, gamma, tap_cs, d,
                             dt_bias, clear_status, clear, nclear);
  };
  if (nclear && softplus) return SSDI8_ERR_UNSUPPORTED;   // (calibration takes the positive time step)
  auto pick = [&](auto sp, auto plain, auto clearing) -> ssdi8_status_t {
    return softplus ? launch(sp) : nclear ? launch(clearing) : launch(plain);
  };
  ssdi8_status_t ls;
  if (d.Q == 256)
    ls = pick(cumsum_kernel<8, true, false>, cumsum_kernel<8, false, false>, cumsum_kernel<8, false, true>);
  else if (d.Q == 128)
    ls = pick(cumsum_kernel<4, true, false>, cumsum_kernel<4, false, false>, cumsum_kernel<4, false, true>);
  else
    ls = pick(cumsum_kernel<2, true, false>, cumsum_kernel<2, false, false>, cumsum_kernel<2, false, true>);
  if (ls != SSDI8_OK) return ls;
  SSDI8_LAUNCH_CHECK();
  return SSDI8_OK;
}

}  // namespace ssdi8
