// Entry quantiser of the SSD layer: the convolution output of a Mamba-2 block is one tensor
// xBC [T][D + 2 G N] (x, then B, then C along the last axis).  One pass reads it (fp32, fp16 or
// bf16) and writes the three int8 tensors the layer consumes, with static step sizes: x per
// channel, B and C per group (quantised once on the group axis at layer entry, before any
// broadcast to heads; Section 4.2 "Quantization of B,C"; Eq. 1 for every element:
// q = rne(fdiv(float(v), alpha)) saturated).  HBM-bound: a thread owns four consecutive columns
// of the concatenated row and walks a slab of rows with several loads in flight.
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "kernels.h"

namespace ssdi8 {
namespace {

constexpr int EROWS = 8;

template <typename T> struct Vec4;
template <> struct Vec4<float> {
  typedef float4 raw;
  static __device__ __forceinline__ float4 cvt(const float4& v) { return v; }
};
template <> struct Vec4<__half> {
  typedef uint2 raw;
  static __device__ __forceinline__ float4 cvt(const uint2& v) {
    const float2 a = __half22float2(*reinterpret_cast<const __half2*>(&v.x));
    const float2 b = __half22float2(*reinterpret_cast<const __half2*>(&v.y));
    return make_float4(a.x, a.y, b.x, b.y);
  }
};
template <> struct Vec4<__nv_bfloat16> {
  typedef uint2 raw;
  static __device__ __forceinline__ float4 cvt(const uint2& v) {
    // bf16 -> fp32 is a 16-bit shift (exact)
    return make_float4(__uint_as_float(v.x << 16), __uint_as_float(v.x & 0xffff0000u),
                       __uint_as_float(v.y << 16), __uint_as_float(v.y & 0xffff0000u));
  }
};

// RAGGED: the row count is no multiple of eight (batches of a decode step).  The last rows then have their loads in flight
// together as well: one by one they end behind everything else, blocks having few rows (us, one by one / together: 5 rows of
// 5376 bf16 2.4 / 1.7, 2047 rows of fp32 8.7 / 7.1).  An instance of its own, because the registers this takes cost the
// common case (8960 rows of bf16 21.9 / 23.3).
template <typename T, bool RAGGED>
__global__ void __launch_bounds__(128) quant_entry_kernel(const typename Vec4<T>::raw* __restrict__ in,
                                                          const float* __restrict__ s_x,
                                                          const float* __restrict__ s_B,
                                                          const float* __restrict__ s_C,
                                                          uint32_t* __restrict__ xq, uint32_t* __restrict__ Bq,
                                                          uint32_t* __restrict__ Cq, i64 T_, int D, int GN, int N,
                                                          int rows_per_block) {
  pdl_launch_dependents();
  pdl_wait();
  const int W4 = (D + 2 * GN) / 4;
  const int q = blockIdx.x * 128 + threadIdx.x;
  if (q >= W4) return;
  const int col = 4 * q;
  float4 s;
  uint32_t* out;
  int ow4, oq;  // output row width and position, in 4-byte words
  if (col < D) {
    s = *reinterpret_cast<const float4*>(s_x + col);
    out = xq; ow4 = D / 4; oq = q;
  } else if (col < D + GN) {
    const float a = s_B[(col - D) / N];
    s = make_float4(a, a, a, a);
    out = Bq; ow4 = GN / 4; oq = (col - D) / 4;
  } else {
    const float a = s_C[(col - D - GN) / N];
    s = make_float4(a, a, a, a);
    out = Cq; ow4 = GN / 4; oq = (col - D - GN) / 4;
  }
  const Step4 st = step4(s);
  const i64 r0 = (i64)blockIdx.y * rows_per_block;
  const i64 r1 = r0 + rows_per_block < T_ ? r0 + rows_per_block : T_;
  i64 r = r0;
  for (; r + EROWS <= r1; r += EROWS) {
    typename Vec4<T>::raw v[EROWS];
#pragma unroll
    for (int u = 0; u < EROWS; ++u) v[u] = __ldcs(in + (r + u) * W4 + q);
    if (st.usable) {
#pragma unroll
      for (int u = 0; u < EROWS; ++u) out[(r + u) * ow4 + oq] = code4(Vec4<T>::cvt(v[u]), st);
    } else {
#pragma unroll 1
      for (int u = 0; u < EROWS; ++u) out[(r + u) * ow4 + oq] = code4_by_division(Vec4<T>::cvt(in[(r + u) * W4 + q]), s);
    }
  }
  if (!RAGGED) {   // (not entered; without a loop here the compiler keeps fewer of the loads above in flight, 24.5 us for 21.9)
    for (; r < r1; ++r) {
      const float4 v = Vec4<T>::cvt(__ldcs(in + r * W4 + q));
      out[r * ow4 + oq] = st.usable ? code4(v, st) : code4_by_division(v, s);
    }
  } else if (r < r1) {
    typename Vec4<T>::raw v[EROWS - 1];
#pragma unroll
    for (int u = 0; u < EROWS - 1; ++u)
      if (r + u < r1) v[u] = __ldcs(in + (r + u) * W4 + q);
#pragma unroll
    for (int u = 0; u < EROWS - 1; ++u)
      if (r + u < r1) {
        const float4 f = Vec4<T>::cvt(v[u]);
        out[(r + u) * ow4 + oq] = st.usable ? code4(f, st) : code4_by_division(f, s);
      }
  }
}

}  // namespace

ssdi8_status_t launch_quantize_entry(const void* xBC, int dtype, i64 T_, int D, int G, int N, const float* s_x,
                                     const float* s_B, const float* s_C, int8_t* xq, int8_t* Bq, int8_t* Cq,
                                     cudaStream_t st) {
  if (T_ == 0) return SSDI8_OK;
  const int GN = G * N, W4 = (D + 2 * GN) / 4;
  const int gx = (W4 + 127) / 128;
  i64 want = (148 * 32 + gx - 1) / gx;
  i64 rows = (T_ + want - 1) / want;
  // at least one round of EROWS loads in flight per thread.  (At least four rounds left the decode step's 64 rows on 22
  // blocks, 8.5 us at 5376 columns; with this and programmatic dependent launch of the step's three kernels the
  // decode step of 64 sequences x 80 heads takes 62 instead of 69.6 us.)
  rows = (rows + EROWS - 1) / EROWS * EROWS;
  dim3 grid(gx, (unsigned)((T_ + rows - 1) / rows));
  auto X = reinterpret_cast<uint32_t*>(xq);
  auto Bo = reinterpret_cast<uint32_t*>(Bq);
  auto Co = reinterpret_cast<uint32_t*>(Cq);
  auto launch = [&](auto kernel, auto* in) -> ssdi8_status_t {
    return launch_configured(kernel, grid, dim3(128), 0, kStreamCarveout, false, st, in, s_x, s_B, s_C, X, Bo, Co, T_, D, GN,
                             N, (int)rows);
  };
  auto pick = [&](auto t, auto* in) -> ssdi8_status_t {
    using E = decltype(t);
    return T_ % EROWS ? launch(quant_entry_kernel<E, true>, in) : launch(quant_entry_kernel<E, false>, in);
  };
  if (dtype == 0) return pick(float{}, static_cast<const float4*>(xBC));
  if (dtype == 1) return pick(__half{}, static_cast<const uint2*>(xBC));
  return pick(__nv_bfloat16{}, static_cast<const uint2*>(xBC));
}

}  // namespace ssdi8
