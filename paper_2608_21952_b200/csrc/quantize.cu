// Activation quantiser (Eq. 1): uniform symmetric 8-bit with one step size per channel
// of the view in[R][Ch][I].  HBM-bound: 16-byte loads, 4-byte packed stores, every warp
// instruction fully coalesced; absmax by per-thread running maxima, warp shuffles and
// one order-independent atomicMax on the (non-negative) binary32 bit pattern.
#include "cumsum.cuh"

namespace ssdi8 {
namespace {

constexpr int QT = 256;      // threads per block
constexpr int QUNROLL = 4;   // float4 loads in flight per thread

// ---- quantise, I == 1: 4 consecutive elements are 4 consecutive channels.  A thread owns one
// float4 column (its four step sizes stay in registers) and walks a slab of rows with QROWS
// independent 16-byte loads in flight; a warp reads 512 and writes 128 contiguous bytes per row.
constexpr int QROWS = 8;
// FIX: the step sizes were just formed by an absmax kernel; an all-zero channel has 0 there and gets 1 (every
// block reads 0 or 1 and takes 1, the first row of blocks writes it).
template <bool FIX>
__global__ void __launch_bounds__(128, 8) quant_ch_fastest(const float4* __restrict__ in, float4* scale,
                                                        uint32_t* __restrict__ out, i64 R, int ch4,
                                                        int rows_per_block) {
  pdl_launch_dependents();
  pdl_wait();
  const int q = blockIdx.x * 128 + threadIdx.x;
  if (q >= ch4) return;
  float4 s = scale[q];
  if (FIX && (s.x == 0.f || s.y == 0.f || s.z == 0.f || s.w == 0.f)) {
    s = make_float4(s.x == 0.f ? 1.f : s.x, s.y == 0.f ? 1.f : s.y, s.z == 0.f ? 1.f : s.z, s.w == 0.f ? 1.f : s.w);
    if (blockIdx.y == 0) scale[q] = s;
  }
  const Step4 st = step4(s);
  const i64 r0 = (i64)blockIdx.y * rows_per_block;
  const i64 r1 = r0 + rows_per_block < R ? r0 + rows_per_block : R;
  if (!st.usable) {   // abnormal step sizes: row by row
    for (i64 r = r0; r < r1; ++r) __stcs(out + r * ch4 + q, code4_by_division(__ldcs(in + r * ch4 + q), s));
    return;
  }
  i64 r = r0;
  for (; r + QROWS <= r1; r += QROWS) {
    float4 v[QROWS];
#pragma unroll
    for (int u = 0; u < QROWS; ++u) v[u] = __ldcs(in + (r + u) * ch4 + q);
#pragma unroll
    for (int u = 0; u < QROWS; ++u) __stcs(out + (r + u) * ch4 + q, code4(v[u], st));
  }
  if (r < r1) {   // the last rows, their loads in flight together too
    float4 v[QROWS];
#pragma unroll
    for (int u = 0; u < QROWS - 1; ++u)
      if (r + u < r1) v[u] = __ldcs(in + (r + u) * ch4 + q);
#pragma unroll
    for (int u = 0; u < QROWS - 1; ++u)
      if (r + u < r1) __stcs(out + (r + u) * ch4 + q, code4(v[u], st));
  }
}

// ---- the layer's three static quantisers (x per channel; B and C per group) as one launch.  Every
// tensor is a matrix of R rows; a block covers up to 128 float4 columns and, where a row is narrower
// than that, several rows per pass, so that a warp still reads 512 contiguous bytes.  The jobs of the
// narrow tensors come first in the grid: they are placed at once and finish under the wide one.
struct QuantJob {
  const float4* in; const float* scale; uint32_t* out;
  int ch4;          // float4 per row
  int tpr;          // threads per row (a power of two <= 128)
  int gx;           // column blocks per row
  int shift;        // step size of channel c = scale[c >> shift]
  int first_block;  // of this job in the grid
  int rows;         // rows per block
};
struct QuantJobs { QuantJob job[3]; i64 R; };

__device__ __forceinline__ void quant_block(const QuantJobs& a, const int blk) {
  const int jb = blk >= a.job[2].first_block ? 2 : blk >= a.job[1].first_block ? 1 : 0;
  const QuantJob& j = a.job[jb];
  const int rel = blk - j.first_block;
  const int bx = rel % j.gx, by = rel / j.gx;
  const int tr = threadIdx.x / j.tpr;          // row of this thread within a pass
  const int rpp = 128 / j.tpr;                 // rows per pass
  const int q = bx * j.tpr + (threadIdx.x & (j.tpr - 1));
  if (q >= j.ch4) return;
  float4 s;
  if (j.shift == 0) {
    s = __ldg(reinterpret_cast<const float4*>(j.scale) + q);
  } else {
    const float g = __ldg(j.scale + ((q * 4) >> j.shift));   // 4 consecutive channels share a group
    s = make_float4(g, g, g, g);
  }
  const Step4 st = step4(s);
  const i64 r0 = (i64)by * j.rows + tr;
  const i64 r1 = (i64)(by + 1) * j.rows < a.R ? (i64)(by + 1) * j.rows : a.R;
  if (r0 >= r1) return;
  // (the launcher keeps every tensor below 2^31 float4, so 32-bit element indices do)
  const uint32_t stride = (uint32_t)(rpp * j.ch4);   // float4 (and code words) between two passes
  uint32_t e = (uint32_t)r0 * (uint32_t)j.ch4 + (uint32_t)q;
  int left = (int)((r1 - r0 + rpp - 1) / rpp);       // passes this thread takes
  const float4* __restrict__ in = j.in;
  uint32_t* __restrict__ out = j.out;
  for (; left >= QROWS; left -= QROWS, e += QROWS * stride) {
    float4 v[QROWS];
#pragma unroll
    for (int u = 0; u < QROWS; ++u) v[u] = __ldcs(in + (e + u * stride));
    if (st.usable) {
#pragma unroll
      for (int u = 0; u < QROWS; ++u) out[e + u * stride] = code4(v[u], st);
    } else {
#pragma unroll 1
      for (int u = 0; u < QROWS; ++u) out[e + u * stride] = code4_by_division(in[e + u * stride], s);
    }
  }
  // (a layer's token count is a multiple of 64, which leaves no rest; the short form keeps the registers from spilling)
  for (; left > 0; --left, e += stride) out[e] = code4_by_division(__ldcs(in + e), s);
}

__global__ void __launch_bounds__(128, 8) quant_jobs(const QuantJobs a) {
  pdl_launch_dependents();
  // Programmatic dependent launch, right behind ChunkCumsum of the same layer, which waits for ITS predecessor before
  // it lets this kernel be scheduled, and whose outputs this kernel does not touch: the blocks start at once and work
  // beside it.  The wait stands at the end of the grid's last block (one waiting block is enough, and a
  // wait in every block would keep the early ones resident until ChunkCumsum has finished): it keeps
  // "this kernel complete" implying "ChunkCumsum complete" for the state kernel that follows, and by then
  // it returns at once.
  quant_block(a, (int)blockIdx.x);
  if (blockIdx.x == gridDim.x - 1) pdl_wait();
}

// ---- ChunkCumsum and the three quantisers of a layer as one launch: the first ncum blocks take four heads of a chunk each
// (hblocks blocks to a chunk).  See launch_lead for where it is taken.
template <int TPL>
__global__ void __launch_bounds__(128, 8) lead_kernel(const QuantJobs a, const cumsum::Args c, int ncum, int hblocks) {
  __shared__ __align__(16) float dts[4 * (32 * TPL + 4)];
  pdl_wait();
  pdl_launch_dependents();
  const int blk = (int)blockIdx.x;
  if (blk >= ncum) {
    quant_block(a, blk - ncum);
    return;
  }
  if (c.status && blk == 0 && threadIdx.x == 0) *c.status = 0;
  const int bk = blk / hblocks;
  cumsum::chunk_of_heads<TPL, false>(dts, 4, (blk - bk * hblocks) * 4, bk % c.d.c, bk / c.d.c, c);
}

// ---- quantise, I % 4 == 0: 4 consecutive elements share a channel
template <bool FIX>
__global__ void __launch_bounds__(QT) quant_inner(const float4* __restrict__ in, float* scale,
                                                  uint32_t* __restrict__ out, uint32_t n4,
                                                  uint32_t I4, uint32_t Ch) {
  pdl_launch_dependents();
  pdl_wait();
  uint32_t base = blockIdx.x * (QT * QUNROLL) + threadIdx.x;
#pragma unroll
  for (int u = 0; u < QUNROLL; ++u) {
    uint32_t e = base + u * QT;
    if (e < n4) {
      float4 v = __ldcs(in + e);
      const uint32_t ch = (e / I4) % Ch;
      float al = scale[ch];
      if (FIX && al == 0.f) {
        al = 1.f;
        if (e < I4 * Ch) scale[ch] = al;   // the first row
      }
      const float4 a4 = make_float4(al, al, al, al);
      const Step4 st = step4(a4);
      out[e] = st.usable ? code4(v, st) : code4_by_division(v, a4);
    }
  }
}

// ---- absmax, I == 1.  A thread owns 4 channels and every fourth row of the block's, with AROWS loads in flight; the four
// threads of a channel meet in shared memory, so that a block of many rows leaves one atomic per channel (an atomic per thread of
// 24 rows: 171 on each of 5120 addresses at 4096 rows; the calibration of 2 x 2048 x 80 heads 91.5 against 88.0 us, of 5 x 2304 x 16
// 105.3 against 84.3, calls in a row; this kernel alone at 65536 rows x 64 channels 53 against 19, at 16384 x 5120 120.8 against
// 115.5).  The loads
// leave their lines in L2 for the quantiser that follows.
constexpr int AROWS = 4, AGROUPS = 4;
__global__ void __launch_bounds__(128 * AGROUPS, 3) absmax_ch_fastest(const float4* __restrict__ in,
                                                                      uint32_t* __restrict__ bits, i64 R, int ch4,
                                                                      int rows_per_block) {
  __shared__ float4 best[AGROUPS - 1][128];
  pdl_launch_dependents();
  pdl_wait();
  const int t = threadIdx.x & 127, g = threadIdx.x >> 7;
  const int q = blockIdx.x * 128 + t;
  const i64 r0 = (i64)blockIdx.y * rows_per_block;
  const i64 r1 = r0 + rows_per_block < R ? r0 + rows_per_block : R;
  float4 m = make_float4(0.f, 0.f, 0.f, 0.f);
  auto take = [&](const float4& v) {
    m.x = fmaxf(m.x, fabsf(v.x)); m.y = fmaxf(m.y, fabsf(v.y));
    m.z = fmaxf(m.z, fabsf(v.z)); m.w = fmaxf(m.w, fabsf(v.w));
  };
  if (q < ch4) {
    i64 r = r0 + g;
    for (; r + (AROWS - 1) * AGROUPS < r1; r += AROWS * AGROUPS) {
      float4 v[AROWS];
#pragma unroll
      for (int u = 0; u < AROWS; ++u) v[u] = __ldg(in + (r + u * AGROUPS) * ch4 + q);
#pragma unroll
      for (int u = 0; u < AROWS; ++u) take(v[u]);
    }
    for (; r < r1; r += AGROUPS) take(__ldg(in + r * ch4 + q));
  }
  if (g > 0) best[g - 1][t] = m;
  __syncthreads();
  if (g > 0 || q >= ch4) return;
#pragma unroll
  for (int k = 0; k < AGROUPS - 1; ++k) take(best[k][t]);
  // step size of this partial maximum: fdiv by a positive constant is monotone, so the
  // maximum of the step sizes is the step size of the maximum
  atomicMax(bits + 4 * q + 0, __float_as_uint(__fdiv_rn(m.x, 127.0f)));
  atomicMax(bits + 4 * q + 1, __float_as_uint(__fdiv_rn(m.y, 127.0f)));
  atomicMax(bits + 4 * q + 2, __float_as_uint(__fdiv_rn(m.z, 127.0f)));
  atomicMax(bits + 4 * q + 3, __float_as_uint(__fdiv_rn(m.w, 127.0f)));
}

// ---- absmax, I % 4 == 0.  Block (x = row split, y = channel) reduces its rows of one channel.
__global__ void __launch_bounds__(QT) absmax_inner(const float4* __restrict__ in,
                                                   uint32_t* __restrict__ bits, i64 R, int Ch, int I4,
                                                   int rows_per_block) {
  __shared__ float red[QT / 32];
  pdl_launch_dependents();
  pdl_wait();
  int ch = blockIdx.y;
  i64 r0 = (i64)blockIdx.x * rows_per_block;
  i64 r1 = r0 + rows_per_block < R ? r0 + rows_per_block : R;
  i64 cnt = (r1 - r0) * I4;
  float m = 0.f;
  for (i64 e = threadIdx.x; e < cnt; e += QT) {
    i64 r = r0 + e / I4;
    int i = (int)(e % I4);
    float4 v = __ldg(in + (r * Ch + ch) * I4 + i);
    m = fmaxf(fmaxf(fmaxf(m, fabsf(v.x)), fmaxf(fabsf(v.y), fabsf(v.z))), fabsf(v.w));
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
#pragma unroll
    for (int w = 1; w < QT / 32; ++w) m = fmaxf(m, red[w]);
    atomicMax(bits + ch, __float_as_uint(__fdiv_rn(m, 127.0f)));
  }
}

// ---- calibrate mode in one launch: a cluster of eight CTAs holds all rows of a column block (I == 1: 8 float4 wide) or of a channel
// (I % 4 == 0) in shared memory, its CTAs exchange their largest magnitudes, and the codes are formed from shared memory: a tensor is read
// once, in one launch instead of three (clear, absmax, codes).  It pays where the whole grid is resident at once and no CTA has much to
// hold; otherwise the three launches, which overlap, use the memory better.  ssdi8_quantize_act, us, three launches / one: 4096 rows
// x 512 channels 12.6 / 7.4, 4096 x 1024 13.9 / 8.0, 512 x 512 7.2 / 4.2, 12800 x 512 25.2 / 19.2, but 12800 x 1024 25.2 / 30.4, 4096 x 5120 27.5 / 28.9,
// 8192 x 5120 55 / 84; channels of 128 elements: 256 rows x 1 7.6 / 3.3, 1024 x 1 7.2 / 5.1, 1024 x 8 9.2 / 6.4, 1024 x 32 12.6 / 7.9, but 2048 x 1
// 7.4 / 8.7, 4096 x 1 9.1 / 14.4.
constexpr int kCluster = 8, kHeldRows = 1600;   // CTAs; rows of a column block that one of them holds at most (200 KB)
// the step size that the three launches leave: 1 where the quotient is 0, as it also is for magnitudes below 63.5 of the smallest number
__device__ __forceinline__ float step_of_channel(float m) {
  const float al = __fdiv_rn(m, 127.0f);
  return al == 0.f ? 1.f : al;
}
__device__ __forceinline__ float remote_float(const float* own, int rank) {   // that of another CTA of the cluster
  uint32_t a = (uint32_t)__cvta_generic_to_shared(own);
  float v;
  asm volatile("mapa.shared::cluster.u32 %0, %0, %1;" : "+r"(a) : "r"(rank));
  asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ void copy16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void copies_done() { asm volatile("cp.async.wait_all;" ::: "memory"); }

__global__ void __cluster_dims__(kCluster, 1, 1) __launch_bounds__(QT)
calibrate_ch_fastest(const float4* __restrict__ in, float* __restrict__ scale, uint32_t* __restrict__ out, i64 R, int ch4, int rows) {
  extern __shared__ __align__(16) float4 tile[];   // [rows][8]; a thread reads what it has copied itself
  __shared__ float part[QT / 32][32], mine[32], step[32];
  pdl_launch_dependents();
  pdl_wait();
  const int tid = threadIdx.x, j = tid & 7, rank = blockIdx.x;   // (the grid is one cluster wide)
  const int q = blockIdx.y * 8 + j;
  const i64 r0 = (i64)rank * rows;
  const int n = (int)(q >= ch4 || r0 >= R ? 0 : R - r0 < rows ? R - r0 : rows);
  const float4* src = in + r0 * ch4 + q;
  for (int r = tid >> 3; r < n; r += QT / 8) copy16(tile + r * 8 + j, src + (i64)r * ch4);
  copies_done();
  float4 m = make_float4(0.f, 0.f, 0.f, 0.f);
  for (int r = tid >> 3; r < n; r += QT / 8) {
    const float4 v = tile[r * 8 + j];
    m.x = fmaxf(m.x, fabsf(v.x)); m.y = fmaxf(m.y, fabsf(v.y));
    m.z = fmaxf(m.z, fabsf(v.z)); m.w = fmaxf(m.w, fabsf(v.w));
  }
#pragma unroll
  for (int o = 8; o < 32; o <<= 1) {
    m.x = fmaxf(m.x, __shfl_xor_sync(0xffffffffu, m.x, o)); m.y = fmaxf(m.y, __shfl_xor_sync(0xffffffffu, m.y, o));
    m.z = fmaxf(m.z, __shfl_xor_sync(0xffffffffu, m.z, o)); m.w = fmaxf(m.w, __shfl_xor_sync(0xffffffffu, m.w, o));
  }
  if ((tid & 31) < 8) *reinterpret_cast<float4*>(&part[tid >> 5][4 * j]) = m;
  __syncthreads();
  if (tid < 32) {
    float a = part[0][tid];
#pragma unroll
    for (int w = 1; w < QT / 32; ++w) a = fmaxf(a, part[w][tid]);
    mine[tid] = a;
  }
  cluster_sync();
  if (tid < 32) {
    float a = 0.f;
#pragma unroll
    for (int c = 0; c < kCluster; ++c) a = fmaxf(a, remote_float(&mine[tid], c));
    const float al = step_of_channel(a);
    step[tid] = al;
    if (rank == 0 && blockIdx.y * 32 + tid < ch4 * 4) scale[blockIdx.y * 32 + tid] = al;
  }
  __syncthreads();
  cluster_arrive();   // (this CTA has read the others' maxima)
  const float4 a4 = *reinterpret_cast<const float4*>(&step[4 * j]);
  const Step4 st = step4(a4);
  uint32_t* dst = out + r0 * ch4 + q;
  for (int r = tid >> 3; r < n; r += QT / 8)
    __stcs(dst + (i64)r * ch4, st.usable ? code4(tile[r * 8 + j], st) : code4_by_division(tile[r * 8 + j], a4));
  cluster_wait();
}

constexpr int kInnerThreads = 1024, kInnerHeld = 8;   // threads of a CTA, float4 of each at most
__global__ void __cluster_dims__(kCluster, 1, 1) __launch_bounds__(kInnerThreads)
calibrate_inner(const float4* __restrict__ in, float* __restrict__ scale, uint32_t* __restrict__ out, int R, int Ch, int I4, int rows) {
  extern __shared__ __align__(16) float4 tile[];   // [<= kInnerHeld][kInnerThreads]; a thread reads what it has copied itself
  __shared__ float part[kInnerThreads / 32], mine, step;
  pdl_launch_dependents();
  pdl_wait();
  const int tid = threadIdx.x, rank = blockIdx.x, ch = blockIdx.y;
  const int r0 = rank * rows, r1 = min(R, r0 + rows);
  // element tid + u kInnerThreads of the CTA's rows of this channel is float4 i of row r
  const int dr = kInnerThreads / I4, di = kInnerThreads % I4;
  auto walk = [&](auto&& f) {
    int r = r0 + tid / I4, i = tid % I4;
    for (int u = 0; r < r1; ++u) {
      f(u, ((i64)r * Ch + ch) * I4 + i);
      r += dr;
      i += di;
      if (i >= I4) {
        i -= I4;
        ++r;
      }
    }
  };
  walk([&](int u, i64 e) { copy16(tile + u * kInnerThreads + tid, in + e); });
  copies_done();
  float m = 0.f;
  walk([&](int u, i64) {
    const float4 v = tile[u * kInnerThreads + tid];
    m = fmaxf(fmaxf(fmaxf(m, fabsf(v.x)), fmaxf(fabsf(v.y), fabsf(v.z))), fabsf(v.w));
  });
  auto largest = [](float v) { return __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(v))); };   // v >= 0
  m = largest(m);
  if ((tid & 31) == 0) part[tid >> 5] = m;
  __syncthreads();
  if (tid < 32) {
    m = largest(part[tid]);
    if (tid == 0) mine = m;
  }
  cluster_sync();
  if (tid < 32) {
    m = largest(tid < kCluster ? remote_float(&mine, tid) : 0.f);
    if (tid == 0) {
      step = step_of_channel(m);
      if (rank == 0) scale[ch] = step;
    }
  }
  __syncthreads();
  cluster_arrive();
  const float al = step;
  const float4 a4 = make_float4(al, al, al, al);
  const Step4 st = step4(a4);
  walk([&](int u, i64 e) {
    const float4 v = tile[u * kInnerThreads + tid];
    out[e] = st.usable ? code4(v, st) : code4_by_division(v, a4);
  });
  cluster_wait();
}

}  // namespace

ssdi8_status_t launch_quantize(const float* in, i64 R, i64 Ch, i64 I, float* scale, int mode,
                               int8_t* out, cudaStream_t st) {
  const i64 n4 = R * Ch * I / 4;
  if (n4 == 0) return SSDI8_OK;
  uint32_t* bits = reinterpret_cast<uint32_t*>(scale);
  ssdi8_status_t ls;
  if (mode == 1) {
    const int sms = sm_count();
    if (sms == 0) return SSDI8_ERR_CUDA;
    const i64 rows = (R + kCluster - 1) / kCluster, held = (rows * (I / 4) + kInnerThreads - 1) / kInnerThreads;
    const i64 per_sm = rows <= kHeldRows ? (224 * 1024) / (rows * 128 + 4 * 1024) : 0;
    if (I == 1 && 10 * (Ch / 4) <= 9 * sms * (per_sm < 4 ? per_sm : 4)) {
      const int ch4 = (int)(Ch / 4);
      return launch_sized(calibrate_ch_fastest, dim3(kCluster, (unsigned)((ch4 + 7) / 8)), dim3(QT), (size_t)rows * 128, (size_t)kHeldRows * 128,
                          -1, false, st, reinterpret_cast<const float4*>(in), scale, reinterpret_cast<uint32_t*>(out), R, ch4, (int)rows);
    }
    if (I > 1 && (held <= 4 ? kCluster * Ch <= 2 * sms : held <= kInnerHeld && Ch >= 4 && kCluster * Ch <= sms))
      return launch_sized(calibrate_inner, dim3(kCluster, (unsigned)Ch), dim3(kInnerThreads), (size_t)held * kInnerThreads * 16,
                          (size_t)kInnerHeld * kInnerThreads * 16, -1, false, st, reinterpret_cast<const float4*>(in), scale,
                          reinterpret_cast<uint32_t*>(out), (int)R, (int)Ch, (int)(I / 4), (int)rows);
  }
  if (mode == 1 || mode == 2) {
    if (mode == 1 && (ls = launch_clear_words(scale, Ch, st)) != SSDI8_OK) return ls;
    if (I == 1) {
      int ch4 = (int)(Ch / 4);
      int gx = (ch4 + 127) / 128;
      // one wave of blocks, each with as many rows as that leaves it (at least a few rounds of loads); where the columns alone
      // are more than half a wave, several waves, the last of which is a small part (128 rows x 230400 channels 44.0 us as
      // one block per 512 channels, 39.8 as six; 1024 rows 355 and 325)
      const i64 want = gx > (148 * 3) / 2 ? 6 : (148 * 3) / gx;
      i64 rows = (R + want - 1) / want;
      if (rows < 2 * AROWS * AGROUPS) rows = 2 * AROWS * AGROUPS;
      rows = (rows + AROWS * AGROUPS - 1) / (AROWS * AGROUPS) * (AROWS * AGROUPS);
      int gy = (int)((R + rows - 1) / rows);
      ls = launch_configured(absmax_ch_fastest, dim3(gx, gy), dim3(128 * AGROUPS), 0, kStreamCarveout, false, st,
                             reinterpret_cast<const float4*>(in), bits, R, ch4, (int)rows);
    } else {
      int I4 = (int)(I / 4);
      i64 want = (148 * 8 + Ch - 1) / Ch;
      i64 rows = (R + want - 1) / want;
      i64 min_rows = (QT * 4 + I4 - 1) / I4;
      if (rows < min_rows) rows = min_rows;
      int gx = (int)((R + rows - 1) / rows);
      // (no carve-out asked for, here and for the codes: a tensor this narrow, B or C, follows x, whose clusters hold their rows in shared memory, and
      // an SM that changes its split first has to run empty.  Calibration calls of 2048 tokens x 24 heads 50.2 -> 45.0 us, 1280 x 8 43.6 -> 38.5)
      ls = launch_configured(absmax_inner, dim3(gx, (unsigned)Ch), dim3(QT), 0, -1, false, st,
                             reinterpret_cast<const float4*>(in), bits, R, (int)Ch, I4, (int)rows);
    }
    if (ls != SSDI8_OK) return ls;
  }
  if (!out) return SSDI8_OK;
  const bool fix = mode == 1;   // an all-zero channel: alpha = 1
  if (I == 1) {
    const int ch4 = (int)(Ch / 4);
    const int gx = (ch4 + 127) / 128;
    // slabs of rows: enough blocks to fill the machine several times over, at least 16 rows each (at least 32 left 2560 to 5120
    // channels of a few thousand rows on one wave and a bit: calibration of 5 x 2304 x 16 heads 84.3 against 79.1 us, 2 x 2048 x
    // 80 88.0 against 86.4, calls in a row)
    i64 want = (148 * 32 + gx - 1) / gx;
    i64 rows = (R + want - 1) / want;
    if (rows < 16) rows = 16;
    rows = (rows + QROWS - 1) / QROWS * QROWS;
    const int gy = (int)((R + rows - 1) / rows);
    return launch_configured(fix ? quant_ch_fastest<true> : quant_ch_fastest<false>, dim3(gx, gy), dim3(128), 0,
                             kStreamCarveout, false, st, reinterpret_cast<const float4*>(in),
                             reinterpret_cast<float4*>(scale), reinterpret_cast<uint32_t*>(out), R, ch4, (int)rows);
  }
  const unsigned grid = (unsigned)((n4 + QT * QUNROLL - 1) / (QT * QUNROLL));
  return launch_configured(fix ? quant_inner<true> : quant_inner<false>, dim3(grid), dim3(QT), 0, -1, false, st,
                           reinterpret_cast<const float4*>(in), scale, reinterpret_cast<uint32_t*>(out), (uint32_t)n4,
                           (uint32_t)(I / 4), (uint32_t)Ch);
}

namespace {

// the jobs of a layer; returns the number of blocks, 0 where an index would not fit
int make_jobs(QuantJobs& a, const float* x, const float* B, const float* C, i64 T_, int D, int G, int N, const float* s_x,
              const float* s_B, const float* s_C, int8_t* xq, int8_t* Bq, int8_t* Cq) {
  if (T_ * D / 4 >= ((i64)1 << 31) || T_ * G * N / 4 >= ((i64)1 << 31)) return 0;
  a.R = T_;
  int shift = 0;
  while ((1 << shift) < N) ++shift;   // N is a power of two here (the caller checks)
  auto fill = [&](QuantJob& j, const float* in, const float* sc, int8_t* out, int width, int sh, int first) {
    j.in = reinterpret_cast<const float4*>(in);
    j.scale = sc;
    j.out = reinterpret_cast<uint32_t*>(out);
    j.ch4 = width / 4;
    j.tpr = 128;
    while (j.tpr / 2 >= j.ch4 && j.tpr > 1) j.tpr /= 2;
    j.gx = (j.ch4 + j.tpr - 1) / j.tpr;
    j.shift = sh;
    j.first_block = first;
    // short slabs: blocks that live a few microseconds each, so that a kernel running beside this one finds
    // free slots all the time (a slab is at least one full round of QROWS passes)
    j.rows = QROWS * (128 / j.tpr) < 16 ? 16 : QROWS * (128 / j.tpr);
    return first + j.gx * (int)((T_ + j.rows - 1) / j.rows);
  };
  int nb = fill(a.job[0], B, s_B, Bq, G * N, shift, 0);
  nb = fill(a.job[1], C, s_C, Cq, G * N, shift, nb);
  return fill(a.job[2], x, s_x, xq, D, 0, nb);
}

}  // namespace

ssdi8_status_t launch_lead(const Dims& d, const LayerInputs& in, const float* dt, const float* A, float* pack, float* gamma,
                           const float* s_x, const float* s_B, const float* s_C, int8_t* xq, int8_t* Bq, int8_t* Cq,
                           int32_t* clear_status, cudaStream_t st) {
  QuantJobs a;
  const i64 T = (i64)d.b * d.L;
  const int nb = make_jobs(a, in.x, in.B, in.C, T, d.H * d.P, d.G, d.N, s_x, s_B, s_C, xq, Bq, Cq);
  if (nb == 0) return SSDI8_ERR_UNSUPPORTED;
  const int hblocks = (d.H + 3) / 4;
  const i64 ncum = (i64)hblocks * d.c * d.b;
  // One launch or two, by tokens x heads.  One saves a launch, which is what the smallest layers consist of, and where the blocks of
  // both fill the device a few times over ChunkCumsum's run in the gaps of the quantisers'; in between ChunkCumsum is on the
  // critical path and its own launch has the shorter chain (more warps a block, more registers), and with many waves the
  // quantisers alone keep the memory busier.  Of the smallest, one or two chunks and chunks of 256 have two: there the chain of
  // ChunkCumsum is what the state kernel waits for.  Layer calls in a row, us, two launches / one (G = 1 where
  // not stated):
  //   smallest, chunks of 64:  256 tokens x 4 heads 15.8 / 15.1, 512 x 4 17.0 / 16.6, 1024 x 4 18.1 / 18.2; one chunk x 6 13.3 / 13.7;
  //     1024 x 8 19.7 / 21.3.  Of 128: 512 x 4 16.8 / 16.4, 256 x 4 15.1 / 15.3, 1024 x 4 18.4 / 18.2, 512 x 24 19.6 / 20.0.  Of 256:
  //     256 x 4 17.0 / 18.0, 1024 x 4 18.4 / 18.5, 256 x 16 18.0 / 19.2
  //   128 to 512 thousand, chunks of 64:  2 x 2688 x 38 96.4 / 96.0, 5 x 6784 x 8 (G 4) 208.2 / 206.9, 4 x 3392 x 28 195.6 / 181.8, 8 x 1024 x
  //     80 (beyond) 190.3 / 190.3, but 3 x 1408 x 50 (N 128) 100.3 / 103.6.  Of 128: 7 x 2816 x 9 67.6 / 66.8, 3 x 5376 x 16 (G 8) 143.2 / 142.1,
  //     3 x 1408 x 50 72.2 / 70.8, 8 x 1024 x 80 (beyond) 140.2 / 140.8.  Of 256: 2 x 2048 x 40 51.7 / 51.3, 4 x 8192 x 7 73.8 / 72.8, 8 x 256 x 64
  //     (G 8) 49.2 / 47.6, 2 x 8192 x 16 (G 4) 97.1 / 95.8, but 6 x 1536 x 20 60.0 / 61.5, 8 x 1024 x 20 53.9 / 54.6, 2 x 8192 x 8 with INT8 states
  //     68.6 / 74.8; 8 x 1024 x 80 (beyond) 126.6 / 127.6.  In the mean of 68 drawn sizes one launch is 0.9 % faster, 63 of them gain.
  const i64 th = T * d.H;
  if ((d.Q <= 128 && d.c >= 3 && th <= 4096) || (th >= 128 * 1024 && th <= 512 * 1024)) {
    const cumsum::Args c = {dt, A, pack, gamma, nullptr, nullptr, clear_status, d};
    auto launch = [&](auto kernel) -> ssdi8_status_t {
      return launch_configured(kernel, dim3((unsigned)(nb + ncum)), dim3(128), 0, kStreamCarveout, false, st, a, c, (int)ncum, hblocks);
    };
    return d.Q == 256 ? launch(lead_kernel<8>) : d.Q == 128 ? launch(lead_kernel<4>) : launch(lead_kernel<2>);
  }
  // ChunkCumsum (it reads dt and A only) and the quantisers need nothing of each other.  ChunkCumsum goes
  // first and lets its successor be scheduled once its own wait for the work ahead of the layer is over;
  // the quantisers' launch then starts without a wait and runs beside it, with the wait at the end of its
  // last block (see quant_jobs), so that the state kernel, which waits for the quantisers' launch, has
  // ChunkCumsum complete as well.  One stream, no events.  (ChunkCumsum on a side stream instead: 0.293 against 0.286 ms at
  // batch 8 x 2048 x 80 heads.)
  const ssdi8_status_t s = launch_cumsum(d, dt, A, pack, gamma, nullptr, st, nullptr, false, clear_status);
  if (s != SSDI8_OK) return s;
  return launch_configured(quant_jobs, dim3((unsigned)nb), dim3(128), 0, kStreamCarveout, false, st, a);
}

}  // namespace ssdi8
