// ChunkState + StatePassing fused, chunk-sequential per (batch, head): the fp32 chunk-local
// state never goes to HBM.  For chunk k = 0 .. c-1 of one (b, h):
//   Xs_q[i,p]   = rne(fmul(fmul(float(xq[i,p]), fdiv(s_x, s_xs)), LUT_state[i]))       (Eq. 3)
//   acc_st[n,p] = sum_i Bq[i,n] Xs_q[i,p]            INT8 MMA over the chunk's tokens, INT32 in TMEM
//   loc[p,n]    = fmul(float(acc_st), fmul(s_xs[h,p], s_B[g]))                         (Eq. 4 rescale)
//   hq[k][p,n]  = rne(fmul(S[p,n], fdiv(1, s_h[h,p])))     (state entering chunk k, int8 for ChunkScan1)
//   S[p,n]      = fmaf(Gamma_k, S[p,n], loc[p,n])                                      (Eq. 6)
// and final_state = S after the last chunk.  The accumulator has the state index n on the TMEM lanes, so thread
// (lane n) works on S[., n] of its 32 channels p; the running state is kept in tensor memory beside the
// accumulator (64 more columns, read and written 8 columns at a time), which leaves the threads with few
// registers so that three CTAs fit an SM: the kernel is a chain of short dependent steps per chunk, and what fills an SM is other
// CTAs' chains.  Three warps re-quantise the xq rows up to two chunks ahead, a fourth issues the MMAs
// and requests the tiles by TMA: xq double-buffered across chunks, Bq single-buffered (requested
// when the MMAs of the chunk before have finished); hq leaves through
// a shared-memory tile and one TMA store per chunk.  Same arithmetic, operation for operation,
// as the separate kernels (chunk_state.cu, state_passing.cu).
// I8S = true selects the paper's own state format (Section 4.2, Eq. 4 and Eq. 7): the state is an
// int8 code with the one per-(H,P) scale s_h, the chunk-local state goes INT32 -> INT8 in
// registers, and the recurrence is integer with a fixed-point decay:
//   locq = rne(fmul(float(acc_st), fdiv(fmul(s_xs, s_B), s_h)));  Gq = rne(fmul(Gamma_k, 128))
//   Sq   = sat(locq + ((Gq * Sq + 64) >> 7));  hq[k] = Sq before the update;  final = fmul(float(Sq), s_h)
// CAL = true is the calibration pass: no codes are formed; the largest |S| of every channel over init_state and
// every S_k goes into absmax_h (binary32 bits, one atomic per channel and CTA).  (Against separate ChunkState and
// StatePassing passes over 42 MB of chunk-local states in HBM, 28 + 7 us at batch 2 x 2048 x 80 heads, this takes 22.)
#include "kernels.h"
#include "sm100.cuh"

namespace ssdi8 {
namespace {

using namespace sm100;

struct FusedArgs {
  const float* s_x; const float* s_xs; const float* s_B; const float* s_h; const float* pack;
  const float* gamma; const float* init; float* final_state;
  float* tap_loc; float* tap_prev; int8_t* tap_Xsq; int32_t* tap_acc; int32_t* status; uint32_t* absmax_h; float* s_xs_out;
  Dims d;
  int n_full;  // CTAs below this index own a whole (batch, head); the rest own a quarter (16 channels) of one
};

constexpr int kStateThreads = 256;   // warps 0-7: running state, hq and its TMA stores
constexpr int kQuantThreads = 128;   // warps 8-10: Q(X_scaled), up to two chunks ahead; warp 11: MMA issue, TMA loads
constexpr int kThreads = kStateThreads + kQuantThreads;
constexpr int kRowWarps = 3;
constexpr uint32_t XSTAGE = 16384;                // xq rows [Q][64] of one chunk
constexpr uint32_t OFF_X = 0;                     // two stages
constexpr uint32_t OFF_B = 2 * XSTAGE;            // Bq rows [Q][N] of one chunk (single buffer)
constexpr uint32_t OFF_HQ = OFF_B + 32768;        // [64 p][N] int8 staging of hq
constexpr uint32_t OFF_LUT = OFF_HQ + 8192;       // 2 x [256] floats
constexpr uint32_t OFF_COL = OFF_LUT + 2048;      // [64] loc scale, [64] 1 / s_h, [64] s_x / s_xs
constexpr uint32_t OFF_BAR = OFF_COL + 768;
constexpr uint32_t SMEM_BYTES = OFF_BAR + 64;     // 76 608 bytes: three CTAs per SM
constexpr uint32_t kTmemCols = 128;               // accumulator in columns 0..63, running state in 64..127

enum { B_XFULL = 0, B_BFULL = 2, B_MMA = 3, B_ACC_FREE = 4, B_COUNT = 5 };

__device__ __forceinline__ void named_bar(int id, int nthreads) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(nthreads) : "memory");
}
__device__ __forceinline__ void named_bar_arrive(int id, int nthreads) {
  asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(nthreads) : "memory");
}

// TAPS: any of the intermediate-tensor taps is requested (tests); the production instance carries no tap code
// NCQ: 16-channel chunks of the head this CTA owns (4 = the whole head, 1 = one quarter)
template <bool I8S, bool TAPS, bool CAL, int NCQ>
__device__ __forceinline__ void fused_body(const CUtensorMap& tm_B, const CUtensorMap& tm_x, const CUtensorMap& tm_hq,
                                           const FusedArgs& a, const int unit, const int c0) {
  // (no padding for the 1024-byte alignment the swizzled tiles need: three CTAs fill the SM's shared
  // memory to the last kilobyte; the launcher checks that the kernel uses no static shared memory, so
  // the dynamic part starts at the window's base, and the kernel checks the address itself)
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  constexpr int ncq = NCQ;
  uint8_t* smem = smem_raw;
  if ((smem_u32(smem) & 1023u) != 0) {
    if (threadIdx.x == 0 && a.status) atomicExch(a.status, (int32_t)SSDI8_ERR_ALIGN);
    return;
  }
  const Dims& d = a.d;
  const int Q = d.Q, N = d.N, P = d.P;
  const int h = unit % d.H, b = unit / d.H;
  const int g = h / (d.H / d.G);
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;   // (the shuffle: uniform for the compiler)
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + OFF_BAR);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + B_COUNT);
  uint8_t* sHQ = smem + OFF_HQ;
  float* col_scale = reinterpret_cast<float*>(smem + OFF_COL);
  float* col_invh = col_scale + 64;
  float* col_rx = col_invh + 64;
  const i64 bh = (i64)b * d.H + h;
  const i64 unit0 = bh * d.c;

  // One warp: the slabs of 32 tokens named by m of the xq rows (with LUT_state of the chunk: a global
  // load there would sit on the re-quantisation group's critical path) or of the Bq rows of chunk k
  auto issue_x = [&](int k, uint32_t m) {
    const int s = k & 1;
    const int tok0 = (int)((i64)b * d.L + (i64)k * Q);
    if (elect_one()) {
      mbar_expect_tx(&bars[B_XFULL + s], (uint32_t)(__popc(m) * 32 * 64 + Q * 4));
      bulk_load(smem + OFF_LUT + s * 1024, a.pack + ((unit0 + k) * kPackRows + PACK_LUT) * Q, (uint32_t)(Q * 4),
                &bars[B_XFULL + s]);
#pragma unroll 1
      for (; m; m &= m - 1) {
        const int i0 = (__ffs((int)m) - 1) * 32;
        tma_load_3d(smem + OFF_X + s * XSTAGE + i0 * 64, &tm_x, &bars[B_XFULL + s], 0, h, tok0 + i0);
      }
    }
    __syncwarp();
  };
  auto issue_B = [&](int k, uint32_t m) {   // once the MMAs of chunk k - 1 have finished
    const int tok0 = (int)((i64)b * d.L + (i64)k * Q);
    if (elect_one()) {
      mbar_expect_tx(&bars[B_BFULL], (uint32_t)(__popc(m) * 32 * N));
#pragma unroll 1
      for (; m; m &= m - 1) {
        const int i0 = (__ffs((int)m) - 1) * 32;
        tma_load_3d(smem + OFF_B + i0 * N, &tm_B, &bars[B_BFULL], 0, g, tok0 + i0);
      }
    }
    __syncwarp();
  };

  constexpr int kLoadWarp = kStateThreads / 32 + kRowWarps;
  if (warp == kLoadWarp) {
    if (lane == 0) {
      mbar_init(&bars[B_XFULL], 1);
      mbar_init(&bars[B_XFULL + 1], 1);
      mbar_init(&bars[B_BFULL], 1);
      mbar_init(&bars[B_MMA], 1);
      mbar_init(&bars[B_ACC_FREE], kStateThreads / 32);
      fence_mbar_init();
      tma_prefetch_desc(&tm_B);
      tma_prefetch_desc(&tm_x);
      tma_prefetch_desc(&tm_hq);
    }
    __syncwarp();
  }
  if (warp == 1) tmem_alloc(tmem_slot, kTmemCols);
  pdl_wait();   // everything below reads global memory
  // (after the wait, not before it: ChunkBMM, launched next, reads and writes global memory without waiting
  // for this kernel, so it must not be scheduled before this kernel's predecessors have completed)
  pdl_launch_dependents();
  if (warp == kLoadWarp) {   // all slabs of the first chunk: its LUT_state would have to come first
    issue_x(0, (1u << (Q / 32)) - 1u);
    issue_B(0, (1u << (Q / 32)) - 1u);
  }
  auto step_xs = [&](int p) -> float {   // (the calibration pass is given the maxima of |X_scaled|)
    const float v = a.s_xs[h * P + p];
    return CAL ? step_of_max(__float_as_uint(v)) : v;
  };
  if (tid < 64) {
    const float sx = step_xs(tid), sxb = __fmul_rn(sx, a.s_B[g]);
    if (CAL && b == 0 && tid >= 16 * c0 && tid < 16 * (c0 + ncq)) a.s_xs_out[h * P + tid] = sx;
    if (CAL) {
      col_scale[tid] = sxb;
      col_invh[tid] = 0.f;               // running maximum of the channel
    } else {
      const float sh = a.s_h[h * P + tid];
      col_scale[tid] = I8S ? __fdiv_rn(sxb, sh) : sxb;
      col_invh[tid] = __fdiv_rn(1.0f, sh);
    }
  } else if (tid < 128) {
    col_rx[tid - 64] = __fdiv_rn(a.s_x[h * P + tid - 64], step_xs(tid - 64));
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  if (warp >= kStateThreads / 32) {
    // ------------------------------------------------------------ Q(X_scaled), one chunk ahead of the state warps
    const int qt = tid - kStateThreads;
    constexpr int lq = ncq == 4 ? 2 : 0;  // log2(chunks per row in this CTA's range)
    const int c = c0 + (qt & (ncq - 1));  // 16-byte chunk (16 channels) of every row this thread visits
    float rx[16];
#pragma unroll
    for (int e = 0; e < 16; ++e) rx[e] = col_rx[c * 16 + e];
    // Rows that re-quantise to zero (the sparsity Eq. 3 rests on: LUT_state decays towards the start
    // of a chunk).  fmul is monotone, so with rxm >= |rx| of every channel of this CTA's range,
    // fmul(fmul(127, rxm), |LUT_state[i]|) < 1/2 implies |fmul(fmul(x, rx), LUT_state[i])| < 1/2 for every
    // code x: row i of Q(X_scaled) is all zeros, exactly.  Such a row is stored as zeros without the
    // arithmetic, and a 32-token slab of such rows is left out altogether (no MMA).
    float rxm = 0.f;
#pragma unroll
    for (int e = 0; e < 16; ++e) rxm = fmaxf(rxm, fabsf(rx[e]));
    if (ncq == 4) rxm = fmaxf(rxm, __shfl_xor_sync(0xffffffffu, rxm, 1));
    if (ncq == 4) rxm = fmaxf(rxm, __shfl_xor_sync(0xffffffffu, rxm, 2));
    const float b127 = __fmul_rn(127.0f, rxm);
    // Three of the warps share the live rows of a chunk evenly, up to two chunks ahead; the fourth requests the tiles, the
    // live slabs of them only, and issues the MMAs.  The live slabs are the last ones of a chunk, often two or three: with
    // whole slabs dealt out by position the warp that had most of them was the time of a chunk, and with all of xq
    // and Bq loaded (48 KB per chunk and CTA) the loads of three CTAs took 1.4 us.  The row warps only arrive at
    // the barrier that releases the MMAs, one of two in turn: they are held back by the xq tile of the chunk after next,
    // which is requested when this chunk's MMAs have finished.  A row warp whose wait for a tile
    // has given up is no longer held back by it: from then on it only waits at the barrier, since one that is overrun never
    // fills, and nothing bounds that wait.  (An mbarrier in its place, with a bounded wait, costs 0.14 us per chunk of a lone chain:
    // 2 x 8192 tokens x 7 heads with INT8 states 66.8 -> 71.4 us.)
    // (Batch 8 x 2048 x 80 heads: 48.9 us with slabs dealt out by position, 41.0 this way, 38.7 with the first tiles requested
    // ahead of all other set-up and s_x / s_xs divided once per channel; 4 x 8192 x 128 151, 118, 115.)
    const int qw = warp - kStateThreads / 32, nsl = Q / 32;
    // live slabs of a chunk from its LUT_state: nsl consecutive tokens per lane, 32 / nsl lanes per slab.  A chunk
    // without a live slab opens the accumulator with its last one, all rows of it stored as zeros.
    struct Lut { float4 a, b; };
    auto lut_of_lane = [&](const float* l) -> Lut {
      Lut v = {make_float4(0.f, 0.f, 0.f, 0.f), make_float4(0.f, 0.f, 0.f, 0.f)};
      if (nsl == 2) {
        const float2 u = reinterpret_cast<const float2*>(l)[lane];
        v.a.x = u.x;
        v.a.y = u.y;
      } else {
        v.a = reinterpret_cast<const float4*>(l + lane * nsl)[0];
        if (nsl == 8) v.b = reinterpret_cast<const float4*>(l + lane * nsl)[1];
      }
      return v;
    };
    auto live_slabs = [&](const Lut& v) -> uint32_t {
      auto alive = [&](float l) { return !(__fmul_rn(b127, fabsf(l)) < 0.5f); };
      const bool any = alive(v.a.x) | alive(v.a.y) | alive(v.a.z) | alive(v.a.w) | alive(v.b.x) | alive(v.b.y) | alive(v.b.z) | alive(v.b.w);
      const uint32_t bal = __ballot_sync(0xffffffffu, any);
      const int lps = 32 / nsl;
      const uint32_t m = __ballot_sync(0xffffffffu, lane < nsl && ((bal >> ((lane * lps) & 31)) & ((1u << lps) - 1u)) != 0);
      return m ? m : 1u << (nsl - 1);
    };
    constexpr int kRowStep = 32 * kRowWarps >> lq;
    const float* const lut0 = a.pack + (unit0 * kPackRows + PACK_LUT) * Q;   // LUT_state of chunk 0; the next one kPackRows Q floats on
    const i64 lut_step = (i64)kPackRows * Q;
    if (qw == kRowWarps) {
      uint32_t cur = live_slabs(lut_of_lane(lut0)), next = 0;
      if (d.c > 1) {
        next = live_slabs(lut_of_lane(lut0 + lut_step));
        issue_x(1, next);
      }
      const uint32_t idesc = idesc_s8(N, 64, 1, 1);
#pragma unroll 1
      for (int k = 0; k < d.c; ++k) {
        Lut v = {};
        if (k + 2 < d.c) v = lut_of_lane(lut0 + (k + 2) * lut_step);     // (its latency under the waits)
        named_bar(2 + (k & 1), kQuantThreads);                           // the rows are re-quantised
        mbar_wait_inline<0>(&bars[B_ACC_FREE], (k & 1) ^ 1, a.status);   // the state warps have read the accumulator of chunk k-1
        mbar_wait_inline<0>(&bars[B_BFULL], k & 1, a.status);            // the chunk's Bq rows have landed
        tc_fence_after();
        const uint32_t sBa = smem_u32(smem + OFF_B), sXa = smem_u32(smem + OFF_X + (k & 1) * XSTAGE);
        if (elect_one()) {
#pragma unroll 1
          for (uint32_t m = cur; m; m &= m - 1) {
            const int sl = __ffs((int)m) - 1;
            mma_s8_ss(tmem, tile_desc(sBa + 32 * sl * N, (uint32_t)N), tile_desc(sXa + 32 * sl * 64, 64), idesc, m != cur);
          }
          mma_commit(&bars[B_MMA]);
        }
        __syncwarp();
        if (k + 1 < d.c) {
          mbar_wait_inline<0>(&bars[B_MMA], k & 1, a.status);   // the MMAs of chunk k have read the Bq buffer and its xq stage
          issue_B(k + 1, next);
          cur = next;
          if (k + 2 < d.c) {
            next = live_slabs(v);
            issue_x(k + 2, next);
          }
        }
      }
    } else {
    int k = 0;
#pragma unroll 1
    for (; k < d.c; ++k) {
      const int s = k & 1;
      uint8_t* sX = smem + OFF_X + s * XSTAGE;
      float* lut = reinterpret_cast<float*>(smem + OFF_LUT) + s * 256;
      const i64 tok0 = (i64)b * d.L + (i64)k * Q;
      if (__any_sync(0xffffffffu, !mbar_wait_inline<256>(&bars[B_XFULL + s], (k >> 1) & 1, a.status))) break;
      const uint32_t lm = live_slabs(lut_of_lane(lut));   // (every warp computes the same mask)
      const uint4 zero4 = make_uint4(0u, 0u, 0u, 0u);
      if (TAPS && a.tap_Xsq) {
        for (int i = qt >> lq; i < Q; i += kRowStep)
          if (!((lm >> (i >> 5)) & 1u)) *reinterpret_cast<uint4*>(a.tap_Xsq + ((tok0 + i) * d.H + h) * P + c * 16) = zero4;
      }
#pragma unroll 1
      for (int r = qt >> lq, m = (int)lm;; r += kRowStep) {   // r: row among the live ones
        for (; r >= 32; r -= 32) m &= m - 1;
        if (m == 0) break;
        const int i = (__ffs(m) - 1) * 32 + r;
        uint4* ptr = reinterpret_cast<uint4*>(sX + swz_off((uint32_t)i, (uint32_t)c, 64));
        const float l = lut[i];
        if (__fmul_rn(b127, fabsf(l)) < 0.5f) {
          *ptr = zero4;
          if (TAPS && a.tap_Xsq) *reinterpret_cast<uint4*>(a.tap_Xsq + ((tok0 + i) * d.H + h) * P + c * 16) = zero4;
          continue;
        }
        const uint4 w4 = *ptr;
        const uint32_t ww[4] = {w4.x ^ 0x80808080u, w4.y ^ 0x80808080u, w4.z ^ 0x80808080u, w4.w ^ 0x80808080u};
        const float2 l2 = make_float2(l, l);
        uint32_t o[4];
#pragma unroll
        for (int w = 0; w < 4; ++w) {
          uint32_t q4[4];
#pragma unroll
          for (int e = 0; e < 4; e += 2) {
            const float2 xf = __fadd2_rn(
                make_float2(__uint_as_float(__byte_perm(ww[w], 0x4B400000u, 0x7650u + e)),
                            __uint_as_float(__byte_perm(ww[w], 0x4B400000u, 0x7651u + e))),
                make_float2(-kMagicIn, -kMagicIn));
            const uint2 c2 = rne_clamp_bits2(__fmul2_rn(__fmul2_rn(xf, make_float2(rx[w * 4 + e], rx[w * 4 + e + 1])), l2));
            q4[e] = c2.x;
            q4[e + 1] = c2.y;
          }
          o[w] = pack4_bits(q4[0], q4[1], q4[2], q4[3]);
        }
        const uint4 v = make_uint4(o[0], o[1], o[2], o[3]);
        *ptr = v;
        if (TAPS && a.tap_Xsq) *reinterpret_cast<uint4*>(a.tap_Xsq + ((tok0 + i) * d.H + h) * P + c * 16) = v;
      }
      fence_async_smem();
      named_bar_arrive(2 + s, kQuantThreads);
    }
    for (; k < d.c; ++k) named_bar(2 + (k & 1), kQuantThreads);   // (a wait has given up)
    }
  } else {
    // ------------------------------------------------------------ state warps
    // M = 128: accumulator row n on TMEM lane n; M = 64: row n on lane (n % 16) + 32 (n / 16),
    // i.e. the first 16 lanes of each warp's quarter
    const int q = warp & 3, ch = warp >> 2;
    constexpr int npp = 8 * ncq;             // channels per thread
    const int cb = 16 * c0 + ch * npp;       // first channel of this thread
    const bool ok = (N == 128) || (lane < 16);
    const int n = (N == 128) ? q * 32 + lane : q * 16 + lane;
    // the running state S[p, n]: fp32, or (I8S) the integer code, in tensor-memory columns 64 + p of lane n
    const uint32_t tlane = tmem + ((uint32_t)(q * 32) << 16);
    const uint32_t tS = tlane + 64u + (uint32_t)cb;
    float smax[CAL ? 32 : 1];   // CAL: running maxima of |S[p, n]| over the chunks
#pragma unroll
    for (int p0 = 0; p0 < 32; p0 += 8) {
      if (p0 < npp) {
        int sv[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          const float v = (a.init && ok) ? a.init[(bh * P + cb + p0 + e) * N + n] : 0.f;
          sv[e] = I8S ? (int)(int8_t)(rne_clamp_bits(__fmul_rn(v, col_invh[(cb + p0 + e) & 63])) & 0xffu) : __float_as_int(v);
        }
        if (CAL) {
#pragma unroll
          for (int e = 0; e < 8; ++e) smax[CAL ? p0 + e : 0] = fmaxf(fabsf(__int_as_float(sv[e])), 0.f);   // (a NaN counts for nothing)
        }
        tmem_st8(tS + (uint32_t)p0, sv);
      }
    }
    tmem_st_wait();
#pragma unroll 1
    for (int k = 0; k < d.c; ++k) {
      const float gam = a.gamma[unit0 + k];
      if (tid < ncq && k > 0) tma_store_wait_read();  // last chunk's hq store has read the staging tile
      named_bar(1, kStateThreads);  // also: every state thread has read the accumulator of chunk k-1
      // ---- hq[k] = codes of the state entering this chunk (and the prev tap).  They are formed here, ahead
      // of the wait for the chunk's MMAs, from a second read of the state; forming them in the update pass of
      // the chunk before, while the new values are in registers, puts them behind that wait on the chain of
      // the chunk and was measured slower (0.0568 against 0.0536 ms at batch 8 x 2048 x 80 heads).
      if (!CAL) {
        const i64 obase = (((((i64)b * d.c + k) * d.H + h) * P) + cb) * N + n;
        // batches of 8: all loads of a batch before its byte stores (a byte store may alias anything,
        // so interleaving them would serialise the loop on shared-memory latency).  The tensor-memory
        // loads are warp-wide; lanes without a state row (N = 64) skip what follows them.
#pragma unroll
        for (int p0 = 0; p0 < 32; p0 += 8) {
          if (p0 < npp) {
            int sv[8];
            tmem_ld8(tS + (uint32_t)p0, sv);
            tmem_ld_wait();
            if (ok) {
              uint32_t code[8];
              // (cb is a multiple of 8: the eight reciprocals are two 16-byte loads)
              const float4 i0 = *reinterpret_cast<const float4*>(col_invh + cb + p0);
              const float4 i1 = *reinterpret_cast<const float4*>(col_invh + cb + p0 + 4);
              const float ih[8] = {i0.x, i0.y, i0.z, i0.w, i1.x, i1.y, i1.z, i1.w};
#pragma unroll
              for (int e = 0; e < 8; e += 2) {
                if (I8S) {
                  code[e] = (uint32_t)sv[e];
                  code[e + 1] = (uint32_t)sv[e + 1];
                } else {
                  const uint2 c2 = rne_clamp_bits2(__fmul2_rn(make_float2(__int_as_float(sv[e]), __int_as_float(sv[e + 1])),
                                                              make_float2(ih[e], ih[e + 1])));
                  code[e] = c2.x;
                  code[e + 1] = c2.y;
                }
              }
              uint8_t* hrow = sHQ + (cb + p0) * N + n;
#pragma unroll
              for (int e = 0; e < 8; ++e, hrow += N) *hrow = (uint8_t)code[e];
              if (TAPS && !I8S && a.tap_prev) {
#pragma unroll
                for (int e = 0; e < 8; ++e) a.tap_prev[obase + (i64)(p0 + e) * N] = __int_as_float(sv[e]);
              }
            }
          }
        }
      }
      fence_async_smem();
      // one warp polls for the MMAs of this chunk; the barrier passes their completion on to the others
      if (warp == 0) mbar_wait_inline<256>(&bars[B_MMA], k & 1, a.status);
      named_bar(1, kStateThreads);
      // ---- hq[k] leaves by TMA
      if (tid < ncq && !CAL) {
        const int j = c0 + tid;              // 16 channels (rows of hq) per store
        tma_store_2d(&tm_hq, sHQ + 16 * j * N, 0, (int)(((((i64)b * d.c + k) * d.H + h) * P) + 16 * j));
        tma_store_commit();
      }
      // ---- epilogue of the MMA: S = fmaf(Gamma_k, S, loc), 8 channels at a time
      tc_fence_after();
#pragma unroll
      for (int hf = 0; hf < 4; ++hf) {       // 8 channels at a time
        if (hf < ncq) {
        int acc[8], sv[8];
        tmem_ld8(tlane + (uint32_t)(cb + hf * 8), acc);
        tmem_ld8(tS + (uint32_t)(hf * 8), sv);
        tmem_ld_wait();
        if (ok) {
          const i64 obase = (((((i64)b * d.c + k) * d.H + h) * P) + cb + hf * 8) * N + n;
          const float4 c0v = *reinterpret_cast<const float4*>(col_scale + cb + hf * 8);
          const float4 c1v = *reinterpret_cast<const float4*>(col_scale + cb + hf * 8 + 4);
          const float cscale[8] = {c0v.x, c0v.y, c0v.z, c0v.w, c1v.x, c1v.y, c1v.z, c1v.w};
#pragma unroll
          for (int e = 0; e < 8; e += 2) {
            const float2 af = __fadd2_rn(make_float2(__int_as_float(acc[e] + 0x4B400000), __int_as_float(acc[e + 1] + 0x4B400000)),
                                         make_float2(-kMagicOut, -kMagicOut));   // exact for |acc| < 2^22
            const float2 l2 = __fmul2_rn(af, make_float2(cscale[e], cscale[e + 1]));
            if (TAPS && a.tap_acc) {
              a.tap_acc[obase + (i64)e * N] = acc[e];
              a.tap_acc[obase + (i64)(e + 1) * N] = acc[e + 1];
            }
            if (I8S) {
              const int Gq = __float2int_rn(__fmul_rn(gam, 128.0f));
#pragma unroll
              for (int j = 0; j < 2; ++j) {
                const int locq = (int)(int8_t)(rne_clamp_bits(j ? l2.y : l2.x) & 0xffu);
                const int Sn = locq + ((Gq * sv[e + j] + 64) >> 7);
                sv[e + j] = max(-127, min(127, Sn));
              }
            } else {
              if (TAPS && a.tap_loc) {
                a.tap_loc[obase + (i64)e * N] = l2.x;
                a.tap_loc[obase + (i64)(e + 1) * N] = l2.y;
              }
              const float2 s2 = __ffma2_rn(make_float2(gam, gam),
                                           make_float2(__int_as_float(sv[e]), __int_as_float(sv[e + 1])), l2);
              sv[e] = __float_as_int(s2.x);
              sv[e + 1] = __float_as_int(s2.y);
              if (CAL) {
                smax[CAL ? hf * 8 + e : 0] = fmaxf(smax[CAL ? hf * 8 + e : 0], fabsf(s2.x));
                smax[CAL ? hf * 8 + e + 1 : 0] = fmaxf(smax[CAL ? hf * 8 + e + 1 : 0], fabsf(s2.y));
              }
            }
          }
        }
        tmem_st8(tS + (uint32_t)(hf * 8), sv);
      }
      }
      tmem_st_wait();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&bars[B_ACC_FREE]);  // this warp has read the accumulator of chunk k
    }
    if (CAL) {
#pragma unroll
      for (int p = 0; p < 32; ++p) {
        if (p < npp) {
          const uint32_t m = __reduce_max_sync(0xffffffffu, ok ? __float_as_uint(smax[CAL ? p : 0]) : 0u);
          if (lane == (p & 31)) atomicMax(reinterpret_cast<uint32_t*>(col_invh) + cb + p, m);
        }
      }
      named_bar(1, kStateThreads);
      if (tid < 64) atomicMax(a.absmax_h + h * P + tid, reinterpret_cast<const uint32_t*>(col_invh)[tid]);
    }
    if (!CAL && a.final_state) {
#pragma unroll
      for (int p0 = 0; p0 < 32; p0 += 8) {
        if (p0 < npp) {
          int sv[8];
          tmem_ld8(tS + (uint32_t)p0, sv);
          tmem_ld_wait();
          if (ok) {
#pragma unroll
            for (int e = 0; e < 8; ++e)
              a.final_state[(bh * P + cb + p0 + e) * N + n] =
                  I8S ? __fmul_rn((float)sv[e], a.s_h[h * P + cb + p0 + e]) : __int_as_float(sv[e]);
          }
        }
      }
    }
    if (tid < ncq) tma_store_wait_read();
  }
  drain_after_timeout(a.status);
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, kTmemCols);
  }
}

// Column range of a CTA: 16-channel chunks c0 .. c0 + ncq - 1 of one head.  Whole heads first, then
// heads in quarters, for a short remainder or a small workload (see the launcher; operand tiles and the MMA stay
// full width: only the re-quantisation, the state update and the hq rows are restricted to the range).
template <bool I8S, bool TAPS, bool CAL>
__global__ void __launch_bounds__(kThreads, CAL ? 2 : 3)
chunk_state_pass_tc(const __grid_constant__ CUtensorMap tm_B, const __grid_constant__ CUtensorMap tm_x,
                    const __grid_constant__ CUtensorMap tm_hq, const FusedArgs a) {
  if ((int)blockIdx.x < a.n_full) {
    fused_body<I8S, TAPS, CAL, 4>(tm_B, tm_x, tm_hq, a, (int)blockIdx.x, 0);
  } else {
    const int r = (int)blockIdx.x - a.n_full;
    fused_body<I8S, TAPS, CAL, 1>(tm_B, tm_x, tm_hq, a, a.n_full + (r >> 2), r & 3);
  }
}

}  // namespace

ssdi8_status_t launch_chunk_state_passing(const Dims& d, const int8_t* xq, const int8_t* Bq,
                                          const float* s_x, const float* s_xs, const float* s_B,
                                          const float* s_h, const float* pack, const float* gamma,
                                          const float* init, int8_t* hq, float* final_state,
                                          float* tap_loc, float* tap_prev, int8_t* tap_Xsq,
                                          int32_t* tap_acc, int32_t* status, bool int8_state,
                                          cudaStream_t st, uint32_t* absmax_h, float* s_xs_out) {
  const uint64_t T = (uint64_t)d.b * d.L;
  CUtensorMap tm_B, tm_x, tm_hq;
  {
    uint64_t dims[3] = {(uint64_t)d.N, (uint64_t)d.G, T};
    uint64_t str[2] = {(uint64_t)d.N, (uint64_t)d.G * d.N};
    uint32_t box[3] = {(uint32_t)d.N, 1, 32};
    if (!encode_tensor_map(&tm_B, Bq, 1, 3, dims, str, box, d.N)) return SSDI8_ERR_CUDA;
  }
  {
    uint64_t dims[3] = {(uint64_t)d.P, (uint64_t)d.H, T};
    uint64_t str[2] = {(uint64_t)d.P, (uint64_t)d.H * d.P};
    uint32_t box[3] = {64, 1, 32};
    if (!encode_tensor_map(&tm_x, xq, 1, 3, dims, str, box, 64)) return SSDI8_ERR_CUDA;
  }
  {
    uint64_t dims[2] = {(uint64_t)d.N, (uint64_t)d.b * d.c * d.H * d.P};
    uint64_t str[1] = {(uint64_t)d.N};
    uint32_t box[2] = {(uint32_t)d.N, 16};
    if (!encode_tensor_map(&tm_hq, hq, 1, 2, dims, str, box, 0)) return SSDI8_ERR_CUDA;
  }
  // (batch, head) units over the CTA slots of the device, 3 per SM.  (The calibration instance has two per SM; it follows
  // the same rule, whose lines were measured on the others.)
  const int sms = sm_count();
  if (sms == 0) return SSDI8_ERR_CUDA;
  const int units = d.H * d.b, slots = 3 * sms;
  // Whole (batch, head) units wherever the device is filled: a partly filled last wave of whole units runs faster per
  // CTA and costs less than the same units cut into more CTAs (592 units on 444 slots: 36.7 us whole, 41.9 with the last
  // 148 in quarters).  Quarter-width CTAs have the shorter chain per chunk (a quarter of the state per thread), so they
  // take a remainder of less than an eighth of a wave (512 tokens x 24 heads: 5.1 us, 7.1 whole) and, where all
  // of them fit the device beside the next kernel's first CTAs and a chain has four chunks or more, the whole workload
  // (Algorithm 2, us, whole / quarters: 2048 tokens x 80 heads 50.4 / 47.6, 2 x 2048 x 50 54.0 / 52.0, 1408 x 70 in chunks of
  // 128 43.8 / 40.4, 1024 x 80 36.6 / 35.5; but with one or two chunks 3 x 256 x 37 24.4 / 26.0, 512 x 100 29.9 / 30.5, and
  // 2048 x 111 55.8 / 56.7).
  int n_full = units / slots * slots;
  const bool quarters = 8 * (units - n_full) <= slots || (n_full == 0 && d.c >= 4 && 4 * units <= slots - slots / 10);
  if (!quarters) n_full = units;
  FusedArgs a = {s_x, s_xs, s_B, s_h, pack, gamma, init, final_state, tap_loc, tap_prev, tap_Xsq, tap_acc,
                 status, absmax_h, s_xs_out, d, n_full};
  const size_t smem = SMEM_BYTES;
  const unsigned grid = (unsigned)(n_full + 4 * (units - n_full));
  const bool taps = tap_loc || tap_prev || tap_Xsq || tap_acc;
  auto launch = [&](auto kernel) -> ssdi8_status_t {
    return launch_configured(kernel, dim3(grid), dim3(kThreads), smem, -1, true, st, tm_B, tm_x, tm_hq, a);
  };
  ssdi8_status_t ls;
  if (absmax_h)
    ls = launch(chunk_state_pass_tc<false, false, true>);
  else if (int8_state)
    ls = taps ? launch(chunk_state_pass_tc<true, true, false>) : launch(chunk_state_pass_tc<true, false, false>);
  else
    ls = taps ? launch(chunk_state_pass_tc<false, true, false>) : launch(chunk_state_pass_tc<false, false, false>);
  if (ls != SSDI8_OK) return ls;
  SSDI8_LAUNCH_CHECK();
  return SSDI8_OK;
}

}  // namespace ssdi8
