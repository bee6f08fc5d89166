// ChunkState + StatePassing fused, chunk-sequential per (batch, head): the fp32 chunk-local
// state never goes to HBM.  For chunk k = 0 .. c-1 of one (b, h):
//   Xs_q[i,p]   = rne(fmul(fmul(float(xq[i,p]), fdiv(s_x, s_xs)), LUT_state[i]))       (Eq. 3)
//   acc_st[p,n] = sum_i Xs_q[i,p] Bq[i,n]            INT8 MMA over the chunk's tokens, INT32 in TMEM
//   loc[p,n]    = fmul(float(acc_st), fmul(s_xs[h,p], s_B[g]))                         (Eq. 4 rescale)
//   hq[k][p,n]  = rne(fmul(S[p,n], fdiv(1, s_h[h,p])))     (state entering chunk k, int8 for ChunkScan1)
//   S[p,n]      = fmaf(Gamma_k, S[p,n], loc[p,n])                                      (Eq. 6)
// and final_state = S after the last chunk.  The kernel is bound by instruction issue where every SM holds three CTAs and by the
// chain of a chunk (MMAs -> accumulator -> update) where it holds one, so both are kept short:
//   * The accumulator has the 64 channels on its rows (M = 64, 16 tensor-memory lanes per warp quarter) and is read in the
//     16 x 256-bit form, which gives all 32 threads of a warp work: a thread has two channels and pairs of neighbouring n.  The
//     running state stays in registers (32 of them at N = 128), the scales of a channel too, and codes leave two at a time.
//   * Tokens arrive in slabs of 64 (xq, Bq and LUT_state of each), live slabs only, through a ring of four or six, so that tiles
//     are requested and re-quantised ahead of the chain; LUT_state of the chunks reaches the loading warp four chunks ahead (read
//     from global memory a chunk ahead, its latency was the time of a chunk of a lone CTA).
// (Against n on the lanes, the state in tensor memory, a byte store per code, a shared-memory load per scale and whole chunks
// of xq and Bq, ncu, us and million warp instructions: 8 x 2048 x 80 heads 43.3 -> 40.2, 25.3 -> 16.8; 4 x 8192 x 128 121 -> 107;
// 3 x 1408 x 50 22.8 -> 18.7; calibration of 2 x 2048 x 80 22.2 -> 18.2.  Calls: 229.4 -> 225, 816 -> 797, 65.7 -> 53.2, 81.4 -> 75.7.)
// Roles: eight state warps, which also form Q(X_scaled), in place, or two warps for that (see Geo), MMA issue, TMA loads.  hq leaves through two shared-memory tiles, one
// TMA store per chunk.  Same arithmetic, operation for operation, as the separate kernels (chunk_state.cu, state_passing.cu).
// I8S = true selects the paper's own state format (Section 4.2, Eq. 4 and Eq. 7): the state is an
// int8 code with the one per-(H,P) scale s_h, the chunk-local state goes INT32 -> INT8 in
// registers, and the recurrence is integer with a fixed-point decay:
//   locq = rne(fmul(float(acc_st), fdiv(fmul(s_xs, s_B), s_h)));  Gq = rne(fmul(Gamma_k, 128))
//   Sq   = sat(locq + ((Gq * Sq + 64) >> 7));  hq[k] = Sq before the update;  final = fmul(float(Sq), s_h)
// CAL = true is the calibration pass: no codes are formed; the largest |S| of every channel over init_state and
// every S_k goes into absmax_h (binary32 bits, one atomic per channel and CTA).  (Against separate ChunkState and
// StatePassing passes over 42 MB of chunk-local states in HBM, 28 + 7 us at batch 2 x 2048 x 80 heads, this takes 18.)
#include <type_traits>

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
  int n_full;  // CTAs below this index own a whole (batch, head); the rest own `slice` columns of the state of one
  int slice;   // 32 or 64
};

constexpr int kStateWarps = 8, kStateThreads = 32 * kStateWarps;
constexpr int kSlab = 64;                         // tokens of a slab
constexpr int kLutAhead = 4;                      // LUT_state of so many chunks is under way to the loading warp
enum { SLAB_LAST = 1 };                           // of its chunk (the word also has the slab's index from bit 8; the warps that need the chunk's count chunks)

// FEW: up to two CTAs per SM (one chunk of 256: one).  A CTA alone on its SM is a chain of latencies, the longest where decay is slow and most slabs live: the
// state warps quantise Q(X_scaled) themselves, all eight at a slab, one chunk ahead, behind a ring of six slabs.  With three
// CTAs per SM what counts is that the chains overlap: two warps of their own quantise, and the ring has four slabs (all of a
// chunk of 256).  Layer calls, us, eight state warps / two of their own: 3 x 1408 x 50 56.5 / 58.8, calibration of 2 x 2048 x 80 heads
// 77.4 / 79.7, but 8 x 2048 x 80 228.7 / 224.8, 4 x 8192 x 128 803 / 791, 5 x 1792 x 80 119.3 / 118.7.
template <bool FEW>
struct Geo {
  static constexpr int kRowWarps = FEW ? 0 : 2, kSlots = FEW ? 6 : 4;
  static constexpr int kMmaWarp = kStateWarps + kRowWarps, kLoadWarp = kMmaWarp + 1, kThreads = 32 * (kLoadWarp + 1);
  static constexpr uint32_t OFF_X = 0;                             // kSlots x [kSlab][64]   xq rows
  static constexpr uint32_t OFF_B = OFF_X + kSlots * kSlab * 64;   // kSlots x [kSlab][NS]   Bq rows (NS: state columns of the CTA)
  static constexpr uint32_t OFF_HQ = OFF_B + kSlots * kSlab * 128; // 2 x [64 p][NS] int8 staging of hq
  static constexpr uint32_t OFF_LUT = OFF_HQ + 2 * 8192;           // kSlots x [kSlab] floats
  static constexpr uint32_t OFF_COL = OFF_LUT + kSlots * kSlab * 4;   // [64] loc scale, [64] 1 / s_h, [64] s_x / s_xs
  static constexpr uint32_t OFF_CHUNK = OFF_COL + 768;             // kLutAhead x [Q] floats: LUT_state of whole chunks, for the loading warp
  static constexpr uint32_t OFF_INFO = OFF_CHUNK + kLutAhead * 1024;   // kSlots words by the loading warp
  static constexpr uint32_t OFF_BAR = OFF_INFO + 32;
  enum { B_FULL = 0, B_READY = kSlots, B_FREE = 2 * kSlots, B_ACC = 3 * kSlots, B_ACC_FREE = B_ACC + 2, B_LUT = B_ACC_FREE + 2,
         B_COUNT = B_LUT + kLutAhead };
  static constexpr uint32_t SMEM_BYTES = OFF_BAR + 8 * B_COUNT + 16;   // 96 768 bytes, two CTAs per SM; 71 632, three
  static_assert((FEW ? 2 : 3) * (SMEM_BYTES + 1024) <= 228 * 1024, "CTAs of an SM");
};
// More than half of an SM's shared memory, asked for where there is a CTA per SM or less (and the start does not count for more, see the launcher): the scheduler, which starts CTAs beside those of the
// kernel before wherever these have left room, would put up to three on one SM, each of them slower for it.  (Likewise the ring of six:
// 3 x 1408 x 50 56.5 us with three to an SM, 53.4 with two; 3 x 2048 x 80 98.7 / 94.7, 1 x 1024 x 128 (G 8) 41.3 / 40.7.)
constexpr uint32_t kSmemAlone = 120 * 1024;
// the lowest n of 32 bits, n from 1 on (1 << 32, of the lanes of a chunk's only slab, is not defined)
__host__ __device__ constexpr uint32_t low_bits(int n) { return 0xffffffffu >> (32 - n); }
static_assert(low_bits(32) == 0xffffffffu && low_bits(16) == 0xffffu && low_bits(8) == 0xffu, "a slab has 32, 16 or 8 lanes of LUT_state");
// position in a ring of slabs
template <int SLOTS>
struct Ring {
  int slot = 0;
  uint32_t phase = 0;
  __device__ __forceinline__ void next() {
    if (++slot == SLOTS) {
      slot = 0;
      phase ^= 1u;
    }
  }
};

// TAPS: any of the intermediate-tensor taps is requested (tests); the production instance carries no tap code
// N: state columns of a head; NS: of this CTA (all, or a slice from n_base on)
template <bool I8S, bool TAPS, bool CAL, bool FEW, int N, int NS>
__device__ __forceinline__ void fused_body(const CUtensorMap& tm_B, const CUtensorMap& tm_x, const CUtensorMap& tm_hq,
                                           const FusedArgs& a, const int unit, const int n_base) {
  // (no padding for the 1024-byte alignment the swizzled tiles need: the launcher checks that the kernel uses no static
  // shared memory, so the dynamic part starts at the window's base, and the kernel checks the address itself)
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  using G = Geo<FEW>;
  constexpr int kMmaWarp = G::kMmaWarp, kLoadWarp = G::kLoadWarp, kThreads = G::kThreads;
  constexpr uint32_t OFF_X = G::OFF_X, OFF_B = G::OFF_B, OFF_LUT = G::OFF_LUT;
  constexpr int B_FULL = G::B_FULL, B_READY = G::B_READY, B_FREE = G::B_FREE, B_ACC = G::B_ACC, B_ACC_FREE = G::B_ACC_FREE, B_LUT = G::B_LUT;
  using Pos = Ring<G::kSlots>;
  uint8_t* smem = smem_raw;
  if ((smem_u32(smem) & 1023u) != 0) {
    if (threadIdx.x == 0 && a.status) atomicExch(a.status, (int32_t)SSDI8_ERR_ALIGN);
    return;
  }
  constexpr int NA = NS == 128 ? 1 : 2;                 // accumulators: two where they fit beside those of two more CTAs
  constexpr uint32_t kTmemCols = NS * NA;
  const Dims& d = a.d;
  const int Q = d.Q, P = d.P;
  const int h = unit % d.H, b = unit / d.H;
  const int g = h / (d.H / d.G);
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;   // (the shuffle: uniform for the compiler)
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + G::OFF_BAR);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + G::B_COUNT);
  volatile int* info = reinterpret_cast<volatile int*>(smem + G::OFF_INFO);
  float* col_scale = reinterpret_cast<float*>(smem + G::OFF_COL);
  float* col_invh = col_scale + 64;
  float* col_rx = col_invh + 64;
  const i64 bh = (i64)b * d.H + h;
  const i64 unit0 = bh * d.c;
  const int nsl = Q / kSlab, tpl = Q / 32;     // slabs of a chunk; tokens of a lane that holds LUT_state of a chunk

  // LUT_state of a chunk: tpl consecutive tokens per lane, 32 / nsl lanes per slab
  struct Lut { float4 a, b; };
  auto lut_of_lane = [&](int place) -> Lut {
    Lut v = {make_float4(0.f, 0.f, 0.f, 0.f), make_float4(0.f, 0.f, 0.f, 0.f)};
    const float* l = reinterpret_cast<const float*>(smem + G::OFF_CHUNK) + place * 256 + lane * tpl;
    if (tpl == 2) {
      const float2 u = *reinterpret_cast<const float2*>(l);
      v.a.x = u.x;
      v.a.y = u.y;
    } else {
      v.a = reinterpret_cast<const float4*>(l)[0];
      if (tpl == 8) v.b = reinterpret_cast<const float4*>(l)[1];
    }
    return v;
  };
  // the loading warp: slab sl of chunk k into a slot: the copies, and LUT_state of the slab, from the registers of the
  // chunk's, with the arrival (which may come after the copies' bytes)
  auto copy = [&](int slot, int k, int sl) {
    const int tok = (int)((i64)b * d.L + (i64)k * Q) + kSlab * sl;
    tma_load_3d(smem + OFF_X + slot * (kSlab * 64), &tm_x, &bars[B_FULL + slot], 0, h, tok);
    tma_load_3d(smem + OFF_B + slot * (kSlab * NS), &tm_B, &bars[B_FULL + slot], n_base, g, tok);
  };
  auto describe = [&](int slot, int k, int sl, const Lut& v, bool last, bool copies) {
    const int rel = lane * tpl - kSlab * sl;   // of this lane's tokens in the slab
    if ((uint32_t)rel < (uint32_t)kSlab) {
      float* l = reinterpret_cast<float*>(smem + OFF_LUT) + slot * kSlab + rel;
      if (tpl == 2) {
        *reinterpret_cast<float2*>(l) = make_float2(v.a.x, v.a.y);
      } else {
        reinterpret_cast<float4*>(l)[0] = v.a;
        if (tpl == 8) reinterpret_cast<float4*>(l)[1] = v.b;
      }
    }
    __syncwarp();
    if (elect_one()) {
      info[slot] = (last ? SLAB_LAST : 0) | (sl << 8);
      mbar_expect_tx(&bars[B_FULL + slot], kSlab * 64 + kSlab * NS);   // (an arrival: releases the stores above)
      if (copies) copy(slot, k, sl);
    }
    __syncwarp();
  };

  if (warp == kLoadWarp) {
    if (lane == 0) {
      for (int s = 0; s < G::kSlots; ++s) {
        mbar_init(&bars[B_FULL + s], 1);
        mbar_init(&bars[B_READY + s], FEW ? kStateWarps : G::kRowWarps);
        mbar_init(&bars[B_FREE + s], 1);
      }
      for (int s = 0; s < kLutAhead; ++s) mbar_init(&bars[B_LUT + s], 1);
      for (int s = 0; s < 2; ++s) {
        mbar_init(&bars[B_ACC + s], 1);
        mbar_init(&bars[B_ACC_FREE + s], kStateWarps);
      }
      fence_mbar_init();
      tma_prefetch_desc(&tm_B);
      tma_prefetch_desc(&tm_x);
      tma_prefetch_desc(&tm_hq);
    }
    __syncwarp();
    asm volatile("bar.arrive 2, %0;" ::"n"(kThreads) : "memory");   // (its set-up for the others)
  }
  if (warp == 1) tmem_alloc(tmem_slot, kTmemCols);
  if (warp == 2 && lane < 8) {   // the head's vectors into L2 (which touches no value), two lines of each
    const float* const v = lane < 2 ? a.s_x : lane < 4 ? a.s_xs : lane < 6 ? a.s_h : nullptr;
    if (v) asm volatile("prefetch.global.L2 [%0];" ::"l"(v + h * P + 32 * (lane & 1)));
  }
  // (and the initial state, whose loads stand behind the set-up, a line per state thread: prefill of 5 x 1792 tokens x 80 heads 122.2 -> 119.9
  // us, 8 x 2048 x 80 209.3 -> 206.4, 12 x 64 x 100 52.1 -> 49.5)
  if (a.init && NS == N && tid < P * N / 32)
    asm volatile("prefetch.global.L2 [%0];" ::"l"(a.init + bh * P * N + 32 * tid));
  pdl_wait();   // everything below reads global memory
  // (after the wait, not before it: ChunkBMM, launched next, reads and writes global memory without waiting
  // for this kernel, so it must not be scheduled before this kernel's predecessors have completed)
  pdl_launch_dependents();
  auto step_xs = [&](int p) -> float {   // (the calibration pass is given the maxima of |X_scaled|)
    const float v = a.s_xs[h * P + p];
    return CAL ? step_of_max(__float_as_uint(v)) : v;
  };
  auto alive = [](float bound, float l) { return !(__fmul_rn(bound, fabsf(l)) < 0.5f); };
  // Rows that re-quantise to zero (the sparsity Eq. 3 rests on: LUT_state decays towards the start
  // of a chunk).  fmul is monotone, so with rxm >= |rx| of every channel,
  // fmul(fmul(127, rxm), |LUT_state[i]|) < 1/2 implies |fmul(fmul(x, rx), LUT_state[i])| < 1/2 for every
  // code x: row i of Q(X_scaled) is all zeros, exactly.  Such a row is stored as zeros without the
  // arithmetic, and a slab of such rows is left out altogether: no loads, no MMA.  A
  // chunk without a live slab opens the accumulator with its last one, all rows of it stored as zeros.
  auto row_bound = [&](float rx0, float rx1) -> float {   // the channels of the head, two per lane
    return __fmul_rn(127.0f, __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(fmaxf(fmaxf(0.f, fabsf(rx0)), fabsf(rx1))))));
  };

  if (warp == kLoadWarp) {
    // ------------------------------------------------------------ loads, as many slabs ahead as the ring has places.  This warp
    // forms the bound itself and does not wait for the others' set-up.  Where LUT_state of the first chunk is not known yet: FEW
    // takes all slabs of that chunk (the start of the chain is what counts: 256 tokens x 24 heads 22.55 -> 22.35 us, 3 x 2048 x 80 96.5 -> 95.6), and of
    // all chunks where the ring holds them, so that none of a short call waits for LUT_state and then for its tiles (graphs of layer calls: 192 tokens x 8
    // heads in chunks of 64, N 128, 13.1 -> 12.6 us, 384 x 16 of 128 15.3 -> 14.6; live slabs only in the first chunk too: 13.2, 15.7); the
    // others take only the last one, the likeliest to live.
    const float sx0 = a.s_x[h * P + lane], sx1 = a.s_x[h * P + 32 + lane], xs0 = step_xs(lane), xs1 = step_xs(32 + lane);
    constexpr int kFirst = FEW ? 1 : 0;   // chunk from which on only live slabs are taken
    auto fetch_lut = [&](int k) {
      if (k < d.c && elect_one()) {
        uint64_t* const bar = &bars[B_LUT + (k - kFirst) % kLutAhead];
        mbar_expect_tx(bar, (uint32_t)(Q * 4));
        bulk_load(smem + G::OFF_CHUNK + (k - kFirst) % kLutAhead * 1024, a.pack + ((unit0 + k) * kPackRows + PACK_LUT) * Q,
                  (uint32_t)(Q * 4), bar);
      }
      __syncwarp();
    };
    Pos at;
    const bool whole = FEW && d.c * nsl <= G::kSlots;   // the ring holds the call
    if (FEW) {
#pragma unroll 1
      for (int k = 0; k < (whole ? d.c : kFirst); ++k) {
#pragma unroll 1
        for (int sl = nsl - 1; sl >= 0; --sl, at.next()) {
          if (elect_one()) {
            info[at.slot] = (sl == 0 ? SLAB_LAST : 0) | (sl << 8);
            mbar_expect_tx(&bars[B_FULL + at.slot], kSlab * 64 + kSlab * NS + kSlab * 4);
            copy(at.slot, k, sl);
            bulk_load(smem + OFF_LUT + at.slot * (kSlab * 4), a.pack + ((unit0 + k) * kPackRows + PACK_LUT) * Q + kSlab * sl, kSlab * 4,
                      &bars[B_FULL + at.slot]);
          }
          __syncwarp();
        }
      }
    } else {
      fetch_lut(0);
      if (elect_one()) copy(0, 0, nsl - 1);
      __syncwarp();
    }
    for (int k = FEW ? kFirst : 1; k < kFirst + kLutAhead && !whole; ++k) fetch_lut(k);
    const float bound = row_bound(__fdiv_rn(sx0, xs0), __fdiv_rn(sx1, xs1));
    auto live_slabs = [&](const Lut& v) -> uint32_t {
      if (TAPS) return (1u << nsl) - 1u;
      const bool any = alive(bound, v.a.x) | alive(bound, v.a.y) | alive(bound, v.a.z) | alive(bound, v.a.w) | alive(bound, v.b.x) |
                       alive(bound, v.b.y) | alive(bound, v.b.z) | alive(bound, v.b.w);
      const uint32_t bal = __ballot_sync(0xffffffffu, any);
      const int lps = 32 / nsl;
      return __ballot_sync(0xffffffffu, lane < nsl && ((bal >> ((lane * lps) & 31)) & low_bits(lps)) != 0);
    };
    bool on = true;
#pragma unroll 1
    for (int k = whole ? d.c : kFirst; k < d.c; ++k) {
      const int i = k - kFirst;
      on = __all_sync(0xffffffffu, mbar_wait_inline<0>(&bars[B_LUT + i % kLutAhead], (i / kLutAhead) & 1, a.status));
      if (!on) break;
      const Lut v = lut_of_lane(i % kLutAhead);
      uint32_t m = live_slabs(v);
      const uint32_t top = 1u << (nsl - 1);
      if ((!FEW && k == 0) || m == 0) m |= top;
      bool issued = !FEW && k == 0;                 // (slab `top` then comes first)
#pragma unroll 1
      while (m) {
        const int sl = issued ? nsl - 1 : __ffs((int)m) - 1;
        m &= ~(1u << sl);
        on = __all_sync(0xffffffffu, mbar_wait_inline<0>(&bars[B_FREE + at.slot], at.phase ^ 1, a.status));
        if (!on) break;
        describe(at.slot, k, sl, v, m == 0, !issued);
        issued = false;
        at.next();
      }
      if (!on) break;
      fetch_lut(k + kLutAhead);                     // (every lane's values have gone into the mask and the slabs)
    }
  } else {
  if (tid < 64) {
    const float sx = step_xs(tid), sxb = __fmul_rn(sx, a.s_B[g]);
    if (CAL && b == 0 && n_base == 0) a.s_xs_out[h * P + tid] = sx;
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
  named_bar_sync(2, kThreads);
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  // row `row` of a slab of chunk k, 16 channels (those of lane % 4) of it
  auto quantise_rows = [&](int slot, int inf, int k, int row, float bound) {
    const int c = lane & 3;
    const float l = reinterpret_cast<const float*>(smem + OFF_LUT)[slot * kSlab + row];
    uint4* ptr = reinterpret_cast<uint4*>(smem + OFF_X + slot * (kSlab * 64) + swz_off((uint32_t)row, (uint32_t)c, 64));
    uint4 v = make_uint4(0u, 0u, 0u, 0u);
    if (alive(bound, l)) {
      const uint4 w4 = *ptr;
      const float2 l2 = make_float2(l, l);
      auto four = [&](uint32_t word, int j) -> uint32_t {
        const uint32_t ww = word ^ 0x80808080u;
        const float4 rx = *reinterpret_cast<const float4*>(col_rx + c * 16 + 4 * j);
        auto pair = [&](int e, const float2& r) -> uint2 {
          const float2 xf = __fadd2_rn(make_float2(__uint_as_float(__byte_perm(ww, 0x4B400000u, 0x7650u + e)),
                                                   __uint_as_float(__byte_perm(ww, 0x4B400000u, 0x7651u + e))),
                                       make_float2(-kMagicIn, -kMagicIn));
          return rne_clamp_bits2(__fmul2_rn(__fmul2_rn(xf, r), l2));
        };
        const uint2 q0 = pair(0, make_float2(rx.x, rx.y)), q1 = pair(2, make_float2(rx.z, rx.w));
        return pack4_bits(q0.x, q0.y, q1.x, q1.y);
      };
      v = make_uint4(four(w4.x, 0), four(w4.y, 1), four(w4.z, 2), four(w4.w, 3));
    }
    *ptr = v;
    if (TAPS && a.tap_Xsq)
      *reinterpret_cast<uint4*>(a.tap_Xsq + (((i64)b * d.L + (i64)k * Q + (inf >> 8) * kSlab + row) * d.H + h) * P +
                                c * 16) = v;
  };

  if (warp == kMmaWarp) {
    // ------------------------------------------------------------ MMA issue
    const uint32_t idesc = idesc_s8(64, NS, 1, 1);
    const uint32_t sxa = smem_u32(smem + OFF_X), sba = smem_u32(smem + OFF_B);
    uint32_t open = 0;                     // the chunk's accumulator has been opened
    Pos at;
#pragma unroll 1
    for (int k = 0; k < d.c; at.next()) {
      const int slot = at.slot;
      if (__any_sync(0xffffffffu, !mbar_wait_inline<0>(&bars[B_READY + slot], at.phase, a.status))) break;
      const int inf = info[slot];
      const bool last = (inf & SLAB_LAST) != 0;
      const uint32_t ai = NA == 1 ? 0u : (uint32_t)k & 1u;
      if (!open) mbar_wait_inline<0>(&bars[B_ACC_FREE + ai], ((k / NA) & 1) ^ 1, a.status);   // the state warps have read the chunk that had it
      tc_fence_after();
      if (elect_one()) {
        const uint64_t da = tile_desc(sxa + slot * (kSlab * 64), 64), db = tile_desc(sba + slot * (kSlab * NS), NS);
        mma_s8_ss(tmem + ai * NS, da, db, idesc, open);
        mma_s8_ss(tmem + ai * NS, da + ((32 * 64) >> 4), db + ((32 * NS) >> 4), idesc, 1);
        mma_commit(&bars[B_FREE + slot]);
        if (last) mma_commit(&bars[B_ACC + ai]);
      }
      __syncwarp();
      open = last ? 0u : 1u;
      k += last ? 1 : 0;
    }
  } else if (!FEW && warp >= kStateWarps) {
    // ------------------------------------------------------------ Q(X_scaled) of the slabs, in place: eight rows of a slab at a time
    const float bound = row_bound(col_rx[lane], col_rx[lane + 32]);
    Pos at;
#pragma unroll 1
    for (int k = 0; k < d.c; at.next()) {
      const int slot = at.slot;
      if (__any_sync(0xffffffffu, !mbar_wait_inline<256>(&bars[B_FULL + slot], at.phase, a.status))) break;
      const int inf = info[slot];
#pragma unroll 1
      for (int row = 8 * (warp - kStateWarps) + (lane >> 2); row < kSlab; row += 8 * G::kRowWarps) quantise_rows(slot, inf, k, row, bound);
      fence_async_smem();
      __syncwarp();
      if (lane == 0) mbar_arrive(&bars[B_READY + slot]);
      k += inf & SLAB_LAST;
    }
  } else {
    // ------------------------------------------------------------ state warps.  Accumulator row p on TMEM lane (p % 16) + 32 (p / 16);
    // 16 x 256 bit loads: registers 0, 1 of a group of eight columns hold row lane / 4, columns 2 (lane % 4) and the next,
    // registers 2, 3 the same columns of row lane / 4 + 8
    constexpr int NC = NS / 2, NG = NC / 8;        // columns of a warp, groups of eight
    const int q = warp & 3, ch = warp >> 2;
    const int p0 = 16 * q + (lane >> 2);           // this thread's channels: p0 and p0 + 8
    const int n0 = n_base + ch * NC + 2 * (lane & 3);
    const uint32_t tacc = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(ch * NC);
    const float2 cs0 = make_float2(col_scale[p0], col_scale[p0]), cs1 = make_float2(col_scale[p0 + 8], col_scale[p0 + 8]);
    const float2 ih0 = make_float2(col_invh[p0], col_invh[p0]), ih1 = make_float2(col_invh[p0 + 8], col_invh[p0 + 8]);
    // the running state S[p, n]: fp32, or (I8S) the integer code
    float2 S[2 * NG];
    float smax0 = 0.f, smax1 = 0.f;                // CAL: running maxima of |S[p, n]| (a NaN counts for nothing)
    auto code2 = [&](const float2& v, const float2& ih) -> uint2 {
      return I8S ? make_uint2(__float_as_uint(v.x), __float_as_uint(v.y)) : rne_clamp_bits2(__fmul2_rn(v, ih));
    };
#pragma unroll
    for (int i = 0; i < NG; ++i) {
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        float2 v = a.init ? *reinterpret_cast<const float2*>(a.init + (bh * P + p0 + 8 * r) * N + n0 + 8 * i) : make_float2(0.f, 0.f);
        if (I8S) {
          const uint2 cd = rne_clamp_bits2(__fmul2_rn(v, r ? ih1 : ih0));
          v = make_float2(__int_as_float((int)(int8_t)(cd.x & 0xffu)), __int_as_float((int)(int8_t)(cd.y & 0xffu)));
        }
        if (CAL) (r ? smax1 : smax0) = fmaxf(fmaxf(r ? smax1 : smax0, fabsf(v.x)), fabsf(v.y));
        S[2 * i + r] = v;
      }
    }
    // codes go to row p0 of the staging tile, swizzled for the TMA store: chunk of 16 columns ^ a term of the row that is the same for p0 + 8
    constexpr int kRowShift = NS == 128 ? 0 : NS == 64 ? 1 : 2, kRowMask = NS / 16 - 1;
    const uint32_t hoff = (uint32_t)p0 * NS + ((uint32_t)(((ch * NC / 16) ^ ((p0 >> kRowShift) & kRowMask)) << 4)) + 2u * (lane & 3);
    // ---- (FEW) Q(X_scaled) of a chunk's slabs, in place, one chunk ahead: a warp takes eight rows of each
    const float bound = FEW ? row_bound(col_rx[lane], col_rx[lane + 32]) : 0.f;
    Pos at;
    auto quantise_chunk = [&](int k) {
#pragma unroll 1
      for (int more = 1; more; at.next()) {
        const int slot = at.slot;
        if (__any_sync(0xffffffffu, !mbar_wait_inline<0>(&bars[B_FULL + slot], at.phase, a.status))) return;
        const int inf = info[slot];
        quantise_rows(slot, inf, k, 8 * warp + (lane >> 2), bound);
        fence_async_smem();
        __syncwarp();
        if (lane == 0) mbar_arrive(&bars[B_READY + slot]);
        more = (inf & SLAB_LAST) ^ SLAB_LAST;
      }
    };
    if (FEW) quantise_chunk(0);
#pragma unroll 1
    for (int k = 0; k < d.c; ++k) {
      const float gam = a.gamma[unit0 + k];
      if (FEW && k + 1 < d.c) quantise_chunk(k + 1);
      const uint32_t ai = NA == 1 ? 0u : (uint32_t)k & 1u;
      // ---- hq[k] = codes of the state entering this chunk (and the prev tap), ahead of the wait for the chunk's MMAs
      uint8_t* const hq = smem + G::OFF_HQ + (k & 1) * 8192;
      if (!CAL) {
#pragma unroll
        for (int i = 0; i < NG; ++i) {
          uint8_t* const at = hq + ((hoff ^ (uint32_t)((i >> 1) << 4)) + 8 * (i & 1));
          const uint2 c0 = code2(S[2 * i], ih0), c1 = code2(S[2 * i + 1], ih1);
          *reinterpret_cast<uint16_t*>(at) = (uint16_t)__byte_perm(c0.x, c0.y, 0x0040u);
          *reinterpret_cast<uint16_t*>(at + 8 * NS) = (uint16_t)__byte_perm(c1.x, c1.y, 0x0040u);
        }
        if (TAPS && !I8S && a.tap_prev) {
#pragma unroll
          for (int i = 0; i < 2 * NG; ++i)
            *reinterpret_cast<float2*>(a.tap_prev + (((((i64)b * d.c + k) * d.H + h) * P) + p0 + 8 * (i & 1)) * N + n0 + 8 * (i >> 1)) = S[i];
        }
        fence_async_smem();
        if (tid == 0) tma_store_wait_read();     // the store of chunk k - 1: its tile is written again in chunk k + 1
      }
      // one warp polls for the MMAs of this chunk; the barrier passes their completion on to the others
      if (warp == 0) mbar_wait_inline<256>(&bars[B_ACC + ai], (k / NA) & 1, a.status);
      named_bar_sync(1, kStateThreads);
      if (tid == 0 && !CAL) {                    // hq[k] leaves by TMA
        tma_store_2d(&tm_hq, hq, n_base, (int)((((i64)b * d.c + k) * d.H + h) * P));
        tma_store_commit();
      }
      // ---- epilogue of the MMA: S = fmaf(Gamma_k, S, loc), 16 columns at a time
      tc_fence_after();
      const float2 g2 = make_float2(gam, gam);
      const int Gq = I8S ? __float2int_rn(__fmul_rn(gam, 128.0f)) : 0;
#pragma unroll
      for (int i0 = 0; i0 < NG; i0 += 2) {
        int acc[8];
        tmem_ld_16x256_x2(tacc + ai * NS + 8 * i0, acc);
        tmem_ld_wait();
        if (i0 + 2 == NG) {                        // this warp has read the accumulator
          tc_fence_before();
          if (lane == 0) mbar_arrive(&bars[B_ACC_FREE + ai]);
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {              // two columns of one row each
          const int i = i0 + (j >> 1);
          const float2 af = __fadd2_rn(make_float2(__int_as_float(acc[2 * j] + 0x4B400000), __int_as_float(acc[2 * j + 1] + 0x4B400000)),
                                       make_float2(-kMagicOut, -kMagicOut));   // exact for |acc| < 2^22
          const float2 l2 = __fmul2_rn(af, j & 1 ? cs1 : cs0);
          float2& sv = S[2 * i + (j & 1)];
          if (TAPS) {
            const i64 o = (((((i64)b * d.c + k) * d.H + h) * P) + p0 + 8 * (j & 1)) * N + n0 + 8 * i;
            if (a.tap_acc) *reinterpret_cast<int2*>(a.tap_acc + o) = make_int2(acc[2 * j], acc[2 * j + 1]);
            if (!I8S && a.tap_loc) *reinterpret_cast<float2*>(a.tap_loc + o) = l2;
          }
          if (I8S) {
            const uint2 lq = rne_clamp_bits2(l2);     // 0x4B400000 + locq
            auto next = [&](float s, uint32_t l) -> float {
              return __int_as_float(max(-127, min(127, (int)l + ((Gq * __float_as_int(s) + 64) >> 7) - 0x4B400000)));
            };
            sv = make_float2(next(sv.x, lq.x), next(sv.y, lq.y));
          } else {
            sv = __ffma2_rn(g2, sv, l2);
          }
          if (CAL) (j & 1 ? smax1 : smax0) = fmaxf(fmaxf(j & 1 ? smax1 : smax0, fabsf(sv.x)), fabsf(sv.y));
        }
      }
    }
    if (CAL) {
#pragma unroll
      for (int o = 1; o < 4; o <<= 1) {
        smax0 = fmaxf(smax0, __shfl_xor_sync(0xffffffffu, smax0, o));
        smax1 = fmaxf(smax1, __shfl_xor_sync(0xffffffffu, smax1, o));
      }
      if ((lane & 3) == 0) {
        atomicMax(reinterpret_cast<uint32_t*>(col_invh) + p0, __float_as_uint(smax0));
        atomicMax(reinterpret_cast<uint32_t*>(col_invh) + p0 + 8, __float_as_uint(smax1));
      }
      named_bar_sync(1, kStateThreads);
      if (tid < 64) atomicMax(a.absmax_h + h * P + tid, reinterpret_cast<const uint32_t*>(col_invh)[tid]);
    }
    if (!CAL && a.final_state) {
      const float sh0 = I8S ? a.s_h[h * P + p0] : 0.f, sh1 = I8S ? a.s_h[h * P + p0 + 8] : 0.f;
#pragma unroll
      for (int i = 0; i < 2 * NG; ++i) {
        float2 v = S[i];
        if (I8S) v = make_float2(__fmul_rn((float)__float_as_int(v.x), i & 1 ? sh1 : sh0), __fmul_rn((float)__float_as_int(v.y), i & 1 ? sh1 : sh0));
        *reinterpret_cast<float2*>(a.final_state + (bh * P + p0 + 8 * (i & 1)) * N + n0 + 8 * (i >> 1)) = v;
      }
    }
    if (tid == 0 && !CAL) tma_store_wait_read();
  }
  tc_fence_before();
  }
  drain_after_timeout(a.status);
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(*tmem_slot, kTmemCols);
  }
}

// Whole heads first, then heads in slices of 32 or 64 state columns, for a short remainder or a small workload (see the launcher; a
// slice re-quantises all channels of the head itself and has the MMA, the state update and the hq columns of its own columns only).
template <bool I8S, bool TAPS, bool CAL, bool FEW, int N>
__global__ void __launch_bounds__(Geo<FEW>::kThreads, FEW ? 2 : 3)
chunk_state_pass_tc(const __grid_constant__ CUtensorMap tm_B, const __grid_constant__ CUtensorMap tm_x,
                    const __grid_constant__ CUtensorMap tm_hq, const __grid_constant__ CUtensorMap tm_Bs,
                    const __grid_constant__ CUtensorMap tm_hqs, const FusedArgs a) {
  if ((int)blockIdx.x < a.n_full) {
    fused_body<I8S, TAPS, CAL, FEW, N, N>(tm_B, tm_x, tm_hq, a, (int)blockIdx.x, 0);
  } else {
    const int r = (int)blockIdx.x - a.n_full;
    // (32 of 128 columns: few units only, see the launcher.  Written the other way round, 32 ahead of 64, slices of 64 take 3 % longer: layer 3 x 1024 x 24 heads
    // 29.6 -> 30.5 us, 3 x 1792 x 20 34.4 -> 35.3)
    if (N == 128 && (!FEW || a.slice == 64)) {
      if constexpr (N == 128) fused_body<I8S, TAPS, CAL, FEW, N, 64>(tm_Bs, tm_x, tm_hqs, a, a.n_full + r / 2, r % 2 * 64);
    } else {
      if constexpr (N == 64 || FEW) fused_body<I8S, TAPS, CAL, FEW, N, 32>(tm_Bs, tm_x, tm_hqs, a, a.n_full + r / (N / 32), r % (N / 32) * 32);
    }
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
  CUtensorMap tm_B, tm_x, tm_hq, tm_Bs, tm_hqs;   // (the last two: of a slice)
  auto maps = [&](CUtensorMap& mB, CUtensorMap& mh, int cols) -> bool {
    uint64_t dims[3] = {(uint64_t)d.N, (uint64_t)d.G, T};
    uint64_t str[2] = {(uint64_t)d.N, (uint64_t)d.G * d.N};
    uint32_t box[3] = {(uint32_t)cols, 1, kSlab};
    uint64_t hdims[2] = {(uint64_t)d.N, (uint64_t)d.b * d.c * d.H * d.P};
    uint64_t hstr[1] = {(uint64_t)d.N};
    uint32_t hbox[2] = {(uint32_t)cols, 64};
    return encode_tensor_map(&mB, Bq, 1, 3, dims, str, box, cols) && encode_tensor_map(&mh, hq, 1, 2, hdims, hstr, hbox, cols);
  };
  {
    uint64_t dims[3] = {(uint64_t)d.P, (uint64_t)d.H, T};
    uint64_t str[2] = {(uint64_t)d.P, (uint64_t)d.H * d.P};
    uint32_t box[3] = {64, 1, kSlab};
    if (!encode_tensor_map(&tm_x, xq, 1, 3, dims, str, box, 64)) return SSDI8_ERR_CUDA;
  }
  // (batch, head) units over the CTA slots of the device, 3 per SM.
  const int sms = sm_count();
  if (sms == 0) return SSDI8_ERR_CUDA;
  const int units = d.H * d.b, slots = 3 * sms;
  // Whole heads wherever the device is filled; a remainder of less than an eighth of a wave goes in slices, whose
  // chain per chunk is shorter (prefill of 6 x 2048 tokens x 80 heads, 36 of 480: whole 161.6 us, slices of 64 160.5, of 32 163.4).  Few units of some chunks go in slices of 64, the longest chains of them in 32 (graphs of layer calls,
  // us, whole / slices of 64 / of 32): N 128: 1024 tokens x 32 heads 22.0 / 20.7 / 21.6, 1024 x 96 32.8 / 32.2 / 36.1, 3 x 512 x 12 (chunks of
  // 128) 19.4 / 19.0 / 20.9, 128 x 12 (of 64) 13.6 / 12.9 / 12.8, 2048 x 80 46.8 / 45.5 / 54.7, 2 x 8192 x 8 (INT8 states) 74.7 / 66.6 / 63.1; but
  // 256 x 64 17.7 / 18.5 / 20.1, 128 x 64 (of 128) 14.2 / 15.7 / 16.5, 3 x 2048 x 80 92 / 101 / 112.  With two or three chunks up to two units to
  // five SMs: 768 x 36 20.8 / 18.9 / -, 384 x 42 (of 128) 17.3 / 16.4 / -, 256 x 48 (of 128) 16.2 / 15.0 / -, 512 x 12 16.6 / 16.2 / 16.8, but 128 x 54 (of 64) 13.7 /
  // 14.4 / -, 768 x 74 24.6 / 26.8 / -, 192 x 74 (of 64) 17.4 / 18.6 / -.
  // N 64, from four chunks on: 768 x 60 28.7 / - / 27.9, 256 x 32 (of 64) 16.4 / - / 15.6, 2048 x 60 44.9 / - / 44.6; with fewer whole heads: 128 x 60
  // (of 64) 13.3 / - / 14.6, 256 x 74 (of 128) 16.4 / - / 17.6, 512 x 36 17.9 / - / 19.2.  The calibration, which forms no codes, takes slices of N 128 from twelve chunks
  // on (calls, whole / slices: 1280 x 48 43.0 / 45.3, 1024 x 32 36.0 / 38.1, 1280 x 48 (of 128) 48.3 / 51.4, but 4096 x 8 53.7 / 52.8).
  int n_full = units / slots * slots, slice = d.N == 128 ? 64 : 32;
  const int last = units - n_full;
  if (n_full > 0) {
    if (8 * last > slots) n_full = units;
  } else if (d.N == 128 && (!absmax_h || d.c >= 12) && (d.c >= 4 ? 3 * units <= 2 * sms : d.c >= 2 && 5 * units <= 2 * sms)) {
    slice = d.c >= 12 && 4 * units <= sms ? 32 : 64;
  } else if (!(d.N == 64 && d.c >= 4 && 2 * units <= sms)) {
    n_full = units;
  }
  if (!maps(tm_B, tm_hq, d.N)) return SSDI8_ERR_CUDA;
  if (n_full == units) {
    tm_Bs = tm_B;
    tm_hqs = tm_hq;
  } else if (!maps(tm_Bs, tm_hqs, slice)) {
    return SSDI8_ERR_CUDA;
  }
  FusedArgs a = {s_x, s_xs, s_B, s_h, pack, gamma, init, final_state, tap_loc, tap_prev, tap_Xsq, tap_acc,
                 status, absmax_h, s_xs_out, d, n_full, slice};
  const unsigned grid = (unsigned)(n_full + d.N / slice * (units - n_full));
  const bool taps = tap_loc || tap_prev || tap_Xsq || tap_acc;
  // (FEW; but of one chunk of 256 two warps of their own quantise faster where SMs have two CTAs, all four slabs of a CTA being there at once.  Layer calls in a
  // row, FEW / two warps: 2 x 256 x 108 with 16-bit y 27.3 / 26.0 us, 2 x 256 x 130 27.2 / 25.7, 256 x 296 29.4 / 27.4, 256 x 150 23.6 / 24.3; prefill of 2 x 256 x 108
  // 28.4 / 29.1.  Not in the calibration, which forms no codes beside it)
  const bool few = (int)grid <= 2 * sms && !(d.Q == 256 && d.c == 1 && (int)grid > sms && !absmax_h);
  // (kSmemAlone; not for one chunk, nor for two or three of N 128 where more than four SMs in five get a CTA: the start is what counts there, and CTAs of that
  // size wait for the SMs that the kernel before still holds.  With / without: 256 tokens x 148 heads N 128 22.1 / 19.8 us, 64 x 100 (of 64) N 64
  // 13.6 / 13.1, 512 x 148 N 128 29.4 / 27.4, 768 x 148 33.9 / 32.2; but 128 x 48 (of 64) N 128 14.5 / 15.3, 384 x 148 (of 128) N 64 22.3 / 22.8)
  const bool alone = (int)grid <= sms && d.c > 1 && !(d.N == 128 && d.c <= 3 && 5 * (int)grid > 4 * sms);
  auto launch = [&](auto few_c, auto kernel) -> ssdi8_status_t {
    using G = Geo<decltype(few_c)::value>;
    const size_t smem = alone ? kSmemAlone : G::SMEM_BYTES;
    return launch_sized(kernel, dim3(grid), dim3(G::kThreads), smem, decltype(few_c)::value ? kSmemAlone : smem, 100, true, st, tm_B, tm_x, tm_hq,
                        tm_Bs, tm_hqs, a);
  };
  auto pick = [&](auto few_c, auto n) -> ssdi8_status_t {
    constexpr bool F = decltype(few_c)::value;
    constexpr int N = decltype(n)::value;
    if (absmax_h) return launch(few_c, chunk_state_pass_tc<false, false, true, F, N>);
    if (int8_state)
      return taps ? launch(few_c, chunk_state_pass_tc<true, true, false, F, N>) : launch(few_c, chunk_state_pass_tc<true, false, false, F, N>);
    return taps ? launch(few_c, chunk_state_pass_tc<false, true, false, F, N>) : launch(few_c, chunk_state_pass_tc<false, false, false, F, N>);
  };
  auto pick_n = [&](auto few_c) -> ssdi8_status_t {
    return d.N == 128 ? pick(few_c, std::integral_constant<int, 128>{}) : pick(few_c, std::integral_constant<int, 64>{});
  };
  const ssdi8_status_t ls = few ? pick_n(std::true_type{}) : pick_n(std::false_type{});
  if (ls != SSDI8_OK) return ls;
  SSDI8_LAUNCH_CHECK();
  return SSDI8_OK;
}

}  // namespace ssdi8
