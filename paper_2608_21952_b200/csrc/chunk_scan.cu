// ChunkScan1 + ChunkScan2 + output sum (Algorithm 2 modules 5, 6) on tcgen05 tensor cores:
// a persistent, warp-specialised kernel, one CTA per SM.
// Per (batch, chunk, head) and 128-row tile of the chunk:
//   acc_off[i,p]  = sum_n Cq[i,n] hq[p,n]                 INT8 MMA, INT32 accumulator in TMEM
//   Mq[i,j]       = per-row re-quantised CBq[i,j] dt_j exp(cs_i - cs_j), j <= i   (see ssdi8.h)
//   acc_diag[i,p] = sum_j Mq[i,j] xq[j,p]                 INT8 MMA, second TMEM accumulator
//   y = exp(cs_i) s_C s_h acc_off + (s_cb rowmax_i / 127) s_x acc_diag + D s_x xq + corr
// Roles (28 warps): warps 0 and 2 issue the TMA loads (CBq K-major, the per-token scalar pack of
// ChunkCumsum and the head's per-column vectors; hq K-major and xq MN-major, once per chunk), a
// tile of the chunk each; warps 1 and 3 issue the MMAs of the two contractions, warp 1 loads Cq as
// well; warps 4-19 build Mq in place over CBq, as two groups of 8 warps that take alternate chunks
// (two threads per output row in adjacent lanes, so a warp owns 16 rows and needs no block barrier
// for the row maximum); warps 20-27 read the
// accumulators, form y and store it through a swizzled staging tile with TMA (128-byte rows), as two
// groups of 4 warps on alternate tiles, so one group's per-tile bookkeeping and waits run under the
// other's arithmetic.  Four accumulator pairs, an xq and an hq buffer per chunk (shared by the chunk's two
// tiles) and an 8-deep ring for what the mask warps hand to the epilogue keep the mask and the MMAs
// of the next tiles independent of the epilogue of the current ones.  Every buffer has its own
// "free" barrier, released by whoever reads it last (tcgen05.commit for MMA operands), so loads run
// several tiles ahead.  What bounds the kernel (0.113 ms with binary32 y at batch 8 x 2048 x 80 heads, 0.103 with 16-bit
// y) are the epilogue groups, busy 85 to 90 % of the time, and close behind them the mask groups, the round trip of the one
// Cq buffer and the DRAM writes of y: without the mask 0.111 ms, without mask and y stores 0.0725.  Issue slots are two
// thirds used (78 M warp instructions), so it is written to issue little all the same: in each group one warp polls the
// mbarriers and the others wait at a hardware barrier, the wait loop is one out-of-line function, the tile walk has no
// divisions, and the code is kept small enough for the instruction cache (every role executes different code).
// The pipeline around it is built so that no role waits for another's order: a timeline of one CTA had the
// mask groups waiting 2.6 us of every 6.6 for CBq buffers, which waited for in-order MMAs, which waited for
// xq, whose buffer the epilogue gave back last; with the loads of the two tiles of a chunk on
// two producers, the scalar pack and hq requested a chunk ahead, xq given back early and the MMA issue
// in uniform registers the same arithmetic takes 0.113 instead of 0.125 ms.
// No multicast; bounded waits.
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <type_traits>

#include "kernels.h"
#include "scan_common.cuh"
#include "sm100.cuh"

namespace ssdi8 {
namespace {

using namespace sm100;
using namespace scan;

struct ScanArgs {
  const float* s_x; const float* s_C; const float* s_cb; const float* s_h;
  const float* pack; const float* D; const float* corr;
  uint8_t* y;       // [b*L][H][P] binary32 or 16-bit
  int32_t* status;
  ScanTaps taps;
  Dims d;
  UnitWalk w;       // CTA j takes units j, j + grid, j + 2 grid, ...
};

constexpr int kWarps = 28, kThreads = kWarps * 32;
constexpr int kMaskWarp0 = 4, kGroupWarps = 8;
constexpr int kEpiWarp0 = 20, kEpiWarps = 8, kEpiGroupWarps = 4;
constexpr uint32_t kTmemCols = 512;  // four accumulator pairs: acc_off at 128 a, acc_diag at 128 a + 64
// shared memory (bytes, from a 1024-byte aligned base)
constexpr uint32_t OFF_CB = 0;          // ring of 4: two 2-panel buffers, two 1-panel buffers
constexpr uint32_t OFF_C = 98304;       // [128][N]
constexpr uint32_t OFF_H = 114688;      // ring of 2 x [64][N], one per chunk: hq comes from HBM, requested a chunk ahead
constexpr uint32_t H_BYTES = 8192;
constexpr uint32_t OFF_X = 131072;      // ring of 2 x [256][64]: the xq rows of a chunk
constexpr uint32_t OFF_YST = 163840;    // 8 warps x [32][128 B] y staging
constexpr uint32_t OFF_TOK = OFF_YST + 32768;   // ring of 4, one per chunk, read by the mask warps: Q floats each of cs, dt, woff, atok, and what is used of the bounds row
constexpr uint32_t TOK_BYTES = 4096 + 608;
// ring of 8 x what the epilogue needs of a tile: [128] row maxima and [128] cs_i, written by the
// mask warps, and the head's s_x, s_h and correction vectors ([64] each, bulk-loaded).  Eight deep so
// that the mask of a tile never waits for the epilogue of an earlier one (four deep: 0.141 against 0.125 ms).
constexpr uint32_t OFF_ROW = OFF_TOK + 4 * TOK_BYTES;
constexpr uint32_t ROW_BYTES = 2048, ROW_COLS = 1024, ROW_SCAL = 1792;   // scalars: s_C of the group, D of the head, s_cb
constexpr uint32_t OFF_BAR = OFF_ROW + 8 * ROW_BYTES;
constexpr uint32_t SMEM_BYTES = OFF_BAR + 512;   // 232 320 bytes

__device__ __forceinline__ uint32_t cb_offset(int idx) { return scan::cb_offset(OFF_CB, idx); }

enum { B_CB_FULL = 0, B_CB_FREE = 4, B_MQ = 8, B_C_FULL = 12, B_C_FREE = 13, B_X_FULL = 14, B_X_FREE = 16,
       B_H_FULL = 18, B_H_FREE = 20, B_TOK_FULL = 22, B_TOK_FREE = 26, B_ACC = 30, B_ACC_FREE = 34, B_ROW_FULL = 38,
       B_ROW_FREE = 46, B_COUNT = 54 };


__device__ __forceinline__ uint32_t row_phase(int n) { return (uint32_t)(n >> 3) & 1u; }

// four codes rn(a g), the exact product rounded once to the nearest integer (ties to even): for
// |a g| < 2^22 that integer sits in the low bits of fma(a, g, 1.5 * 2^23); callers guarantee
// |a g| < 127.5.  (One fused operation by definition: a packed multiply followed by a packed add of
// the rounding constant is not an alternative, the assembler contracts that pair into this very
// fused operation, which differs from the two-step result wherever the rounded product is a tie.)
__device__ __forceinline__ uint32_t pack4_rn_product(float2 a, float2 b, float2 g) {
  const float2 ra = __ffma2_rn(a, g, make_float2(kMagicOut, kMagicOut));
  const float2 rb = __ffma2_rn(b, g, make_float2(kMagicOut, kMagicOut));
  return __byte_perm(__byte_perm(__float_as_uint(ra.x), __float_as_uint(ra.y), 0x0040u),
                     __byte_perm(__float_as_uint(rb.x), __float_as_uint(rb.y), 0x0040u), 0x5410u);
}

// ---- the masked operand of one tile, in place over CBq.  Two threads per output row, in
// adjacent lanes, so a warp owns 16 rows that share their own sub-block I16 = i / 16 (everything
// below is warp-uniform up to values) and the row maximum needs one shuffle, no block barrier.  Every
// sub-block (16 columns) is split 8/8 between the two threads.  Sub-block I16 is the row's own: running
// product of per-token decays (the thread with the lower columns first runs the product through the upper
// ones).  Earlier sub-blocks use the column weights woff and one factor f = fmul(dec_i, gtab[c]) each,
// dec_i the row's decay to the end of the sub-block before its own; later ones are zero.
//
// The own and the nearest earlier sub-block are straight-line code: they decide the row maximum of
// nearly every row, and their products stay in registers until the codes are formed.  Of the farther
// ones, work that decides no output bit is skipped.  bound[c] = b127[c] gtab[c], one sub-block per lane,
// bounds |t| gtab[c] over sub-block c, so with R = the warp's largest dec_i / (row maximum so far) a
// sub-block with bound[c] R <= 1 raises no row maximum, and with R = the warp's largest dec_i inv_i one
// with bound[c] R < 1/2 rounds to zero in every row; both with a slack of 1e-5, far above the few
// binary32 roundings (and the approximate reciprocal) on either side.  One ballot so names the sub-blocks
// to visit.  Where cs increases somewhere in the chunk (b127[16] is +inf then) dec_i and gtab are not
// bounded by 1, products may leave the binary32 range, and every sub-block is visited.
// (Against a walk that tested one sub-block after the other, nearest first, 16 columns per thread: 86.5 against 97.1 M
// warp instructions, 0.125 against 0.139 ms at batch 8 x 2048 x 80 heads.)
template <bool TAPS>
__device__ __forceinline__ void mask_tile(uint8_t* sCB, const float* tokbuf, float* rowbuf, int rb, int lane, int TM, uint32_t RBQ,
                                          const Tile& t, const ScanArgs& a) {
  const int Q = a.d.Q;
  const float* cs_s = tokbuf;
  const float* dt_s = tokbuf + Q;
  const float* woff_s = tokbuf + 2 * Q;
  const float* atok_s = tokbuf + 3 * Q;
  const float* b127_s = tokbuf + 4 * Q;
  const int r = rb * 16 + (lane >> 1), q2 = lane & 1;   // the warp's block of 16 rows
  if (rb * 16 >= TM) return;         // whole warps (TM is a multiple of 16)
  const int i = t.it * TM + r;       // row within the chunk
  const int I16 = (t.it * TM >> 4) + rb, ri = lane >> 1;
  const uint32_t cshift = RBQ == 128 ? 3u : 2u;  // log2(sub-blocks per panel row)
  uint8_t* const rowbase = sCB + (RBQ == 128 ? (uint32_t)r * 128u : (uint32_t)r * 64u);
  const uint32_t rx = RBQ == 128 ? ((uint32_t)r & 7u) : (((uint32_t)r >> 1) & 3u);  // swizzle term of the row
  auto chunk_ptr = [&](int c) -> uint8_t* {
    const uint32_t pn = (uint32_t)c >> cshift, cc = (uint32_t)c & ((1u << cshift) - 1u);
    return rowbase + pn * PANEL + ((cc ^ rx) << 4);
  };
  auto half_ptr = [&](int c) -> uint2* { return reinterpret_cast<uint2*>(chunk_ptr(c)) + q2; };   // this thread's 8 columns
  constexpr uint32_t kAll = 0xffffffffu;
  const float cs_i = cs_s[i];
  const float* const gtab = b127_s + 32 + ((I16 * (I16 - 1)) >> 1);
  // eight products cb w of an earlier sub-block and their largest magnitude
  auto products = [&](int c, float2 (&p)[4]) -> float {
    const uint2 w2 = *half_ptr(c);
    const float4* wo = reinterpret_cast<const float4*>(woff_s + c * 16 + q2 * 8);
    const float4 o0 = wo[0], o1 = wo[1];
    const uint32_t x0 = w2.x ^ 0x80808080u, x1 = w2.y ^ 0x80808080u;
    p[0] = __fmul2_rn(unpack2(x0, 0), make_float2(o0.x, o0.y));
    p[1] = __fmul2_rn(unpack2(x0, 2), make_float2(o0.z, o0.w));
    p[2] = __fmul2_rn(unpack2(x1, 0), make_float2(o1.x, o1.y));
    p[3] = __fmul2_rn(unpack2(x1, 2), make_float2(o1.z, o1.w));
    float m = 0.f;
#pragma unroll
    for (int k = 0; k < 4; ++k) m = fmaxf(fmaxf(m, fabsf(p[k].x)), fabsf(p[k].y));
    return m;
  };
  float2 tv[4], tn[4];               // t of this thread's half of the own and of the nearest earlier sub-block
  float rmax = 0.f, dec = 0.f, bound = 0.f;
  if (I16 > 0) {
    dec = exp32(__fsub_rn(cs_i, cs_s[I16 * 16 - 1]));
    rmax = __fmul_rn(products(I16 - 1, tn), dec);   // gtab[I16 - 1] = 1
    if (lane < I16 - 1) bound = __fmul_rn(b127_s[lane], gtab[lane]);
  }
  {
    // own sub-block, right to left: E[i,i] = 1, E[i,j] = fmul(E[i,j+1], a_{j+1}).  Straight-line code: the
    // product starts as 0 and is set to 1 where the row meets its diagonal, so the columns past it, which
    // carry no weight, raise no row maximum and the 16 rows of the warp do not diverge.
    const uint2 w2 = *half_ptr(I16);
    const uint32_t ww[2] = {w2.x ^ 0x80808080u, w2.y ^ 0x80808080u};
    const float* ab = atok_s + I16 * 16;   // a_m of the sub-block at ab[m]
    const int e0 = q2 * 8;
    float E = 0.f;
    {
      // the thread with the lower columns first runs the product through the upper ones: columns 15 .. 8
      const float4 p2 = *reinterpret_cast<const float4*>(ab + 8), p3 = *reinterpret_cast<const float4*>(ab + 12);
      const float au[7] = {p2.y, p2.z, p2.w, p3.x, p3.y, p3.z, p3.w};   // a_9 .. a_15
      const int rm = q2 ? 32 : ri;         // (the other thread keeps 0 here: its own run starts at column 15)
      E = rm == 15 ? 1.0f : 0.f;
#pragma unroll
      for (int m = 14; m >= 8; --m) E = rm == m ? 1.0f : __fmul_rn(E, au[m - 8]);
    }
    const float4 h0 = *reinterpret_cast<const float4*>(ab + e0), h1 = *reinterpret_cast<const float4*>(ab + e0 + 4);
    const float hn[8] = {h0.y, h0.z, h0.w, h1.x, h1.y, h1.z, h1.w, ab[8]};   // a_{e0+k+1}; the last one meets E = 0 when e0 = 8
    const float4 d0 = *reinterpret_cast<const float4*>(dt_s + I16 * 16 + e0);
    const float4 d1 = *reinterpret_cast<const float4*>(dt_s + I16 * 16 + e0 + 4);
    const float dv[8] = {d0.x, d0.y, d0.z, d0.w, d1.x, d1.y, d1.z, d1.w};
    const int rr = ri - e0;                // this thread's columns k <= rr are on or below the diagonal
    float Ev[8];
#pragma unroll
    for (int k = 7; k >= 0; --k) {
      E = k == rr ? 1.0f : __fmul_rn(E, hn[k]);
      Ev[k] = E;
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      tv[k] = __fmul2_rn(unpack2(ww[k >> 1], 2 * (k & 1)),
                         __fmul2_rn(make_float2(dv[2 * k], dv[2 * k + 1]), make_float2(Ev[2 * k], Ev[2 * k + 1])));
      rmax = fmaxf(fmaxf(rmax, fabsf(tv[k].x)), fabsf(tv[k].y));
    }
  }
  rmax = fmaxf(rmax, __shfl_xor_sync(kAll, rmax, 1));
  const bool mono = b127_s[16] < __int_as_float(0x7f800000);
  auto warp_max = [&](float v) { return __uint_as_float(__reduce_max_sync(kAll, __float_as_uint(v))); };   // v >= 0
  constexpr float kSlack = 1.00001f;
  const uint32_t all = I16 > 1 ? (1u << (I16 - 1)) - 1u : 0u;   // the farther sub-blocks
  if (I16 > 1) {
    float rcp;
    asm("rcp.approx.f32 %0, %1;" : "=f"(rcp) : "f"(rmax));
    const float R = warp_max(__fmul_rn(dec, fminf(rcp, 3.0e38f)));   // (a row of zeros so far: any bound but 0 is above it)
    uint32_t m = __ballot_sync(kAll, __fmul_rn(bound, R) * kSlack > 1.0f);
    if (!mono) m = all;
    if (m) {
      do {
        const int c = 31 - __clz(m);
        m ^= 1u << c;
        float2 p[4];
        const float pm = products(c, p);
        rmax = fmaxf(rmax, __fmul_rn(pm, __fmul_rn(dec, gtab[c])));
      } while (m);
      rmax = fmaxf(rmax, __shfl_xor_sync(kAll, rmax, 1));
    }
  }
  const float inv = (rmax >= 1e-30f) ? __fdiv_rn(127.0f, rmax) : 0.f;
  int8_t* mq_tap = nullptr;
  if (TAPS && a.taps.Mq) mq_tap = a.taps.Mq + ((((i64)t.b * a.d.c + t.k) * a.d.H + t.h) * Q + i) * Q;
  if (q2 == 0) {
    rowbuf[r] = rmax;                   // read by the epilogue warps, with cs_i (they take its
    rowbuf[128 + r] = cs_i;             // exponential: the mask warps set the pace of the kernel)
    if (TAPS && a.taps.rowmax) a.taps.rowmax[(t.tok0 + i) * a.d.H + t.h] = rmax;
  }
  // (the sub-blocks after the row's own arrive as zeros: ChunkBMM writes them so)
  auto store = [&](int c, const float2 (&p)[4], float g, uint32_t keep0 = ~0u, uint32_t keep1 = ~0u) {
    const float2 g2 = make_float2(g, g);
    const uint2 v = make_uint2(pack4_rn_product(p[0], p[1], g2) & keep0, pack4_rn_product(p[2], p[3], g2) & keep1);
    *half_ptr(c) = v;
    if (TAPS && mq_tap) *reinterpret_cast<uint2*>(mq_tap + c * 16 + q2 * 8) = v;
  };
  {
    // Codes past the diagonal are cleared by their bytes: their E is 0, but 0 times a dt that is not finite is not, and a
    // token must not reach the rows before it whatever its dt.
    const int live = 8 * (ri - q2 * 8 + 1);   // bits of this thread's columns on or below the diagonal
    store(I16, tv, inv, __funnelshift_lc(~0u, 0u, max(live, 0)), __funnelshift_lc(~0u, 0u, max(live - 32, 0)));
  }
  const float di = __fmul_rn(dec, inv);
  if (I16 > 0) store(I16 - 1, tn, di);
  if (I16 > 1) {
    uint32_t m = __ballot_sync(kAll, __fmul_rn(bound, warp_max(di)) * kSlack >= 0.5f);
    if (!mono) m = all;
#pragma unroll 1
    for (int c = I16 - 2 - q2; c >= 0; c -= 2) {   // 16 columns of zeros per thread, alternately
      if ((m >> c) & 1u) continue;
      *reinterpret_cast<uint4*>(chunk_ptr(c)) = make_uint4(0u, 0u, 0u, 0u);
      if (TAPS && mq_tap) *reinterpret_cast<uint4*>(mq_tap + c * 16) = make_uint4(0u, 0u, 0u, 0u);
    }
#pragma unroll 1
    while (m) {
      const int c = 31 - __clz(m);
      m ^= 1u << c;
      float2 p[4];
      products(c, p);
      store(c, p, __fmul_rn(__fmul_rn(dec, gtab[c]), inv));
    }
  }
}

// CORR: a mean-correction vector is given; TAPS: intermediate tensors are written out (tests);
// YT: format of y (0 binary32, 1 fp16, 2 bf16: rounded to nearest even on the way to the staging tile);
// BIGQ: chunks of 128 tokens or more (128-row tiles with 128-byte CBq rows: the tile geometry, which
// every role's address arithmetic depends on, is then known at compile time)
template <bool CORR, bool TAPS, int YT, bool BIGQ>
__global__ void __launch_bounds__(kThreads, 1)
chunk_scan_tc(const __grid_constant__ CUtensorMap tm_C, const __grid_constant__ CUtensorMap tm_h,
              const __grid_constant__ CUtensorMap tm_x, const __grid_constant__ CUtensorMap tm_cb,
              const __grid_constant__ CUtensorMap tm_y, const ScanArgs a) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  // (no padding for the 1024-byte alignment the swizzled tiles need: the kernel takes all of the SM's shared
  // memory; the launcher checks that it uses no static shared memory, so that the dynamic part starts at the
  // window's base, and the kernel checks the address itself)
  uint8_t* smem = smem_raw;
  if ((smem_u32(smem) & 1023u) != 0) {
    if (threadIdx.x == 0 && a.status) atomicExch(a.status, (int32_t)SSDI8_ERR_ALIGN);
    return;
  }
  const Dims& d = a.d;
  const int Q = d.Q, N = d.N, P = d.P;
  const int TM = BIGQ ? 128 : Q;           // valid rows of a tile
  const int ntpu = BIGQ ? Q / 128 : 1;     // tiles per (batch, chunk, head)
  const uint32_t RBN = N, RBQ = BIGQ ? 128u : (uint32_t)Q;   // row bytes of the N-contracted and Q-contracted tiles
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;   // (the shuffle: uniform for the compiler)
  // tiles of this CTA: its units blockIdx.x, blockIdx.x + gridDim.x, ..., ntpu tiles each
  const int n_end = tiles_of_cta(a.w, (int)blockIdx.x, (int)gridDim.x, ntpu);
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + OFF_BAR);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + B_COUNT);
  Tile* first_tile = reinterpret_cast<Tile*>(bars + B_COUNT + 2);   // 448 .. 496 of the 512 bytes

  if (tid == 0) {
    for (int s = 0; s < 4; ++s) {
      mbar_init(&bars[B_CB_FULL + s], 1);
      mbar_init(&bars[B_CB_FREE + s], 1);
      mbar_init(&bars[B_MQ + s], kGroupWarps);
      mbar_init(&bars[B_TOK_FULL + s], 1);
      mbar_init(&bars[B_TOK_FREE + s], kGroupWarps);
      mbar_init(&bars[B_ACC + s], 2);      // both issuers' commits
      mbar_init(&bars[B_ACC_FREE + s], kEpiGroupWarps);
    }
    for (int s = 0; s < 8; ++s) {
      mbar_init(&bars[B_ROW_FULL + s], 1 + kGroupWarps);   // the column vectors and the mask warps' row scalars
      mbar_init(&bars[B_ROW_FREE + s], kEpiGroupWarps);
    }
    mbar_init(&bars[B_C_FULL], 1);
    mbar_init(&bars[B_C_FREE], 1);
    for (int s = 0; s < 2; ++s) {
      mbar_init(&bars[B_H_FULL + s], 1);
      mbar_init(&bars[B_H_FREE + s], 1);
      mbar_init(&bars[B_X_FULL + s], 1);
      mbar_init(&bars[B_X_FREE + s], (ntpu == 1 ? kEpiGroupWarps : kEpiWarps) + 1);  // the epilogue warps of the chunk's tiles and the MMAs
    }
    fence_mbar_init();
    tma_prefetch_desc(&tm_C); tma_prefetch_desc(&tm_h); tma_prefetch_desc(&tm_x);
    tma_prefetch_desc(&tm_cb); tma_prefetch_desc(&tm_y);
    *first_tile = decode_unit((int)blockIdx.x, d, TM);
  }
  pdl_launch_dependents();
  if (warp == 1) tmem_alloc(tmem_slot, kTmemCols);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = __shfl_sync(0xffffffffu, *tmem_slot, 0);
  pdl_wait();   // every role below reads or writes global memory

  if (warp == 0 || warp == 2) {
    // ------------------------------------------------------------ TMA producers.  Warp 0 serves the first tile of
    // every chunk (hq, CBq panel, scalar pack), warp 2 the second (xq rows, CBq panels); each also the tile's column
    // vectors.  The buffers of the two kinds of tile become free in an order that depends on how the mask
    // groups happen to run, and a single in-order producer let the first tile's loads wait behind the
    // second's: both mask groups waited 40 % of their time for CBq and the scalar pack.
    if (lane == 0) {
      const int mine = warp >> 1;          // tile of the chunk whose loads this warp issues (warp 2: xq as well)
      Tile t = *first_tile;
      // four rows of the pack and of the bounds row 32 + n (n - 1) / 2 entries, n = Q / 16 sub-blocks
      const uint32_t tok_bytes = (uint32_t)(16 * Q + (((32 + (Q >> 4) * ((Q >> 4) - 1) / 2) * 4 + 15) & ~15));
#pragma unroll 1
      for (int n0 = 0; n0 < n_end; n0 += ntpu, next_head(t, d, a.w, TM, ntpu)) {
        const int tg = t.h / a.w.hpg;   // group of the head (one division per chunk in this one thread)
        const int xs = x_index(n0, ntpu);
        const uint32_t xph = x_phase(n0, ntpu);
        if (mine == 0) {
          // the scalar pack of the chunk for the mask warps (four chunks deep: ahead of the wait for a CBq buffer)
          const int u = ntpu == 1 ? n0 : n0 >> 1, ts = u & 3;
          mbar_wait(&bars[B_TOK_FREE + ts], ((u >> 2) & 1) ^ 1, a.status);
          mbar_expect_tx(&bars[B_TOK_FULL + ts], tok_bytes);
          bulk_load(smem + OFF_TOK + ts * TOK_BYTES, a.pack + t.unit * kPackRows * Q, tok_bytes, &bars[B_TOK_FULL + ts]);
          mbar_wait(&bars[B_H_FREE + xs], xph ^ 1, a.status);
          mbar_expect_tx(&bars[B_H_FULL + xs], (uint32_t)(64 * N));
          tma_load_2d(smem + OFF_H + xs * H_BYTES, &tm_h, &bars[B_H_FULL + xs], 0, (int)((((i64)t.b * d.c + t.k) * d.H + t.h) * P));
        } else {
          mbar_wait(&bars[B_X_FREE + xs], xph ^ 1, a.status);
          mbar_expect_tx(&bars[B_X_FULL + xs], (uint32_t)(Q * 64));
          for (int j0 = 0; j0 < Q; j0 += TM)
            tma_load_3d(smem + OFF_X + xs * 16384 + j0 * 64, &tm_x, &bars[B_X_FULL + xs], 0, t.h, (int)(t.tok0 + j0));
        }
        if (mine >= ntpu) continue;
        const int n = n0 + mine, ci = cb_index(n, mine, ntpu);
        // the tile's three scalars, fetched here so that their latency is not in the epilogue's chain
        const float sc0 = a.s_C[tg], sc1 = a.D ? a.D[t.h] : 0.f, sc2 = a.s_cb[tg];
        mbar_wait(&bars[B_CB_FREE + ci], ((n >> 2) & 1) ^ 1, a.status);
        const int npanel = BIGQ ? mine + 1 : 1;
        mbar_expect_tx(&bars[B_CB_FULL + ci], (uint32_t)(npanel * TM * RBQ));
        for (int pn = 0; pn < npanel; ++pn)
          tma_load_2d(smem + cb_offset(ci) + pn * PANEL, &tm_cb, &bars[B_CB_FULL + ci], pn * (int)RBQ,
                      (int)((((i64)t.b * d.c + t.k) * d.G + tg) * Q + mine * TM));
        // the head's per-column vectors for the epilogue (read once per 8-column piece: from global
        // memory each read would be a long-latency load in its chain)
        const int r8 = n & 7;
        mbar_wait(&bars[B_ROW_FREE + r8], row_phase(n) ^ 1, a.status);
        uint8_t* cols = smem + OFF_ROW + r8 * ROW_BYTES + ROW_COLS;
        float* sc = reinterpret_cast<float*>(smem + OFF_ROW + r8 * ROW_BYTES + ROW_SCAL);
        sc[0] = sc0;
        sc[1] = sc1;
        sc[2] = sc2;
        mbar_expect_tx(&bars[B_ROW_FULL + r8], (uint32_t)((CORR ? 3 : 2) * P * 4));   // (an arrival: releases the stores above)
        bulk_load(cols, a.s_x + t.h * P, (uint32_t)(P * 4), &bars[B_ROW_FULL + r8]);
        bulk_load(cols + 256, a.s_h + t.h * P, (uint32_t)(P * 4), &bars[B_ROW_FULL + r8]);
        if (CORR) bulk_load(cols + 512, a.corr + t.h * P, (uint32_t)(P * 4), &bars[B_ROW_FULL + r8]);
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------ C h: this thread loads the one Cq buffer itself,
    // as soon as its MMAs of the tile before have read it, and issues the MMAs.  (The MMAs of the two
    // contractions have an issuer each: an issue is a chain of dependent instructions of one thread, and a single
    // thread that issued the 8 or 12 MMAs of a tile in turn took 1.0 us per tile with nothing else in its way,
    // half of the tile's time.)
    {   // (the whole warp runs the loop, see elect_one: one lane alone kept every descriptor in per-thread registers, 80 ns per MMA)
      const uint32_t idesc_off = idesc_s8(128, 64, 0, 0);
      const uint32_t sbase = smem_u32(smem);
      const uint64_t da = tile_desc(sbase + OFF_C, RBN);
      Tile t = *first_tile;
#pragma unroll 1
      for (int n = 0; n < n_end; ++n, next_tile(t, d, a.w, TM, ntpu)) {
        const int a4 = n & 3, xs = x_index(n, ntpu);
        const uint64_t db = tile_desc(sbase + OFF_H + xs * H_BYTES, RBN);
        const uint32_t acc = tmem + (uint32_t)a4 * 128u;
        const int tg = t.h / a.w.hpg;
        mbar_wait(&bars[B_C_FREE], (n & 1) ^ 1, a.status);
        if (elect_one()) {
          mbar_expect_tx(&bars[B_C_FULL], (uint32_t)(TM * N));
          tma_load_3d(smem + OFF_C, &tm_C, &bars[B_C_FULL], 0, tg, (int)(t.tok0 + t.it * TM));
        }
        __syncwarp();
        mbar_wait(&bars[B_ACC_FREE + a4], ((n >> 2) & 1) ^ 1, a.status);
        mbar_wait(&bars[B_H_FULL + xs], x_phase(n, ntpu), a.status);
        mbar_wait(&bars[B_C_FULL], n & 1, a.status);
        tc_fence_after();
        if (elect_one()) {
          // descriptors advance by a constant per 32-byte K step (their low bits are the address >> 4)
          mma_s8_ss(acc, da, db, idesc_off, 0);
          mma_s8_ss(acc, da + 2, db + 2, idesc_off, 1);
          if (N == 128) {
            mma_s8_ss(acc, da + 4, db + 4, idesc_off, 1);
            mma_s8_ss(acc, da + 6, db + 6, idesc_off, 1);
          }
          mma_commit(&bars[B_C_FREE]);
          if (t.it + 1 == ntpu) mma_commit(&bars[B_H_FREE + xs]);   // the chunk's last tile
          mma_commit(&bars[B_ACC + a4]);
        }
        __syncwarp();
      }
    }
  } else if (warp == 3) {
    // ------------------------------------------------------------ MMA issuer: Mq x
    {
      const uint32_t idesc_diag = idesc_s8(128, 64, 0, 1);
      const uint32_t sbase = smem_u32(smem);
#pragma unroll 1
      for (int n = 0; n < n_end; ++n) {
        const int it = ntpu == 1 ? 0 : (n & 1);   // a CTA's first tile is the first of its unit
        const int ci = cb_index(n, it, ntpu), a4 = n & 3, xs = x_index(n, ntpu);
        const uint32_t ph4 = (n >> 2) & 1;
        const uint32_t acc = tmem + (uint32_t)a4 * 128u + 64u;
        const uint64_t da = tile_desc(sbase + cb_offset(ci), RBQ), db = tile_desc(sbase + OFF_X + xs * 16384, 64);
        mbar_wait(&bars[B_ACC_FREE + a4], ph4 ^ 1, a.status);
        mbar_wait(&bars[B_X_FULL + xs], x_phase(n, ntpu), a.status);
        mbar_wait(&bars[B_MQ + ci], ph4, a.status);
        tc_fence_after();
        constexpr uint64_t kStepX = (32 * 64) >> 4;   // 32 tokens of x
        if (elect_one()) {
          mma_s8_ss(acc, da, db, idesc_diag, 0);
          mma_s8_ss(acc, da + 2, db + kStepX, idesc_diag, 1);
          if (BIGQ) {
            mma_s8_ss(acc, da + 4, db + 2 * kStepX, idesc_diag, 1);
            mma_s8_ss(acc, da + 6, db + 3 * kStepX, idesc_diag, 1);
            if (it) {   // the second panel of 128 columns
#pragma unroll
              for (uint32_t q = 0; q < 4; ++q)
                mma_s8_ss(acc, da + (PANEL >> 4) + 2 * q, db + (4 + q) * kStepX, idesc_diag, 1);
            }
          }
          mma_commit(&bars[B_CB_FREE + ci]);
          mma_commit(&bars[B_ACC + a4]);
          if (it + 1 == ntpu) mma_commit(&bars[B_X_FREE + xs]);   // the chunk's last tile
        }
        __syncwarp();
      }
    }
  } else if (warp < kEpiWarp0) {
    // ------------------------------------------------------------ mask warps.  With two tiles per chunk, group g
    // takes the chunks c = g, g + 2, ... of this CTA, both tiles: warp w builds the 16-row block w of the
    // first tile and block 7 - w of the second, which is the same number of 16-column sub-blocks for every
    // warp over a chunk (the causal rows grow with the row index); the group meets once per tile, though, so each
    // tile lasts as long as its slowest warp.  With one tile per chunk the groups alternate tiles.
    const int g = (warp - kMaskWarp0) / kGroupWarps;
    const int w = (warp - kMaskWarp0) % kGroupWarps;
    // A CTA of one chunk (all of them where there are no more chunks than SMs): a tile each.  With both tiles on the first group
    // the second one was idle: prefill of 256 tokens x 24 heads 25.6 -> 24.5 us, calls in a row.
    const bool one = ntpu == 2 && n_end == 2;
    Tile t = *first_tile;
    if (one && g) {
      t.it = 1;
      t.KJ = 2 * TM;
    } else if (g) {
      next_head(t, d, a.w, TM, ntpu);
    }
#pragma unroll 1
    for (int n = one ? g : g * ntpu; n < n_end; ++n) {
      const int ci = cb_index(n, t.it, ntpu), r8 = n & 7;
      const int u = ntpu == 1 ? n : n >> 1, ts = u & 3;   // the chunk's scalar pack
      const uint32_t ph4 = (n >> 2) & 1;
      const int rb = t.it ? kGroupWarps - 1 - w : w;
      // one warp of the group polls (the scalar pack, the CBq tile, and the epilogue of the tile that
      // used the row slot); the others wait at a hardware barrier, which costs no issue slots
      if (w == 0 && lane < 3) {
        const int bi = lane == 0 ? B_TOK_FULL + ts : lane == 1 ? B_CB_FULL + ci : B_ROW_FREE + r8;
        mbar_wait(&bars[bi], lane == 2 ? (row_phase(n) ^ 1) : lane == 1 ? ph4 : ((u >> 2) & 1), a.status);
      }
      named_bar_sync(1 + g, kGroupWarps * 32);
      mask_tile<TAPS>(smem + cb_offset(ci), reinterpret_cast<const float*>(smem + OFF_TOK + ts * TOK_BYTES),
                      reinterpret_cast<float*>(smem + OFF_ROW + r8 * ROW_BYTES), rb, lane, TM, RBQ, t, a);
      fence_async_smem();
      __syncwarp();
      const bool last = t.it + 1 == ntpu;   // the scalar pack serves both tiles of the chunk
      if (lane < (last ? 3 : 2)) mbar_arrive(&bars[lane == 0 ? B_MQ + ci : lane == 1 ? B_ROW_FULL + r8 : B_TOK_FREE + ts]);
      if (one) break;
      if (!last) {             // the chunk's second tile
        t.it = 1;
        t.KJ = 2 * TM;
      } else {                 // skip the other group's chunk (or tile)
        next_head(t, d, a.w, TM, ntpu);
        next_head(t, d, a.w, TM, ntpu);
        n += ntpu;
      }
    }
  } else {
    // ------------------------------------------------------------ epilogue warps: two groups of four take
    // alternate tiles; warp q of a group owns rows 32 q .. of the tile and all 64 columns
    const int ew = warp - kEpiWarp0;
    const int eg = ew / kEpiGroupWarps;     // group: tiles n = eg, eg + 2, ...
    const int q = warp & 3;                 // TMEM lane quarter this warp may read
    const int er = q * 32 + lane;           // row of the tile
    uint8_t* ystage = smem + OFF_YST + ew * 4096;   // [32][128 B], 16-byte chunks swizzled by the row
    uint8_t* srow = ystage + lane * 128;
    constexpr int PPR = YT ? 8 : 4;         // 8-column pieces per round (128 bytes of y per row)
    Tile t = *first_tile;
    if (eg) next_tile(t, d, a.w, TM, ntpu);
#pragma unroll 1
    for (int n = eg; n < n_end; n += 2) {
      const int ci = cb_index(n, t.it, ntpu), a4 = n & 3, xs = x_index(n, ntpu);
      const uint32_t ph4 = (n >> 2) & 1;
      const float* row = reinterpret_cast<const float*>(smem + OFF_ROW + (n & 7) * ROW_BYTES);
      const uint8_t* sX = smem + OFF_X + xs * 16384;
      const float4* ssx = reinterpret_cast<const float4*>(row + ROW_COLS / 4);
      const float4* ssh = ssx + 16;
      const float4* sco = ssx + 32;
      const bool ok = er < TM;
      const int ei = t.it * TM + er;
      // The row of x for the skip term goes to registers before the accumulators are waited for, and the warp
      // hands its share of the buffer back: were it read (and released) with the accumulators, the load of the
      // chunk after next would wait for the end of this epilogue, and with it the MMAs, the CBq buffers and the
      // mask of that chunk.
      uint4 xr[4];
      mbar_wait(&bars[B_X_FULL + xs], x_phase(n, ntpu), a.status);
#pragma unroll
      for (int j = 0; j < 4; ++j)
        xr[j] = ok ? *reinterpret_cast<const uint4*>(sX + swz_off((uint32_t)ei, (uint32_t)j, 64)) : make_uint4(0u, 0u, 0u, 0u);
      // (the fence: nothing has consumed the loads yet, and an arrival alone does not order them ahead of the next TMA
      // load into the buffer, which is another proxy's write.  Behind a warp's own backlog of global stores they were still
      // waiting when that load landed, and the skip term was that of the chunk after next.)
      fence_async_smem();
      __syncwarp();
      if (lane == 0) mbar_arrive(&bars[B_X_FREE + xs]);
      // two lanes of one warp of the group poll side by side, one barrier each: the accumulators and the row
      // slot (the head's column vectors and the row scalars written by the mask warps; not the mask barrier of
      // the CBq buffer, which may complete a second time before this group gets here); the other warps wait at
      // a hardware barrier, which costs no issue slots
      if (q == 0 && lane < 2) mbar_wait(&bars[lane == 0 ? B_ACC + a4 : B_ROW_FULL + (n & 7)], lane == 0 ? ph4 : row_phase(n), a.status);
      named_bar_sync(3 + eg, kEpiGroupWarps * 32);
      tc_fence_after();
      const float sC = row[ROW_SCAL / 4], Dh = row[ROW_SCAL / 4 + 1], scb = row[ROW_SCAL / 4 + 2];
      const float dec = ok ? exp32(row[128 + er]) * sC : 0.f;
      const float sm = ok ? scb * row[er] * (1.0f / 127.0f) : 0.f;
      const float2 dec2 = make_float2(dec, dec), sm2 = make_float2(sm, sm), Dh2 = make_float2(Dh, Dh);
      const uint32_t tbase = tmem + (uint32_t)a4 * 128u + ((uint32_t)(q * 32) << 16);
#pragma unroll                             // (the piece index folds into addresses and registers)
      for (int pc = 0; pc < 8; ++pc) {       // 8 columns at a time (keeps the accumulators in registers)
        int acc_o[8], acc_d[8];
        tmem_ld8(tbase + pc * 8, acc_o);
        tmem_ld8(tbase + 64 + pc * 8, acc_d);
        const uint4& x4 = xr[pc >> 1];
        const uint32_t xw[2] = {(pc & 1 ? x4.z : x4.x) ^ 0x80808080u, (pc & 1 ? x4.w : x4.y) ^ 0x80808080u};
        float2 v[4];
        tmem_ld_wait();
#pragma unroll
        for (int cc = 0; cc < 2; ++cc) {
          const float4 sx4 = ssx[pc * 2 + cc], sh4 = ssh[pc * 2 + cc];
          const float4 co4 = CORR ? sco[pc * 2 + cc] : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
          for (int e2 = 0; e2 < 2; ++e2) {
            const int pp = cc * 4 + e2 * 2;
            const float2 sx2 = e2 ? make_float2(sx4.z, sx4.w) : make_float2(sx4.x, sx4.y);
            const float2 sh2 = e2 ? make_float2(sh4.z, sh4.w) : make_float2(sh4.x, sh4.y);
            const float2 co2 = e2 ? make_float2(co4.z, co4.w) : make_float2(co4.x, co4.y);
            const float2 xv = unpack2(xw[cc], e2 * 2);
            const float2 ao = make_float2((float)acc_o[pp], (float)acc_o[pp + 1]);
            const float2 ad = make_float2((float)acc_d[pp], (float)acc_d[pp + 1]);
            // y = s_x (s_M acc_diag + D x) + s_h (dec acc_off) + corr: five packed operations
            const float2 u2 = __ffma2_rn(sm2, ad, __fmul2_rn(Dh2, xv));
            const float2 r2 = __ffma2_rn(sx2, u2, co2);
            v[cc * 2 + e2] = __ffma2_rn(sh2, __fmul2_rn(dec2, ao), r2);
          }
        }
        // the staging tile must have been read by the last store: waited for here, with this piece's arithmetic done
        if ((pc & (PPR - 1)) == 0) {
          if (lane == 3) tma_store_wait_read();
          __syncwarp();
        }
        if (ok) {
          if (YT == 0) {  // 4 values = one 16-byte chunk
#pragma unroll
            for (int cc = 0; cc < 2; ++cc)
              *reinterpret_cast<float4*>(srow + ((((pc & 3) * 2 + cc) ^ (lane & 7)) << 4)) =
                  make_float4(v[cc * 2].x, v[cc * 2].y, v[cc * 2 + 1].x, v[cc * 2 + 1].y);
          } else {        // 8 values = one 16-byte chunk
            uint32_t h[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              if (YT == 1) {
                const __half2 hv = __floats2half2_rn(v[e].x, v[e].y);
                h[e] = *reinterpret_cast<const uint32_t*>(&hv);
              } else {
                const __nv_bfloat162 bv = __floats2bfloat162_rn(v[e].x, v[e].y);
                h[e] = *reinterpret_cast<const uint32_t*>(&bv);
              }
            }
            *reinterpret_cast<uint4*>(srow + ((pc ^ (lane & 7)) << 4)) = make_uint4(h[0], h[1], h[2], h[3]);
          }
          if (TAPS && (a.taps.acc_off || a.taps.acc_diag)) {
            const i64 o = ((t.tok0 + ei) * d.H + t.h) * P + pc * 8;
#pragma unroll
            for (int pp = 0; pp < 8; ++pp) {
              if (a.taps.acc_off) a.taps.acc_off[o + pp] = acc_o[pp];
              if (a.taps.acc_diag) a.taps.acc_diag[o + pp] = acc_d[pp];
            }
          }
        }
        if ((pc & (PPR - 1)) == PPR - 1) {   // 128 bytes of every row are staged: store them
          if (pc == 7) tc_fence_before();
          fence_async_smem();
          __syncwarp();
          if (pc == 7 && lane < 2) {         // one release each, side by side
            mbar_arrive(&bars[lane == 0 ? B_ACC_FREE + a4 : B_ROW_FREE + (n & 7)]);
          } else if (lane == 3 && q * 32 < TM) {
            tma_store_3d(&tm_y, ystage, (pc / PPR) * 32, t.h, (int)(t.tok0 + t.it * TM + q * 32));
            tma_store_commit();
          }
        }
      }
      if (ntpu == 2) {   // the same tile of the next head
        const int it = t.it;
        next_head(t, d, a.w, TM, ntpu);
        t.it = it;
        t.KJ = (it + 1) * TM;
      } else {
        next_tile(t, d, a.w, TM, ntpu);
        next_tile(t, d, a.w, TM, ntpu);
      }
    }
    if (lane == 3) tma_store_wait_read();
  }
  tc_fence_before();
  drain_after_timeout(a.status);
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, kTmemCols);
  }
}

}  // namespace

ssdi8_status_t launch_chunk_scan(const Dims& d, const int8_t* xq, const int8_t* Cq,
                                 const int8_t* CBq, const int8_t* hq, const float* s_x,
                                 const float* s_C, const float* s_cb, const float* s_h,
                                 const float* pack, const float* D,
                                 const float* corr, void* y, int ydt, int32_t* status, const ScanTaps& taps,
                                 cudaStream_t st) {
  const int TM = d.Q < 128 ? d.Q : 128;
  const uint64_t T = (uint64_t)d.b * d.L;
  CUtensorMap tm_C, tm_h, tm_x, tm_cb, tm_y;
  {
    uint64_t dims[3] = {(uint64_t)d.N, (uint64_t)d.G, T};
    uint64_t str[2] = {(uint64_t)d.N, (uint64_t)d.G * d.N};
    uint32_t box[3] = {(uint32_t)d.N, 1, (uint32_t)TM};
    if (!encode_tensor_map(&tm_C, Cq, 1, 3, dims, str, box, d.N)) return SSDI8_ERR_CUDA;
  }
  {
    uint64_t dims[2] = {(uint64_t)d.N, (uint64_t)d.b * d.c * d.H * d.P};
    uint64_t str[1] = {(uint64_t)d.N};
    uint32_t box[2] = {(uint32_t)d.N, 64};
    if (!encode_tensor_map(&tm_h, hq, 1, 2, dims, str, box, d.N)) return SSDI8_ERR_CUDA;
  }
  {
    uint64_t dims[3] = {(uint64_t)d.P, (uint64_t)d.H, T};
    uint64_t str[2] = {(uint64_t)d.P, (uint64_t)d.H * d.P};
    uint32_t box[3] = {64, 1, (uint32_t)TM};
    if (!encode_tensor_map(&tm_x, xq, 1, 3, dims, str, box, 64)) return SSDI8_ERR_CUDA;
  }
  {
    uint64_t dims[2] = {(uint64_t)d.Q, (uint64_t)d.b * d.c * d.G * d.Q};
    uint64_t str[1] = {(uint64_t)d.Q};
    uint32_t box[2] = {(uint32_t)TM, (uint32_t)TM};
    if (!encode_tensor_map(&tm_cb, CBq, 1, 2, dims, str, box, TM)) return SSDI8_ERR_CUDA;
  }
  {
    const uint64_t eb = ydt ? 2 : 4;  // bytes per element of y
    uint64_t dims[3] = {(uint64_t)d.P, (uint64_t)d.H, T};
    uint64_t str[2] = {(uint64_t)d.P * eb, (uint64_t)d.H * d.P * eb};
    uint32_t box[3] = {ydt ? 64u : 32u, 1, 32};   // 128 bytes of a row per store
    if (!encode_tensor_map(&tm_y, y, (int)eb, 3, dims, str, box, 128)) return SSDI8_ERR_CUDA;
  }
  const int sms = sm_count();
  if (sms == 0) return SSDI8_ERR_CUDA;
  UnitWalk walk;
  int grid_i = 0;
  if (!make_unit_walk(d, TM, sms, &walk, &grid_i)) return SSDI8_ERR_SHAPE;
  ScanArgs a = {s_x, s_C, s_cb, s_h, pack, D, corr, static_cast<uint8_t*>(y), status, taps, d, walk};
  const size_t smem = SMEM_BYTES;
  const unsigned grid = (unsigned)grid_i;
  const bool tp = taps.acc_off || taps.rowmax || taps.Mq || taps.acc_diag;
  auto launch = [&](auto kernel) -> ssdi8_status_t {
    return launch_configured(kernel, dim3(grid), dim3(kThreads), smem, -1, true, st, tm_C, tm_h, tm_x, tm_cb, tm_y, a);
  };
  if (tp && ydt) return SSDI8_ERR_UNSUPPORTED;  // the taps come with binary32 y only
  const bool big = d.Q >= 128;
  auto pick = [&](auto corr_c, auto big_c) -> ssdi8_status_t {
    constexpr bool C = decltype(corr_c)::value, B = decltype(big_c)::value;
    if (tp) return launch(chunk_scan_tc<C, true, 0, B>);
    if (ydt == 0) return launch(chunk_scan_tc<C, false, 0, B>);
    if (ydt == 1) return launch(chunk_scan_tc<C, false, 1, B>);
    return launch(chunk_scan_tc<C, false, 2, B>);
  };
  ssdi8_status_t ls;
  if (corr)
    ls = big ? pick(std::true_type{}, std::true_type{}) : pick(std::true_type{}, std::false_type{});
  else
    ls = big ? pick(std::false_type{}, std::true_type{}) : pick(std::false_type{}, std::false_type{});
  if (ls != SSDI8_OK) return ls;
  SSDI8_LAUNCH_CHECK();
  return SSDI8_OK;
}

}  // namespace ssdi8
