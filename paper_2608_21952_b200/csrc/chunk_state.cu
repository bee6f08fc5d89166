// ChunkState with the sparse-aware reformulation (Eq. 3) and the INT32 rescale (Eq. 4) on
// tcgen05 tensor cores.  One CTA per (batch, chunk, head):
//   LUT_state[i] = fmul(dt_i, exp32(fsub(cs_last, cs_i)))        (row 4 of the ChunkCumsum pack)
//   Xs_q[i,p]    = rne(fmul(fmul(float(xq[i,p]), fdiv(s_x, s_xs)), LUT_state[i]))   in place in smem
//   acc_st[n,p]  = sum_i Bq[i,n] Xs_q[i,p]     INT8 MMA over the tokens of the chunk, INT32 in TMEM
//   loc[p,n]     = fmul(float(acc_st), fmul(s_xs[h,p], s_B[g]))
// Both operands are token-major in HBM, i.e. MN-major for this contraction: TMA stages them
// as they are and the MMA reads them through MN-major descriptors (no transposes anywhere).
// The accumulator is held with the state index n on the TMEM lanes, so that each warp store
// of the epilogue writes 32 consecutive n of one p: full 128-byte lines of loc[p][n].
// The forward pass takes this kernel where there are too few (batch, head) pairs to fill the device with
// chunk-sequential ones (see fwd_phases).
// PASS: the eight chunks of a (batch, head) are a cluster.  The chunk-local states stay in shared memory, and once all of
// them are there each CTA takes an eighth of the (p, n) through all chunks (Eq. 5-6, as state_passing.cu does, operation for
// operation), reading the others' by way of distributed shared memory: no second launch, and no 32 KB per chunk out to L2 and
// back (layer calls: 512 tokens x 4 heads 17.0 -> 16.0 us, 2048 x 24 29.5 -> 28.4; and with the epilogue's scales in shared memory, the
// MMAs issued from uniform registers and the pass's operands fetched under them, 14.9 and 27.95).  The chunk count and the share of a thread
// are constants: written for up to eight chunks it took 94 registers instead of 72, and with two CTAs on every SM ChunkBMM no longer found room beside
// them (prefill of 1024 tokens x 37 heads 30.8 -> 26.8 us, 28.4 with two launches before; 2048 x 36 38.7 -> 33.9, 1024 x 4 18.2 -> 17.85).
#include "kernels.h"
#include "sm100.cuh"

namespace ssdi8 {
namespace {

using namespace sm100;

struct StateArgs {
  const float* s_x; const float* s_xs; const float* s_B; const float* pack;
  float* loc; int8_t* tap_Xsq; int32_t* tap_acc; int32_t* status;
  Dims d;
  const float* s_h; const float* gamma; const float* init; float* final_state; int8_t* hq;   // PASS
};

constexpr int kThreads = 256;
constexpr uint32_t OFF_B = 0;        // [Q][N]  Bq rows (token-major)
constexpr uint32_t OFF_X = 32768;    // [Q][64] xq rows -> Xs_q in place
constexpr uint32_t OFF_F = 49152;    // lut[256], s_x / s_xs [64], s_xs s_B [64], bars, tmem slot
constexpr uint32_t SMEM_BYTES = OFF_F + 256 * 4 + 128 * 4 + 64;

constexpr int kCluster = 8;   // chunks, CTAs of a cluster (PASS)

template <bool PASS>
__global__ void __launch_bounds__(kThreads, PASS ? 2 : 3)
chunk_state_tc(const __grid_constant__ CUtensorMap tm_B, const __grid_constant__ CUtensorMap tm_x,
               const StateArgs a) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  const Dims& d = a.d;
  const int Q = d.Q, N = d.N, P = d.P;
  const int TQ = Q < 128 ? Q : 128;  // rows per TMA box
  const int h = PASS ? blockIdx.y : blockIdx.x, k = PASS ? blockIdx.x : blockIdx.y, b = blockIdx.z;   // (PASS: the cluster is along x)
  const int g = h / (d.H / d.G);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const i64 tok0 = (i64)b * d.L + (i64)k * Q;
  uint8_t* sB = smem + OFF_B;
  uint8_t* sX = smem + OFF_X;
  float* lut = reinterpret_cast<float*>(smem + OFF_F);
  float* rxs = lut + 256;
  float* scale = rxs + 64;
  uint64_t* bars = reinterpret_cast<uint64_t*>(scale + 64);  // [0] operands landed, [1] MMA done
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2);

  if (tid == 0) {
    mbar_init(&bars[0], 1);
    mbar_init(&bars[1], 1);
    fence_mbar_init();
    tma_prefetch_desc(&tm_B);
    tma_prefetch_desc(&tm_x);
  }
  if (warp == 1) tmem_alloc(tmem_slot, 64);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  // (the wait ahead of the trigger: ChunkBMM, launched next, reads and writes global memory without waiting for this
  // kernel, so it must not be scheduled before this kernel's predecessors have completed)
  pdl_wait();
  pdl_launch_dependents();
  if (tid == 0) {
    mbar_expect_tx(&bars[0], (uint32_t)(Q * 64 + Q * N));
    for (int i0 = 0; i0 < Q; i0 += TQ) {
      tma_load_3d(sX + i0 * 64, &tm_x, &bars[0], 0, h, (int)(tok0 + i0));
      tma_load_3d(sB + i0 * N, &tm_B, &bars[0], 0, g, (int)(tok0 + i0));
    }
  }
  if (tid < Q) lut[tid] = a.pack[((((i64)b * d.H + h) * d.c + k) * kPackRows + PACK_LUT) * Q + tid];
  if (tid >= kThreads - 64) {   // one division per channel (each thread's own sixteen were a third of the kernel's instructions)
    const int p = tid - (kThreads - 64);
    const float sxs = a.s_xs[h * P + p];
    rxs[p] = __fdiv_rn(a.s_x[h * P + p], sxs);
    scale[p] = __fmul_rn(sxs, a.s_B[g]);   // (read from global memory in the epilogue they stood behind the MMAs)
  }
  __syncthreads();
  // per-column factors of this thread's 16 channels (16-byte chunk c of every row it visits)
  const int c = tid & 3;
  float rx[16];
#pragma unroll
  for (int e = 0; e < 16; e += 4) {
    const float4 v = *reinterpret_cast<const float4*>(rxs + c * 16 + e);
    rx[e] = v.x; rx[e + 1] = v.y; rx[e + 2] = v.z; rx[e + 3] = v.w;
  }
  // rows that re-quantise to zero, by the bound of the fused kernel (chunk_state_pass.cu): stored as zeros
  // without the arithmetic, and a 32-token slab of such rows issues no MMA
  float rxm = 0.f;
#pragma unroll
  for (int e = 0; e < 16; ++e) rxm = fmaxf(rxm, fabsf(rx[e]));
  rxm = fmaxf(rxm, __shfl_xor_sync(0xffffffffu, rxm, 1));
  rxm = fmaxf(rxm, __shfl_xor_sync(0xffffffffu, rxm, 2));
  const float b127 = __fmul_rn(127.0f, rxm);
  uint32_t live = 0;   // slabs with a row that does not (in the issuing warp)
  if (warp == 0) {
    for (int sl = 0; sl < Q / 32; ++sl)
      if (__any_sync(0xffffffffu, !(__fmul_rn(b127, fabsf(lut[sl * 32 + lane])) < 0.5f))) live |= 1u << sl;
    if (live == 0) live = 1u;
  }
  mbar_wait(&bars[0], 0, a.status);

  // ---- X_scaled, re-quantised in place (thread: chunk c of rows tid/4, tid/4 + 64, ...)
  for (int i = tid >> 2; i < Q; i += kThreads / 4) {
    uint4* ptr = reinterpret_cast<uint4*>(sX + swz_off((uint32_t)i, (uint32_t)c, 64));
    const float l = lut[i];
    if (__fmul_rn(b127, fabsf(l)) < 0.5f) {
      *ptr = make_uint4(0u, 0u, 0u, 0u);
      if (a.tap_Xsq) *reinterpret_cast<uint4*>(a.tap_Xsq + ((tok0 + i) * d.H + h) * P + c * 16) = make_uint4(0u, 0u, 0u, 0u);
      continue;
    }
    const uint4 w4 = *ptr;
    const uint32_t ww[4] = {w4.x ^ 0x80808080u, w4.y ^ 0x80808080u, w4.z ^ 0x80808080u, w4.w ^ 0x80808080u};
    uint32_t o[4];
#pragma unroll
    for (int w = 0; w < 4; ++w) {
      uint32_t q4[4];
#pragma unroll
      for (int e = 0; e < 4; ++e)
        q4[e] = rne_clamp_bits(__fmul_rn(__fmul_rn(s8_to_f32(ww[w], e), rx[w * 4 + e]), l));
      o[w] = pack4_bits(q4[0], q4[1], q4[2], q4[3]);
    }
    const uint4 v = make_uint4(o[0], o[1], o[2], o[3]);
    *ptr = v;
    if (a.tap_Xsq) *reinterpret_cast<uint4*>(a.tap_Xsq + ((tok0 + i) * d.H + h) * P + c * 16) = v;
  }
  fence_async_smem();
  __syncthreads();

  // ---- acc[n][p] = sum_i Bq[i][n] Xs_q[i][p]: A = Bq (MN-major, M = N states), B = Xs_q (MN-major)
  const uint32_t tmem = *tmem_slot;
  if (warp == 0) {   // (the descriptors are formed by the whole warp, see elect_one)
    tc_fence_after();
    const uint32_t idesc = idesc_s8(N, 64, 1, 1);
    const uint32_t sBa = smem_u32(sB), sXa = smem_u32(sX);
    uint32_t first = 0;
    if (elect_one()) {
#pragma unroll 1
      for (uint32_t m = live; m; m &= m - 1) {
        const int s = __ffs((int)m) - 1;
        mma_s8_ss(tmem, tile_desc(sBa + 32 * s * N, (uint32_t)N), tile_desc(sXa + 32 * s * 64, 64), idesc, first);
        first = 1;
      }
      mma_commit(&bars[1]);
    }
  }
  __syncwarp();
  // (PASS) this CTA's eighth of the states, four neighbouring n a thread (128 or 256 threads); what they need from global memory
  // is on its way under the MMAs
  const int units = P * N / 4, u = k * (units / kCluster) + tid;
  const bool mine = PASS && tid < units / kCluster;
  const i64 bh = (i64)b * d.H + h;
  float gam[kCluster], inv_h = 0.f;
  float4 S = make_float4(0.f, 0.f, 0.f, 0.f);
  if (mine) {
#pragma unroll
    for (int j = 0; j < kCluster; ++j) gam[j] = a.gamma[bh * kCluster + j];
    inv_h = __fdiv_rn(1.0f, a.s_h[h * P + 4 * u / N]);
    if (a.init) S = reinterpret_cast<const float4*>(a.init)[bh * units + u];
  }
  mbar_wait(&bars[1], 0, a.status);
  tc_fence_after();

  // ---- epilogue.  M = 128: accumulator row n on TMEM lane n.  M = 64: row n on lane
  // (n % 16) + 32 (n / 16), i.e. the first 16 lanes of each warp's quarter.
  {
    const int q = warp & 3, ch = warp >> 2;
    int acc[32];
    tmem_ld32(tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(ch * 32), acc);
    tmem_ld_wait();
    const bool ok = (N == 128) || (lane < 16);
    const int n = (N == 128) ? q * 32 + lane : q * 16 + lane;
    if (PASS) {   // (over the Bq tile, which the MMAs have read)
      float* loc = reinterpret_cast<float*>(sB) + n;
      if (ok) {
#pragma unroll
        for (int pp = 0; pp < 32; ++pp) {
          const int p = ch * 32 + pp;
          loc[p * N] = __fmul_rn(i22_to_f32(acc[pp]), scale[p]);
        }
      }
    } else if (ok) {
      const i64 obase = ((((i64)b * d.c + k) * d.H + h) * P) * N + n;
#pragma unroll
      for (int pp = 0; pp < 32; ++pp) {
        const int p = ch * 32 + pp;
        a.loc[obase + (i64)p * N] = __fmul_rn(i22_to_f32(acc[pp]), scale[p]);
        if (a.tap_acc) a.tap_acc[obase + (i64)p * N] = acc[pp];
      }
    }
  }
  tc_fence_before();
  if (PASS) {
    cluster_sync();
    if (mine) {
      float4 l[kCluster];
#pragma unroll
      for (int j = 0; j < kCluster; ++j) {
        uint32_t at;
        asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(at) : "r"(smem_u32(sB) + 16u * (uint32_t)u), "r"(j));
        asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
                     : "=f"(l[j].x), "=f"(l[j].y), "=f"(l[j].z), "=f"(l[j].w)
                     : "r"(at)
                     : "memory");
      }
      uint32_t* hq = reinterpret_cast<uint32_t*>(a.hq) + ((i64)b * kCluster * d.H + h) * units + u;
#pragma unroll
      for (int j = 0; j < kCluster; ++j) {
        hq[(i64)j * d.H * units] = pack4_bits(rne_clamp_bits(__fmul_rn(S.x, inv_h)), rne_clamp_bits(__fmul_rn(S.y, inv_h)),
                                              rne_clamp_bits(__fmul_rn(S.z, inv_h)), rne_clamp_bits(__fmul_rn(S.w, inv_h)));
        S.x = __fmaf_rn(gam[j], S.x, l[j].x);
        S.y = __fmaf_rn(gam[j], S.y, l[j].y);
        S.z = __fmaf_rn(gam[j], S.z, l[j].z);
        S.w = __fmaf_rn(gam[j], S.w, l[j].w);
      }
      if (a.final_state) reinterpret_cast<float4*>(a.final_state)[bh * units + u] = S;
    }
    cluster_sync();   // (the others have read this CTA's)
  }
  drain_after_timeout(a.status);
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, 64);
  }
}

}  // namespace

ssdi8_status_t launch_chunk_state(const Dims& d, const int8_t* xq, const int8_t* Bq,
                                  const float* s_x, const float* s_xs, const float* s_B,
                                  const float* pack, float* loc, int8_t* tap_Xsq,
                                  int32_t* tap_acc, int32_t* status, cudaStream_t st, const StatePass* pass) {
  const int TQ = d.Q < 128 ? d.Q : 128;
  const uint64_t T = (uint64_t)d.b * d.L;
  CUtensorMap tm_B, tm_x;
  {
    uint64_t dims[3] = {(uint64_t)d.N, (uint64_t)d.G, T};
    uint64_t str[2] = {(uint64_t)d.N, (uint64_t)d.G * d.N};
    uint32_t box[3] = {(uint32_t)d.N, 1, (uint32_t)TQ};
    if (!encode_tensor_map(&tm_B, Bq, 1, 3, dims, str, box, d.N)) return SSDI8_ERR_CUDA;
  }
  {
    uint64_t dims[3] = {(uint64_t)d.P, (uint64_t)d.H, T};
    uint64_t str[2] = {(uint64_t)d.P, (uint64_t)d.H * d.P};
    uint32_t box[3] = {64, 1, (uint32_t)TQ};
    if (!encode_tensor_map(&tm_x, xq, 1, 3, dims, str, box, 64)) return SSDI8_ERR_CUDA;
  }
  StateArgs a = {s_x, s_xs, s_B, pack, loc, tap_Xsq, tap_acc, status, d, nullptr, nullptr, nullptr, nullptr, nullptr};
  const size_t smem = SMEM_BYTES + 1024;
  if (!pass) return launch_configured(chunk_state_tc<false>, dim3(d.H, d.c, d.b), dim3(kThreads), smem, -1, false, st, tm_B, tm_x, a);
  if (d.c != kCluster) return SSDI8_ERR_SHAPE;
  a.s_h = pass->s_h;
  a.gamma = pass->gamma;
  a.init = pass->init;
  a.final_state = pass->final_state;
  a.hq = pass->hq;
  return launch_clustered(chunk_state_tc<true>, dim3(kCluster, d.H, d.b), kCluster, dim3(kThreads), smem, st, tm_B, tm_x, a);
}

}  // namespace ssdi8
