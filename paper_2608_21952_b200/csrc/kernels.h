// Host-side launchers of the SSDi8 kernels (internal to the library).
#pragma once
#include "common.cuh"

#include <utility>

namespace ssdi8 {

// kernel<<<grid, block, smem, st>>>(args...) with programmatic stream serialization allowed: the
// kernel may be scheduled while its predecessor in the stream drains (see pdl_wait in common.cuh).  cluster: CTAs of a
// cluster along x, where the kernel does not say so itself (0 or 1: none)
template <typename... KArgs, typename... Args>
inline cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, int cluster, dim3 block, size_t smem, cudaStream_t st,
                              Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  if (cluster > 1) {
    at[1].id = cudaLaunchAttributeClusterDimension;
    at[1].val.clusterDim.x = (unsigned)cluster;
    at[1].val.clusterDim.y = at[1].val.clusterDim.z = 1;
    cfg.numAttrs = 2;
  }
  return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}

// Launch attributes of a kernel (largest dynamic shared memory, preferred share of shared memory in percent or -1),
// set at its first launch on a device and remembered per kernel and device (launch_state.cu; set on
// every call they are 1.2 us of the 14.7 us of host time of a layer call).  check_static: fail if the
// kernel uses static shared memory (kernels that need their dynamic part at the window's base).
cudaError_t kernel_ready(const void* kernel, size_t smem, int carveout, bool check_static);
void kernel_forget(const void* kernel);   // the device was reset under us: set the attributes again
// (smem_most: the largest that any launch of the kernel asks for)
template <typename... KArgs, typename... Args>
inline ssdi8_status_t launch_any(void (*kernel)(KArgs...), dim3 grid, int cluster, dim3 block, size_t smem, size_t smem_most, int carveout,
                                 bool check_static, cudaStream_t st, Args&&... args) {
  const void* k = reinterpret_cast<const void*>(kernel);
  for (int attempt = 0; attempt < 2; ++attempt) {
    if (kernel_ready(k, smem_most, carveout, check_static) != cudaSuccess) break;
    if (launch_pdl(kernel, grid, cluster, block, smem, st, args...) == cudaSuccess) return SSDI8_OK;
    kernel_forget(k);
  }
  (void)cudaGetLastError();
  return SSDI8_ERR_CUDA;
}
template <typename... KArgs, typename... Args>
inline ssdi8_status_t launch_sized(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, size_t smem_most, int carveout,
                                   bool check_static, cudaStream_t st, Args&&... args) {
  return launch_any(kernel, grid, 0, block, smem, smem_most, carveout, check_static, st, std::forward<Args>(args)...);
}
template <typename... KArgs, typename... Args>
inline ssdi8_status_t launch_clustered(void (*kernel)(KArgs...), dim3 grid, int cluster, dim3 block, size_t smem, cudaStream_t st,
                                       Args&&... args) {
  return launch_any(kernel, grid, cluster, block, smem, smem, -1, false, st, std::forward<Args>(args)...);
}
template <typename... KArgs, typename... Args>
inline ssdi8_status_t launch_configured(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, int carveout,
                                        bool check_static, cudaStream_t st, Args&&... args) {
  return launch_sized(kernel, grid, block, smem, smem, carveout, check_static, st, std::forward<Args>(args)...);
}
int sm_count();   // of the current device (0 on failure)

// L1 / shared memory split of the streaming kernels that lead a layer (ChunkCumsum, the quantisers), in percent
// of shared memory: 64 KB of 228.  Launched through programmatic dependent launch right behind ChunkScan they
// would otherwise inherit its split (28 KB of L1), too little for the loads a streaming kernel keeps in flight
// (8 blocks x 128 threads x 128 bytes = 131 KB): layer step at batch 8 x 2048 x 80 heads, calls back to back,
// 0.300 ms without and 0.279 ms with the preference (1.03 and 0.94 ms at batch 4 x 8192 x 128 heads); 0, 14, 44
// and 58 percent are within 2 % of it.
constexpr int kStreamCarveout = 28;

ssdi8_status_t launch_quantize(const float* in, i64 R, i64 Ch, i64 I, float* scale, int mode,
                               int8_t* out, cudaStream_t st);

// The head of a layer step: ChunkCumsum, and the three static quantisers (x [T][H P] with H P step sizes, B and C [T][G N] with G
// step sizes each), as one launch or two.  clear_status: a status word that is set to 0, or NULL.
struct LayerInputs {
  const float* x; const float* B; const float* C;
};
ssdi8_status_t launch_lead(const Dims& d, const LayerInputs& in, const float* dt, const float* A, float* pack, float* gamma,
                           const float* s_x, const float* s_B, const float* s_C, int8_t* xq, int8_t* Bq, int8_t* Cq,
                           int32_t* clear_status, cudaStream_t st);

// Per-(batch, head, chunk) pack of kPackRows rows of Q floats: cs, dt, woff, atok, wmax, lut (see
// cumsum.cu); element (u, row, i) at pack[(u * kPackRows + row) * Q + i], u = (b*H + h)*c + k.
constexpr int kPackRows = 6;
enum { PACK_CS = 0, PACK_DT = 1, PACK_WOFF = 2, PACK_ATOK = 3, PACK_WMAX = 4, PACK_LUT = 5 };

// xBC [T][D + 2 G N] (dtype 0 fp32, 1 fp16, 2 bf16) -> xq [T][D], Bq, Cq [T][G N], static step sizes
ssdi8_status_t launch_quantize_entry(const void* xBC, int dtype, i64 T_, int D, int G, int N, const float* s_x,
                                     const float* s_B, const float* s_C, int8_t* xq, int8_t* Bq, int8_t* Cq,
                                     cudaStream_t st);

// ssdi8_chunk_scan_fwd's body; clear_status = false leaves the status word alone (the host pipeline clears it once for all
// its slices).  layer: the layer step, which quantises these (16-byte aligned) into a->xq, Bq and Cq first; all modules run then
ssdi8_status_t fwd_phases(const ssdi8_dims_t* dims, const ssdi8_fwd_args_t* a, uint32_t flags, void* workspace,
                          size_t workspace_bytes, void* stream, bool clear_status, const LayerInputs* layer = nullptr);

// pack [b,H,c,6,Q], gamma [b,H,c], tap_cs [b,H,c,Q] or NULL; clear_status: a status word the kernel sets to 0, or NULL;
// clear: so many words that it sets to 0 before the next kernel may be scheduled
// softplus: dt is the raw time step, dt = softplus(dt + dt_bias[h]) is applied first (dt_bias may be NULL)
ssdi8_status_t launch_cumsum(const Dims& d, const float* dt, const float* A, float* pack,
                             float* gamma, float* tap_cs, cudaStream_t st, const float* dt_bias = nullptr,
                             bool softplus = false, int32_t* clear_status = nullptr, uint32_t* clear = nullptr,
                             int nclear = 0);
ssdi8_status_t launch_softplus_dt(const float* dt_raw, const float* dt_bias, float* out, i64 rows, int H,
                                  cudaStream_t st);

// acc_cb (tap, may be NULL), CBq (may be NULL when s_cb is NULL), absmax_acc: per-group
// running max of |acc_cb| over the causal half (calibration; may be NULL).  after_state_kernel: the launch
// directly follows launch_chunk_state_passing (or launch_absmax_xs) in the same stream and may run beside it (see bmm.cu)
ssdi8_status_t launch_bmm(const Dims& d, const int8_t* Cq, const int8_t* Bq, const float* s_C,
                          const float* s_B, const float* s_cb, int8_t* CBq, int32_t* tap_acc,
                          uint32_t* absmax_acc, int32_t* status, cudaStream_t st, bool after_state_kernel = false);

// pass: ChunkState and StatePassing of eight chunks in one launch (loc and the taps unused)
struct StatePass {
  const float* s_h; const float* gamma; const float* init; float* final_state; int8_t* hq;
};
ssdi8_status_t launch_chunk_state(const Dims& d, const int8_t* xq, const int8_t* Bq,
                                  const float* s_x, const float* s_xs, const float* s_B,
                                  const float* pack, float* loc, int8_t* tap_Xsq,
                                  int32_t* tap_acc, int32_t* status, cudaStream_t st, const StatePass* pass = nullptr);

// ChunkState and StatePassing in one chunk-sequential kernel (loc never leaves the chip).  absmax_h (calibration):
// per-channel running max (binary32 bits) of |S| over init and every S_k; s_xs then holds the maxima of |X_scaled|, whose step
// sizes go to s_xs_out, and no other output is written
ssdi8_status_t launch_chunk_state_passing(const Dims& d, const int8_t* xq, const int8_t* Bq,
                                          const float* s_x, const float* s_xs, const float* s_B,
                                          const float* s_h, const float* pack, const float* gamma,
                                          const float* init, int8_t* hq, float* final_state,
                                          float* tap_loc, float* tap_prev, int8_t* tap_Xsq,
                                          int32_t* tap_acc, int32_t* status, bool int8_state,
                                          cudaStream_t st, uint32_t* absmax_h = nullptr, float* s_xs_out = nullptr);

// forward: in place of the fused state kernel (codes of a NaN)
ssdi8_status_t launch_state_passing(const Dims& d, const float* loc, const float* gamma,
                                    const float* init, const float* s_h, float* prev,
                                    float* final_state, int8_t* hq, cudaStream_t st, bool forward = false);

struct ScanTaps {
  int32_t* acc_off; float* rowmax; int8_t* Mq; int32_t* acc_diag;
};

// the same with the paper's FP16 ChunkScan2 operand
ssdi8_status_t launch_chunk_scan_f16(const Dims& d, const int8_t* xq, const int8_t* Cq,
                                     const int8_t* CBq, const int8_t* hq, const float* s_x, const float* s_C,
                                     const float* s_cb, const float* s_h, const float* pack, const float* D,
                                     const float* corr, void* y, int ydt, int32_t* status, cudaStream_t st);

ssdi8_status_t launch_chunk_scan(const Dims& d, const int8_t* xq, const int8_t* Cq,
                                 const int8_t* CBq, const int8_t* hq, const float* s_x,
                                 const float* s_C, const float* s_cb, const float* s_h,
                                 const float* pack, const float* D,
                                 const float* corr, void* y, int ydt, int32_t* status,
                                 const ScanTaps& taps, cudaStream_t st);

ssdi8_status_t launch_ssd_step(const Dims& d, const int8_t* xq, const float* s_x,
                               const int8_t* Bq, const float* s_B, const int8_t* Cq,
                               const float* s_C, const float* dt, const float* A, const float* D,
                               const float* corr, float* state, float* y, cudaStream_t st);

// Eq. 8: corr[ch] = eta * mean_r (y[r][ch] - yq[r][ch]); partial holds kMeanCorrMaxSlabs * Ch doubles
constexpr int kMeanCorrMaxSlabs = 256;
int mean_correction_slabs(i64 R);
ssdi8_status_t launch_mean_correction(const float* y, const float* yq, i64 R, i64 Ch, float eta, float* corr,
                                      double* partial, cudaStream_t st);

// measurement aid and self-test (selftest.cu): `nbatch` batches of int8_mma_peak_batch() MMAs of
// M 128 x N 256 x K 32 on every SM (ctas = number of CTAs launched); a bounded wait that runs out
ssdi8_status_t launch_int8_mma_peak(int nbatch, int32_t* status, int* ctas, cudaStream_t st);
int int8_mma_peak_batch();
ssdi8_status_t launch_bounded_wait_expires(int32_t* status, cudaStream_t st);

// calibration (calibrate.cu): per-channel running max of |X_scaled|; words set to 0; step sizes from maxima (s_h: binary32
// absmax; s_cb: int32 absmax of acc_cb, times s_C s_B), 1 where a maximum is 0
ssdi8_status_t launch_absmax_xs(const Dims& d, const int8_t* xq, const float* s_x, const float* pack, uint32_t* absmax,
                                cudaStream_t st);
ssdi8_status_t launch_clear_words(void* a, i64 n, cudaStream_t st);
ssdi8_status_t launch_finalize_scales(const uint32_t* max_h, float* s_h, i64 n, const uint32_t* max_cb, float* s_cb, i64 nq,
                                      const float* s_C, const float* s_B, cudaStream_t st);

}  // namespace ssdi8
