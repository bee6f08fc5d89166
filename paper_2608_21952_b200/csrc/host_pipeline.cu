// The layer step as one call: Eq. 1 quantisation of fp32 x, B, C with static step sizes and the SSD
// layer forward (Algorithm 2).
// ssdi8_layer_fwd (device buffers): one chain on the caller's stream, linked by programmatic dependent
// launch.  ChunkCumsum reads dt and A only, so the quantisers' launch behind it starts without waiting
// for it and works beside it; the state kernel, ChunkBMM and ChunkScan follow.
// ssdi8_layer_fwd_host (host buffers): the same, one slice at a time, a slice being a run of chunks of one batch
// element (the state after it goes on to the next slice, in its exact binary32 or code value) or a few whole
// elements where they are small.  The host->device copies of the next slices and the device->host copy of the
// outputs of the ones before run on two copy streams while the kernels of a slice run on the caller's
// stream: the host link is busy in both directions for the whole call.  Only stream and event
// plumbing lives here; every arithmetic step is a kernel of this library.
#include <mutex>

#include "kernels.h"

namespace ssdi8 {
namespace {

constexpr int kStages = 3;   // slices in flight: arriving, computing, leaving
constexpr int kBlocks = 2;   // buffers of B, C and dt
constexpr uint32_t kLayerFlags = SSDI8_FLAG_FP16_OPERAND | SSDI8_FLAG_INT8_STATE | SSDI8_FLAG_Y_FP16 | SSDI8_FLAG_Y_BF16;

inline size_t up256(size_t v) { return (v + 255) & ~(size_t)255; }

// How the host pipeline cuts a call.  (Measured at one size, below; the limits of 2 and 8 MB are not, beyond the results being
// right on both sides of them.)  The pipeline fills with two slices' copies in and drains with two slices'
// copies out exposed, so slices are small; but a slice's kernels are a chain of about 30 us whatever its size, and a
// copy costs a few microseconds beside its bytes, so they are not smaller than kMinSlice of x.  Measured on PCIe 5
// x16 at 3 x 1024 tokens x 80 heads (63 MB of x in and of y out, 1.15 ms each way with the link to itself): a
// twelfth of the call per slice 1.87 ms, an eighth 1.92, a twentieth 1.88; whole elements 2.01.
// B, C and dt are small beside x: they cross in pieces of several slices.
struct Cut {
  int nb, Lt;        // elements and tokens per slice: nb > 1 only with Lt = L
  int per_elem;      // slices per element (1 when a slice is whole elements)
  int nslices;
  int block;         // slices per piece of B, C and dt
};
constexpr size_t kMinSlice = (size_t)2 << 20, kMaxSlice = (size_t)8 << 20;
Cut make_cut(const ssdi8_dims_t& d) {
  Cut c;
  const size_t x_elem = (size_t)d.seqlen * d.nheads * d.headdim * 4;
  size_t target = x_elem * d.batch / 12;
  target = target < kMinSlice ? kMinSlice : target > kMaxSlice ? kMaxSlice : target;
  if (x_elem <= target) {
    const size_t fit = target / x_elem;
    c.nb = fit < (size_t)d.batch ? (int)fit : d.batch;
    c.Lt = d.seqlen;
    c.per_elem = 1;
    c.nslices = (d.batch + c.nb - 1) / c.nb;
    c.block = 1;
    return c;
  }
  const int chunks = d.seqlen / d.chunk;
  int per = (int)((x_elem + target / 2) / target);       // about target bytes each, whole chunks, equal but for the last
  per = per < 1 ? 1 : per > chunks ? chunks : per;
  const int cps = (chunks + per - 1) / per;
  c.nb = 1;
  c.Lt = cps * d.chunk;
  c.per_elem = (chunks + cps - 1) / cps;
  c.nslices = d.batch * c.per_elem;
  const size_t small = ((size_t)2 * d.ngroups * d.dstate + d.nheads) * 4 * c.Lt;
  const size_t block = ((size_t)2 << 20) / small;
  c.block = block < 1 ? 1 : block > (size_t)c.per_elem ? c.per_elem : (int)block;
  return c;
}
ssdi8_dims_t slice_dims(const ssdi8_dims_t& d, int nb, int Lt) {
  ssdi8_dims_t s = d;
  s.batch = nb;
  s.seqlen = Lt;
  return s;
}

struct StageBuf {
  float *x, *y;
  float* fin;          // state after the slice: read by the next one, or copied out
  int8_t *xq, *Bq, *Cq;
};
struct BlockBuf {
  float *B, *C, *dt;
};
struct Layout {
  StageBuf st[kStages];
  BlockBuf blk[kBlocks];
  void* ws;
  int32_t* status;
  size_t ws_bytes, total;
};
Layout make_layout(const ssdi8_dims_t& d, const Cut& c, uint8_t* base, uint32_t flags) {
  Layout lo;
  const size_t T = (size_t)c.nb * c.Lt;   // tokens of a slice
  const size_t nx = T * d.nheads * d.headdim, nb = T * d.ngroups * d.dstate, ndt = T * d.nheads;
  const size_t nfin = (size_t)c.nb * d.nheads * d.headdim * d.dstate;
  size_t o = 0;
  auto take = [&](size_t bytes) { uint8_t* p = base + o; o = up256(o + bytes); return p; };
  for (StageBuf& s : lo.st) {
    s.x = reinterpret_cast<float*>(take(nx * 4));
    s.y = reinterpret_cast<float*>(take(nx * 4));
    s.fin = reinterpret_cast<float*>(take(nfin * 4));
    s.xq = reinterpret_cast<int8_t*>(take(nx));
    s.Bq = reinterpret_cast<int8_t*>(take(nb));
    s.Cq = reinterpret_cast<int8_t*>(take(nb));
  }
  for (BlockBuf& k : lo.blk) {
    k.B = reinterpret_cast<float*>(take(nb * 4 * c.block));
    k.C = reinterpret_cast<float*>(take(nb * 4 * c.block));
    k.dt = reinterpret_cast<float*>(take(ndt * 4 * c.block));
  }
  lo.status = reinterpret_cast<int32_t*>(take(256));
  const ssdi8_dims_t ds = slice_dims(d, c.nb, c.Lt);
  lo.ws_bytes = ssdi8_workspace_bytes(&ds, flags);
  lo.ws = take(lo.ws_bytes);
  lo.total = o;
  return lo;
}

// Copy streams and events of the host-buffer entry point, made once per device and kept for the life of the process.  All
// calls on a device share them, so a call holds `enqueue` while it enqueues: a wait for an event means the last record ahead
// of it, and two calls whose records and waits mixed would wait for each other's kernels instead of their own.
struct Plumbing {
  bool ready = false;
  std::mutex enqueue;
  cudaStream_t s_in = nullptr, s_out = nullptr;
  cudaEvent_t start = nullptr, in_done[kStages] = {}, cmp_done[kStages] = {}, out_done[kStages] = {}, blk_done[kBlocks] = {},
              gate[2] = {};
};
Plumbing g_plumb[64];
std::mutex g_plumb_mu;   // two threads may make their first call on a device at once

ssdi8_status_t get_plumbing(Plumbing** out) {
  int dev = 0;
  SSDI8_CUDA_CHECK(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64) return SSDI8_ERR_CUDA;
  Plumbing& p = g_plumb[dev];
  std::lock_guard<std::mutex> lock(g_plumb_mu);
  if (!p.ready) {
    SSDI8_CUDA_CHECK(cudaStreamCreateWithFlags(&p.s_in, cudaStreamNonBlocking));
    SSDI8_CUDA_CHECK(cudaStreamCreateWithFlags(&p.s_out, cudaStreamNonBlocking));
    auto make = [](cudaEvent_t& e) { return cudaEventCreateWithFlags(&e, cudaEventDisableTiming); };
    SSDI8_CUDA_CHECK(make(p.start));
    for (cudaEvent_t& e : p.in_done) SSDI8_CUDA_CHECK(make(e));
    for (cudaEvent_t& e : p.cmp_done) SSDI8_CUDA_CHECK(make(e));
    for (cudaEvent_t& e : p.out_done) SSDI8_CUDA_CHECK(make(e));
    for (cudaEvent_t& e : p.blk_done) SSDI8_CUDA_CHECK(make(e));
    for (cudaEvent_t& e : p.gate) SSDI8_CUDA_CHECK(make(e));
    p.ready = true;
  }
  *out = &p;
  return SSDI8_OK;
}

// Leaves the caller's stream behind the copy streams when a call ends early: copies that it has enqueued still read
// and write the caller's buffers.
struct JoinOnError {
  Plumbing* p;
  cudaStream_t st;
  bool armed = true;
  ~JoinOnError() {
    if (!armed) return;
    for (cudaStream_t side : {p->s_in, p->s_out})
      if (cudaEventRecord(p->start, side) == cudaSuccess) (void)cudaStreamWaitEvent(st, p->start, 0);
  }
};

struct LayerWs {
  int8_t *xq, *Bq, *Cq;
  void* ws;
  size_t ws_bytes, total;
};
LayerWs layer_ws(const ssdi8_dims_t& d, uint8_t* base, uint32_t flags) {
  LayerWs w;
  const size_t nx = (size_t)d.batch * d.seqlen * d.nheads * d.headdim;
  const size_t nb = (size_t)d.batch * d.seqlen * d.ngroups * d.dstate;
  size_t o = 0;
  auto take = [&](size_t bytes) { uint8_t* p = base + o; o = up256(o + bytes); return p; };
  w.xq = reinterpret_cast<int8_t*>(take(nx));
  w.Bq = reinterpret_cast<int8_t*>(take(nb));
  w.Cq = reinterpret_cast<int8_t*>(take(nb));
  w.ws_bytes = ssdi8_workspace_bytes(&d, flags);
  w.ws = take(w.ws_bytes);
  w.total = o;
  return w;
}

// quantisers + forward on device tensors, int8 tensors and workspace given; clear_status: the status word is set
// to 0 first (the host pipeline clears it once for all its slices)
ssdi8_status_t layer_step(const ssdi8_dims_t& d, const ssdi8_layer_args_t& a, const float* x, const float* B,
                          const float* C, const float* dt, const float* init, float* y, float* fin,
                          int32_t* status, int8_t* xq, int8_t* Bq, int8_t* Cq, void* ws, size_t ws_bytes,
                          uint32_t flags, cudaStream_t st, bool clear_status) {
  ssdi8_fwd_args_t f = {};
  f.xq = xq; f.Bq = Bq; f.Cq = Cq;
  f.s_x = a.s_x; f.s_B = a.s_B; f.s_C = a.s_C;
  f.dt = dt; f.A = a.A; f.D = a.D; f.corr = a.corr;
  f.s_xs = a.s_xs; f.s_cb = a.s_cb; f.s_h = a.s_h;
  f.init_state = init; f.y = y; f.final_state = fin; f.status = status;
  // (the three quantisers are one launch: it needs a power-of-two N, which every supported N is, and 16-byte
  // aligned tensors, which the entry points have checked or provide themselves)
  if ((d.dstate & (d.dstate - 1)) != 0) return SSDI8_ERR_UNSUPPORTED;
  const LayerInputs in = {x, B, C};
  return fwd_phases(&d, &f, flags & kLayerFlags, ws, ws_bytes, st, clear_status, &in);
}

bool layer_args_ok(const ssdi8_layer_args_t* a) {
  return a->x && a->B && a->C && a->dt && a->A && a->s_x && a->s_B && a->s_C && a->s_xs && a->s_cb && a->s_h && a->y;
}

}  // namespace
}  // namespace ssdi8

using namespace ssdi8;

extern "C" {

size_t ssdi8_layer_fwd_workspace_bytes(const ssdi8_dims_t* dims, uint32_t flags) {
  if (!dims || dims->batch <= 0 || (flags & ~kLayerFlags)) return 0;
  if (ssdi8_workspace_bytes(dims, flags) == 0) return 0;
  return layer_ws(*dims, nullptr, flags).total;
}

ssdi8_status_t ssdi8_layer_fwd(const ssdi8_dims_t* dims, const ssdi8_layer_args_t* a, void* workspace,
                               size_t workspace_bytes, uint32_t flags, void* stream) {
  if (!dims || !a || !workspace) return SSDI8_ERR_NULL;
  if (!layer_args_ok(a)) return SSDI8_ERR_NULL;
  if (flags & ~kLayerFlags) return SSDI8_ERR_UNSUPPORTED;
  const size_t need = ssdi8_layer_fwd_workspace_bytes(dims, flags);
  if (need == 0) return SSDI8_ERR_SHAPE;
  if (workspace_bytes < need) return SSDI8_ERR_WORKSPACE;
  if (reinterpret_cast<uintptr_t>(workspace) & 255) return SSDI8_ERR_ALIGN;
  // the quantisers read x, B and C sixteen bytes at a time (the other tensors are checked by the forward pass,
  // also before anything is enqueued)
  if ((reinterpret_cast<uintptr_t>(a->x) | reinterpret_cast<uintptr_t>(a->B) | reinterpret_cast<uintptr_t>(a->C)) & 15)
    return SSDI8_ERR_ALIGN;
  const LayerWs w = layer_ws(*dims, static_cast<uint8_t*>(workspace), flags);
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  return layer_step(*dims, *a, a->x, a->B, a->C, a->dt, a->init_state, a->y, a->final_state, a->status, w.xq, w.Bq,
                    w.Cq, w.ws, w.ws_bytes, flags, st, true);
}

size_t ssdi8_layer_fwd_host_scratch_bytes(const ssdi8_dims_t* dims, uint32_t flags) {
  if (!dims || dims->batch <= 0) return 0;
  if (ssdi8_workspace_bytes(dims, flags) == 0) return 0;   // unsupported dimensions or flags
  return make_layout(*dims, make_cut(*dims), nullptr, flags).total;
}

ssdi8_status_t ssdi8_layer_fwd_host(const ssdi8_dims_t* dims, const ssdi8_layer_args_t* a, void* scratch,
                                    size_t scratch_bytes, uint32_t flags, void* stream) {
  if (!dims || !a || !scratch) return SSDI8_ERR_NULL;
  if (!layer_args_ok(a)) return SSDI8_ERR_NULL;
  if (flags & ~kLayerFlags) return SSDI8_ERR_UNSUPPORTED;
  const size_t need = ssdi8_layer_fwd_host_scratch_bytes(dims, flags);
  if (need == 0) return SSDI8_ERR_SHAPE;
  if (scratch_bytes < need) return SSDI8_ERR_WORKSPACE;
  if (reinterpret_cast<uintptr_t>(scratch) & 255) return SSDI8_ERR_ALIGN;
  const Cut c = make_cut(*dims);
  const Layout lo = make_layout(*dims, c, static_cast<uint8_t*>(scratch), flags);
  Plumbing* p = nullptr;
  ssdi8_status_t s = get_plumbing(&p);
  if (s != SSDI8_OK) return s;
  std::lock_guard<std::mutex> lock(p->enqueue);
  cudaStream_t s_cmp = static_cast<cudaStream_t>(stream);
  const size_t L = dims->seqlen, D = (size_t)dims->nheads * dims->headdim, H = dims->nheads;
  const size_t GN = (size_t)dims->ngroups * dims->dstate, nstate = D * dims->dstate;   // state of an element
  const size_t yb = (flags & (SSDI8_FLAG_Y_FP16 | SSDI8_FLAG_Y_BF16)) ? 2 : 4;  // bytes per element of y
  // everything below is ordered after the work already in the caller's stream
  SSDI8_CUDA_CHECK(cudaMemsetAsync(lo.status, 0, sizeof(int32_t), s_cmp));
  SSDI8_CUDA_CHECK(cudaEventRecord(p->start, s_cmp));
  SSDI8_CUDA_CHECK(cudaStreamWaitEvent(p->s_in, p->start, 0));
  SSDI8_CUDA_CHECK(cudaStreamWaitEvent(p->s_out, p->start, 0));
  JoinOnError join{p, s_cmp};

  struct Slice {
    size_t b0, t0, nb, Lt, tok0, T;   // first element, first token in it, elements, tokens of each; the same over all tokens
    bool last;                        // of its elements
  };
  auto slice_of = [&](int i) {
    Slice v;
    const int part = i % c.per_elem;
    v.b0 = (size_t)(i / c.per_elem) * c.nb;
    v.t0 = (size_t)part * c.Lt;
    v.nb = (size_t)c.nb < dims->batch - v.b0 ? (size_t)c.nb : dims->batch - v.b0;
    v.Lt = (size_t)c.Lt < L - v.t0 ? (size_t)c.Lt : L - v.t0;
    v.tok0 = v.b0 * L + v.t0;
    v.T = v.nb * v.Lt;                // contiguous in every host tensor
    v.last = part + 1 == c.per_elem;
    return v;
  };
  // outputs of slice i, not before `gate` (an event of the input stream, or none)
  auto send_out = [&](int i, cudaEvent_t gate) -> ssdi8_status_t {
    const Slice v = slice_of(i);
    const int st = i % kStages;
    SSDI8_CUDA_CHECK(cudaStreamWaitEvent(p->s_out, p->cmp_done[st], 0));
    if (gate) SSDI8_CUDA_CHECK(cudaStreamWaitEvent(p->s_out, gate, 0));
    SSDI8_CUDA_CHECK(cudaMemcpyAsync(reinterpret_cast<uint8_t*>(a->y) + v.tok0 * D * yb, lo.st[st].y, v.T * D * yb,
                                     cudaMemcpyDeviceToHost, p->s_out));
    if (v.last && a->final_state)
      SSDI8_CUDA_CHECK(cudaMemcpyAsync(a->final_state + v.b0 * nstate, lo.st[st].fin, v.nb * nstate * 4,
                                       cudaMemcpyDeviceToHost, p->s_out));
    SSDI8_CUDA_CHECK(cudaEventRecord(p->out_done[st], p->s_out));
    return SSDI8_OK;
  };
  int blocks = 0;         // pieces of B, C and dt sent so far
  size_t blk_tok0 = 0;    // first token (over the whole batch) of the present piece
  for (int i = 0; i < c.nslices; ++i) {
    const Slice v = slice_of(i);
    const int part = i % c.per_elem, st = i % kStages;
    const StageBuf& sb = lo.st[st];
    // a new piece of B, C and dt: once the kernels of the piece that had its buffer are through
    if (part % c.block == 0) {
      const BlockBuf& k = lo.blk[blocks % kBlocks];
      const size_t left = v.nb * (L - v.t0), most = (size_t)c.block * c.Lt * v.nb, bt = most < left ? most : left;
      if (blocks >= kBlocks) SSDI8_CUDA_CHECK(cudaStreamWaitEvent(p->s_in, p->blk_done[blocks % kBlocks], 0));
      SSDI8_CUDA_CHECK(cudaMemcpyAsync(k.dt, a->dt + v.tok0 * H, bt * H * 4, cudaMemcpyHostToDevice, p->s_in));
      SSDI8_CUDA_CHECK(cudaMemcpyAsync(k.B, a->B + v.tok0 * GN, bt * GN * 4, cudaMemcpyHostToDevice, p->s_in));
      SSDI8_CUDA_CHECK(cudaMemcpyAsync(k.C, a->C + v.tok0 * GN, bt * GN * 4, cudaMemcpyHostToDevice, p->s_in));
      blk_tok0 = v.tok0;
      ++blocks;
    }
    const int kb = (blocks - 1) % kBlocks;
    const size_t off = v.tok0 - blk_tok0;   // of the slice in its piece, in tokens
    // x of the slice: the kernels of slice i - kStages have finished with this stage
    if (i >= kStages) SSDI8_CUDA_CHECK(cudaStreamWaitEvent(p->s_in, p->cmp_done[st], 0));
    SSDI8_CUDA_CHECK(cudaEventRecord(p->gate[i & 1], p->s_in));
    SSDI8_CUDA_CHECK(cudaMemcpyAsync(sb.x, a->x + v.tok0 * D, v.T * D * 4, cudaMemcpyHostToDevice, p->s_in));
    SSDI8_CUDA_CHECK(cudaEventRecord(p->in_done[st], p->s_in));
    // kernels of the slice: its inputs have arrived, and y and the state of slice i - kStages have left
    SSDI8_CUDA_CHECK(cudaStreamWaitEvent(s_cmp, p->in_done[st], 0));
    if (i >= kStages) SSDI8_CUDA_CHECK(cudaStreamWaitEvent(s_cmp, p->out_done[st], 0));
    const float* init = part > 0 ? lo.st[(i - 1) % kStages].fin : a->init_state ? a->init_state + v.b0 * nstate : nullptr;
    float* fin = (a->final_state || !v.last) ? sb.fin : nullptr;
    const ssdi8_dims_t ds = slice_dims(*dims, (int)v.nb, (int)v.Lt);
    s = layer_step(ds, *a, sb.x, lo.blk[kb].B + off * GN, lo.blk[kb].C + off * GN, lo.blk[kb].dt + off * H, init, sb.y, fin,
                   lo.status, sb.xq, sb.Bq, sb.Cq, lo.ws, lo.ws_bytes, flags, s_cmp, false);
    if (s != SSDI8_OK) return s;
    SSDI8_CUDA_CHECK(cudaEventRecord(p->cmp_done[st], s_cmp));
    if (v.last || (part + 1) % c.block == 0) SSDI8_CUDA_CHECK(cudaEventRecord(p->blk_done[kb], s_cmp));
    // The outputs of slice i - 2 leave together with the copy in of slice i, not when they are ready: a copy in that
    // becomes due while a copy out is under way was seen to start only when that has ended (the link then
    // carries one direction half of the time: 1.9 ms for 63 MB each way in twelve slices, 1.53 ms when the two
    // start together, 1.15 ms for one direction alone).
    if (i >= 2 && (s = send_out(i - 2, p->gate[i & 1])) != SSDI8_OK) return s;
  }
  for (int i = c.nslices < 2 ? 0 : c.nslices - 2; i < c.nslices; ++i)
    if ((s = send_out(i, nullptr)) != SSDI8_OK) return s;
  // the caller's stream ends after the last copies (one stream, in order: its last event covers all)
  SSDI8_CUDA_CHECK(cudaEventRecord(p->start, p->s_out));
  SSDI8_CUDA_CHECK(cudaStreamWaitEvent(s_cmp, p->start, 0));
  join.armed = false;
  if (a->status)
    SSDI8_CUDA_CHECK(cudaMemcpyAsync(a->status, lo.status, sizeof(int32_t), cudaMemcpyDeviceToHost, s_cmp));
  return SSDI8_OK;
}

}  // extern "C"
