// Host state of the launches: which kernels have had their attributes set on which device, and the SM counts.
#include <atomic>

#include "kernels.h"

namespace ssdi8 {
namespace {

// One slot per kernel, found by its address; bit d of `devices` is set once the attributes are in place on device
// d.  Filled without a lock: two threads that meet at a first launch both set the same attributes.
struct Slot {
  std::atomic<const void*> kernel{nullptr};
  std::atomic<uint64_t> devices{0};
};
constexpr int kSlots = 128;   // the library has about a hundred kernels, most of them with attributes
Slot g_slots[kSlots];

Slot* find_slot(const void* kernel) {
  size_t i = (reinterpret_cast<uintptr_t>(kernel) >> 4) * 0x9E3779B97F4A7C15ull >> 57;
  for (int probe = 0; probe < kSlots; ++probe, i = (i + 1) & (kSlots - 1)) {
    const void* seen = g_slots[i].kernel.load(std::memory_order_acquire);
    if (seen == kernel) return &g_slots[i];
    if (seen == nullptr) {
      if (g_slots[i].kernel.compare_exchange_strong(seen, kernel) || seen == kernel) return &g_slots[i];
    }
  }
  return nullptr;   // (full: the attributes are then set on every call)
}

std::atomic<int> g_sms[64];

}  // namespace

cudaError_t kernel_ready(const void* kernel, size_t smem, int carveout, bool check_static) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  Slot* s = dev < 64 ? find_slot(kernel) : nullptr;
  if (s && (s->devices.load(std::memory_order_acquire) >> dev & 1)) return cudaSuccess;
  if (check_static) {
    cudaFuncAttributes fa;
    if ((e = cudaFuncGetAttributes(&fa, kernel)) != cudaSuccess) return e;
    if (fa.sharedSizeBytes != 0) return cudaErrorInvalidConfiguration;
  }
  if (smem > 0 && (e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) != cudaSuccess)
    return e;
  if (carveout >= 0 &&
      (e = cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, carveout)) != cudaSuccess)
    return e;
  if (s) s->devices.fetch_or(1ull << dev, std::memory_order_release);
  return cudaSuccess;
}

void kernel_forget(const void* kernel) {
  (void)cudaGetLastError();
  if (Slot* s = find_slot(kernel)) s->devices.store(0, std::memory_order_release);
}

int sm_count() {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0) return 0;
  int n = dev < 64 ? g_sms[dev].load(std::memory_order_relaxed) : 0;
  if (n == 0) {
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
    if (dev < 64) g_sms[dev].store(n, std::memory_order_relaxed);
  }
  return n;
}

}  // namespace ssdi8
