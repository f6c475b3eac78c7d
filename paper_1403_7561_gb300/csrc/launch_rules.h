// Rules of launches that need neither the device nor the mesh (host only, no CUDA).
#pragma once

#include <atomic>

namespace qcad {

// FP32 Gram (gram32_kernel): tiles of 32 rows after which a thread's FP32 sums enter its double-float
// ones. Of a tile's eight chunks of four rows the first of `groups` row groups sums ceil(8 / groups), so
// no FP32 sum runs over more than 32 rows (after `groups` tiles it were 48 for six groups, that is for
// blocks of 13 to 16 columns).
inline int gram32_flush_tiles(int groups) { return 8 / ((8 + groups - 1) / groups); }

// Function attributes (the opt-in to more than 48 KB of shared memory) belong to a device: set() runs at
// the first launch on each and again where it failed.
struct PerDevice {
  static constexpr int MAX = 64;
  std::atomic<bool> done[MAX] = {};
};
template <class F>
void once_per_device(PerDevice& state, int device, F set) {
  const bool kept = device >= 0 && device < PerDevice::MAX;
  if (kept && state.done[device].load(std::memory_order_acquire)) return;
  if (set() && kept) state.done[device].store(true, std::memory_order_release);
}

}  // namespace qcad
