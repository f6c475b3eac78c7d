// Rules of launches that need neither the device nor the mesh (host only, no CUDA).
#pragma once

#include <atomic>

namespace qcad {

// FP32 Gram (gram32_kernel): tiles of 32 rows after which a thread's FP32 sums enter its double-float
// ones. Of a tile's eight chunks of four rows the first of `groups` row groups sums ceil(8 / groups), so
// no FP32 sum runs over more than 32 rows (after `groups` tiles it were 48 for six groups, that is for
// blocks of 13 to 16 columns).
inline int gram32_flush_tiles(int groups) { return 8 / ((8 + groups - 1) / groups); }

// Element layers of the subdomain whose moments (27 doubles per element) fit the assembly's scratch of
// 64 MB; at least two, which a row needs.
inline int hm_slab_layers(int nx, int ny, int nz) {
  const long long fit = (64LL << 20) / (27LL * 8 * nx * ny);
  const int slab = (int)(fit < nz ? fit : nz);
  return slab < 2 ? (nz < 2 ? nz : 2) : slab;
}
// The next slab of the assembly, from node plane p0 of nz element layers: the layers [e0, e1) whose moments
// are formed and the node planes [p0, p1) whose rows they complete.
struct HmSlab {
  int e0, e1, p0, p1;
};
inline HmSlab hm_next_slab(int p0, int nz, int slab) {
  HmSlab r;
  r.p0 = p0;
  r.e0 = p0 > 0 ? p0 - 1 : 0;
  r.e1 = r.e0 + slab < nz ? r.e0 + slab : nz;
  r.p1 = r.e1 == nz ? nz + 1 : r.e1;
  return r;
}

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
