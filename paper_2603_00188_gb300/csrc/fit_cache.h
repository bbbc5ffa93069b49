// How many clusters of the selection kernel are resident at once, remembered
// between launches: the occupancy query takes the host 5 us, and a launch
// compares up to nine cluster sizes.  Plain C++, no CUDA.
#pragma once

#include <algorithm>
#include <atomic>
#include <cstdint>

namespace stl {

// CTAs of `dyn` bytes of dynamic shared memory to an SM of `sm` bytes, `fixed`
// bytes of static and reserved shared memory each (allocated in 128-byte
// units), at most `most`.
inline int ctas_per_sm(int sm, int fixed, int dyn, int most) {
  return std::min(most, sm / ((fixed + dyn + 127) & ~127));
}

// The most dynamic shared memory (a multiple of 16 bytes, at most `cap`) with
// which `occ` CTAs still share an SM.  Every size of the same `occ` is asked
// for as this one, so that what is remembered does not depend on which size
// came first.
inline int largest_dynamic(int sm, int fixed, int occ, int cap) {
  return std::min(cap, (((sm / occ) & ~127) - fixed) & ~15);
}

// Answers by (device, cluster size, CTAs per SM), each with the context it was
// given in: a context may be limited to a part of the SMs, so another
// context's answer does not count.  "None fit" is not remembered.  A slot is
// one word, so threads need no lock: they read a whole answer or an older one.
template <int Devices, int Clusters, int Occ>
class FitCache {
 public:
  // -1: not known
  int get(int dev, int c, int occ, uint64_t ctx) const {
    if (dev < 0 || dev >= Devices || c > Clusters || occ > Occ || ctx == 0) return -1;
    const uint64_t v = slot_[dev][c][occ].load(std::memory_order_relaxed);
    return v != 0 && (v >> 16) == ctx ? (int)(v & 0xffffu) : -1;
  }
  void put(int dev, int c, int occ, uint64_t ctx, int fit) {
    if (dev < 0 || dev >= Devices || c > Clusters || occ > Occ || ctx == 0 || ctx >> 48 || fit < 1 || fit > 0xffff)
      return;
    slot_[dev][c][occ].store(ctx << 16 | (uint64_t)fit, std::memory_order_relaxed);
  }

 private:
  std::atomic<uint64_t> slot_[Devices][Clusters + 1][Occ + 1] = {};
};

}  // namespace stl
