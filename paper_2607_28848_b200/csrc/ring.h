// Place of a role in a ring of shared-memory stages.  Plain C++, so that the arithmetic runs on the host too.
#pragma once

#include <cstdint>

#ifdef __CUDACC__
#define MLORA_HD __host__ __device__ __forceinline__
#else
#define MLORA_HD inline
#endif

namespace mlora {

// Slot and lap parity of the next use.  Use number u takes slot u % n; the barrier "full" of that slot completes one phase
// per use, the phase of use u having parity (u / n) & 1.
struct Ring {
  int n, slot = 0;
  uint32_t parity = 0;
  int used = 0;                  // uses that next() has left behind, counted up to n
  MLORA_HD explicit Ring(int stages) : n(stages) {}
  MLORA_HD void next() {
    if (++slot == n) { slot = 0; parity ^= 1; }
    if (used < n) ++used;
  }
  // The uses whose loads may still be in flight - the last ones of every slot used so far, newest first; not the one the
  // role stands at, which it has not begun - as f(slot, parity of the use's phase).
  template <typename F>
  MLORA_HD void last_uses(F f) const {
    int s = slot;
    uint32_t p = parity;
    for (int i = 0; i < used; ++i) {
      if (--s < 0) { s = n - 1; p ^= 1; }
      f(s, p);
    }
  }
};

}  // namespace mlora
