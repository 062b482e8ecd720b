// Clusters of more CTAs than the device can place at once are not launched: a GPU that is partitioned (fewer SMs per GPC) holds
// smaller ones, or none.
#pragma once
#include <cstdint>

namespace purekv {

// The largest cluster size, from `want` down by halves, of which at least one fits (`at_once(size)`: how many do); 1 if none does.
template <typename AtOnce>
inline int32_t cluster_that_fits(int32_t want, AtOnce at_once) {
  int32_t c = want;
  while (c > 1 && at_once(c) < 1) c /= 2;
  return c;
}

#ifdef __CUDACC__
// How many clusters of this launch fit on the device at once, in the context and partition of its stream; 0 if none, or if the
// device cannot say.  (0.2 us of host time.)
template <typename Kernel>
inline int32_t clusters_at_once(Kernel kernel, const cudaLaunchConfig_t& cfg) {
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) != cudaSuccess) {
    (void)cudaGetLastError();
    return 0;
  }
  return n;
}
#endif

}  // namespace purekv
