// launch_table.h -- what a kernel needs once per device before it is launched: the
// opt-in to its dynamic shared memory and the number of resident blocks per SM
// for each ring depth.
#pragma once
#include <cuda_runtime.h>

#include <atomic>

namespace lbm {

// One table per kernel instantiation (a function-local static).  Both values belong to
// a device, so a second GPU of the process has its own row; an entry is one
// atomic word written after the opt-in, so that host threads may launch at the same
// time (two that find it empty both do the same work).  Asking the runtime at every launch
// instead costs the host about as much as a step of a 64^2 lattice takes.
struct LaunchTable {
  static constexpr int kDevices = 16, kDepths = 9;
  std::atomic<int> per_sm[kDevices][kDepths];
  LaunchTable() {
    for (auto& d : per_sm)
      for (auto& v : d) v.store(0, std::memory_order_relaxed);
  }

  // Resident blocks per SM of the kernel on `device` at ring depth `depth`.
  // opt_in() sets the function attribute and occupancy(&n) asks for the number; both act
  // on the current device, which is `device`.
  template <class OptIn, class Occupancy>
  cudaError_t get(int device, int depth, OptIn opt_in, Occupancy occupancy, int* blocks) {
    std::atomic<int>* slot =
        device >= 0 && device < kDevices && depth >= 0 && depth < kDepths ? &per_sm[device][depth] : nullptr;
    int n = slot ? slot->load(std::memory_order_acquire) : 0;
    if (n == 0) {
      cudaError_t e = opt_in();
      if (e == cudaSuccess) e = occupancy(&n);
      if (e != cudaSuccess) return e;
      if (n < 1) return cudaErrorInvalidConfiguration;
      if (slot) slot->store(n, std::memory_order_release);
    }
    *blocks = n;
    return cudaSuccess;
  }
};

}  // namespace lbm
