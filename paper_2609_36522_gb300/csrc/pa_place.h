// Where a caller's buffer lies, and whether a solver's kernels may take it
// there (pa_init's x_init, the x_out of a result or poll). Otherwise it goes
// through copies, which take a stream and buffers of any device.
#pragma once

#include <stddef.h>
#include <stdint.h>

namespace pa {

// [p, p + n) and [q, q + m) share no byte.
inline bool apart(const void* p, size_t n, const void* q, size_t m) {
  const uintptr_t a = reinterpret_cast<uintptr_t>(p), b = reinterpret_cast<uintptr_t>(q);
  return a + n <= b || b + m <= a;
}

// A kernel goes to the solver's stream, so the buffer and the calling thread's
// current device both have to be the solver's.
inline bool kernels_reach(bool device_memory, int mem_dev, int current_dev, int solver_dev) {
  return device_memory && mem_dev == solver_dev && current_dev == solver_dev;
}

}  // namespace pa
