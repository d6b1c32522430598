// smem_limit.cuh -- a kernel's dynamic shared-memory limit, raised by whichever
// handle needs more.  Plain C++ without CUDA types, so that the host compiler
// can build it for the CPU tests.
#pragma once
#include <mutex>

namespace gnm {

inline std::mutex& limit_mutex() {
  static std::mutex m;
  return m;
}

// Raise a limit to at least `smem`: get(&current) and set(smem) return an error
// code, 0 for success.  The limit belongs to the kernel, not to a handle, so it
// is only ever raised: another handle may have opted in to more.  Handles may
// be created in several threads, so reading and setting are one step.
template <class Get, class Set>
auto raise_limit(Get get, Set set, int smem) -> decltype(set(smem)) {
  std::lock_guard<std::mutex> lock(limit_mutex());
  int current = 0;
  const auto e = get(&current);
  if (e || current >= smem) return e;
  return set(smem);
}

}  // namespace gnm
