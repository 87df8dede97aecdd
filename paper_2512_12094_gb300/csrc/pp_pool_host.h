// How much memory that nothing uses the library's pool may keep mapped.  Plain C++ (no
// CUDA), so that the CPU tests can compile it.
#pragma once

#include <algorithm>
#include <cstddef>

namespace pppool {

// Kept whatever else runs: mapping a gigabyte anew takes 0.8 ms and giving it back
// 1.35, which small jobs one after the other would pay each time.
constexpr size_t kKeepAlways = (size_t)1 << 30;
// Kept when a context ends, for the next one.
constexpr size_t kKeepBetween = (size_t)8 << 30;

// Bytes to keep of `unused` ones.  Another program of the device, or another allocator
// of this one, can have what is left of it: a quarter of the device stays free for
// them, or all that would be free without the pool's spare memory.  Where that much
// is free, a context that goes on keeps what it had (the scratch of its next layer).
inline size_t keep(size_t unused, size_t device_free, size_t device_total, bool context_ends) {
  if (unused <= kKeepAlways) return unused;
  if (device_free < device_total / 4) return kKeepAlways;
  return context_ends ? std::min(unused, kKeepBetween) : unused;
}

}  // namespace pppool
