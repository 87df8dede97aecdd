// How much memory that nothing uses the library's pool may keep mapped beyond the most
// that tables have taken: what the scratch of layers has added to it.  Plain C++ (no
// CUDA), so that the CPU tests can compile it.
#pragma once

#include <algorithm>
#include <cstddef>

namespace pppool {

// Kept whatever else runs: mapping a gigabyte anew takes 0.8 ms and giving it back
// 1.35, which small jobs one after the other would pay each time.
constexpr size_t kKeepAlways = (size_t)1 << 30;
// Scratch of a layer after which the pool is looked at, and with which a context had one
// the end of which looks: asking takes some 25 us, 3 % of a layer of 512 columns on 10
// qubits, whose scratch is 1.3 GB, and 1 % of a job of 45 sites and 100 columns.
constexpr size_t kLargeScratch = (size_t)4 << 30;
constexpr size_t kSmallScratch = (size_t)256 << 20;
// Kept when a context ends, for the next one.
constexpr size_t kKeepBetween = (size_t)8 << 30;

// Bytes to keep of `unused` ones.  A quarter of the device stays free for other
// programs and allocators, or all that would be free without this pool's spare memory.
// Where that much is free, a context that goes on keeps what it had: its next layer
// takes the like again.
inline size_t keep(size_t unused, size_t device_free, size_t device_total, bool context_ends) {
  if (unused <= kKeepAlways) return unused;
  if (device_free < device_total / 4) return kKeepAlways;
  return context_ends ? std::min(unused, kKeepBetween) : unused;
}

}  // namespace pppool
