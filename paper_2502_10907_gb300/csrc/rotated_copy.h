// Whether an FP64 system keeps a second copy of its blocks in the form its
// matvec multiplies with (apply.cu), 32 bytes per entry; pure host C++.
#pragma once

#include <cstddef>

namespace mtf {

// Without the copy the matvec takes 1.26 times as long with 2 right-hand
// sides, 1.5 times with one (split sphere of 11 rings), but nothing else may be
// refused for it: it is kept only while seven eighths of the device stay free
// beside it, so that all copies together never take more than a sixteenth of
// the memory (the blocks they copy take as much).  free_bytes: with the blocks
// allocated, the copy not.
constexpr bool keep_rotated_copy(size_t copy_bytes, size_t free_bytes, size_t total_bytes) {
  return free_bytes >= copy_bytes && free_bytes - copy_bytes >= total_bytes - total_bytes / 8;
}

}  // namespace mtf
