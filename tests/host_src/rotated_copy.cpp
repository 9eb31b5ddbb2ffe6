// Host checks of the rule for the optional copy of an FP64 system's blocks
// (rotated_copy.h): sizes on a device of 284,208 MiB, and systems added until
// the device is full.
#include <cstdio>
#include <initializer_list>
#include "rotated_copy.h"

int main() {
  const size_t GiB = size_t(1) << 30, total = size_t(284208) << 20;
  struct { size_t copy, used; bool keep; } cases[] = {
      {GiB / 2, GiB, true},               // an ordinary system on an empty device
      {17 * GiB, 17 * GiB, true},         // one eighth of the device, blocks and copy
      {18 * GiB, 18 * GiB, false},        // above it
      {150 * GiB, 150 * GiB, false},      // blocks in more than half of the device
      {GiB / 2, 200 * GiB, false},        // a full device
      {GiB, total - GiB / 2, false},      // less free than the copy
      {0, 0, true},
  };
  for (const auto& c : cases)
    if (mtf::keep_rotated_copy(c.copy, total - c.used, total) != c.keep)
      return std::printf("copy %zu used %zu\n", c.copy, c.used), 1;
  // many systems: as many fit as without copies but for a sixteenth of the device
  for (size_t block : {GiB / 64, GiB, 5 * GiB, 30 * GiB, 100 * GiB}) {
    size_t used = 0, copies = 0, n = 0;
    while (used + block <= total) {
      used += block;
      ++n;
      if (mtf::keep_rotated_copy(block, total - used, total)) {
        used += block;
        copies += block;
      }
    }
    if (copies > total / 16) return std::printf("copies %zu of %zu\n", copies, total), 1;
    if (n < (total - total / 16) / block) return std::printf("%zu systems of %zu\n", n, block), 1;
  }
  std::printf("ok\n");
  return 0;
}
