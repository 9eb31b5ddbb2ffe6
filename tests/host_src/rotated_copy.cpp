// Host checks of the rule for the optional copy of an FP64 system's blocks
// (rotated_copy.h): sizes on a device of 284,208 MiB, systems added until the
// device is full and taken away again, and a budget shared by threads.
#include <cstdio>
#include <memory>
#include <thread>
#include <vector>
#include "rotated_copy.h"

int main() {
  const size_t GiB = size_t(1) << 30, total = size_t(284208) << 20;
  struct { size_t copy, used; bool keep; } cases[] = {
      {GiB / 2, GiB, true},               // an ordinary system on an empty device
      {GiB / 2, 200 * GiB, true},         // and beside a large solve's workspaces
      {17 * GiB, 17 * GiB, true},         // a sixteenth of the device
      {18 * GiB, 18 * GiB, false},        // above it
      {150 * GiB, 150 * GiB, false},      // blocks in more than half of the device
      {GiB, total - 7 * GiB, false},      // more than an eighth of what is free
      {GiB, total - GiB / 2, false},      // more than what is free
      {0, 0, true},
  };
  for (const auto& c : cases) {
    mtf::RotatedBudget b;
    const bool keep = mtf::rotated_copy_fits(c.copy, total - c.used) && b.take(c.copy, total);
    if (keep != c.keep) return std::printf("copy %zu used %zu\n", c.copy, c.used), 1;
  }
  // many systems: as many fit as without copies but for a sixteenth of the device
  const size_t sizes[] = {GiB / 64, GiB, 5 * GiB, 30 * GiB, 100 * GiB};
  for (size_t block : sizes) {
    mtf::RotatedBudget b;
    std::vector<std::unique_ptr<mtf::RotatedShare>> shares;
    size_t used = 0, n = 0;
    while (used + block <= total) {
      used += block;
      ++n;
      shares.emplace_back(new mtf::RotatedShare);
      if (mtf::rotated_copy_fits(block, total - used) && shares.back()->take(b, block, total)) used += block;
    }
    if (b.used() > total / 16) return std::printf("copies %zu of %zu\n", b.used(), total), 1;
    if (n < (total - total / 16) / block) return std::printf("%zu systems of %zu\n", n, block), 1;
    shares.clear();
    if (b.used() != 0) return std::printf("%zu left\n", b.used()), 1;
  }
  // threads that take and give: never above the cap, nothing left behind
  mtf::RotatedBudget b;
  std::vector<std::thread> th;
  std::vector<int> bad(8, 0);
  for (int q = 0; q < 8; ++q)
    th.emplace_back([&, q] {
      for (int k = 0; k < 20000; ++k) {
        mtf::RotatedShare s;
        s.take(b, (1 + (k * 7 + q) % 5) * GiB, total);
        if (b.used() > total / 16) bad[size_t(q)] = 1;
      }
    });
  for (auto& t : th) t.join();
  for (int v : bad)
    if (v) return std::printf("above the cap\n"), 1;
  if (b.used() != 0) return std::printf("%zu left by threads\n", b.used()), 1;
  std::printf("ok\n");
  return 0;
}
