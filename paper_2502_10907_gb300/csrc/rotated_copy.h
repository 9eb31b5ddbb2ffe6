// Whether an FP64 system keeps a second copy of its blocks in the form its
// matvec multiplies with (apply.cu), 32 bytes per entry; pure host C++.
//
// Without the copy the matvec takes 1.26 times as long with 2 right-hand
// sides, 1.5 times with one (split sphere of 11 rings), but nothing else may be
// refused for it.  It is kept while it takes at most an eighth of the free
// memory and all copies on the device together at most a sixteenth of the
// device: small next to what is left, and bounded however many systems there
// are.  (A line at the device's fill alone, seven eighths free, was tried: a
// program with the workspaces of one large solve lost the copy of a 455 MB
// system, 5.4 -> 4.7 solves per second.)
#pragma once

#include <atomic>
#include <cstddef>

namespace mtf {

// free_bytes: with the blocks allocated, the copy not
constexpr bool rotated_copy_fits(size_t copy_bytes, size_t free_bytes) { return copy_bytes <= free_bytes / 8; }

// Bytes of all rotated copies on one device; any thread.
class RotatedBudget {
 public:
  bool take(size_t bytes, size_t total_bytes) {
    const size_t cap = total_bytes / 16;
    size_t now = used_.load();
    do {
      if (bytes > cap || now > cap - bytes) return false;
    } while (!used_.compare_exchange_weak(now, now + bytes));
    return true;
  }
  void give(size_t bytes) { used_ -= bytes; }
  size_t used() const { return used_.load(); }

 private:
  std::atomic<size_t> used_{0};
};

// A system's share of its device's budget, given back with the system.
struct RotatedShare {
  RotatedBudget* budget = nullptr;
  size_t bytes = 0;
  RotatedShare() = default;
  RotatedShare(const RotatedShare&) = delete;
  RotatedShare& operator=(const RotatedShare&) = delete;
  ~RotatedShare() { give(); }
  bool take(RotatedBudget& b, size_t n, size_t total_bytes) {
    give();
    if (!b.take(n, total_bytes)) return false;
    budget = &b;
    bytes = n;
    return true;
  }
  void give() {
    if (budget) budget->give(bytes);
    budget = nullptr;
    bytes = 0;
  }
};

}  // namespace mtf
