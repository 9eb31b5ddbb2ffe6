// Takes the optional copy of an FP64 system's blocks away, as the library does
// where memory is short (test_gpu_rotated_copy.py).
#include "common.h"

extern "C" int drop_rotated(mtf_system sys) {
  const bool had = sys->d_rot64.p != nullptr;
  sys->d_rot64.p = nullptr;  // (left to the process)
  sys->d_rot64.n = 0;
  sys->rot64_share.give();
  sys->rot64_off = true;
  return had;
}
