// A device table of float64 values that depends on one parameter: storage on
// first use, built again when the parameter changes.  Where the storage cannot
// be had, the caller's form without the table serves, and the allocation is
// not tried again (a failing cudaMalloc in every solve would cost more than
// the table gains).
#pragma once

#include <cmath>

namespace kfbi {

struct LazyTable {
  double* p = nullptr;
  double key = 0.0;
  bool failed = false;

  // alloc() -> pointer or nullptr; build(pointer) enqueues the table for k
  template <class Alloc, class Build>
  double* get(double k, const Alloc& alloc, const Build& build) {
    if (p == nullptr) {
      if (failed) return nullptr;
      p = alloc();
      failed = p == nullptr;
      if (failed) return nullptr;
      key = std::nan("");
    }
    if (!(key == k)) {
      build(p);
      key = k;
    }
    return p;
  }
};

}  // namespace kfbi
