// Host run of LazyTable with a fake allocation: prints one line per request,
// "<served> <allocations so far> <builds so far> <key of the last build>".
// argv[1]: 1 = the allocation succeeds, 0 = it fails; the rest: keys.
#include <cstdio>
#include <cstdlib>

#include "lazy_table.cuh"

int main(int argc, char** argv) {
  const bool have = std::atoi(argv[1]) != 0;
  double storage = 0.0, last = -1.0;
  int allocs = 0, builds = 0;
  kfbi::LazyTable t;
  for (int i = 2; i < argc; ++i) {
    const double key = std::atof(argv[i]);
    double* p = t.get(
        key, [&]() -> double* { return ++allocs, have ? &storage : nullptr; },
        [&](double*) { ++builds, last = key; });
    std::printf("%d %d %d %g\n", p == &storage, allocs, builds, last);
  }
  return 0;
}
