// Prints what largest_cluster (host_internal.h) makes of a device that runs clusters up to
// a size, with and without sizes beyond the portable 8.  Host code only; built with nvcc and
// run by tests/test_cluster_host.py.
#include <cstdio>

#include "host_internal.h"

int main() {
  for (int most : {16, 8, 4, 2, 1, 0}) {
    auto runs = [&](int size) { return size <= most; };
    const int wide = nbldpc_host::largest_cluster(true, runs), portable = nbldpc_host::largest_cluster(false, runs);
    std::printf("%d %d %d\n", most, wide, portable);
  }
  return 0;
}
