// Prints the FP64 plane kernel's block for every supported grid and request: N IB -> ib threads.
#include <cstdio>
#include <initializer_list>

#include "plane_block.h"

int main() {
  for (int n : {8, 10, 12, 16, 18, 20, 24, 25, 27, 30, 32, 36, 40})
    for (int ib = 1; ib <= 64; ++ib) {
      const ltmp2::PlaneBlock b = ltmp2::plane_block_f64(n, ib);
      std::printf("%d %d %d %d\n", n, ib, b.ib, b.threads);
    }
  return 0;
}
