// Host check of the co-densities' exponents (csrc/fixed.cuh): prints the number of norms whose exponent
// is below a smaller norm's, whose bound fails, and the exponents of 0, NaN and infinity.
#include <cmath>
#include <cstdio>

#include "fixed.cuh"

int main() {
  int falls = 0, bound = 0, last = -1 << 30;
  for (int e = -1074; e <= 996; ++e)
    for (int k = 0; k < 64; ++k) {
      const double x = std::ldexp(1.0 + k / 64.0, e);
      const int f = ltmp2::fx_exponent(x);
      if (f < last) ++falls;
      if (!(std::ldexp(1.0, f) > std::sqrt(x))) ++bound;
      last = f;
    }
  std::printf("%d %d %d %d %d\n", falls, bound, ltmp2::fx_exponent(0.0), ltmp2::fx_exponent(std::nan("")) == ltmp2::kFxNotFinite,
              ltmp2::fx_exponent(INFINITY) == ltmp2::kFxNotFinite);
  return 0;
}
