// Host program of tests/test_ck_host.py: which 64-bit values fx_split_any and fx_split_wide take as operands.  Prints
// for each: values below the limit that were refused, values above it that were let through, largest of those
// in units of 2^61.
#include <cmath>
#include <cstdio>
#include <random>

#include "fixed.cuh"

using namespace shweno;

int main() {
  std::mt19937_64 rng(7);
  for (int wide = 0; wide < 2; ++wide) {
    const double limit = std::ldexp(1.0, wide ? 60 : 59);
    long refused = 0, passed = 0;
    double worst = 0.0;
    auto check = [&](int64_t z) {
      FxRange r{0};
      if (wide) fx_split_wide(z, r);
      else fx_split_any(z, r);
      const double m = std::fabs((double)z);
      if (m < limit * (1.0 - 1e-9) && r.bad()) ++refused;
      if (m > limit * (1.0 + 1e-9) && !r.bad()) {
        ++passed;
        worst = std::fmax(worst, m / std::ldexp(1.0, 61));
      }
    };
    for (int k = 0; k < 4096; ++k)  // every multiple of 1/512 up to +-4, and a value beside it
      for (int64_t off : {(int64_t)0, (int64_t)(rng() >> 12)}) {
        check((int64_t)((uint64_t)(k - 2048) << 52) + off);
        check(INT64_MAX - off);
        check(INT64_MIN + off);
      }
    for (int n = 0; n < 1000000; ++n) check((int64_t)rng());
    std::printf("%ld %ld %g\n", refused, passed, worst);
  }
}
