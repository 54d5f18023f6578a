// Sums of many equal terms in two words of fixed point (fixpt.cuh), as the
// blocks of a gradient's sum add them, against the exact product.
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <initializer_list>

#include "../paper_0902_0699_gb300/csrc/fixpt.cuh"

int main() {
  const double xs[] = {0.0, 0.5, 0.499999, -0.499999, 0.25, 12345.4375, -987654321.4999, 549755813888.375, -0x1p38, 1e-9};
  for (long long n : {1ll, 4096ll, 65536ll, 1ll << 20})
    for (double x : xs) {
      unsigned long long hi = 0, lo = 0;  // wraps as the device's atomics do
      for (long long i = 0; i < n; ++i) {
        long long h, l;
        qc::fx_split(x, h, l);
        hi += (unsigned long long)h;
        lo += (unsigned long long)l;
      }
      const double got = qc::fx_join((long long)hi, (long long)lo);
      const long double want = (long double)x * (long double)n;
      // half a unit of the low word a term, and one rounding of the result
      const long double tol = n * 0x1p-37L + 0x1p-53L * std::fabs((double)want);
      if (std::fabs((double)(got - want)) > tol) {
        std::printf("n = %lld, x = %.17g: %.17g instead of %.17Lg\n", n, x, got, want);
        return 1;
      }
    }
  std::puts("ok");
  return 0;
}
