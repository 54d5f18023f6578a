// Running double-float dot products (ff.cuh) as a Hamiltonian pass forms them:
// a complex diagonal's two products, then up to 96 flips of two products each,
// the low word moved up after every second flip.
#include <cmath>
#include <cstdio>
#include <initializer_list>
#include <random>

#include "../paper_0902_0699_gb300/csrc/ff.cuh"

int main() {
  using namespace qc;
  std::mt19937_64 g(7);
  std::normal_distribution<double> nd;
  for (int kind = 0; kind < 3; ++kind)
    for (int rep = 0; rep < 20000; ++rep) {
      ffacc A{0.f, 0.f};
      long double want = 0, mag = 0;
      auto mac = [&]() {
        double a = nd(g) * 1e-2, b = nd(g) * 1e-3;
        if (kind == 1) a = std::fabs(a), b = std::fabs(b);   // no cancellation
        if (kind == 2) a *= std::exp2((int)(g() % 40) - 20);  // terms of very different sizes
        ffacc_add(A, ff_from_d(a), ff_from_d(b));
        want += (long double)a * b;
        mag += std::fabs((long double)a * b);
      };
      mac(), mac();
      for (int k = 0; k < 96; ++k) {
        mac(), mac();
        if (k & 1) ffacc_norm(A);
      }
      const ff r = ffacc_result(A);
      const long double err = std::fabs((long double)r.hi + (long double)r.lo - want);
      if (err > 0x1p-44L * mag) {
        std::printf("kind %d: error 2^%.2f of the terms' sizes\n", kind, std::log2((double)(err / mag)));
        return 1;
      }
    }
  std::puts("ok");
  return 0;
}
