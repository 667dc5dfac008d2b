// Host-side check of the FP64 segment weight (vet_exp64.h) against long
// double: over optical depths of every size, at the table's and the forms'
// seams, and that what its premise does not cover is refused.
// Prints "ok" or the failure.
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <limits>
#include <random>
#include <vector>

#include "vet_exp64.h"

int main() {
  std::vector<double> tab(vet::kExp64TableDoubles);
  vet::exp64_fill_table(tab.data());
  const long double ln2 = 0.693147180559945309417232121458176568L;
  std::mt19937_64 rng(3);
  std::uniform_real_distribution<double> U(0.0, 1.0);
  double worst = 0.0, worst_x = 0.0;
  long refused = 0, count = 0;
  auto check = [&](double kappa, double len) {
    double w;
    bool thin;
    ++count;
    if (!vet::exp64_weight(kappa, len, (float)(1024.0 * len), tab.data(), w, thin)) {
      ++refused;
      return true;
    }
    const long double y = (long double)kappa * (long double)len;
    const long double want = thin ? std::expm1(y * ln2) : std::exp2(y);
    if (want == 0.0L) return w == 0.0;
    const double err = (double)(std::fabs((long double)w - want) / std::fabs(want));
    if (err > worst) {
      worst = err;
      worst_x = (double)-y;
    }
    // thin: r, F, q, the table's E ln2 and T, the product and w, each half an
    // ulp at most; thick: q is below 2^-10 of w, so E and w alone count
    return err <= (thin ? 4.0 : 2.5) * 1.2e-16;
  };
  // depths log-uniform over [1e-25, 690], with lengths and opacities of any scale
  for (int i = 0; i < 4000000; ++i) {
    const double x = std::exp(std::log(1e-25) + U(rng) * (std::log(690.0) - std::log(1e-25)));
    const double len = -std::exp((U(rng) - 0.5) * 60.0);
    if (!check(x * 1.4426950408889634 / -len, len)) return std::printf("depth %g: off by %g\n", x, worst), 1;
  }
  if (refused) return std::printf("%ld of %ld refused\n", refused, count), 1;
  // every seam: depths within rounding of half-integer multiples of the step, and the form's change
  for (int n = 0; n < 3000; ++n)
    for (int d = -3; d <= 3; ++d) {
      double y = (n + 0.5) / 1024.0;
      for (int s = 0; s < (d < 0 ? -d : d); ++s) y = std::nextafter(y, d < 0 ? 0.0 : 10.0);
      if (!check(y, -1.0)) return std::printf("seam %d %d: off by %g\n", n, d, worst), 1;
    }
  if (refused) return std::printf("%ld refused at seams\n", refused), 1;
  // kappa = 0 and tiny depths: exact
  double w;
  bool thin;
  if (!vet::exp64_weight(0.0, -0.3, -0.3f * 1024, tab.data(), w, thin) || w != 0.0 || !thin) return std::printf("zero\n"), 1;
  for (double k : {1e-300, 1e-40, 1e-30}) {
    if (!vet::exp64_weight(k, -1.0, -1024.f, tab.data(), w, thin) || !thin) return std::printf("tiny refused\n"), 1;
    if (std::fabs(w + (double)(k * ln2)) > 2.3e-16 * k) return std::printf("tiny %g\n", k), 1;
  }
  // refused: not a number, infinite, beyond the range, growing, FP32 out of range
  const double inf = std::numeric_limits<double>::infinity(), nan = std::numeric_limits<double>::quiet_NaN();
  const double bad[][2] = {{nan, -1.0}, {inf, -1.0}, {1e4, -1.0}, {1e300, -1.0}, {-1.0, -1.0}, {-5000.0, -1.0}, {1e-50, -1e50}, {inf, -0.0}};
  for (auto &b : bad)
    if (vet::exp64_weight(b[0], b[1], (float)(1024.0 * b[1]), tab.data(), w, thin))
      return std::printf("accepted %g %g\n", b[0], b[1]), 1;
  std::printf("ok %.3g at depth %.3g\n", worst, worst_x);
  return 0;
}
