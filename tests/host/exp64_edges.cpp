// Host-side check of the FP64 segment weight (vet_exp64.h) where its premise
// just holds or just fails: remainders out to the bound that it checks, and
// opacities that are negative or a negative zero, which are either refused or
// right.  Built with the undefined-behaviour sanitizer where there is one.
// Prints "ok" or the failure.
#include <cmath>
#include <cstdio>
#include <random>
#include <vector>

#include "vet_exp64.h"

int main() {
  std::vector<double> tab(vet::kExp64TableDoubles);
  vet::exp64_fill_table(tab.data());
  const long double ln2 = 0.693147180559945309417232121458176568L;
  double w, reached = 0.0, worst = 0.0;
  bool thin;
  long accepted = 0;
  // the bound of exp64_check.cpp: every rounding half an ulp at most
  auto right = [&](double kappa, double len, float lens) {
    if (!vet::exp64_weight(kappa, len, lens, tab.data(), w, thin)) return true;
    ++accepted;
    const long double y = (long double)kappa * (long double)len, want = thin ? std::expm1(y * ln2) : std::exp2(y);
    const double err = want == 0.0L ? (w == 0.0 ? 0.0 : 1.0) : (double)(std::fabs((long double)w - want) / std::fabs(want));
    worst = std::fmax(worst, err);
    return err <= (thin ? 4.0 : 2.5) * 1.2e-16;
  };
  // a step chosen up to a whole one off: remainders of up to 1.5 steps, accepted to 2^-10.5 (0.71)
  std::mt19937_64 rng(5);
  std::uniform_real_distribution<double> U(0.0, 1.0);
  for (int i = 0; i < 2000000; ++i) {
    const double steps = 2.0 + U(rng) * 700000.0 * U(rng) * U(rng), off = 2.0 * U(rng) - 1.0, len = -std::exp2(10.0 * (U(rng) - 0.5));
    const double kappa = steps / 1024.0 / -len;
    const long before = accepted;
    if (!right(kappa, len, (float)(1024.0 * len * (1.0 + off / steps)))) return std::printf("%g steps, %g off: %g\n", steps, off, worst), 1;
    if (accepted > before) reached = std::fmax(reached, std::fabs(off));
  }
  if (!(reached > 0.7 && reached < 1.25)) return std::printf("offsets reached %g steps\n", reached), 1;
  for (double kappa : {-0.0, -1e-300, -1e-40, -1e-38, -1e-30, -1e-10, -1e-5, -1e-3, -0.1, -1.0, -3e38, -1e300})
    for (double len : {-1e-10, -1e-3, -0.3, -1.0, -100.0})
      if (!right(kappa, len, (float)(1024.0 * len))) return std::printf("kappa %g len %g: %g\n", kappa, len, worst), 1;
  std::printf("ok %.3g, steps off by up to %.3f\n", worst, reached);
  return 0;
}
