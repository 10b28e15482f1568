// ten_log10 on the host against the long double logarithm: the largest error in
// units in the last place of the FP32 result, over ratios of every size and
// close to one.
#include <cmath>
#include <cstdio>
#include <random>

#include "../paper_2604_02624_gb300/csrc/dos_decibel.cuh"

int main() {
  std::mt19937_64 rng(3);
  std::uniform_real_distribution<double> u(0.0, 1.0);
  double worst = 0.0, at = 0.0;
  for (int i = 0; i < 4000000; ++i) {
    double x = std::exp((u(rng) - 0.5) * 30.0);
    if (i % 4 == 1) x = 0.5 + 1.5 * u(rng);
    if (i % 4 == 2) x = 1.0 + (u(rng) - 0.5) * std::exp(-30.0 * u(rng));
    if (i % 4 == 3) x = std::ldexp((u(rng) < 0.5 ? 2.0 / 3.0 : 1.0) + 1e-6 * (u(rng) - 0.5), (int)(u(rng) * 40) - 20);
    const long double want = 10.0L * log10l((long double)x);
    const float got = dos::ten_log10(x);
    const float w = std::fabs((float)want);
    const double ulp = (double)std::nextafterf(w, INFINITY) - (double)w;
    const double err = std::fabs((double)(((long double)got - want) / (long double)ulp));
    if (err > worst) worst = err, at = x;
  }
  const bool edges = dos::ten_log10(1.0) == 0.f && std::isinf(dos::ten_log10(INFINITY)) && std::isinf(dos::ten_log10(0.0)) &&
                     std::isnan(dos::ten_log10(NAN)) && dos::ten_log10(1e-300) == -3000.f;
  std::printf("%.4f ulp at %.17g%s\n", worst, at, edges ? "" : " (edges wrong)");
  return !edges || worst > 0.55;
}
