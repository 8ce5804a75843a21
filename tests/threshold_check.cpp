// unit_threshold against the FP64 decision it stands for: u * W < a for
// u = k * 2^-24, over values drawn per seed and the edges of the type.
#include <cmath>
#include <cstdio>
#include <limits>
#include <random>
#include <string>
#include <vector>

#include "ipt_internal.h"

int main() {
  std::mt19937_64 rng(7);
  std::uniform_real_distribution<double> un(0.0, 1.0);
  std::vector<std::pair<double, double>> cases;
  const double inf = std::numeric_limits<double>::infinity(), nan = std::nan("");
  for (double W : {0.0, 5e-324, 1e-310, 1e-45, 1e-30, 0.37, 1.0, 16777216.0, 3e38, 1e39, 1e300, inf, nan})
    for (double f : {0.0, 5e-324, 0x1p-24, 0x1p-23, 0.1, 0.5, 1.0 - 0x1p-53, 1.0, 1.5}) cases.push_back({f * W, W});
  for (double p : {-1.0, nan, inf, 0x1p-25, 1.0 + 0x1p-52}) cases.push_back({p, 1.0});
  for (int i = 0; i < 20000; ++i) {
    const double W = std::exp(60.0 * un(rng) - 30.0);
    const double a = i % 3 ? W * un(rng) : std::floor(un(rng) * 16777216.0) * 0x1p-24 * W;
    cases.push_back({a, i % 5 ? W : 1.0});
  }
  for (const auto& c : cases) {
    const float T = ipt::unit_threshold(c.first, c.second);
    const double kt = (double)T * 16777216.0;
    if (!(kt >= 0.0 && kt <= 16777216.0) || kt != std::floor(kt)) {
      std::printf("threshold %g of (%g, %g) is no multiple of 2^-24\n", T, c.first, c.second);
      return 1;
    }
    std::vector<int> ks = {0, 1, 16777214, 16777215};
    for (int d = -20; d <= 20; ++d) ks.push_back((int)kt + d);
    for (int j = 0; j < 20; ++j) ks.push_back((int)(un(rng) * 16777216.0));
    for (int k : ks) {
      if (k < 0 || k > 16777215) continue;
      const float u = (float)k * (1.0f / 16777216.0f);
      if (((double)u * c.second < c.first) != (u < T)) {
        std::printf("u = %d * 2^-24, a = %g, W = %g: threshold %g decides otherwise\n", k, c.first, c.second, T);
        return 1;
      }
    }
  }
  return 0;
}
