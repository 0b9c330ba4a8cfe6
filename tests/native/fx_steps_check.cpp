// Host driver of the FP64 operator's integer steps (csrc/fx_steps.h).  Reads,
// per site: "site <hops> <exponent of the links' unit, or 9999 for the one the
// range check gives>" and for each hop 18 link doubles and 6 vector doubles
// (all hexadecimal floats); prints the six sums of the site, or "range" where
// the steps hand it to the FP64 loop.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <vector>

#include "fx_steps.h"

struct V2 {
  double x, y;
};
struct Entry {
  int x, y, z, w;
};

static double next() {
  char buf[64];
  if (std::scanf("%63s", buf) != 1) std::exit(1);
  return std::strtod(buf, nullptr);
}

int main() {
  using namespace stag::fxd;
  int hops, kexp;
  while (std::scanf(" site %d %d", &hops, &kexp) == 2) {
    std::vector<double> in(24 * (size_t)hops);
    for (auto& v : in) v = next();
    if (kexp == 9999) {
      double row = 0, most = 0;
      for (int i = 0; i < 3; ++i) {
        double sum = 0;
        for (int t = 0; t < hops; ++t) {
          double n2 = 0;
          for (int k = 0; k < 6; ++k) n2 += in[24 * t + 6 * i + k] * in[24 * t + 6 * i + k];
          row = std::max(row, std::sqrt(n2));
          sum += std::sqrt(n2);
        }
        most = std::max(most, sum);
      }
      kexp = unit_exponent(row, most);
    }
    Sums S;
    init(S);
    for (int t = 0; t < hops; ++t) {
      const double* f = &in[24 * t];
      Entry w[9];
      for (int e = 0; e < 9; ++e) {
        fixed_entry(f[2 * e], kexp, w[e].x, w[e].y);
        fixed_entry(f[2 * e + 1], kexp, w[e].z, w[e].w);
      }
      V2 psi[3];
      for (int c = 0; c < 3; ++c) psi[c] = V2{f[18 + 2 * c], f[19 + 2 * c]};
      hop(S, psi, [&](int e) { return w[e]; });
    }
    V2 out[3];
    if (!result(S, kexp, out)) {
      std::puts("range");
      continue;
    }
    for (const auto& v : out) std::printf("%a %a ", v.x, v.y);
    std::puts("");
  }
  return 0;
}
