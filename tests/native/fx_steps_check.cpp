// Host driver of the FP64 operator's integer steps (csrc/fx_steps.h).  Reads,
// per site: "site <hops> <unit>" and for each hop 18 link doubles and 6 vector
// doubles (all hexadecimal floats); prints the six sums of the site, or
// "range" where the steps hand it to the FP64 loop.  <unit>: the exponent of
// every matrix's unit, 9999 for the one matrix_exponent gives, 7777 for the
// sums in doubles, one multiply-add after the other.
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
    if (kexp == 7777) {
      for (int i = 0; i < 3; ++i) {
        double re = 0, im = 0;
        for (int t = 0; t < hops; ++t)
          for (int j = 0; j < 3; ++j) {
            const double* w = &in[24 * t + 6 * i + 2 * j];
            const double* v = &in[24 * t + 18 + 2 * j];
            re = std::fma(-w[1], v[1], std::fma(w[0], v[0], re));
            im = std::fma(w[1], v[0], std::fma(w[0], v[1], im));
          }
        std::printf("%a %a ", re, im);
      }
      std::puts("");
      continue;
    }
    Sums S;
    init(S);
    for (int t = 0; t < hops; ++t) {
      const double* f = &in[24 * t];
      Entry w[9];
      double m[18];
      std::copy(f, f + 18, m);
      const int k = kexp == 9999 ? matrix_exponent(m) : kexp;
      for (int e = 0; e < 9; ++e) {
        fixed_entry(f[2 * e], k, w[e].x, w[e].y);
        fixed_entry(f[2 * e + 1], k, w[e].z, w[e].w);
      }
      V2 psi[3];
      for (int c = 0; c < 3; ++c) psi[c] = V2{f[18 + 2 * c], f[19 + 2 * c]};
      hop(S, psi, k, [&](int e) { return w[e]; });
    }
    V2 out[3];
    if (!result(S, out)) {
      std::puts("range");
      continue;
    }
    for (const auto& v : out) std::printf("%a %a ", v.x, v.y);
    std::puts("");
  }
  return 0;
}
