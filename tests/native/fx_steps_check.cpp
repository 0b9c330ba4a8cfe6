// Host driver of the FP64 operator's integer steps (csrc/fx_steps.h).  Reads,
// per site: "site <hops> <exponent of the links' unit>" and for each hop 18
// link doubles and 6 vector doubles (all hexadecimal floats); prints the six
// sums of the site, or "range" where the steps hand it to the FP64 loop.
#include <cstdio>
#include <cstdlib>

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
    Sums S;
    init(S);
    for (int t = 0; t < hops; ++t) {
      Entry w[9];
      for (auto& e : w) {
        const double re = next(), im = next();
        fixed_entry(re, kexp, e.x, e.y);
        fixed_entry(im, kexp, e.z, e.w);
      }
      V2 psi[3];
      for (auto& v : psi) {
        v.x = next();
        v.y = next();
      }
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
