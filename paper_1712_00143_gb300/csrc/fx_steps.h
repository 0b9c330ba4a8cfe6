// fx_steps.h -- the integer steps of the fixed-point forms, without CUDA types,
// so that a host program can run them too: the wide multiply-adds, the split
// of a 64-bit value into two words, and the FP64 operator's running sums over
// the hops of a site (dslash_fx.cuh).
#pragma once
#include <cmath>
#include <cstring>

#ifdef __CUDACC__
#define STAG_FX __host__ __device__ __forceinline__
#else
#define STAG_FX inline
#endif
#ifdef __CUDA_ARCH__
#define STAG_UNROLL _Pragma("unroll")
#else
#define STAG_UNROLL
#endif

namespace stag {
namespace fx {

// Inline PTX: from C the compiler forms some of these as a 64-bit product and
// an addition (1.3 times the time of a matrix product).  Sums are modulo 2^64.
STAG_FX void wmad(long long& acc, int a, int b) {
#ifdef __CUDA_ARCH__
  asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(acc) : "r"(a), "r"(b));
#else
  acc = (long long)((unsigned long long)acc + (unsigned long long)((long long)a * b));
#endif
}
STAG_FX long long wmul(int a, int b) {
#ifdef __CUDA_ARCH__
  long long r;
  asm("mul.wide.s32 %0, %1, %2;" : "=l"(r) : "r"(a), "r"(b));
  return r;
#else
  return (long long)a * b;
#endif
}
// a + b and a - b modulo 2^64
STAG_FX long long add64(long long a, long long b) {
  return (long long)((unsigned long long)a + (unsigned long long)b);
}
STAG_FX long long sub64(long long a, long long b) {
  return (long long)((unsigned long long)a - (unsigned long long)b);
}

// int64 in units of 2^-60 -> (h, l): h = round(s / 2^30), l = s - h 2^30
STAG_FX void split1(long long s, int& h, int& l) {
  h = (int)((s + (1LL << 29)) >> 30);
  l = ((int)((unsigned)s << 2)) >> 2;
}
STAG_FX long long join1(int h, int l) { return ((long long)h << 30) + l; }

STAG_FX unsigned long long bits_of(double v) {
#ifdef __CUDA_ARCH__
  return (unsigned long long)__double_as_longlong(v);
#else
  unsigned long long b;
  std::memcpy(&b, &v, sizeof(b));
  return b;
#endif
}
STAG_FX double double_of_bits(unsigned long long b) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double((long long)b);
#else
  double v;
  std::memcpy(&v, &b, sizeof(v));
  return v;
#endif
}
STAG_FX int leading_zeros(unsigned long long a) {
#ifdef __CUDA_ARCH__
  return __clzll((long long)a);
#else
  return a ? __builtin_clzll(a) : 64;
#endif
}

// s 2^k, rounded to nearest; the result must be a normal number (or s = 0)
STAG_FX double double_of(long long s, int k) {
  const unsigned long long a0 = s < 0 ? 0ull - (unsigned long long)s : (unsigned long long)s;
  const int z = leading_zeros(a0);
  const unsigned long long a = a0 << (z & 63);
  const unsigned long long m = (a >> 11) + ((a >> 10) & 1);  // 53 bits, leading bit at 52
  unsigned long long b = ((unsigned long long)(unsigned)(1023 + 62 - z + k) << 52) + m;
  b = a0 == 0 ? 0 : b;
  return double_of_bits(b | ((unsigned long long)s & 0x8000000000000000ull));
}

}  // namespace fx

namespace fxd {

// The unit of a link matrix is 2^k with the smallest k for which no row's norm
// passes 1.25 units.  That keeps in range the 32-bit sum of an entry's two
// parts (1.25 sqrt 2 < 2) and a row's three cross products (see hop: 1.25
// sqrt 2 sqrt 3 2^61 + 3 2^58 < 2^63); every matrix is known to 2^-61 of at
// most 1.6 times its own largest row norm, FP64's entries to 2^-53.
// NO_MATRIX: all entries are zero.  BAD_MATRIX: an exponent beyond +-100 (or
// an infinity, or a NaN); the field then stays in doubles.
constexpr int NO_MATRIX = -128, BAD_MATRIX = 127;

// |v| 2^-e as a float, without an FP64 instruction; below 2^-126: 0.  |v| < 2^(e + 1).
STAG_FX float scaled_float(double v, int e) {
  const unsigned long long b = fx::bits_of(v) & 0x7fffffffffffffffull;
  const int k = (int)(b >> 52) - e;  // biased exponent of the result (+ 0: that of a double)
  const unsigned u = k < 897 ? 0u : ((unsigned)(k - 896) << 23) | ((unsigned)(b >> 29) & 0x7fffffu);
#ifdef __CUDA_ARCH__
  return __uint_as_float(u);
#else
  float f;
  std::memcpy(&f, &u, sizeof(f));
  return f;
#endif
}

STAG_FX int matrix_exponent(const double (&v)[18]) {
  int mx = 0;
  unsigned any = 0;
  STAG_UNROLL
  for (int i = 0; i < 18; ++i) {
    const unsigned long long b = fx::bits_of(v[i]);
    const int h = (int)(b >> 32) & 0x7fffffff;
    mx = mx > h ? mx : h;
    any |= (unsigned)h | (unsigned)b;
  }
  if (any == 0) return NO_MATRIX;
  const int e = (mx >> 20) - 1023;  // the largest entry's exponent
  if (e < -100 || e > 100) return BAD_MATRIX;
  float row = 0.f;
  STAG_UNROLL
  for (int i = 0; i < 3; ++i) {
    float n2 = 0.f;
    STAG_UNROLL
    for (int j = 0; j < 6; ++j) {
      const float a = scaled_float(v[6 * i + j], e);
      n2 += a * a;
    }
    row = row > n2 ? row : n2;
  }
  // row norms of up to 1.25, 2.5 and 5 (an entry's parts are below 2: at most 2 sqrt 6)
  return e + (row <= 1.5625f ? 0 : row <= 6.25f ? 1 : 2);
}

// One link entry in units of 2^kexp, |v| <= 1.25 2^kexp: v = (h 2^-30 + l 2^-60) 2^kexp, rounded to nearest.
STAG_FX void fixed_entry(double v, int kexp, int& h, int& l) {
  const unsigned long long b = fx::bits_of(v);
  const int r = 1023 + kexp - (int)((b >> 52) & 0x7ff);  // >= 0
  const unsigned long long m = ((b & 0xfffffffffffffull) | 0x10000000000000ull) << 8;
  const long long q = r > 62 ? 0 : r > 0 ? (long long)((m + (1ull << (r - 1))) >> r) : (long long)m;
  fx::split1((long long)b < 0 ? -q : q, h, l);
}

// The running sums of one site.  p[row] = {sum ar br, sum ai bi, sum (ar + ai)
// (br + bi)}, cross sums folded in, modulo 2^64: only the differences re = p0
// - p1 and im = p2 - p0 - p1 are bounded (dslash_fx.cuh), and only they are
// shifted or converted.
struct Sums {
  long long p[3][3];
  int eb;        // biased exponent of the unit (0: nothing met)
  unsigned any;  // 0 while every component seen through a matrix was an exact zero
};

STAG_FX void init(Sums& S) {
  for (int i = 0; i < 3; ++i)
    for (int q = 0; q < 3; ++q) S.p[i][q] = 0;
  S.eb = 0;
  S.any = 0;
}
STAG_FX long long real_sum(const Sums& S, int i) { return fx::sub64(S.p[i][0], S.p[i][1]); }
STAG_FX long long imag_sum(const Sums& S, int i) { return fx::sub64(fx::sub64(S.p[i][2], S.p[i][0]), S.p[i][1]); }

// S in units raised to 2^(eb - 1023).  The third sum may have passed 2^63, so
// the differences are shifted, and the sums replaced by others that have them.
STAG_FX void raise(Sums& S, int eb) {
  const int sh = eb - S.eb > 63 ? 63 : eb - S.eb;
  STAG_UNROLL
  for (int i = 0; i < 3; ++i) {
    const long long re = real_sum(S, i) >> sh, im = imag_sum(S, i) >> sh;
    S.p[i][0] = re;
    S.p[i][1] = 0;
    S.p[i][2] = fx::add64(im, re);
  }
  S.eb = eb;
}

// One component (h, l) in units of 2^-30, 2^-60 of 2^(eb - 1023); its exponent is at most eb - 4.
STAG_FX void component(double v, int eb, int& h, int& l) {
  const unsigned long long b = fx::bits_of(v);
  const int hi = (int)(b >> 32);
  int r = eb - ((hi >> 20) & 0x7ff);
  r = r > 63 ? 63 : r;
  const unsigned long long m = (((b & 0xfffffffffffffull) | 0x10000000000000ull) << 8) >> r;
  const int s = hi >> 31;
  h = ((int)(m >> 30) ^ s) - s;
  l = ((int)((unsigned)m & 0x3fffffffu) ^ s) - s;
}

// One hop: psi[3] with .x and .y, kexp the exponent of its matrix (NO_MATRIX:
// the hop counts for nothing, unless psi is not finite), link(e) the matrix
// entry e = 3 row + column as {re.h, re.l, im.h, im.l}.  The sums' unit follows
// the largest vector times its matrix's unit.
template <class V2, class Link> STAG_FX void hop(Sums& S, const V2 (&psi)[3], int kexp, Link link) {
  int mx = 0;
  unsigned any = 0;
  STAG_UNROLL
  for (int c = 0; c < 3; ++c) {
    const unsigned long long x = fx::bits_of(psi[c].x), y = fx::bits_of(psi[c].y);
    const int a = (int)(x >> 32) & 0x7fffffff, b = (int)(y >> 32) & 0x7fffffff, ab = a > b ? a : b;
    mx = mx > ab ? mx : ab;
    any |= (unsigned)a | (unsigned)b | (unsigned)x | (unsigned)y;
  }
  kexp = kexp == NO_MATRIX ? -4000 : kexp;
  const int ec = mx >= 0x7ff00000 ? 8000 : (mx >> 20) + kexp;
  S.any |= ec >= -1000 ? any : 0u;
  if (ec + 4 > S.eb) raise(S, ec + 4);
  const int eb = S.eb - kexp;
  int rh[3], rl[3], ih[3], il[3], sh[3], sl[3];
  STAG_UNROLL
  for (int c = 0; c < 3; ++c) {
    component(psi[c].x, eb, rh[c], rl[c]);
    component(psi[c].y, eb, ih[c], il[c]);
    sh[c] = rh[c] + ih[c];
    sl[c] = rl[c] + il[c];
  }
  // a row's cross sums, in units of 2^-90 (their high words alone, 2^-58, made
  // a single product less accurate than FP64's): |rl|, |il| < 2^30 and |rh|,
  // |ih| < 2^27, so |sl| < 2^31 and |sh| < 2^28
  STAG_UNROLL
  for (int i = 0; i < 3; ++i) {
    long long m1 = 1LL << 29, m2 = m1, m3 = m1;  // rounds them to 2^-60
    STAG_UNROLL
    for (int j = 0; j < 3; ++j) {
      const auto w = link(3 * i + j);
      const int th = w.x + w.z, tl = w.y + w.w;
      fx::wmad(S.p[i][0], w.x, rh[j]);
      fx::wmad(m1, w.x, rl[j]);
      fx::wmad(m1, w.y, rh[j]);
      fx::wmad(S.p[i][1], w.z, ih[j]);
      fx::wmad(m2, w.z, il[j]);
      fx::wmad(m2, w.w, ih[j]);
      fx::wmad(S.p[i][2], th, sh[j]);
      fx::wmad(m3, th, sl[j]);
      fx::wmad(m3, tl, sh[j]);
    }
    S.p[i][0] = fx::add64(S.p[i][0], m1 >> 30);
    S.p[i][1] = fx::add64(S.p[i][1], m2 >> 30);
    S.p[i][2] = fx::add64(S.p[i][2], m3 >> 30);
  }
}

// Exponents of the unit for which every value on the way is a normal number.
constexpr int MIN_EB = 256, MAX_EB = 1900;

// The site's sum as doubles; false: exponents out of range.
template <class V2> STAG_FX bool result(const Sums& S, V2* out) {
  const int k = S.eb - 1083;
  STAG_UNROLL
  for (int i = 0; i < 3; ++i) {
    out[i].x = fx::double_of(real_sum(S, i), k);
    out[i].y = fx::double_of(imag_sum(S, i), k);
  }
  return S.eb >= MIN_EB && S.eb <= MAX_EB;
}

}  // namespace fxd
}  // namespace stag
