// dslash_fx.cuh -- the FP64 hop sum on the integer pipe.
//
// The FP64 operator needs 573 FP64 multiply-adds per site, which at 2.2 per
// clock and SM take 2.8 times as long as its 2400 bytes take from HBM.  Here
// the sixteen link-times-vector products run in the exact fixed-point
// arithmetic of fx.cuh (81 wide integer multiply-adds per hop) and the
// operator is bound by HBM again: 32^4, one half 214 us (0.88 of the copy
// rate; integer pipe 45 % busy) against 522 us in FP64.
//
// Links: the handle's FP64 copy holds, in place of two doubles, {re.h, re.l,
// im.h, im.l} with entry = (h 2^-30 + l 2^-60) 2^kexp, |entry| < 2^kexp
// (links.cu converts a field when its range allows).
// Vectors stay doubles in memory.  A site's sum runs in units of 2^-60 2^E
// with E set by the largest neighbour component met so far (E = eb - 1023,
// |component| < 2^(E-2)); a larger one raises E and shifts the sums down,
// which after the first neighbour is rare.  The neighbours' small components
// are thus known to 2^-60 of the largest, FP64's rounded sums to 2^-53 of it.
// The two spare bits and the bound on the link rows that links.cu checks
// (sum over hops of the row norms <= 9) keep every sum below 2^63:
// 9 sqrt(2) sqrt(6) / 4 2^60 < 7.8 2^60.
// Neighbours with exponents near the ends of the double range (infinities,
// NaN and subnormals among them) take an FP64 loop over the same links.
#pragma once
#include "fx.cuh"
#include "internal.h"

namespace stag {

template <int P> struct DslashArgs;
// NL tag of the fixed-point form of the FP64 links (9 stored entries per Naik hop)
constexpr int kNLFixed = 10;

namespace fxd {

struct Sums {
  long long p[3][3];  // [row]: sum ar br, sum ai bi, sum (ar + ai)(br + bi); cross sums folded in
  int eb;             // biased exponent of the unit (0: nothing met)
  unsigned any;       // 0 while every component was an exact zero
};

__device__ __forceinline__ void init(Sums& S) {
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int q = 0; q < 3; ++q) S.p[i][q] = 0;
  S.eb = 0;
  S.any = 0;
}

// S in units raised to 2^(eb - 1023)
__device__ __forceinline__ void raise(Sums& S, int eb) {
  const int sh = eb - S.eb > 63 ? 63 : eb - S.eb;
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int q = 0; q < 3; ++q) S.p[i][q] >>= sh;
  S.eb = eb;
}

// One component (h, l) in units of 2^-30, 2^-60 of 2^(eb - 1023); its exponent is at most eb - 3.
__device__ __forceinline__ void component(double v, int eb, int& h, int& l) {
  const int hi = __double2hiint(v);
  const unsigned lo = (unsigned)__double2loint(v);
  const unsigned mh = ((unsigned)hi & 0xfffffu) | 0x100000u;
  int r = eb - ((hi >> 20) & 0x7ff);
  r = r > 63 ? 63 : r;
  const unsigned long long m = ((unsigned long long)__funnelshift_l(lo, mh, 8) << 32 | (lo << 8)) >> r;
  const int s = hi >> 31;
  h = ((int)(m >> 30) ^ s) - s;
  l = ((int)((unsigned)m & 0x3fffffffu) ^ s) - s;
}

// The hop t = 4 mu + kind (kind: +1, -1, +3, -3), its nine link entries read row by row.
__device__ __forceinline__ void hop(Sums& S, const int4* __restrict__ L, int Vh, const double2 (&psi)[3]) {
  int mx = 0;
  unsigned any = 0;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const int a = __double2hiint(psi[c].x) & 0x7fffffff, b = __double2hiint(psi[c].y) & 0x7fffffff;
    mx = max(mx, max(a, b));
    any |= (unsigned)a | (unsigned)b | (unsigned)__double2loint(psi[c].x) | (unsigned)__double2loint(psi[c].y);
  }
  S.any |= any;
  const int ec = mx >> 20;
  if (ec + 3 > S.eb) raise(S, ec + 4);
  int rh[3], rl[3], ih[3], il[3], sh[3], sl[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    component(psi[c].x, S.eb, rh[c], rl[c]);
    component(psi[c].y, S.eb, ih[c], il[c]);
    sh[c] = rh[c] + ih[c];
    sl[c] = rl[c] + il[c];
  }
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    long long m1 = 0x80000000LL, m2 = m1, m3 = m1;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      const int4 w = __ldg(L + (size_t)(3 * i + j) * Vh);
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
    S.p[i][0] += (long long)(int)(m1 >> 32) * 4;
    S.p[i][1] += (long long)(int)(m2 >> 32) * 4;
    S.p[i][2] += (long long)(int)(m3 >> 32) * 4;
  }
}

// FP64 loop over the same links (rare): the sums whose exponents leave the fixed-point range.
template <class Args> __device__ __noinline__ void site_fp64(const Args& a, int s, double2* out) {
  const Coord c = cb_coords(a.g, s, a.out_parity);
  const double scale = __longlong_as_double((long long)(1023 + a.kexp) << 52);
  for (int i = 0; i < 3; ++i) out[i] = make_double2(0.0, 0.0);
#pragma unroll 1
  for (int t = 0; t < 16; ++t) {
    const int k = ((t & 2) ? 3 : 1) * ((t & 1) ? -1 : 1);
    double2 psi[3];
    SpinorLoad<64>::ld(a.in, cb_neighbour(a.g, s, c, t >> 2, k), psi);
    const int4* L = (const int4*)a.links + (size_t)t * 9 * a.g.Vh + STAG_BOUND(s, a.g.Vh, BOUND_LINK);
#pragma unroll 1
    for (int i = 0; i < 3; ++i)
#pragma unroll 1
      for (int j = 0; j < 3; ++j) {
        const int4 w = __ldg(L + (size_t)(3 * i + j) * a.g.Vh);
        const double2 e = make_double2(scale * ((double)w.x * 0x1p-30 + (double)w.y * 0x1p-60),
                                       scale * ((double)w.z * 0x1p-30 + (double)w.w * 0x1p-60));
        cmac(out[i], e, psi[j]);
      }
  }
}

// Exponents of the unit for which every value on the way is a normal number.
constexpr int MIN_EB = 256, MAX_EB = 1900;

// the site's sum as doubles; false: exponents out of range
__device__ __forceinline__ bool result(const Sums& S, int kexp, double2 out[3]) {
  const bool ok = S.eb >= MIN_EB && S.eb <= MAX_EB;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const int k = S.eb - 1083 + kexp;
    out[i].x = fx::double_of(S.p[i][0] - S.p[i][1], k);
    out[i].y = fx::double_of(S.p[i][2] - S.p[i][0] - S.p[i][1], k);
  }
  return ok;
}

// hops [t0, t1) of site s
template <class Args> __device__ __forceinline__ void hops(Sums& S, const Args& a, int s, const Coord& c, int t0, int t1) {
  const int Vh = a.g.Vh;
#pragma unroll 1
  for (int t = t0; t < t1; ++t) {
    const int k = ((t & 2) ? 3 : 1) * ((t & 1) ? -1 : 1);
    double2 psi[3];
    SpinorLoad<64>::ld(a.in, cb_neighbour(a.g, s, c, t >> 2, k), psi);
    hop(S, (const int4*)a.links + (size_t)t * 9 * Vh + STAG_BOUND(s, Vh, BOUND_LINK), Vh, psi);
  }
}

template <class Args> __device__ __forceinline__ void finish(const Sums& S, const Args& a, int s, double2 out[3]) {
  if (!result(S, a.kexp, out)) {
    if (S.any == 0) {
#pragma unroll
      for (int i = 0; i < 3; ++i) out[i] = make_double2(0.0, 0.0);
    } else {
      site_fp64(a, s, out);
    }
  }
}

template <class Args> __device__ __forceinline__ void site(const Args& a, int s, double2 out[3]) {
  Sums S;
  init(S);
  hops(S, a, s, cb_coords(a.g, s, a.out_parity), 0, 16);
  finish(S, a, s, out);
}

// Few sites: a block of 128 threads takes 8 sites, one hop of one site per
// thread (lane = 8 (hop % 4) + site, warp = hop / 4), and adds the sixteen
// sums by shuffles and through shared memory.  Call with all threads of the
// block; thread 8 k + i < 48 returns true with component k (re, im of the
// three colours) of site i in out, unless that site is past the end.
template <class Args> __device__ __forceinline__ bool component16(const Args& a, int s0, int end, double& out) {
  __shared__ long long sm[4][6][8];
  __shared__ int se[4][8];
  __shared__ unsigned sa[4][8];
  const int tid = threadIdx.x, w = tid >> 5, ls = tid & 7, t = 4 * w + ((tid >> 3) & 3);
  Sums S;
  init(S);
  int s = s0 + ls;
  if (s < end) hops(S, a, s, cb_coords(a.g, s, a.out_parity), t, t + 1);
  long long v[6];
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    v[2 * i] = S.p[i][0] - S.p[i][1];
    v[2 * i + 1] = S.p[i][2] - S.p[i][0] - S.p[i][1];
  }
#pragma unroll
  for (int o = 8; o <= 16; o += 8) {
    const int eb = max(S.eb, __shfl_xor_sync(0xffffffffu, S.eb, o));
    const int d = eb - S.eb, sh = d > 63 ? 63 : d;
    S.eb = eb;
    S.any |= __shfl_xor_sync(0xffffffffu, S.any, o);
#pragma unroll
    for (int i = 0; i < 6; ++i) {
      v[i] >>= sh;
      v[i] += __shfl_xor_sync(0xffffffffu, v[i], o);
    }
  }
  if ((tid & 31) < 8) {
#pragma unroll
    for (int i = 0; i < 6; ++i) sm[w][i][ls] = v[i];
    se[w][ls] = S.eb;
    sa[w][ls] = S.any;
  }
  __syncthreads();
  const int k = tid >> 3;
  if (k >= 6 || s >= end) return false;
  const int eb = max(max(se[0][ls], se[1][ls]), max(se[2][ls], se[3][ls]));
  long long sum = 0;
  unsigned any = 0;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int d = eb - se[q][ls];
    sum += sm[q][k][ls] >> (d > 63 ? 63 : d);
    any |= sa[q][ls];
  }
  if (eb >= MIN_EB && eb <= MAX_EB) {
    out = fx::double_of(sum, eb - 1083 + a.kexp);
  } else if (any == 0) {
    out = 0.0;
  } else {
    double2 d[3];
    site_fp64(a, s, d);
    out = k == 0 ? d[0].x : k == 1 ? d[0].y : k == 2 ? d[1].x : k == 3 ? d[1].y : k == 4 ? d[2].x : d[2].y;
  }
  return true;
}

}  // namespace fxd
}  // namespace stag
