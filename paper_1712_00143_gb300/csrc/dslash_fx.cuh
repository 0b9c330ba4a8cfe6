// dslash_fx.cuh -- the FP64 hop sum on the integer pipe.
//
// The FP64 operator needs 573 FP64 multiply-adds per site, which at 2.2 per
// clock and SM take 2.8 times as long as its 2400 bytes take from HBM.  Here
// the sixteen link-times-vector products run in the exact fixed-point
// arithmetic of fx.cuh (81 wide integer multiply-adds per hop) and the
// operator is bound by HBM again: 32^4, one half 216 us (0.87 of the copy
// rate; integer pipe 45 % busy) against 522 us in FP64.
//
// Links: the handle's FP64 copy holds, in place of two doubles, {re.h, re.l,
// im.h, im.l} with entry = (h 2^-30 + l 2^-60) 2^k, and one byte k per matrix
// (fx_steps.h says how k is chosen; links.cu converts a field).
// Vectors stay doubles in memory.  A site's sum runs in units of 2^-60 2^E
// with E set by the largest product of a neighbour's largest component and its
// matrix's unit met so far (E = eb - 1023; a component of matrix unit 2^k is
// below 2^(E - k - 3)); a larger one raises E and shifts the sums down.  A
// neighbour seen through a zero matrix sets no unit.
// A site's real and imaginary sums stay below 2^63: 16 hops x 1.25 x sqrt(6) /
// 8 2^60 < 6.2 2^60.  The three sums they are made of (Gauss) are kept modulo
// 2^64.
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

// FP64 loop over the same links (rare): the sums whose exponents leave the fixed-point range.
template <class Args> __device__ __noinline__ void site_fp64(const Args& a, int s, double2* out) {
  const Coord c = cb_coords(a.g, s, a.out_parity);
  for (int i = 0; i < 3; ++i) out[i] = make_double2(0.0, 0.0);
#pragma unroll 1
  for (int t = 0; t < 16; ++t) {
    const int k = ((t & 2) ? 3 : 1) * ((t & 1) ? -1 : 1);
    double2 psi[3];
    SpinorLoad<64>::ld(a.in, cb_neighbour(a.g, s, c, t >> 2, k), psi);
    const int at = STAG_BOUND(s, a.g.Vh, BOUND_LINK);
    const int4* L = (const int4*)a.links + (size_t)t * 9 * a.g.Vh + at;
    const double scale = __longlong_as_double((long long)(1023 + __ldg(a.kexp + (size_t)at * 16 + t)) << 52);
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

// hop t of site s, kexp the exponent of its matrix
template <class Args>
__device__ __forceinline__ void hop_of(Sums& S, const Args& a, int s, const Coord& c, int t, int kexp) {
  const int Vh = a.g.Vh, k = ((t & 2) ? 3 : 1) * ((t & 1) ? -1 : 1);
  double2 psi[3];
  SpinorLoad<64>::ld(a.in, cb_neighbour(a.g, s, c, t >> 2, k), psi);
  const int4* L = (const int4*)a.links + (size_t)t * 9 * Vh + STAG_BOUND(s, Vh, BOUND_LINK);
  hop(S, psi, kexp, [&](int e) { return __ldg(L + (size_t)e * Vh); });
}

template <class Args> __device__ __forceinline__ void finish(const Sums& S, const Args& a, int s, double2 out[3]) {
  if (!result(S, out)) {
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
  const Coord c = cb_coords(a.g, s, a.out_parity);
  // the sixteen exponents in one load ahead of the hops (a byte per hop, which
  // each hop's conversion waits for, cost 6 % at 32^4)
  uint4 k = __ldg((const uint4*)a.kexp + STAG_BOUND(s, a.g.Vh, BOUND_LINK));
#pragma unroll 1
  for (int t = 0; t < 16; ++t) {
    hop_of(S, a, s, c, t, (int)(signed char)(k.x & 0xffu));
    k.x = __funnelshift_r(k.x, k.y, 8);
    k.y = __funnelshift_r(k.y, k.z, 8);
    k.z = __funnelshift_r(k.z, k.w, 8);
    k.w >>= 8;
  }
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
  if (s < end)
    hop_of(S, a, s, cb_coords(a.g, s, a.out_parity), t, __ldg(a.kexp + (size_t)STAG_BOUND(s, a.g.Vh, BOUND_LINK) * 16 + t));
  long long v[6];
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    v[2 * i] = real_sum(S, i);
    v[2 * i + 1] = imag_sum(S, i);
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
    out = fx::double_of(sum, eb - 1083);
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
