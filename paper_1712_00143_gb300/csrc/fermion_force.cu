// fermion_force.cu -- the staggered fermion force through the link
// construction, FP64.
//
// The paper benchmarks the HISQ fermion force of the RHMC/RHMD algorithm as
// its third routine (Sec. 4.2).  For the pseudofermion action of a rational
// approximation in partial fractions,
//   S = sum_i alpha_i phi^dag (M + sigma_i)^{-1} phi,   M = m^2 - D_eo D_oe,
// with X_i = (M + sigma_i)^{-1} phi (even sites) and Y_i = D_oe X_i (odd
// sites), a change of the links changes S by sum_i alpha_i 2 Re X_i^dag dD_eo Y_i
//   = sum_{x,mu} Re Tr[dF_mu(x) G^F_mu(x) + dL_mu(x) G^L_mu(x)],
// with the outer products (summed over i, weight alpha_i)
//   x even: G^F_mu(x) =  eta_mu(x) Y(x+mu) X(x)^dag,   G^L: Y(x+3mu) in place of Y(x+mu)
//   x odd:  G^F_mu(x) = -eta_mu(x) X(x+mu) Y(x)^dag,   G^L: X(x+3mu) in place of X(x+mu)
// Pass 1 (k_ff_outer) stores G^F and G^L.  Pass 2 (k_ff_chain) takes the
// chain rule through the fat link F = c1 U + c_st (upper + lower staples) and
// the Naik link L = c3 U U U: for the thin link U_r(y) it gathers
//   Z = c1 G^F_r(y)
//     + c3 [ U_r(y+r) (U_r(y+2r) G^L_r(y) + G^L_r(y-r) U_r(y-r))
//            + G^L_r(y-2r) U_r(y-2r) U_r(y-r) ]
//     + c_st sum_{n != r} [ U_n(y+r) (G^F_r(y+n) U_n(y)^dag + U_r(y+n)^dag G^F_n(y))
//                           + G^F_n(y+r)^dag (U_n(y) U_r(y+n))^dag
//                           + U_n(y-n+r)^dag (G^F_r(y-n) U_n(y-n) + U_r(y-n)^dag G^F_n(y-n)^dag)
//                           + G^F_n(y-n+r) U_r(y-n)^dag U_n(y-n) ]
// (the six places a thin link takes in the staples: middle link of an upper
// and of a lower staple of F_r, first and last link of an upper and of a
// lower staple of F_n), so that dS = sum Re Tr[dU Z], and writes
//   force_r(y) = -TA[U_r(y) Z],  TA(A) = (A - A^dag)/2 - Tr(A - A^dag)/6,
// the convention of the gauge force: U -> exp(eps X) U changes S by
// -eps Re Tr(X force).  36 products of 3x3 complex matrices per link.  Both
// passes run on the integer pipe (fx.cuh) when the links are SU(3) matrices,
// and on the FP64 pipe, which bounds them, otherwise.
#include <cmath>

#include "fx.cuh"

namespace stag {
namespace ffc {
using namespace su3;

constexpr int MAX_TERMS = 32;
struct Alphas {
  double a[MAX_TERMS];
};

__device__ __forceinline__ void ld3(const double2* __restrict__ f, long long cb, double2 v[3]) {
#pragma unroll
  for (int c = 0; c < 3; ++c) v[c] = __ldg(f + cb * 3 + c);
}

// acc += w a b^dag (colour vectors a, b)
__device__ __forceinline__ void outer_acc(M3& acc, double w, const double2 a[3], const double2 b[3]) {
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      const double re = a[i].x * b[j].x + a[i].y * b[j].y, im = a[i].y * b[j].x - a[i].x * b[j].y;
      acc.e[3 * i + j].x = fma(w, re, acc.e[3 * i + j].x);
      acc.e[3 * i + j].y = fma(w, im, acc.e[3 * i + j].y);
    }
}

__device__ __forceinline__ void st3x3(double2* __restrict__ p, const M3& m) {
#pragma unroll
  for (int i = 0; i < 9; ++i) p[i] = m.e[i];
}

// FP64 forms.  With a status word they run only when the integer kernels may
// not, in grids that return at once otherwise.
// One thread per (site x, direction mu), idx = x * 4 + mu: consecutive threads
// write consecutive matrices.  X, Y: [n][V/2][3], checkerboard index lex / 2.
__global__ void __launch_bounds__(128) k_ff_outer(Dims d, long long V, long long Vh, int n, Alphas al,
                                                  const double2* __restrict__ X, const double2* __restrict__ Y,
                                                  double2* __restrict__ GF, double2* __restrict__ GL,
                                                  const int* status) {
  if (status && fx::usable(status)) return;
  for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < 4 * V;
       idx += (long long)gridDim.x * blockDim.x) {
  const int mu = (int)(idx & 3);
  const long long x = idx >> 2;
  const Pos p = pos_of(d, x);
  const int par = (p.c.x + p.c.y + p.c.z + p.c.t) & 1;
  const int below = mu == 0 ? 0 : mu == 1 ? p.c.x : mu == 2 ? p.c.x + p.c.y : p.c.x + p.c.y + p.c.z;
  // eta_mu(x), and the sign of the odd-site terms
  const double sgn = ((below & 1) ? -1.0 : 1.0) * (par ? -1.0 : 1.0);
  const long long n1 = shifted(d, x, p.c, mu, 1) >> 1, n3 = shifted(d, x, p.c, mu, 3) >> 1, here = x >> 1;
  // even x: left field Y at the neighbour, right field X here; odd x: the reverse
  const double2* Fl = par ? X : Y;
  const double2* Fr = par ? Y : X;
  M3 gf = zero3(), gl = zero3();
#pragma unroll 1
  for (int i = 0; i < n; ++i) {
    const double w = sgn * al.a[i];
    double2 r[3], l1[3], l3[3];
    ld3(Fr + (long long)i * Vh * 3, here, r);
    ld3(Fl + (long long)i * Vh * 3, n1, l1);
    ld3(Fl + (long long)i * Vh * 3, n3, l3);
    outer_acc(gf, w, l1, r);
    outer_acc(gl, w, l3, r);
  }
  st3x3(GF + idx * 9, gf);
  st3x3(GL + idx * 9, gl);
  }
}

__device__ __forceinline__ M3 ldG(const double2* __restrict__ G, long long site, int mu) { return ld(G, site, mu); }

// One thread per thin link, idx = r * V + y (a warp shares r).
__global__ void __launch_bounds__(128) k_ff_chain(Dims d, long long V, const double2* __restrict__ U,
                                                  const double2* __restrict__ GF, const double2* __restrict__ GL,
                                                  double2* __restrict__ force, double c1, double cst, double c3,
                                                  const int* status) {
  if (status && fx::usable(status)) return;
  for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < 4 * V;
       idx += (long long)gridDim.x * blockDim.x) {
  const int r = (int)(idx / V);
  const long long y = idx - (long long)r * V;
  const Pos py = pos_of(d, y);
  const Pos pr = step(d, py, r, 1);   // y + r
  const Pos pmr = step(d, py, r, -1);  // y - r
  M3 Z = ldG(GF, y, r);
  scale3(Z, c1);
  // Naik: the link as first, middle and last factor of L_r(y), L_r(y-r), L_r(y-2r)
  {
    const M3 u_mr = ld(U, pmr.lex, r);  // U_r(y-r)
    M3 t = zero3();
    mac_mul(t, ld(U, step(d, pr, r, 1).lex, r), ldG(GL, y, r));  // U_r(y+2r) G^L_r(y)
    mac_mul(t, ldG(GL, pmr.lex, r), u_mr);                        // G^L_r(y-r) U_r(y-r)
    scale3(t, c3);
    mac_mul(Z, ld(U, pr.lex, r), t);
    const Pos pm2 = step(d, pmr, r, -1);  // y - 2r
    M3 w = mul(ldG(GL, pm2.lex, r), ld(U, pm2.lex, r));
    scale3(w, c3);
    mac_mul(Z, w, u_mr);
  }
#pragma unroll 1
  for (int n = 0; n < 4; ++n) {
    if (n == r) continue;
    {
      // staples through y + n and y: A = U_n(y+r), B = U_n(y), C = U_r(y+n)
      const Pos pn = step(d, py, n, 1);
      const M3 B = ld(U, y, n), C = ld(U, pn.lex, r);
      M3 t = zero3();
      mac_mul_dag(t, ldG(GF, pn.lex, r), B);  // G^F_r(y+n) U_n(y)^dag
      mac_dag_mul(t, C, ldG(GF, y, n));       // U_r(y+n)^dag G^F_n(y)
      scale3(t, cst);
      mac_mul(Z, ld(U, pr.lex, n), t);
      M3 w = mul(B, C);
      scale3(w, cst);
      mac_dag_mul_dag(Z, ldG(GF, pr.lex, n), w);  // G^F_n(y+r)^dag (U_n(y) U_r(y+n))^dag
    }
    {
      // staples through y - n: D = U_n(y-n+r), E = U_n(y-n), H = U_r(y-n)
      const Pos pmn = step(d, py, n, -1);
      const Pos pmnr = step(d, pmn, r, 1);
      const M3 E = ld(U, pmn.lex, n), H = ld(U, pmn.lex, r);
      M3 t = zero3();
      mac_mul(t, ldG(GF, pmn.lex, r), E);           // G^F_r(y-n) U_n(y-n)
      mac_dag_mul_dag(t, H, ldG(GF, pmn.lex, n));   // U_r(y-n)^dag G^F_n(y-n)^dag
      scale3(t, cst);
      mac_dag_mul(Z, ld(U, pmnr.lex, n), t);
      M3 w = zero3();
      mac_dag_mul(w, H, E);  // U_r(y-n)^dag U_n(y-n)
      scale3(w, cst);
      mac_mul(Z, ldG(GF, pmnr.lex, n), w);
    }
  }
  const M3 uz = mul(ld(U, y, r), Z);
  M3 a;
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j)
      a.e[3 * i + j] = make_double2(0.5 * (uz.e[3 * i + j].x - uz.e[3 * j + i].x),
                                    0.5 * (uz.e[3 * i + j].y + uz.e[3 * j + i].y));
  const double tr3 = (a.e[0].y + a.e[4].y + a.e[8].y) / 3.0;
  double2* f = force + (y * 4 + r) * 9;
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j)
      f[3 * i + j] = make_double2(-a.e[3 * i + j].x, -(a.e[3 * i + j].y - (i == j ? tr3 : 0.0)));
  }
}

// ------------------------------------------------------------ fixed point
// One field of 12 matrices per site: U_mu in slots 0..3, G^F_mu in 4..7, G^L_mu
// in 8..11.  Every G has its own exponent, G = matrix 2^e with entries up to
// 2^-3 (so that its norm is below 0.54); exponents in tiles like the matrices'.
constexpr int SLOTS = 12, GF0 = 4, GL0 = 8;
constexpr int ZERO_E = -(1 << 20);  // exponent of a zero matrix
__device__ __forceinline__ size_t eat(int slot, int site) {
  return (size_t)((site >> 5) * 8 + slot - GF0) * 32 + (site & 31);
}
inline size_t exps_bytes(long long V) { return (size_t)((V + 31) / 32) * 8 * 32 * sizeof(int); }

struct FxAlphas {
  fx::Coef c[MAX_TERMS];  // alpha = c 2^e, |c| < 1 (0: e = ZERO_E)
  int e[MAX_TERMS];
};

// The three components of a colour vector as v = (h 2^-30 + l 2^-60) 2^e with
// |v| 2^-e < 1/2; e = ZERO_E for a zero vector.  False: exponents so far from 1
// (or not finite) that products of them may leave the double range.
__device__ __forceinline__ bool vector_fx(const double2 (&v)[3], int (&h)[6], int (&l)[6], int& e) {
  int mx = 0;
  unsigned lo = 0;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    mx = max(mx, max(__double2hiint(v[c].x) & 0x7fffffff, __double2hiint(v[c].y) & 0x7fffffff));
    lo |= (unsigned)__double2loint(v[c].x) | (unsigned)__double2loint(v[c].y);
  }
  const int ec = mx >> 20;
  const bool zero = (mx | (int)lo) == 0;
#pragma unroll
  for (int c = 0; c < 6; ++c) {
    const double u = c & 1 ? v[c >> 1].y : v[c >> 1].x;
    const int hi = __double2hiint(u), s = hi >> 31;
    const unsigned b = (unsigned)__double2loint(u), mh = ((unsigned)hi & 0xfffffu) | 0x100000u;
    const int r = ec + 2 - ((hi >> 20) & 0x7ff);
    const unsigned long long m = ((unsigned long long)__funnelshift_l(b, mh, 8) << 32 | (b << 8)) >> (r > 63 ? 63 : r);
    h[c] = ((int)(m >> 30) ^ s) - s;
    l[c] = ((int)((unsigned)m & 0x3fffffffu) ^ s) - s;
  }
  e = zero ? ZERO_E : ec + 2 - 1023;
  return zero || (ec >= 1023 - 200 && ec <= 1023 + 200);
}

// G^F (blockIdx.y = 0) or G^L (1) of a tile of 32 sites, warp = mu.  The sum
// over terms runs in units of 2^-60 2^E with E two above the largest term's
// exponent met so far (32 terms of up to 1/2 fit); 81 wide multiply-adds per
// term against 54 FP64 instructions at 58 clocks.
__global__ void __launch_bounds__(128) k_ff_outer_fx(Dims d, long long V, long long Vh, int n, FxAlphas al,
                                                     const double2* __restrict__ X, const double2* __restrict__ Y,
                                                     int4* __restrict__ T, int* __restrict__ exps,
                                                     int* __restrict__ status) {
  if (!fx::usable(status)) return;
  const int x = blockIdx.x * fx::TS + (threadIdx.x & 31), mu = threadIdx.x >> 5, which = blockIdx.y;
  if (x >= V) return;
  const fx::Site p = fx::site_of(d, x);
  const int par = (p.c.x + p.c.y + p.c.z + p.c.t) & 1;
  const int below = mu == 0 ? 0 : mu == 1 ? p.c.x : mu == 2 ? p.c.x + p.c.y : p.c.x + p.c.y + p.c.z;
  const int neg = ((below ^ par) & 1) ? -1 : 0;  // sign of eta_mu(x), and of the odd-site terms
  // the neighbour one or three steps along mu
  const int L = su3::extent(d, mu), st = (int)su3::stride(d, mu), c0 = p.c.get(mu);
  int w = c0 + (which ? 3 : 1);
  w = w >= L ? w - L : w;
  const long long nb = (x + st * (w - c0)) >> 1, here = x >> 1;
  const double2* Fl = par ? X : Y;
  const double2* Fr = par ? Y : X;
  long long acc[18];
  fx::clear(acc);
  int E = ZERO_E;
  bool ok = true;
#pragma unroll 1
  for (int i = 0; i < n; ++i) {
    double2 v[3];
    int lh[6], ll[6], le, rh[6], rl[6], re;
    ld3(Fl + (long long)i * Vh * 3, nb, v);
    ok = vector_fx(v, lh, ll, le) && ok;
    ld3(Fr + (long long)i * Vh * 3, here, v);
    ok = vector_fx(v, rh, rl, re) && ok;
    const int e = le + re + al.e[i];
    if (e <= ZERO_E / 2) continue;
    // alpha into the right-hand vector
#pragma unroll
    for (int c = 0; c < 6; ++c) fx::split1(fx::scaled(al.c[i], fx::join1(rh[c], rl[c])), rh[c], rl[c]);
    if (e + 2 > E) {
      const int sh = e + 2 - E;
#pragma unroll
      for (int q = 0; q < 18; ++q) acc[q] >>= sh > 63 ? 63 : sh;
      E = e + 2;
    }
    const int dn = E - e > 63 ? 63 : E - e;
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
      for (int b = 0; b < 3; ++b) {
        // l_a conj(r_b): P1 = lr rr, P2 = li ri, P3 = (lr + li)(rr - ri)
        const int A = 2 * a, B = 2 * b;
        const int sh = lh[A] + lh[A + 1], sl = ll[A] + ll[A + 1], th = rh[B] - rh[B + 1], tl = rl[B] - rl[B + 1];
        const long long p1 = fx::wmul(lh[A], rh[B]), p2 = fx::wmul(lh[A + 1], rh[B + 1]), p3 = fx::wmul(sh, th);
        long long m1 = 0x80000000LL, m2 = m1, m3 = m1;
        fx::wmad(m1, lh[A], rl[B]);
        fx::wmad(m1, ll[A], rh[B]);
        fx::wmad(m2, lh[A + 1], rl[B + 1]);
        fx::wmad(m2, ll[A + 1], rh[B + 1]);
        fx::wmad(m3, sh, tl);
        fx::wmad(m3, sl, th);
        const unsigned k1 = (unsigned)(m1 >> 32), k2 = (unsigned)(m2 >> 32), k3 = (unsigned)(m3 >> 32);
        acc[2 * (3 * a + b)] += (p1 + p2 + (long long)(int)(k1 + k2) * 4) >> dn;
        acc[2 * (3 * a + b) + 1] += (p3 - p1 + p2 + (long long)(int)(k3 - k1 + k2) * 4) >> dn;
      }
  }
  if (!ok) atomicOr(status, fx::FX_RANGE);
  // normalised: the largest entry to [2^56, 2^57) in units of 2^-60
  unsigned long long mx = 0;
#pragma unroll
  for (int q = 0; q < 18; ++q) {
    acc[q] = (acc[q] ^ neg) - neg;
    mx |= (unsigned long long)(acc[q] < 0 ? -acc[q] : acc[q]);
  }
  const int up = mx == 0 ? 0 : __clzll((long long)mx) - 7;  // left shift (right if negative)
  fx::FM g;
#pragma unroll
  for (int q = 0; q < 18; ++q) fx::split1(up >= 0 ? acc[q] << up : acc[q] >> -up, g.h[q], g.l[q]);
  const int slot = (which ? GL0 : GF0) + mu;
  fx::st<SLOTS>(T, slot, x, g);
  exps[eat(slot, x)] = mx == 0 ? ZERO_E : E - up;
}

// The chain rule.  The terms of Z are taken in seven groups of five products
//   t = a0 b0 + a1 b1,  w = a2 b2,  Z += a3 t + a4 b4
// (six staples: direction n, upper and lower; then the Naik products), all
// through one product loop whose operands are fetched by slot, site and an
// adjoint flag: the code is one matrix product long.  With upper staples
// B = U_n(y), C = U_r(y+n), lower ones B = U_n(y-n), C = U_r(y-n):
//   t = G^F_r B' + C^dag G',  w = C^dag B',  Z += A' t + G'' w
// in the notation at the top of the file (B' = B^dag or B, and so on).
// Every G is shifted to the largest exponent E among those of its part: the
// staples' eighteen, the Naik products' three, G^F_r(y) (with one exponent for
// all, a part whose coefficient is small or 0 took the others' bits where its G
// is larger).
// The staples' sum (up to 9.6 with G's norm, held halved), c1 G and the Naik
// sum are each brought to full width before their coefficient is applied and
// they are added (add_part), and Z again before the last product: scaling the
// factors by the coefficients instead left the products' rounding at 2^-52 of
// the force.  Z, t and w wait in shared memory, a column per thread.  Bound by
// the integer pipe (67 % busy, three blocks per SM).  20x24x16x28, eight
// terms: conversion 0.05, outer products 0.47, this pass 1.85 ms; the call
// 2.4 ms against 7.4 ms with the FP64 kernels.
struct ChainCoef {
  fx::Coef c[3];  // c1, c_st, c3 = c 2^e, 1/2 <= |c| < 1 (0: e = ZERO_E)
  int e[3];
};
// Shift that brings the largest of the values OR-ed into mx to [2^59, 2^60) (right if negative).
__device__ __forceinline__ int widen(unsigned long long mx) { return mx == 0 ? 0 : __clzll((long long)mx) - 4; }
__device__ __forceinline__ long long shifted(long long v, int up) {
  const int dn = -up > 63 ? 63 : -up;
  return up >= 0 ? v << up : v >> dn;
}
__global__ void __launch_bounds__(128, 3) k_ff_chain_fx(Dims d, long long V, const int4* __restrict__ T,
                                                        const int* __restrict__ exps, const int* __restrict__ status,
                                                        double2* __restrict__ force, ChainCoef cf) {
  if (!fx::usable(status)) return;
  extern __shared__ __align__(16) unsigned char ff_sm[];
  long long(*Z)[128] = (long long(*)[128])ff_sm;  // [18][128]
  int2(*hold)[128] = (int2(*)[128])(Z + 18);       // [36][128]: t, then w, as (h, l)
  double2* out = (double2*)ff_sm;                  // the block's output, at the end
  const long long x0 = (long long)blockIdx.x * fx::TS;
  const int ns = (int)(V - x0 < fx::TS ? V - x0 : fx::TS);
  const int r = threadIdx.x >> 5, lane = threadIdx.x & 31, tid = threadIdx.x;
  double dg[3];
  double2 off[3];
  if (lane < ns) {
    const fx::Site py = fx::site_of(d, (int)x0 + lane), pr = fx::next(d, py, r, 1), pmr = fx::next(d, py, r, -1);
    const int y = py.lex, p2 = fx::next_lex(d, pr, r, 1), pm2 = fx::next_lex(d, pmr, r, -1);
    const int EF = exps[eat(GF0 + r, y)];
    const int EL = max(exps[eat(GL0 + r, y)], max(exps[eat(GL0 + r, pmr.lex)], exps[eat(GL0 + r, pm2)]));
    int E = ZERO_E;  // the common exponent of the part at hand: the staples' first
#pragma unroll 1
    for (int g = 0; g < 6; ++g) {
      const int o = g >> 1, n = o < r ? o : o + 1, low = g & 1;
      const int pn = fx::next_lex(d, py, n, low ? -1 : 1), q = low ? pn : y;
      const int far = low ? fx::next_lex(d, pr, n, -1) : pr.lex;
      E = max(E, max(exps[eat(GF0 + r, pn)], max(exps[eat(GF0 + n, q)], exps[eat(GF0 + n, far)])));
    }
    // the operand in `slot` at `site`; a G in the common exponent
    auto fetch = [&](int slot, int site, int adj) {
      fx::FM m = fx::ld<SLOTS>(T, slot, site);
      if (slot >= GF0) {
        const int e = E - exps[eat(slot, site)], sh = e > 63 ? 63 : e;
        if (__any_sync(__activemask(), sh != 0)) {
#pragma unroll
          for (int q = 0; q < 18; ++q) fx::split1(fx::join1(m.h[q], m.l[q]) >> sh, m.h[q], m.l[q]);
        }
      }
      fx::adjoint_if(m, adj);
      return m;
    };
    int eZ = ZERO_E;  // Z in units of 2^-60 2^eZ
    // Z += coefficient i times the sum in `hold` (units of 2^-60 2^e0)
    auto add_part = [&](int i, int e0) {
      long long(*src)[128] = (long long(*)[128])hold;
      unsigned long long mx = 0;
#pragma unroll 2
      for (int q = 0; q < 18; ++q) {
        const long long v = src[q][tid];
        mx |= (unsigned long long)(v < 0 ? -v : v);
      }
      const int up = widen(mx), e = mx == 0 ? ZERO_E : cf.e[i] + e0 - up;
      const int to = max(eZ, e) + 1, dz = to - eZ > 63 ? 63 : to - eZ, de = to - e > 63 ? 63 : to - e;
#pragma unroll 2
      for (int q = 0; q < 18; ++q)
        Z[q][tid] = (Z[q][tid] >> dz) + (fx::scaled(cf.c[i], shifted(src[q][tid], up)) >> de);
      eZ = to;
    };
#pragma unroll
    for (int q = 0; q < 18; ++q) Z[q][tid] = 0;
#pragma unroll 1
    for (int g = 0; g < 7; ++g) {
      const int naik = g == 6, o = naik ? 0 : g >> 1, n = o < r ? o : o + 1, low = g & 1;
      const int pn = fx::next_lex(d, py, n, low ? -1 : 1), q = low ? pn : y;
      const int far = low ? fx::next_lex(d, pr, n, -1) : pr.lex;
      long long acc[18];
#pragma unroll 1
      for (int j = 0; j < 5; ++j) {
        // a and b of product j (slot < 0: t or w)
        int sa, xa, da = 0, sb, xb, db = 0;
        if (!naik) {
          sa = j == 0 ? GF0 + r : j < 3 ? r : j == 3 ? n : GF0 + n;
          xa = j < 3 ? pn : far;
          da = j == 1 || j == 2 ? -1 : j == 3 ? -low : j == 4 ? low - 1 : 0;
          sb = j == 1 ? GF0 + n : j < 3 ? n : -1;
          xb = q;
          db = j == 1 ? -low : low - 1;
        } else {
          sa = j == 0 || j == 3 ? r : j < 3 ? GL0 + r : -1;
          xa = j == 0 ? p2 : j == 1 ? pmr.lex : j == 2 ? pm2 : pr.lex;
          sb = j == 0 ? GL0 + r : j == 3 ? -1 : r;
          xb = j == 0 ? y : j == 2 ? pm2 : pmr.lex;
        }
        const int2(*held)[128] = hold + (j == 4 ? 18 : 0);
        fx::FM a, b;
        if (sa >= 0) {
          a = fetch(sa, xa, da);
        } else {
#pragma unroll
          for (int e = 0; e < 18; ++e) {
            const int2 v = held[e][tid];
            a.h[e] = v.x;
            a.l[e] = v.y;
          }
        }
        if (sb >= 0) {
          b = fetch(sb, xb, db);
        } else {
#pragma unroll
          for (int e = 0; e < 18; ++e) {
            const int2 v = held[e][tid];
            b.h[e] = v.x;
            b.l[e] = v.y;
          }
        }
        if (j != 1 && j != 4) fx::clear(acc);
        fx::mac(acc, a, b);
        if (j == 1 || j == 2) {
          int2(*to)[128] = hold + (j == 2 ? 18 : 0);
#pragma unroll
          for (int e = 0; e < 18; ++e) {
            int h, l;
            fx::split1(acc[e], h, l);
            to[e][tid] = make_int2(h, l);
          }
        }
      }
      if (!naik) {
#pragma unroll
        for (int e = 0; e < 18; ++e) Z[e][tid] += acc[e] >> 1;
      }
      if (g < 5) continue;
      // the staples' sum, or the Naik sum, with its coefficient; c1 G^F_r(y) in between
      long long(*part)[128] = (long long(*)[128])hold;
#pragma unroll
      for (int e = 0; e < 18; ++e) {
        part[e][tid] = naik ? acc[e] : Z[e][tid];
        if (!naik) Z[e][tid] = 0;
      }
      add_part(naik ? 2 : 1, naik ? E : E + 1);
      if (!naik) {
        E = EF;
        const fx::FM gy = fetch(GF0 + r, y, 0);
#pragma unroll
        for (int e = 0; e < 18; ++e) part[e][tid] = fx::join1(gy.h[e], gy.l[e]);
        add_part(0, E);
        E = EL;
      }
    }
    // force = -TA[U Z]; the differences are exact
    unsigned long long mx = 0;
#pragma unroll 2
    for (int e = 0; e < 18; ++e) {
      const long long v = Z[e][tid];
      mx |= (unsigned long long)(v < 0 ? -v : v);
    }
    const int up = widen(mx);
    fx::FM z;
#pragma unroll
    for (int e = 0; e < 18; ++e) fx::split1(shifted(Z[e][tid], up), z.h[e], z.l[e]);
    long long w[18];
    fx::clear(w);
    fx::mac(w, fx::ld<SLOTS>(T, r, y), z);
    const long long tr = w[1] + w[9] + w[17];
    const int k = eZ - up - 60;  // (no use where every sum is zero)
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      dg[i] = (-1.0 / 3.0) * fx::double_of(3 * w[8 * i + 1] - tr, k);
      const int a = i == 2 ? 1 : 0, b = i == 0 ? 1 : 2, e = 2 * (3 * a + b), f = 2 * (3 * b + a);
      off[i] = make_double2(fx::double_of(w[f] - w[e], k - 1), fx::double_of(-w[e + 1] - w[f + 1], k - 1));
    }
  }
  __syncthreads();  // the sums' memory becomes the output's
  if (lane < ns) {
    double2* o = out + lane * fx::SITE_W + r * 9;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      const int a = i == 2 ? 1 : 0, b = i == 0 ? 1 : 2;
      o[4 * i] = make_double2(0.0, dg[i]);
      o[3 * a + b] = off[i];
      o[3 * b + a] = make_double2(-off[i].x, off[i].y);
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < ns * 36; i += 128) force[x0 * 36 + i] = out[(i / 36) * fx::SITE_W + i % 36];
}

}  // namespace ffc
}  // namespace stag

using namespace stag;

extern "C" int stag_fermion_force(const int dims[4], const void* thin, int n_terms, const void* x_even,
                                  const void* y_odd, const double* alpha, double c1, double c_staple, double c3,
                                  void* force, void* stream) {
  if (!dims || !thin || !x_even || !y_odd || !alpha || !force) return STAG_EINVAL;
  if (n_terms < 1 || n_terms > ffc::MAX_TERMS) return STAG_EINVAL;
  long long V = 1;
  for (int i = 0; i < 4; ++i) {
    if (dims[i] < 4 || dims[i] % 2) return STAG_EINVAL;
    V *= dims[i];
  }
  if (V > (1LL << 31)) return STAG_EINVAL;
  const long long Vh = V / 2;
  const size_t lbytes = (size_t)V * 4 * 9 * sizeof(double2), fbytes = (size_t)n_terms * Vh * 3 * sizeof(double2);
  auto overlap = [](const void* a, size_t na, const void* b, size_t nb) {
    const char *p = (const char*)a, *q = (const char*)b;
    return p < q + nb && q < p + na;
  };
  if (overlap(force, lbytes, thin, lbytes) || overlap(force, lbytes, x_even, fbytes) ||
      overlap(force, lbytes, y_odd, fbytes))
    return STAG_EINVAL;
  ffc::Alphas al{};
  ffc::FxAlphas fa{};
  // the integer kernels take coefficients within 2^+-150 (0 among them)
  bool fixed = true;
  for (int i = 0; i < n_terms; ++i) {
    al.a[i] = alpha[i];
    const double m = std::fabs(alpha[i]);
    fixed = fixed && (m == 0.0 || (m > 0x1p-150 && m < 0x1p150));
    fa.e[i] = ffc::ZERO_E;
    if (fixed && m > 0.0) fa.c[i] = fx::make_coef(std::frexp(alpha[i], &fa.e[i]));
  }
  ffc::ChainCoef cf{};
  const double coef[3] = {c1, c_staple, c3};
  for (int i = 0; i < 3; ++i) {
    const double m = std::fabs(coef[i]);
    fixed = fixed && (m == 0.0 || (m > 0x1p-150 && m < 0x1p150));
    cf.e[i] = ffc::ZERO_E;
    if (fixed && m > 0.0) cf.c[i] = fx::make_coef(std::frexp(coef[i], &cf.e[i]));
  }
  const su3::Dims d{dims[0], dims[1], dims[2], dims[3]};
  cudaStream_t st = (cudaStream_t)stream;
  // Stream-ordered scratch: links, G^F and G^L in fixed point with the
  // exponents (1760 B per site), or G^F and G^L in FP64 (1152 B per site); the
  // FP64 kernels alone if there is no room for the larger.
  const size_t gbytes = fx::field_bytes(V, ffc::SLOTS), ebytes = ffc::exps_bytes(V);
  char* scratch = nullptr;
  if (fixed && cudaMallocAsync((void**)&scratch, 256 + gbytes + ebytes, st) != cudaSuccess) {
    cudaGetLastError();
    scratch = nullptr;
    fixed = false;
  }
  if (!fixed && cudaMallocAsync((void**)&scratch, 256 + 2 * lbytes, st) != cudaSuccess) {
    cudaGetLastError();
    return STAG_ENOMEM;
  }
  fx::Header* hd = (fx::Header*)scratch;
  int* status = &hd->status;
  int4* T = (int4*)(scratch + 256);
  int* exps = (int*)(scratch + 256 + gbytes);
  double2* GF = (double2*)(scratch + 256);
  double2* GL = GF + (size_t)V * 4 * 9;
  const double2 *U = (const double2*)thin, *X = (const double2*)x_even, *Y = (const double2*)y_odd;
  int s = STAG_OK;
  if (fixed) {
    const unsigned tiles = (unsigned)((V + fx::TS - 1) / fx::TS);
    {
      ProfScope ps("fermion_force", st);
      s = fx::launch_fx_links(V, U, T, ffc::SLOTS, 0, hd, st);
    }
    if (!s) {
      ProfScope ps("fermion_force", st);
      ffc::k_ff_outer_fx<<<dim3(tiles, 2), 128, 0, st>>>(d, V, Vh, n_terms, fa, X, Y, T, exps, status);
      s = last_launch_status();
    }
    if (!s) {
      ProfScope ps("fermion_force", st);
      constexpr int smem = 3 * 18 * 128 * sizeof(long long);  // 54 KB, three blocks per SM
      s = cuda_status(cudaFuncSetAttribute(ffc::k_ff_chain_fx, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
      if (!s) ffc::k_ff_chain_fx<<<tiles, 128, smem, st>>>(d, V, T, exps, status, (double2*)force, cf);
      if (!s) s = last_launch_status();
    }
  }
  const long long n = (4 * V + 127) / 128;
  const unsigned grid = fixed ? beside_grid(n) : (unsigned)n;
  const int* when = fixed ? status : nullptr;
  if (!s) {
    ProfScope ps("fermion_force", st);
    ffc::k_ff_outer<<<grid, 128, 0, st>>>(d, V, Vh, n_terms, al, X, Y, GF, GL, when);
    s = last_launch_status();
  }
  if (!s) {
    ProfScope ps("fermion_force", st);
    ffc::k_ff_chain<<<grid, 128, 0, st>>>(d, V, U, GF, GL, (double2*)force, c1, c_staple, c3, when);
    s = last_launch_status();
  }
  const int f = cuda_status(cudaFreeAsync(scratch, st));
  return s ? s : f;
}
