// gauge_force.cu -- the Symanzik one-loop improved gauge force in FP64.
//
// The paper benchmarks the gauge force of the HISQ RHMC/RHMD algorithm next
// to the CG (Sec. 4.2, Figs. 6-8: matrix-matrix products, arithmetic
// intensity 1.1 in MILC's baseline code and above 2.0 with reuse of
// three-link staples).  The action is the Luscher-Weisz form
//   S = beta sum_loops c (1 - Re Tr W / 3)
// over plaquettes (c_pl), 1x2 rectangles (c_rt) and parallelograms (the
// six-link loop a, b, c, -a, -b, -c over three directions; c_pg).  For the
// link U_mu(x), Sigma_mu(x) sums c times the product of the other links of
// every loop through it, each loop oriented to traverse U_mu(x) forward and
// started right after it:
//   plaquettes    [nu s, mu -, nu -s]                            6
//   rectangles    [mu +, nu s, mu -, mu -, nu -s]                6
//                 [nu s, mu -, mu -, nu -s, mu +]                6
//                 [nu s, nu s, mu -, nu -s, nu -s]               6
//   parallelograms [nu s, rho r, mu -, nu -s, rho -r]            24
// (nu, rho distinct and != mu, s, r = +-1), and the force is
//   F_mu(x) = (beta/3) TA[U_mu(x) Sigma_mu(x)],  TA(M) = (M - M^dag)/2 - Tr(M - M^dag)/6,
// so that moving the link as exp(eps X) U changes S by -eps Re Tr(X F).
// The staples are built from a stored table of three-link staples (below): on
// the integer pipe (fx.cuh) when the links are SU(3) matrices, otherwise, and
// when they are all close to 1, by the FP64 kernels.
#include <cmath>

#include "fx.cuh"

namespace stag {
namespace gf {
using namespace su3;

__device__ __forceinline__ M3 dagger(const M3& a) {
  M3 r;
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) r.e[3 * i + j] = make_double2(a.e[3 * j + i].x, -a.e[3 * j + i].y);
  return r;
}

// The link of one step from p (forward: U_dir(p), then p += dir; backward:
// p -= dir, then U_dir(p)^dag).
__device__ __forceinline__ M3 hop_link(const double2* __restrict__ U, const Dims& d, Pos& p, int dir, int sgn) {
  if (sgn > 0) {
    const M3 l = ld(U, p.lex, dir);
    p = step(d, p, dir, 1);
    return l;
  }
  p = step(d, p, dir, -1);
  return dagger(ld(U, p.lex, dir));
}

// ------------------------------------------------------------ staple reuse
// The paper's QOPQDP and QPhiX versions reuse three-link staples (60 % fewer
// flops than MILC's baseline, Sec. 4.2).  Here: one pass stores, for every
// link (y, mu) and plane (nu, s), its plaquette staple
//   T_{mu nu s}(y) = h(y+mu, nu, s) U_mu(y+s nu)^dag h(y+s nu, nu, -s)
// (the path [nu s, mu -, nu -s] from y + mu; h(z, nu, +1) = U_nu(z),
// h(z, nu, -1) = U_nu(z-nu)^dag), 24 per site; the force pass then closes
// every loop through U_mu(x) from at most three factors, the hops next to
// x + mu and x + s nu cancelling between adjacent staples:
//   plaquette        T(x; mu nu s)
//   rectangle 1      U_mu(x+mu) T(x+mu; mu nu s) T(x; mu nu s)
//   rectangle 2      T(x; mu nu s) T(x-mu; mu nu s) U_mu(x-mu)
//   rectangle 3      h(x+mu, nu, s) T(x+s nu; mu nu s) h(x+s nu, nu, -s)
//   parallelogram    h(x+mu, nu, s) T(x+s nu; mu rho r) Q,  Q = T(x; nu rho r) (s = +1)
//                                                          or T(x-nu; nu rho r)^dag (s = -1)
// with the left factor h(x+mu, nu, s) shared by rectangle 3 and the four
// parallelograms of (nu, s): 12 products per link for the table and 60 for
// the force, against 181 when every staple is walked link by link.

// slot of T(y; mu nu s) in the table: [site][mu][nu][s], 9 complex each
__device__ __forceinline__ long long tslot(long long y, int mu, int nu, int s) {
  return (((y * 4 + mu) * 4 + nu) * 2 + (s < 0 ? 1 : 0)) * 9;
}

__device__ __forceinline__ M3 ldT(const double2* __restrict__ T, long long y, int mu, int nu, int s) {
  M3 m;
  const double2* p = T + tslot(y, mu, nu, s);
#pragma unroll
  for (int i = 0; i < 9; ++i) m.e[i] = __ldg(p + i);
  return m;
}

// h(p, dir, sgn) without moving p
__device__ __forceinline__ M3 hop_at(const double2* __restrict__ U, const Dims& d, Pos p, int dir, int sgn) {
  return hop_link(U, d, p, dir, sgn);
}

// T(p0; mu nu s) from the links: the walk [nu s, mu -, nu -s] from p0 + mu
__device__ __forceinline__ M3 staple(const double2* __restrict__ U, const Dims& d, const Pos& p0, int mu, int nu, int s) {
  Pos p = step(d, p0, mu, 1);
  M3 m = hop_link(U, d, p, nu, s);
  m = mul(m, hop_link(U, d, p, mu, -1));
  return mul(m, hop_link(U, d, p, nu, -s));
}

// FP64 form; it and k_gauge_force_reuse run only when the integer kernels do
// not serve (fx::all_fp64), in grids that return at once otherwise.
__global__ void __launch_bounds__(128) k_gf_staples(Dims d, long long V, const double2* __restrict__ U,
                                                    double2* __restrict__ T, const fx::Header* hd, long long cap) {
  if (!fx::all_fp64(hd, fx::NEAR_5, V, cap)) return;
  for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < 24 * V;
       idx += (long long)gridDim.x * blockDim.x) {
    const int k = (int)(idx / V);  // mu * 6 + (other direction index) * 2 + sign
    const long long x = idx - (long long)k * V;
    const int mu = k / 6, o = (k % 6) >> 1, s = (k & 1) ? -1 : 1;
    const int nu = o < mu ? o : o + 1;
    const M3 m = staple(U, d, pos_of(d, x), mu, nu, s);
    double2* out = T + tslot(x, mu, nu, s);
#pragma unroll
    for (int i = 0; i < 9; ++i) out[i] = m.e[i];
  }
}

// acc += c m
__device__ __forceinline__ void axpy3(M3& acc, double c, const M3& m) {
#pragma unroll
  for (int i = 0; i < 9; ++i) {
    acc.e[i].x = fma(c, m.e[i].x, acc.e[i].x);
    acc.e[i].y = fma(c, m.e[i].y, acc.e[i].y);
  }
}

// S += the terms of (nu, s) for the link (p0, mu), with pp = x + mu, pm = x - mu
// and their links U_mu; staples from the table, or from the links where there
// is none.
template <bool TABLE>
__device__ __forceinline__ void add_pair(M3& S, const double2* __restrict__ U, const double2* __restrict__ T, const Dims& d,
                                         const Pos& p0, const Pos& pp, const Pos& pm, const M3& u_pm, const M3& u_mm,
                                         int mu, int nu, int s, double cpl, double crt, double cpg) {
  auto at = [&](const Pos& p, int a, int b, int sign) {
    if (TABLE) return ldT(T, p.lex, a, b, sign);
    return staple(U, d, p, a, b, sign);
  };
  const M3 t0 = at(p0, mu, nu, s);
  axpy3(S, cpl, t0);                                       // plaquette
  axpy3(S, crt, mul(u_pm, mul(at(pp, mu, nu, s), t0)));  // rectangle 1
  axpy3(S, crt, mul(mul(t0, at(pm, mu, nu, s)), u_mm));  // rectangle 2
  // rectangle 3 and the parallelograms share the left factor h(x+mu, nu, s)
  const Pos ps = step(d, p0, nu, s);  // x + s nu
  M3 R = mul(at(ps, mu, nu, s), hop_at(U, d, ps, nu, -s));
#pragma unroll
  for (int i = 0; i < 9; ++i) {
    R.e[i].x *= crt;
    R.e[i].y *= crt;
  }
  const Pos pmn = step(d, p0, nu, -1);  // x - nu (for s = -1)
  if constexpr (TABLE) {
#pragma unroll 1
    for (int rho = 0; rho < 4; ++rho) {
      if (rho == mu || rho == nu) continue;
#pragma unroll 1
      for (int r = -1; r <= 1; r += 2) {
        const M3 a = at(ps, mu, rho, r);
        const M3 q = s > 0 ? at(p0, nu, rho, r) : dagger(at(pmn, nu, rho, r));
        axpy3(R, cpg, mul(a, q));
      }
    }
  } else {
    // the same in a form that lanes of other (mu, nu, s) run together (for the
    // table kernel, whose warps share them, it is 1.5 % slower)
    const Pos pq = s > 0 ? p0 : pmn;
    const int lo = nu < mu ? nu : mu, hi = nu < mu ? mu : nu;
#pragma unroll 1
    for (int j = 0; j < 4; ++j) {
      int rho = j >> 1;
      const int r = (j & 1) ? 1 : -1;
      rho += rho >= lo ? 1 : 0;
      rho += rho >= hi ? 1 : 0;
      const M3 a = at(ps, mu, rho, r);
      M3 q = at(pq, nu, rho, r);
      if (s < 0) q = dagger(q);
      axpy3(R, cpg, mul(a, q));
    }
  }
  axpy3(S, 1.0, mul(hop_at(U, d, pp, nu, s), R));
}

// F_mu(x) = (beta/3) TA[U_mu(x) S]
__device__ __forceinline__ void store_force(const double2* __restrict__ U, double2* __restrict__ F, long long x, int mu,
                                            const M3& S, double beta) {
  const M3 us = mul(ld(U, x, mu), S);
  M3 a;
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j)
      a.e[3 * i + j] = make_double2(0.5 * (us.e[3 * i + j].x - us.e[3 * j + i].x),
                                    0.5 * (us.e[3 * i + j].y + us.e[3 * j + i].y));
  const double tr3 = (a.e[0].y + a.e[4].y + a.e[8].y) / 3.0;
  const double k = beta / 3.0;
  double2* f = F + (x * 4 + mu) * 9;
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j)
      f[3 * i + j] = make_double2(k * a.e[3 * i + j].x, k * (a.e[3 * i + j].y - (i == j ? tr3 : 0.0)));
}

// The links that k_gauge_force_fx has marked (its header says which), without a
// table: eight lanes per link, six of which take one (nu, s) each -- 34 products
// of a chain of 204, which one thread would take 0.6 ms for.
__device__ __forceinline__ void marked_links(const Dims& d, const double2* __restrict__ U, const long long* __restrict__ list,
                                             long long n, double2* __restrict__ F, double beta, double cpl, double crt,
                                             double cpg) {
  const int o = threadIdx.x & 7, per = gridDim.x * 16;
  for (long long i0 = blockIdx.x * 16 + (threadIdx.x >> 5) * 4; i0 < n; i0 += per) {  // (a warp's four links)
    const long long i = i0 + ((threadIdx.x & 31) >> 3);
    const bool in = i < n;
    const long long at = in ? __ldcg(list + i) : 0, x = at >> 2;
    const int mu = (int)(at & 3), q = o >> 1, nu = q < mu ? q : q + 1;
    M3 S = zero3();
    if (in && o < 6) {
      const Pos p0 = pos_of(d, x), pp = step(d, p0, mu, 1), pm = step(d, p0, mu, -1);
      add_pair<false>(S, U, nullptr, d, p0, pp, pm, ld(U, pp.lex, mu), ld(U, pm.lex, mu), mu, nu, (o & 1) ? 1 : -1, cpl, crt,
                      cpg);
    }
#pragma unroll
    for (int w = 1; w < 8; w <<= 1)
#pragma unroll
      for (int e = 0; e < 9; ++e) {
        S.e[e].x += __shfl_down_sync(0xffffffffu, S.e[e].x, w, 8);
        S.e[e].y += __shfl_down_sync(0xffffffffu, S.e[e].y, w, 8);
      }
    if (in && o == 0) store_force(U, F, x, mu, S, beta);
  }
}

// The force from the table, or the marked links alone (in a launch of its own
// that cost small lattices 4 us).
__global__ void __launch_bounds__(128) k_gauge_force_reuse(Dims d, long long V, const double2* __restrict__ U,
                                                           const double2* __restrict__ T, double2* __restrict__ F,
                                                           double beta, double cpl, double crt, double cpg,
                                                           const fx::Header* hd, const long long* __restrict__ list,
                                                           long long cap) {
  if (!fx::all_fp64(hd, fx::NEAR_5, V, cap)) {
    marked_links(d, U, list, (long long)__ldcg(&hd->marked), F, beta, cpl, crt, cpg);
    return;
  }
  for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < 4 * V;
       idx += (long long)gridDim.x * blockDim.x) {
    const int mu = (int)(idx / V);
    const long long x = idx - (long long)mu * V;
    const Pos p0 = pos_of(d, x), pp = step(d, p0, mu, 1), pm = step(d, p0, mu, -1);
    const M3 u_pm = ld(U, pp.lex, mu), u_mm = ld(U, pm.lex, mu);
    M3 S = zero3();
#pragma unroll 1
    for (int nu = 0; nu < 4; ++nu) {
      if (nu == mu) continue;
#pragma unroll 1
      for (int s = -1; s <= 1; s += 2) add_pair<true>(S, U, T, d, p0, pp, pm, u_pm, u_mm, mu, nu, s, cpl, crt, cpg);
    }
    store_force(U, F, x, mu, S, beta);
  }
}

// ------------------------------------------------------------ fixed point
// One field of 28 matrices per site: T(y; mu nu s) in slots 0..23, U_mu in 24..27.
constexpr int SLOTS = 28, U0 = 24;
__device__ __forceinline__ int fslot(int mu, int nu, int s) {
  return mu * 6 + (nu < mu ? nu : nu - 1) * 2 + (s < 0 ? 1 : 0);
}

// The staple table, from the links in slots 24..27 of the same field: a block
// takes 32 sites, its warp w the six staples of mu = w.  T is stored as the
// adjoint of the path walked the other way, A B C with A or C daggered.
__global__ void __launch_bounds__(128, 3) k_gf_staples_fx(Dims d, long long V, int4* __restrict__ T,
                                                          const fx::Header* hd) {
  if (!fx::serve(hd, fx::NEAR_5, V)) return;
  const int x = blockIdx.x * fx::TS + (threadIdx.x & 31);
  const int mu = threadIdx.x >> 5;
  if (x >= V) return;
  const fx::Site p = fx::site_of(d, x), pm = fx::next(d, p, mu, 1);
#pragma unroll 1
  for (int t = 0; t < 6; ++t) {
    const int o = t >> 1, nu = o < mu ? o : o + 1, low = t & 1;
    const int xm = fx::next_lex(d, p, nu, -1), xp = fx::next_lex(d, p, nu, 1);
    fx::FM a = fx::ld<SLOTS>(T, U0 + nu, low ? xm : x);
    fx::adjoint_if(a, -low);
    a = fx::mul(a, fx::ld<SLOTS>(T, U0 + mu, low ? xm : xp));
    fx::FM c = fx::ld<SLOTS>(T, U0 + nu, low ? fx::next_lex(d, pm, nu, -1) : pm.lex);
    fx::adjoint_if(c, low - 1);
    a = fx::mul(a, c);
    fx::adjoint_if(a, -1);
    fx::st<SLOTS>(T, mu * 6 + t, x, a);
  }
}

// The force.  The products are grouped so that a factor common to several
// staples is multiplied once, 51 per link:
//   group 0    U_mu(x+mu) [sum_{nu,s} T(x+mu; mu nu s) T(x; mu nu s)]             rectangles 1
//   group 1    [sum_{nu,s} T(x; mu nu s) T(x-mu; mu nu s)] U_mu(x-mu)             rectangles 2
//   2..7       h(x+mu, nu, s) [c_rt T(x+s nu; mu nu s) h(x+s nu, nu, -s)
//                              + c_pg sum_{rho,r} T(x+s nu; mu rho r) Q]          rectangles 3, parallelograms
// All groups run through the same two matrix products (sum += a b inside a
// group, S += P Q at its end), and what is done per entry runs in loops over
// shared memory: code beyond the instruction cache cost 1.4 issue slots per
// instruction (twelve warps, each at another place).  The coefficients, scaled
// by 2^-k so that |c_pl| 6 + |c_rt| 18 + |c_pg| 24 <= 1, keep S within range.
// Sums that are touched once per group (S, and a group's rectangle 3) wait in
// shared memory, a column per thread: in registers they cost the third block
// of an SM (255 registers, 4.4 ms at 24^4).  The factors of the next product
// are copied to shared memory while one runs (loaded into registers where they
// are used the kernel took 3.57 ms at 24^4, 3.47 so).  Bound by the integer pipe, 67 % busy (ncu),
// the rest additions, address arithmetic and dependences at three warps per scheduler.
// 24^4: conversion 0.07, table 0.68, force 3.5 ms; the call 4.2 ms against
// 21.3 ms with the FP64 kernels.
// Accuracy: about 2^-57 of the coefficients' size, whatever the force.  FP64
// sums do better where they keep the relative accuracy of a small force: around
// a link close to a diagonal matrix of 1, -1, i and -i, whose products are
// exact.  So where a link lies within 3 2^-5 of such a matrix, and the
// off-diagonal entries and the force in U S below 3 2^-6 of the coefficients'
// size, the link is marked and done again in FP64.  (Links exp(i eps H), rms
// error of the force in FP64 and here: eps = 0.08 1.8e-16 and 1.5e-16, eps =
// 0.04 1.7e-16 and 2.4e-16, eps = 0.005 1.8e-16 and 1.8e-15; the rule marks 3,
// 70 and 100 % of the links, and none at eps = 0.3.)
struct ForceCoef {
  fx::Coef pl8, rt8, rt, pg4;  // 8 c_pl, 8 c_rt, c_rt, 4 c_pg, each times 2^-k
  double off, diag;            // beta/3 times 2^(k-60) / 2 and / 3
};
__global__ void __launch_bounds__(128, 3) k_gauge_force_fx(Dims d, long long V, const int4* __restrict__ T,
                                                           fx::Header* hd, long long* __restrict__ list, long long cap,
                                                           double2* __restrict__ F, ForceCoef cf) {
  if (!fx::serve(hd, fx::NEAR_5, V)) return;
  extern __shared__ __align__(16) unsigned char gf_sm[];
  long long(*S)[128] = (long long(*)[128])gf_sm;  // [18][128]
  long long(*lone)[128] = S + 18;                  // a group's rectangle 3
  int4(*A)[128] = (int4(*)[128])(S + 36);          // [9][128]: an item's factors on their way, in A
  int4(*B)[128] = A + 9;                           // and in B; at a group's end the thread's column of B
  // holds the group's sum, then its weighted sum
  auto hold = [&](int e) -> long long* { return (long long*)&B[e >> 1][threadIdx.x] + (e & 1); };
  double2* out = (double2*)gf_sm;                  // the block's output, at the end
  const long long x0 = (long long)blockIdx.x * fx::TS;
  const int ns = (int)(V - x0 < fx::TS ? V - x0 : fx::TS);
  const int mu = threadIdx.x >> 5, lane = threadIdx.x & 31, tid = threadIdx.x;
  double dg[3];    // the force: imaginary parts of the diagonal,
  double2 off[3];  // entries 01, 02, 12
  if (lane < ns) {
    const fx::Site p0 = fx::site_of(d, (int)x0 + lane);
    const fx::Site pp = fx::next(d, p0, mu, 1);
    const int x = p0.lex, xm = fx::next_lex(d, p0, mu, -1);  // x, x - mu; pp = x + mu
    {  // plaquettes
      long long acc[18];
      fx::clear(acc);
#pragma unroll 1
      for (int t = 0; t < 6; ++t) {
        const fx::FM b = fx::ld<SLOTS>(T, mu * 6 + t, x);
#pragma unroll
        for (int e = 0; e < 18; ++e) acc[e] += fx::join1(b.h[e], b.l[e]);
      }
#pragma unroll
      for (int e = 0; e < 18; ++e) S[e][tid] = acc[e];
#pragma unroll 2
      for (int e = 0; e < 18; ++e) {
        S[e][tid] = fx::scaled(cf.pl8, S[e][tid] >> 3);
        lone[e][tid] = 0;
      }
    }
    // copies the factors of item t of group g into the thread's columns of A and B
    auto fetch = [&](int g, int t) {
      const int gt = g < 2 ? 0 : g - 2, go = gt >> 1, gnu = go < mu ? go : go + 1, gs = (gt & 1) ? -1 : 1;
      int sa, sb, xa, xb;
      if (g < 2) {
        sa = sb = mu * 6 + t;
        xa = g == 0 ? pp.lex : x;
        xb = g == 0 ? x : xm;
      } else {
        // ps = x + s nu; x (s > 0) or x - nu
        xa = fx::next_lex(d, p0, gnu, gs);
        xb = gs > 0 ? x : xa;
        if (t == 0) {
          sa = mu * 6 + gt;
          sb = U0 + gnu;
        } else {
          // (rho, r): the two directions other than mu and nu, both signs
          int rho = (t - 1) >> 1;
          const int lo = gnu < mu ? gnu : mu, hi = gnu < mu ? mu : gnu, r = (t & 1) ? 1 : -1;
          rho += rho >= lo ? 1 : 0;
          rho += rho >= hi ? 1 : 0;
          sa = fslot(mu, rho, r);
          sb = fslot(gnu, rho, r);
        }
      }
      fx::copy_column<SLOTS>(&A[0][tid], T, sa, xa);
      fx::copy_column<SLOTS>(&B[0][tid], T, sb, xb);
    };
    fetch(0, 0);
#pragma unroll 1
    for (int g = 0; g < 8; ++g) {
      // group g >= 2: its (nu, s)
      const int gt = g < 2 ? 0 : g - 2, go = gt >> 1, gnu = go < mu ? go : go + 1, gs = (gt & 1) ? -1 : 1;
      long long acc[18];
      fx::clear(acc);
      const int items = g < 2 ? 6 : 5;
#pragma unroll 1
      for (int t = 0; t < items; ++t) {
        fx::wait_columns();
        const fx::FM a = fx::from_column(&A[0][tid]);
        fx::FM b = fx::from_column(&B[0][tid]);
        if (t + 1 < items) fetch(g, t + 1);
        fx::adjoint_if(b, g < 2 ? 0 : (t == 0) == (gs > 0) ? -1 : 0);
        fx::mac(acc, a, b);
        if (g >= 2 && t == 0) {
#pragma unroll
          for (int e = 0; e < 18; ++e) {
            lone[e][tid] = acc[e];
            acc[e] = 0;
          }
        }
      }
#pragma unroll
      for (int e = 0; e < 18; ++e) *hold(e) = acc[e];
      {
        const fx::Coef ca = g < 2 ? cf.rt8 : cf.pg4, cb = cf.rt;
        const int sh = g < 2 ? 3 : 2;
#pragma unroll 2
        for (int e = 0; e < 18; ++e) {
          int h, l;  // lone is 0 for the first two groups
          fx::split1(fx::scaled(ca, *hold(e) >> sh) + fx::scaled(cb, lone[e][tid]), h, l);
          *(int2*)hold(e) = make_int2(h, l);
        }
      }
      // the other factor: U_mu(x+mu), U_mu(x-mu), else h(x+mu, nu, s)
      const int xh = g == 1 ? xm : g == 0 || gs > 0 ? pp.lex : fx::next_lex(d, pp, gnu, -1);
      fx::FM P = fx::ld<SLOTS>(T, U0 + (g < 2 ? mu : gnu), xh), Q;
      fx::adjoint_if(P, g >= 2 && gs < 0 ? -1 : 0);
#pragma unroll
      for (int e = 0; e < 18; ++e) {
        const int2 q = *(const int2*)hold(e);
        Q.h[e] = g == 1 ? P.h[e] : q.x;
        Q.l[e] = g == 1 ? P.l[e] : q.y;
        P.h[e] = g == 1 ? q.x : P.h[e];
        P.l[e] = g == 1 ? q.y : P.l[e];
      }
      if (g < 7) fetch(g + 1, 0);
      fx::clear(acc);
      fx::mac(acc, P, Q);
#pragma unroll
      for (int e = 0; e < 18; ++e) S[e][tid] += acc[e];
    }
    // F = (beta/3) TA[U S]; the differences are exact
    fx::FM s;
#pragma unroll
    for (int e = 0; e < 18; ++e) fx::split1(S[e][tid], s.h[e], s.l[e]);
    long long w[18];
    fx::clear(w);
    fx::mac(w, fx::ld<SLOTS>(T, U0 + mu, x), s);
    const long long tr = w[1] + w[9] + w[17];
    int size = 0;  // the largest off-diagonal entry, in units of 2^-28
    auto top = [](long long v) { return abs((int)(v >> 32)); };
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      const long long di = 3 * w[8 * i + 1] - tr;
      dg[i] = cf.diag * fx::double_of(di, 0);
      const int r = i == 2 ? 1 : 0, c = i == 0 ? 1 : 2;  // entries 01, 02, 12
      const int e = 2 * (3 * r + c), f = 2 * (3 * c + r);
      off[i] = make_double2(cf.off * fx::double_of(w[e] - w[f], 0), cf.off * fx::double_of(w[e + 1] + w[f + 1], 0));
      size = max(size, max(max(top(w[e]), top(w[e + 1])), max(top(w[f]), top(w[f + 1]))));
      size = max(size, top(di) >> 1);  // (a third of it is the force's)
    }
    if (size < 3 << 22 && fx::away(fx::ld<SLOTS>(T, U0 + mu, x)) < 3 << 25) fx::mark(hd, list, cap, 4LL * x + mu);
  }
  __syncthreads();  // the sums' memory becomes the output's
  if (lane < ns) {
    double2* o = out + lane * fx::SITE_W + mu * 9;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      const int r = i == 2 ? 1 : 0, c = i == 0 ? 1 : 2;
      o[4 * i] = make_double2(0.0, dg[i]);
      o[3 * r + c] = off[i];
      o[3 * c + r] = make_double2(-off[i].x, off[i].y);
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < ns * 36; i += 128) F[x0 * 36 + i] = out[(i / 36) * fx::SITE_W + i % 36];
}

}  // namespace gf
}  // namespace stag

using namespace stag;

extern "C" int stag_gauge_force(const int dims[4], const void* thin, void* force, double beta, double c_pl,
                                double c_rt, double c_pg, void* stream) {
  if (!dims || !thin || !force) return STAG_EINVAL;
  long long V = 1;
  for (int i = 0; i < 4; ++i) {
    if (dims[i] < 4 || dims[i] % 2) return STAG_EINVAL;
    V *= dims[i];
  }
  if (V > (1LL << 31)) return STAG_EINVAL;
  const size_t bytes = (size_t)V * 4 * 9 * sizeof(double2);
  const char *p = (const char*)thin, *q = (const char*)force;
  if (p < q + bytes && q < p + bytes) return STAG_EINVAL;
  const su3::Dims d{dims[0], dims[1], dims[2], dims[3]};
  cudaStream_t st = (cudaStream_t)stream;
  // stream-ordered scratch: the FP64 staple table (24 of 32 matrix slots per
  // site, 4608 B), or the fixed-point field (28 matrices, 4032 B) and the list of
  // marked links (up to one in four: one by one they take 2.2 times as long as
  // with the table), whichever form runs
  const long long cap = V;
  const size_t tbytes = (size_t)V * 32 * 9 * sizeof(double2), fbytes = fx::field_bytes(V, gf::SLOTS);
  const size_t lbytes = fbytes + (size_t)cap * sizeof(long long);
  char* scratch = nullptr;
  if (cudaMallocAsync((void**)&scratch, 256 + (tbytes > lbytes ? tbytes : lbytes), st) != cudaSuccess) {
    cudaGetLastError();
    return STAG_ENOMEM;
  }
  fx::Header* hd = (fx::Header*)scratch;
  double2* T = (double2*)(scratch + 256);
  int4* Tf = (int4*)(scratch + 256);
  long long* list = (long long*)(scratch + 256 + fbytes);
  const double2* U = (const double2*)thin;
  // coefficients with a power of two taken out (see k_gauge_force_fx); beyond
  // 2^+-900, with a beta that would make the last factor (ForceCoef) subnormal, or
  // not finite, the FP64 kernels, whose range is wider
  const double big = std::fabs(c_pl) * 6 + std::fabs(c_rt) * 18 + std::fabs(c_pg) * 24;
  const double b = std::fabs(beta);
  const bool fixed = big > 0x1p-900 && big < 0x1p900 && (b == 0.0 || (b > 0x1p-50 && b < 0x1p60));
  int s = fixed ? STAG_OK : cuda_status(cudaMemsetAsync(hd, 0, sizeof(*hd), st));
  if (fixed) {
    int k = 0;
    std::frexp(big, &k);
    gf::ForceCoef cf;
    cf.pl8 = fx::make_coef(std::ldexp(c_pl, 3 - k));
    cf.rt8 = fx::make_coef(std::ldexp(c_rt, 3 - k));
    cf.rt = fx::make_coef(std::ldexp(c_rt, -k));
    cf.pg4 = fx::make_coef(std::ldexp(c_pg, 2 - k));
    cf.off = std::ldexp(beta / 3.0, k - 61);
    cf.diag = std::ldexp(beta / 9.0, k - 60);
    const unsigned tiles = (unsigned)((V + fx::TS - 1) / fx::TS);
    {
      ProfScope ps("gauge_force", st);
      s = fx::launch_fx_links(V, U, Tf, gf::SLOTS, gf::U0, hd, st);
    }
    if (!s) {
      ProfScope ps("gauge_force", st);
      gf::k_gf_staples_fx<<<tiles, 128, 0, st>>>(d, V, Tf, hd);
      s = last_launch_status();
    }
    if (!s) {
      ProfScope ps("gauge_force", st);
      constexpr int smem = 4 * 18 * 128 * sizeof(long long);  // 72 KB, three blocks per SM
      s = cuda_status(cudaFuncSetAttribute(gf::k_gauge_force_fx, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
      if (!s) gf::k_gauge_force_fx<<<tiles, 128, smem, st>>>(d, V, Tf, hd, list, cap, (double2*)force, cf);
      if (!s) s = last_launch_status();
    }
  }
  if (!s) {
    ProfScope ps("gauge_force", st);
    const long long n = (24 * V + 127) / 128;
    gf::k_gf_staples<<<fixed ? beside_grid(n) : (unsigned)n, 128, 0, st>>>(d, V, U, T, hd, cap);
    s = last_launch_status();
  }
  if (!s) {
    ProfScope ps("gauge_force", st);
    const long long n = (4 * V + 127) / 128;
    gf::k_gauge_force_reuse<<<fixed ? beside_grid(n) : (unsigned)n, 128, 0, st>>>(d, V, U, T, (double2*)force, beta, c_pl,
                                                                               c_rt, c_pg, hd, list, cap);
    s = last_launch_status();
  }
  const int f = cuda_status(cudaFreeAsync(scratch, st));
  return s ? s : f;
}
