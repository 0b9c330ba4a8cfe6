// links_build.cu -- the link construction that precedes the operator: fat
// (three-staple) and Naik links from thin links, in FP64 on the GPU.
//
// The paper's production code smears the thin gauge links before the CG
// (HISQ-link smearing, Sec. 1, and its share of the run time in Sec. 2,
// Fig. 1); the workload here uses the three-staple fat link and the Naik
// link:
//   F_mu(x) = c1 U_mu(x) + c_st sum_{nu != mu} [ U_nu(x) U_mu(x+nu) U_nu(x+mu)^dag
//                                               + U_nu(x-nu)^dag U_mu(x-nu) U_nu(x-nu+mu) ]
//   L_mu(x) = c3 U_mu(x) U_mu(x+mu) U_mu(x+2mu)
// One thread per (site, direction): 12 staple products and 2 Naik products
// of 3x3 complex matrices (about 1500 real multiply-adds), inputs from L2
// (each thin link is read by up to 19 threads).  Links that are SU(3) matrices
// go through the fixed-point products of fx.cuh on the integer pipe; any
// other input, and links all close to 1, through the FP64 kernel.
#include <cmath>

#include "fx.cuh"

namespace stag {
namespace lb {
using namespace su3;

// F_mu(x) in FP64
__device__ __forceinline__ M3 fat_link(const Dims& d, const double2* __restrict__ U, const Pos& p, int mu, double c1,
                                       double cst) {
  const Pos pm = step(d, p, mu, 1);
  M3 S = zero3();
#pragma unroll 1
  for (int nu = 0; nu < 4; ++nu) {
    if (nu == mu) continue;
    // upper staple U_nu(x) U_mu(x+nu) U_nu(x+mu)^dag
    {
      const M3 ab = mul(ld(U, p.lex, nu), ld(U, shifted(d, p.lex, p.c, nu, 1), mu));
      mac_mul_dag(S, ab, ld(U, pm.lex, nu));
    }
    // lower staple U_nu(x-nu)^dag U_mu(x-nu) U_nu(x-nu+mu)
    {
      const long long x_mnu = shifted(d, p.lex, p.c, nu, -1);
      const M3 ab = dag_mul(ld(U, x_mnu, nu), ld(U, x_mnu, mu));
      mac_mul(S, ab, ld(U, shifted(d, pm.lex, pm.c, nu, -1), nu));
    }
  }
  const M3 u = ld(U, p.lex, mu);
#pragma unroll
  for (int i = 0; i < 9; ++i) S.e[i] = make_double2(c1 * u.e[i].x + cst * S.e[i].x, c1 * u.e[i].y + cst * S.e[i].y);
  return S;
}
// L_mu(x) = c3 U_mu(x) U_mu(x+mu) U_mu(x+2mu) in FP64
__device__ __forceinline__ M3 naik_link(const Dims& d, const double2* __restrict__ U, const Pos& p, int mu, double c3) {
  const M3 uu = mul(ld(U, p.lex, mu), ld(U, shifted(d, p.lex, p.c, mu, 1), mu));
  M3 l = mul(uu, ld(U, shifted(d, p.lex, p.c, mu, 2), mu));
#pragma unroll
  for (int i = 0; i < 9; ++i) l.e[i] = make_double2(c3 * l.e[i].x, c3 * l.e[i].y);
  return l;
}
__device__ __forceinline__ void st(double2* __restrict__ out, long long link, const M3& m) {
#pragma unroll
  for (int i = 0; i < 9; ++i) out[link * 9 + i] = m.e[i];
}

// FP64 form: bound by the FP64 pipe (10.8 ms at 32^4, 1.2 TFLOP/s).  With a
// header it does the whole field only when the integer kernels do not serve,
// otherwise the fat and Naik links that k_build_links_fx has marked, one per
// thread (in a launch of its own that cost small lattices 3 us).
__global__ void __launch_bounds__(128) k_build_links(Dims d, long long V, const double2* __restrict__ U,
                                                     double2* __restrict__ F, double2* __restrict__ Lk, double c1,
                                                     double cst, double c3, const fx::Header* hd,
                                                     const long long* __restrict__ list, long long cap) {
  const bool all = !hd || fx::all_fp64(hd, fx::NEAR_6, V, cap);
  const long long n = all ? 8 * V : (long long)__ldcg(&hd->marked);
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    long long link;  // 4 site + mu; a warp of the whole field shares mu and the kind
    int kind;
    if (all) {
      const long long q = i / V;
      kind = q >= 4;
      link = 4 * (i - q * V) + (q & 3);
    } else {
      const long long at = __ldcg(list + i);
      kind = (int)(at & 1);
      link = at >> 1;
    }
    const int mu = (int)(link & 3);
    const Pos p = pos_of(d, link >> 2);
    if (kind)
      st(Lk, link, naik_link(d, U, p, mu, c3));
    else
      st(F, link, fat_link(d, U, p, mu, c1, cst));
  }
}

// The fat links (12 products) or the Naik links (2 products) on the integer
// pipe; two launches keep each loop's code small.  A block takes a tile of 32
// sites, its warp w the direction mu = w: link loads are whole 512-byte rows,
// the four directions of a site share their staples' links in L1, and the
// outputs leave through shared memory as one contiguous piece.  The
// coefficients, scaled by 2^-k to at most 1, are applied in fixed point too:
// FP64 instructions at the end would cost a tenth of the whole kernel.  Bound
// by the integer pipe (65 % busy with two blocks per SM; three or four blocks
// measured the same).  24^4: conversion 0.06, fat 0.84, Naik 0.17 ms; the call
// at 32^4 3.46 ms against 10.84 ms with the FP64 kernel.
// Accuracy: half of FP64's error in every matrix's norm.  FP64 does better on
// small off-diagonal entries, which it knows to their own size where the links
// are close to a diagonal matrix; so where the link lies within 3 2^-6 of a
// diagonal matrix of 1, -1, i, -i and the result's off-diagonal entries are
// below 3 2^-7 (of the larger coefficient), the result is marked and done again
// in FP64.  (Off-diagonal entries of fat links from exp(i eps H), rms error in
// FP64 and here: eps = 0.04 1.2e-16 and 1.0e-16, eps = 0.02 1.1e-16 and 2.0e-16,
// eps = 0.005 1.1e-16 and 7.7e-16.)
template <bool FAT>
__global__ void __launch_bounds__(128, FAT ? 2 : 3) k_build_links_fx(Dims d, long long V, const int4* __restrict__ U,
                                                        fx::Header* hd, long long* __restrict__ list, long long cap,
                                                        double2* __restrict__ out, fx::Coef c1, fx::Coef cst, int k) {
  unsigned long long near = 0;
  if (!fx::serve(hd, fx::NEAR_6, V, &near)) return;
  __shared__ double2 sm[fx::TS * fx::SITE_W];
  const long long x0 = (long long)blockIdx.x * fx::TS;
  const int ns = (int)(V - x0 < fx::TS ? V - x0 : fx::TS);
  const int mu = threadIdx.x >> 5, s = threadIdx.x & 31;
  if (s < ns) {
    const fx::Site p = fx::site_of(d, (int)x0 + s), pm = fx::next(d, p, mu, 1);
    double2* o = sm + s * fx::SITE_W + mu * 9;
    long long acc[18];
    fx::clear(acc);
    if constexpr (FAT) {
      // t = 0..5: direction nu, upper (U_nu(x) U_mu(x+nu) U_nu(x+mu)^dag) and
      // lower (U_nu(x-nu)^dag U_mu(x-nu) U_nu(x-nu+mu)) staple
#pragma unroll 1
      for (int t = 0; t < 6; ++t) {
        const int o3 = t >> 1, nu = o3 < mu ? o3 : o3 + 1, low = t & 1;
        const int xm = fx::next_lex(d, p, nu, -1), xp = fx::next_lex(d, p, nu, 1);
        fx::FM a = fx::ld<4>(U, nu, low ? xm : p.lex);
        fx::adjoint_if(a, -low);
        a = fx::mul(a, fx::ld<4>(U, mu, low ? xm : xp));
        fx::FM c = fx::ld<4>(U, nu, low ? fx::next_lex(d, pm, nu, -1) : pm.lex);
        fx::adjoint_if(c, low - 1);
        fx::mac(acc, a, c);
      }
      const fx::FM u = fx::ld<4>(U, mu, p.lex);
#pragma unroll
      for (int e = 0; e < 18; ++e)  // the staple sum, of norm up to 6, enters as an eighth
        acc[e] = fx::scaled(c1, fx::join1(u.h[e], u.l[e])) + fx::scaled(cst, (acc[e] + 4) >> 3);
    } else {
      // U_mu(x) U_mu(x+mu) U_mu(x+2mu)
      fx::FM a = fx::mul(fx::ld<4>(U, mu, p.lex), fx::ld<4>(U, mu, pm.lex));
      fx::mac(acc, a, fx::ld<4>(U, mu, fx::next_lex(d, pm, mu, 1)));
#pragma unroll
      for (int e = 0; e < 18; ++e) acc[e] = fx::scaled(c1, acc[e]);
    }
#pragma unroll
    for (int e = 0; e < 9; ++e) o[e] = make_double2(fx::double_of(acc[2 * e], k), fx::double_of(acc[2 * e + 1], k));
    if (near != 0) {
      int size = 0;  // the largest off-diagonal entry, in units of 2^-28
#pragma unroll
      for (int e = 0; e < 9; ++e)
        if (e % 4) size = max(size, max(abs((int)(acc[2 * e] >> 32)), abs((int)(acc[2 * e + 1] >> 32))));
      if (size < 3 << 21 && fx::away(fx::ld<4>(U, mu, p.lex)) < 3 << 24)
        fx::mark(hd, list, cap, (4LL * p.lex + mu) * 2 + (FAT ? 0 : 1));
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < ns * 36; i += 128) out[x0 * 36 + i] = sm[(i / 36) * fx::SITE_W + i % 36];
}

}  // namespace lb
}  // namespace stag

using namespace stag;

extern "C" int stag_build_links(const int dims[4], const void* thin, void* fat, void* lng, double c1, double c_staple,
                                double c3, void* stream) {
  if (!dims || !thin || !fat || !lng) return STAG_EINVAL;
  long long V = 1;
  for (int i = 0; i < 4; ++i) {
    if (dims[i] < 4 || dims[i] % 2) return STAG_EINVAL;
    V *= dims[i];
  }
  const su3::Dims d{dims[0], dims[1], dims[2], dims[3]};
  if (V > (1LL << 31)) return STAG_EINVAL;
  const size_t bytes = (size_t)V * 4 * 9 * sizeof(double2);
  // the outputs may not overlap the input or each other
  auto overlap = [bytes](const void* a, const void* b) {
    const char *p = (const char*)a, *q = (const char*)b;
    return p < q + bytes && q < p + bytes;
  };
  if (overlap(thin, fat) || overlap(thin, lng) || overlap(fat, lng)) return STAG_EINVAL;
  cudaStream_t st = (cudaStream_t)stream;
  const double2* U = (const double2*)thin;
  const long long cap = 4 * V;  // marked results that the list holds (of 8 V)
  auto fp64 = [&](const fx::Header* hd, const long long* list) {
    ProfScope ps("links", st);
    const long long want = (8 * V + 127) / 128;
    const unsigned grid = hd ? beside_grid(want) : (unsigned)want;
    lb::k_build_links<<<grid, 128, 0, st>>>(d, V, U, (double2*)fat, (double2*)lng, c1, c_staple, c3, hd, list, cap);
    return last_launch_status();
  };
  // Coefficients as fixed point with a power of two taken out; beyond 2^+-900
  // (or not finite) the FP64 kernel, whose range is wider.
  const double big = std::fmax(std::fabs(c1), 8.0 * std::fabs(c_staple)), big3 = std::fabs(c3);
  int k = 0, k3 = 0;
  if (!(big > 0x1p-900 && big < 0x1p900 && big3 > 0x1p-900 && big3 < 0x1p900) || c1 != c1 || c_staple != c_staple)
    return fp64(nullptr, nullptr);
  std::frexp(big, &k);
  std::frexp(big3, &k3);
  // the fixed-point copy of the links and the list (608 B per site) in stream-ordered
  // scratch; without room for it the FP64 kernel does the work
  const size_t fbytes = fx::field_bytes(V, 4);
  char* scratch = nullptr;
  if (cudaMallocAsync((void**)&scratch, 256 + fbytes + (size_t)cap * sizeof(long long), st) != cudaSuccess) {
    cudaGetLastError();
    return fp64(nullptr, nullptr);
  }
  fx::Header* hd = (fx::Header*)scratch;
  int4* Uf = (int4*)(scratch + 256);
  long long* list = (long long*)(scratch + 256 + fbytes);
  const unsigned tiles = (unsigned)((V + fx::TS - 1) / fx::TS);
  const fx::Coef none{0, 0};
  int s;
  {
    ProfScope ps("links", st);
    s = fx::launch_fx_links(V, U, Uf, 4, 0, hd, st);
  }
  if (!s) {
    ProfScope ps("links", st);
    lb::k_build_links_fx<true><<<tiles, 128, 0, st>>>(d, V, Uf, hd, list, cap, (double2*)fat, fx::make_coef(std::ldexp(c1, -k)),
                                                      fx::make_coef(std::ldexp(c_staple, 3 - k)), k - 60);
    s = last_launch_status();
  }
  if (!s) {
    ProfScope ps("links", st);
    lb::k_build_links_fx<false><<<tiles, 128, 0, st>>>(d, V, Uf, hd, list, cap, (double2*)lng,
                                                       fx::make_coef(std::ldexp(c3, -k3)), none, k3 - 60);
    s = last_launch_status();
  }
  if (!s) s = fp64(hd, list);
  const int f = cuda_status(cudaFreeAsync(scratch, st));
  return s ? s : f;
}
