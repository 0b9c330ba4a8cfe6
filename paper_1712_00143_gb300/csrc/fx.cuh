// fx.cuh -- 3x3 complex matrix products of FP64-class accuracy on the integer
// pipe, for fields of SU(3) links.
//
// GB300 retires 2.2 FP64 multiply-adds per clock and SM and 32 integer ones
// of 32 x 32 + 64 bits, which are exact, so a product of link matrices is
// computed in fixed point.  A number |v| <= 1 is held as
//   v = h 2^-30 + l 2^-60,   h, l signed 32-bit, |l| <= 2^29,
// that is, to 2^-60 (FP64 rounds numbers near 1 to 2^-53), and
//   a b = (h_a h_b) 2^-60 + (h_a l_b + l_a h_b) 2^-90 + O(2^-62):
// three multiply-adds into two 64-bit sums.  Of the cross sum m only the high
// word is kept (2^-58, rounded), which needs no 64-bit shift.  A complex
// product takes three real ones (Gauss): with P1 = sum ar br, P2 = sum ai bi,
// P3 = sum (ar + ai)(br + bi), the real part is P1 - P2 and the imaginary
// part P3 - P1 - P2, all exact in the h sums.  Error of an entry: about 2^-58,
// thirty times below that of the FP64 chain of six multiply-adds.
// One product costs a warp 1.3 k clocks of an SM quarter (81 x 3 wide
// multiply-adds at 4 clocks each, the rest on the ALU pipe beside them;
// measured; 1.5 k with four real products per complex one), against 6.3 k in
// FP64.
//
// Range.  Every factor is unitary to 2^-12 or a product of such (checked for
// the input links, see k_fx_links), so rows and columns have norm <= 1.01;
// by Cauchy-Schwarz an entry's h sums stay below 2^61.1, and its cross sums,
// with |ar + ai| and |br + bi| of row norm sqrt 2, below 2 sqrt(2) sqrt(3)
// 2^60 < 2^62.4.
#pragma once
#include "fx_steps.h"
#include "su3.cuh"

namespace stag {
namespace fx {

using su3::Dims;

// One matrix: entry e = 3 row + column, [2 e] real, [2 e + 1] imaginary part.
struct FM {
  int h[18], l[18];
};

// One entry of a b, in units of 2^-60.
__device__ __forceinline__ void entry(const FM& a, const FM& b, int i, int j, long long& re, long long& im) {
  constexpr long long half = 0x80000000LL;  // rounds the high word of a cross sum
  long long p1, p2, p3, m1 = half, m2 = half, m3 = half;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const int e = 2 * (3 * i + k), f = 2 * (3 * k + j);
    const int sh = a.h[e] + a.h[e + 1], sl = a.l[e] + a.l[e + 1];
    const int th = b.h[f] + b.h[f + 1], tl = b.l[f] + b.l[f + 1];
    if (k == 0) {
      p1 = wmul(a.h[e], b.h[f]);
      p2 = wmul(a.h[e + 1], b.h[f + 1]);
      p3 = wmul(sh, th);
    } else {
      wmad(p1, a.h[e], b.h[f]);
      wmad(p2, a.h[e + 1], b.h[f + 1]);
      wmad(p3, sh, th);
    }
    wmad(m1, a.h[e], b.l[f]);
    wmad(m1, a.l[e], b.h[f]);
    wmad(m2, a.h[e + 1], b.l[f + 1]);
    wmad(m2, a.l[e + 1], b.h[f + 1]);
    wmad(m3, sh, tl);
    wmad(m3, sl, th);
  }
  // high words, units of 2^-58; the differences are below 2^31 whatever the terms (unsigned: modulo 2^32)
  const unsigned c1 = (unsigned)(m1 >> 32), c2 = (unsigned)(m2 >> 32), c3 = (unsigned)(m3 >> 32);
  re = p1 - p2 + (long long)(int)(c1 - c2) * 4;
  im = p3 - p1 - p2 + (long long)(int)(c3 - c1 - c2) * 4;
}

// a b
__device__ __forceinline__ FM mul(const FM& a, const FM& b) {
  FM c;
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      long long re, im;
      entry(a, b, i, j, re, im);
      const int e = 2 * (3 * i + j);
      split1(re, c.h[e], c.l[e]);
      split1(im, c.h[e + 1], c.l[e + 1]);
    }
  return c;
}

// s (units of 2^-60) += a b; up to seven products of unitary matrices fit
__device__ __forceinline__ void mac(long long (&s)[18], const FM& a, const FM& b) {
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      long long re, im;
      entry(a, b, i, j, re, im);
      const int e = 2 * (3 * i + j);
      s[e] += re;
      s[e + 1] += im;
    }
}

__device__ __forceinline__ void clear(long long (&s)[18]) {
#pragma unroll
  for (int i = 0; i < 18; ++i) s[i] = 0;
}

// ------------------------------------------------------------ coefficients
// A coefficient |c| <= 1 in the same form, and c s for |s| <= 2^60.
struct Coef {
  int h, l;
};
__device__ __forceinline__ long long scaled(Coef c, long long s) {
  int h, l;
  split1(s, h, l);
  long long p = wmul(c.h, h), m = 0x80000000LL;
  wmad(m, c.h, l);
  wmad(m, c.l, h);
  return p + ((long long)(int)(m >> 32) << 2);
}
// Host: c = coefficient 2^k with a common k for a set of coefficients.
inline Coef make_coef(double c) {  // |c| <= 1
  Coef r;
  const double s = c * 0x1p30;
  const long long h = (long long)(s < 0 ? s - 0.5 : s + 0.5);
  r.h = (int)h;
  r.l = (int)((s - (double)h) * 0x1p30);
  return r;
}

// ------------------------------------------------------------ field layout
// Tiles of 32 consecutive sites; in a tile, one row of 32 int4 {re.h, re.l,
// im.h, im.l} per entry: [site / 32][slot][entry][site % 32].  A warp's loads
// over consecutive sites are whole 512-byte rows, and the nine entries of a
// matrix lie at constant offsets from one address.
constexpr int TS = 32;
inline size_t field_bytes(long long V, int slots) { return (size_t)((V + TS - 1) / TS) * TS * slots * 9 * sizeof(int4); }
__device__ __forceinline__ size_t row0(int slots, int site, int slot) {
  return (size_t)((site >> 5) * slots + slot) * 288 + (site & 31);
}
template <int SLOTS> __device__ __forceinline__ FM ld(const int4* __restrict__ f, int slot, int site) {
  FM m;
  const int4* p = f + row0(SLOTS, site, slot);
#pragma unroll
  for (int e = 0; e < 9; ++e) {
    const int4 q = __ldg(p + e * 32);
    m.h[2 * e] = q.x;
    m.l[2 * e] = q.y;
    m.h[2 * e + 1] = q.z;
    m.l[2 * e + 1] = q.w;
  }
  return m;
}
// A matrix copied asynchronously into the thread's own column of a [9][128]
// block of int4 in shared memory, and read from there: no other thread is
// waited for.
template <int SLOTS> __device__ __forceinline__ void copy_column(int4* col, const int4* __restrict__ f, int slot, int site) {
  const int4* p = f + row0(SLOTS, site, slot);
  const unsigned to = (unsigned)__cvta_generic_to_shared(col);
#pragma unroll
  for (int e = 0; e < 9; ++e)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(to + e * 2048), "l"(p + e * 32) : "memory");
}
__device__ __forceinline__ void wait_columns() { asm volatile("cp.async.wait_all;" ::: "memory"); }
__device__ __forceinline__ FM from_column(const int4* col) {
  FM m;
#pragma unroll
  for (int e = 0; e < 9; ++e) {
    const int4 q = col[e * 128];
    m.h[2 * e] = q.x;
    m.l[2 * e] = q.y;
    m.h[2 * e + 1] = q.z;
    m.l[2 * e + 1] = q.w;
  }
  return m;
}
template <int SLOTS> __device__ __forceinline__ void st(int4* __restrict__ f, int slot, int site, const FM& m) {
  int4* p = f + row0(SLOTS, site, slot);
#pragma unroll
  for (int e = 0; e < 9; ++e) p[e * 32] = make_int4(m.h[2 * e], m.l[2 * e], m.h[2 * e + 1], m.l[2 * e + 1]);
}
// m, or its adjoint (adj: 0 or -1): one code path for factors that are daggered
// in some terms of a loop keeps the loop inside the instruction cache.
__device__ __forceinline__ void adjoint_if(FM& m, int adj) {
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    m.h[8 * i + 1] = (m.h[8 * i + 1] ^ adj) - adj;
    m.l[8 * i + 1] = (m.l[8 * i + 1] ^ adj) - adj;
#pragma unroll
    for (int j = i + 1; j < 3; ++j) {
      const int e = 2 * (3 * i + j), f = 2 * (3 * j + i);
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        const int eh = m.h[e + c], el = m.l[e + c], fh = m.h[f + c], fl = m.l[f + c], sg = c ? adj : 0;
        m.h[e + c] = ((adj ? fh : eh) ^ sg) - sg;
        m.l[e + c] = ((adj ? fl : el) ^ sg) - sg;
        m.h[f + c] = ((adj ? eh : fh) ^ sg) - sg;
        m.l[f + c] = ((adj ? el : fl) ^ sg) - sg;
      }
    }
  }
}

// A site's index and coordinates in 32 bits (the entry points take at most 2^31
// sites): 64-bit index products would run on the wide multiply-add pipe.
struct Site {
  int lex;
  su3::C4 c;
};
__device__ __forceinline__ Site site_of(const Dims& d, int x) {
  Site p;
  p.lex = x;
  const int r = x / d.L0, q = r / d.L1;
  p.c.x = x - r * d.L0;
  p.c.y = r - q * d.L1;
  p.c.t = q / d.L2;
  p.c.z = q - p.c.t * d.L2;
  return p;
}
// The index of p moved by k = +-1 along mu (periodic).
__device__ __forceinline__ int next_lex(const Dims& d, const Site& p, int mu, int k) {
  const int L = su3::extent(d, mu), v = p.c.get(mu);
  const int st = mu == 0 ? 1 : mu == 1 ? d.L0 : mu == 2 ? d.L0 * d.L1 : d.L0 * d.L1 * d.L2;
  const int w = v + k;
  return p.lex + st * ((w >= L ? w - L : w < 0 ? w + L : w) - v);
}
__device__ __forceinline__ Site next(const Dims& d, const Site& p, int mu, int k) {
  Site q = p;
  q.lex = next_lex(d, p, mu, k);
  const int L = su3::extent(d, mu);
  int w = p.c.get(mu) + k;
  w = w >= L ? w - L : w < 0 ? w + L : w;
  q.c.x = mu == 0 ? w : q.c.x;
  q.c.y = mu == 1 ? w : q.c.y;
  q.c.z = mu == 2 ? w : q.c.z;
  q.c.t = mu == 3 ? w : q.c.t;
  return q;
}

// ------------------------------------------------------------ canonical fields
// A block of 128 threads takes one tile of 32 sites; warp w the direction
// mu = w of each.  The canonical field [V][4][3][3] of those sites is one
// contiguous 18 KB piece, moved through shared memory with whole-warp
// contiguous accesses; there a site takes 592 B (37 16-byte words, odd: the
// eight threads of a 128-bit access phase fall in different bank groups).
constexpr int SITE_W = 37;

// Bits of *status.  Set by k_fx_links: some link is not unitary to 2^-12 (or
// not finite); some link is at least 2^-5 away from the unit matrix.  Set by a
// later kernel: some other input's exponent is out of range.
enum : int { FX_NOT_UNITARY = 1, FX_AWAY = 2, FX_RANGE = 4 };
// The integer kernels run on FX_AWAY alone.  Links all close to the unit
// matrix stay on the FP64 kernels: their small entries, and a force made of
// them, would be known to 2^-58 absolute where FP64 keeps 2^-53 relative.
__device__ __forceinline__ bool usable(const int* status) { return __ldcg(status) == FX_AWAY; }

// The distance of m from the diagonal matrices of 1, -1, i, -i, in units of 2^-30.
__device__ __forceinline__ int away(const FM& m) {
  int d = 0;
#pragma unroll
  for (int e = 0; e < 9; ++e) {
    const int re = abs(m.h[2 * e]), im = abs(m.h[2 * e + 1]);
    d = max(d, e % 4 == 0 ? min(re, im) : max(re, im));
  }
  return d;
}

// What a call's scratch starts with: the status word, the count of single
// results that the integer kernels leave to the FP64 ones, and the counts of
// links within 3 2^-6 and 3 2^-5 of a diagonal matrix of 1, -1, i, -i.
struct Header {
  int status;
  unsigned long long marked;
  unsigned long long near[2];
};
enum : int { NEAR_6 = 0, NEAR_5 = 1 };
// Whether the integer kernels run.  Where more than half of the links are near
// (at the distance at which a routine marks its results) they would leave most
// of the work to the FP64 kernels anyway.
__device__ __forceinline__ bool serve(const Header* hd, int which, long long V, unsigned long long* count = nullptr) {
  const unsigned long long n = __ldcg(&hd->near[which]);  // (both words are asked for before either is waited for)
  const bool ok = usable(&hd->status);
  if (count) *count = n;
  return ok & ((long long)n <= 2 * V);
}
__device__ __forceinline__ void mark(Header* hd, long long* __restrict__ list, long long cap, long long item) {
  const unsigned long long n = atomicAdd(&hd->marked, 1ull);
  if ((long long)n < cap) list[n] = item;
}
// The FP64 kernels do the whole field when the integer kernels may not, or have
// marked more results than the list holds.
__device__ __forceinline__ bool all_fp64(const Header* hd, int which, long long V, long long cap) {
  return !serve(hd, which, V) || (long long)__ldcg(&hd->marked) > cap;
}

// Fixed-point copy of the thin links [V][4][3][3] into slots slot0 + mu of a
// field with `slots` slots, and *hd (fx.cu).
int launch_fx_links(long long V, const double2* U, int4* out, int slots, int slot0, Header* hd, cudaStream_t st);

}  // namespace fx
}  // namespace stag
