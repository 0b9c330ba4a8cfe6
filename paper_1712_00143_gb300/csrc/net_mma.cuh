// net_mma.cuh -- the preconditioner network's 16 -> 16 layers and every weight
// gradient on the tensor cores, straight from registers.
//
// A layer computes pre_c(x) = sum_d sum_c' W[d][c][c'] (T_d h_c')(x).  Its
// products are small (per site six rows x 16 channels x 16 channels, nine
// directions): with tcgen05 the transported channels had to be written to
// shared memory as an operand, waited for and handed over at two barriers per
// direction, and that staging, not the products, took the time (366 us at
// 24^4, tensor pipe 2 % busy, three CTAs per SM).  mma.sync m16n8k16 takes the
// operand from the registers in which the transports are computed:
//   a warp takes 8 sites; lane 4 g + t holds, of site g, the channel pairs t
//   and t + 4 (channels 2t, 2t+1, 2t+8, 2t+9).  For one colour the real parts
//   are rows 0..7 and the imaginary parts rows 8..15 of the 16 x 16 A operand,
//   whose fragment is then exactly what the lane has; the accumulator's
//   fragment gives the lane the same two channel pairs of the output, so that
//   gate and stores need no exchange either.
// Every warp works by itself: no barrier after the start, its gather running
// three directions ahead in shared memory of its own.
// The transports enter as two bfloat16 parts (16 bits), products and sums are
// FP32.  The unit truncates its sums, and over a chain of them that shrinks
// every result by the same few 2^-22, which a gradient, a sum over all sites,
// keeps while the sites' own errors average out.  So in training a product
// starts from zero for each direction, the low parts first, and is added with
// rounding outside: gradient at 16 x 20 x 12 x 24 3.0e-7 from the 64-bit one
// against 3.4e-6, for 3.5 % more time per layer.  Applied as a preconditioner
// the network's values are as good either way (4.2e-6 and 4.5e-6), and the
// products are summed in one chain.
#pragma once
#include "net_tc.cuh"

namespace stag {
namespace nm {

__device__ __forceinline__ void mma(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                    uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
// transpose of an 8 x 8 matrix of 16-bit values held two per lane
__device__ __forceinline__ uint32_t trans(uint32_t a) {
  uint32_t d;
  asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(d) : "r"(a));
  return d;
}

// Two values as three bfloat16 parts each (24 significant bits): part 0 + part 1
// is tc::split2's pair.
__device__ __forceinline__ void split3(float a, float b, uint32_t (&p)[3]) {
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    p[k] = *reinterpret_cast<const uint32_t*>(&h);
    a -= __low2float(h);
    b -= __high2float(h);
  }
}

// The two hop matrices of direction mu at site s: +mu (d = 1 + 2 mu) and -mu (d = 2 + 2 mu).
__device__ __forceinline__ void load_hops(const NetGeom& ng, int p, int s, int mu, float2 (&w)[2][9]) {
  const uint4* src = (p ? ng.links[1] : ng.links[0]) + (size_t)(mu * ng.cpm >> 1) * ng.g.Vh + s;
#pragma unroll
  for (int j = 0; j < 9; ++j) {
    const uint4 c = __ldg(src + (size_t)j * ng.g.Vh);
    w[2 * j / 9][2 * j % 9] = make_float2(__uint_as_float(c.x), __uint_as_float(c.y));
    w[(2 * j + 1) / 9][(2 * j + 1) % 9] = make_float2(__uint_as_float(c.z), __uint_as_float(c.w));
  }
}

// Channel pairs t and t + 4 of one site's record: [pair][channel of the pair][colour].
// A 16-channel record is stored as the 16-byte words [half q][word k][t]: word
// k (two colour components) of pair t + 4 q, so that a load or store of one
// word by the four lanes of a site is 64 contiguous bytes.  (With a pair's
// three words in a row every access touched twice the sectors.)
struct Pairs {
  float2 v[2][2][3];
};
__device__ __forceinline__ Pairs load_pairs(const float2* rec, int t) {
  Pairs r;
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const float4* f = (const float4*)rec + 12 * q + t;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const float4 u = __ldg(f + 4 * k);
      r.v[q][(2 * k) / 3][(2 * k) % 3] = make_float2(u.x, u.y);
      r.v[q][(2 * k + 1) / 3][(2 * k + 1) % 3] = make_float2(u.z, u.w);
    }
  }
  return r;
}
__device__ __forceinline__ void store_pairs(float2* rec, int t, const Pairs& r) {
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    float4* f = (float4*)rec + 12 * q + t;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const float2 a = r.v[q][(2 * k) / 3][(2 * k) % 3], b = r.v[q][(2 * k + 1) / 3][(2 * k + 1) % 3];
      f[4 * k] = make_float4(a.x, a.y, b.x, b.y);
    }
  }
}

// Colour i of the pair q after the hop w (or as it is): {re, re', im, im'} of its two channels.
__device__ __forceinline__ float4 transported(const Pairs& v, const float2 (&w)[9], int q, int i) {
  float2 x[2];
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    x[c] = make_float2(0.f, 0.f);
#pragma unroll
    for (int j = 0; j < 3; ++j) cmac(x[c], w[3 * i + j], v.v[q][c][j]);
  }
  return make_float4(x[0].x, x[1].x, x[0].y, x[1].y);
}

// ---- the gather, three directions ahead
// A lane copies the six words it will read itself (cp.async into its own
// column of shared memory: no other lane is waited for), and the warp's lanes
// together the nine words of each site's two hop matrices of a direction mu.
// (Loads straight into registers left the layer waiting for L2: 206 us at 24^4
// at four warps per scheduler; there are no registers for a second set.  With
// the copies ahead it takes 180 us, scheduler 62 % busy with the split and the
// transports, two blocks per SM at 95 KB of shared memory and 111 registers.)
constexpr int TW = 8;  // warps per block of the thin weight gradients
constexpr int STAGES = 3;
struct WarpStage {
  float4 v[STAGES][6][32];  // [stage][word][lane]
  uint4 w[2][9][8];         // [slot][chunk][site]
};
__device__ __forceinline__ void copy16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(tc::smem_u32(dst)), "l"(src) : "memory");
}

// Walks (group of 8 sites, direction 0..8) and issues one direction's copies
// per step; consumers follow in the same order.
struct Gather {
  const NetGeom& ng;
  const float2* act;
  WarpStage* st;
  int grp, step, total, per;  // current group, groups per step, all groups, groups per parity
  int lane, d = 0, stage = 0, slot = 0, p = 0, s = 0;
  Coord c;
  __device__ __forceinline__ Gather(const NetGeom& ng_, const float2* a, WarpStage* st_, int first, int step_)
      : ng(ng_), act(a), st(st_), grp(first), step(step_), lane(threadIdx.x & 31) {
    per = (ng.g.Vh + 7) / 8;
    total = 2 * per;
  }
  __device__ __forceinline__ void issue() {
    if (grp < total) {
      const int Vh = ng.g.Vh;
      if (d == 0) {
        p = grp >= per;
        s = (grp - p * per) * 8 + (lane >> 2);
        s = s < Vh ? s : Vh - 1;
        c = cb_coords(ng.g, s, p);
      }
      const int mu = (d - 1) >> 1;
      const int ns = d == 0 ? s : cb_neighbour(ng.g, s, c, mu, (d & 1) ? 1 : -1);
      const float4* f = (const float4*)act_ptr(act, 16, Vh, d ? 1 - p : p, ns) + (lane & 3);
#pragma unroll
      for (int k = 0; k < 6; ++k) copy16(&st->v[stage][k][lane], f + 12 * (k / 3) + 4 * (k % 3));
      if (d & 1) {
        // chunks t, t + 4, t + 8 of this lane's site
        const uint4* src = (p ? ng.links[1] : ng.links[0]) + (size_t)(mu * ng.cpm >> 1) * Vh + s;
#pragma unroll
        for (int j = 0; j < 3; ++j) {
          const int k = (lane & 3) + 4 * j;
          if (k < 9) copy16(&st->w[slot][k][lane >> 2], src + (size_t)k * Vh);
        }
        slot ^= 1;
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
    stage = stage == STAGES - 1 ? 0 : stage + 1;
    if (++d == NET_NDIR) {
      d = 0;
      grp += step;
    }
  }
  __device__ __forceinline__ static void wait() {  // the oldest direction in flight has arrived, for the whole warp
    asm volatile("cp.async.wait_group %0;" ::"n"(STAGES - 1) : "memory");
    __syncwarp();
  }
  __device__ __forceinline__ static void drain() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }
};
__device__ __forceinline__ Pairs staged_pairs(const WarpStage* st, int stage, int lane) {
  Pairs r;
#pragma unroll
  for (int q = 0; q < 2; ++q)
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const float4 u = st->v[stage][3 * q + k][lane];
      r.v[q][(2 * k) / 3][(2 * k) % 3] = make_float2(u.x, u.y);
      r.v[q][(2 * k + 1) / 3][(2 * k + 1) % 3] = make_float2(u.z, u.w);
    }
  return r;
}
// hop matrix k (0: +mu, 1: -mu) of the lane's site: entries 9 k .. 9 k + 8 of the slot's eighteen
template <int K> __device__ __forceinline__ void staged_hop(const WarpStage* st, int slot, int site, float2 (&w)[9]) {
#pragma unroll
  for (int j = 4 * K; j < 5 + 4 * K; ++j) {
    const uint4 c = st->w[slot][j][site];
    const int e = 2 * j - 9 * K;
    if (e >= 0) w[e] = make_float2(__uint_as_float(c.x), __uint_as_float(c.y));
    if (e + 1 < 9) w[e + 1] = make_float2(__uint_as_float(c.z), __uint_as_float(c.w));
  }
}

// The weights as B fragments, one uint4 per direction and lane: {b0, b1} of
// output channels 0..7, then 8..15.  transpose: the adjoint layer's, sign(d)
// W[partner(d)][c'][c].
__device__ __forceinline__ void stage_weights(uint4* sB, const __nv_bfloat16* __restrict__ W, int transpose) {
  for (int i = threadIdx.x; i < NET_NDIR * 32; i += blockDim.x) {
    const int d = i >> 5, g = (i >> 2) & 7, t = i & 3;
    uint32_t b[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int c = (k >> 1) * 8 + g, cp = 2 * t + (k & 1) * 8;  // output channel; input channels cp, cp + 1
      uint32_t lo, hi;
      if (!transpose) {
        lo = __bfloat16_as_ushort(W[(d * 16 + c) * 16 + cp]);
        hi = __bfloat16_as_ushort(W[(d * 16 + c) * 16 + cp + 1]);
      } else {
        const int dd = d == 0 ? 0 : ((d & 1) ? d + 1 : d - 1);
        const uint32_t sg = d ? 0x8000u : 0u;
        lo = __bfloat16_as_ushort(W[(dd * 16 + cp) * 16 + c]) ^ sg;
        hi = __bfloat16_as_ushort(W[(dd * 16 + cp + 1) * 16 + c]) ^ sg;
      }
      b[k] = lo | hi << 16;
    }
    sB[i] = make_uint4(b[0], b[1], b[2], b[3]);
  }
}

// A field's own-site channel pairs as the transposed parts of a product over
// sites: part k, colour i, {re, im} x {pair t, pair t + 4} -> word
// ((k 3 + i) 2 + (0: pair t, 1: pair t + 4)) 2 + (0: re, 1: im).
__device__ __forceinline__ void site_operand(const Pairs& h, uint32_t (&o)[36]) {
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      uint32_t re[3], im[3];
      split3(h.v[q][0][i].x, h.v[q][1][i].x, re);
      split3(h.v[q][0][i].y, h.v[q][1][i].y, im);
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        o[((k * 3 + i) * 2 + q) * 2] = trans(re[k]);
        o[((k * 3 + i) * 2 + q) * 2 + 1] = trans(im[k]);
      }
    }
}

// d[nt] += sum over the 8 sites and (re, im) of colour i: a (channels or
// directions m: transposed parts [part]{re t, re t+4, im t, im t+4}) times the
// site operand (parts b[part][nt]{re, im}).  Six products of parts carry 24 bits
// of each factor; the five small ones, the smallest first, have a sum of their
// own, and both are added with rounding.
__device__ __forceinline__ void outer(float (&d)[2][4], const uint32_t (&a)[3][4], const uint2 (&b)[3][2]) {
#pragma unroll
  for (int nt = 0; nt < 2; ++nt) {
    float s[4] = {0.f, 0.f, 0.f, 0.f}, m[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int n = 2; n > 0; --n)
#pragma unroll
      for (int k = 0; k <= n; ++k) mma(s, a[k][0], a[k][1], a[k][2], a[k][3], b[n - k][nt].x, b[n - k][nt].y);
    mma(m, a[0][0], a[0][1], a[0][2], a[0][3], b[0][nt].x, b[0][nt].y);
#pragma unroll
    for (int e = 0; e < 4; ++e) d[nt][e] += m[e] + s[e];
  }
}
// acc += s, rounded to nearest
__device__ __forceinline__ void add(float (&acc)[2][4], const float (&s)[2][4]) {
#pragma unroll
  for (int nt = 0; nt < 2; ++nt)
#pragma unroll
    for (int e = 0; e < 4; ++e) acc[nt][e] += s[nt][e];
}

constexpr int FW = 8;    // warps per block of the forward layer
constexpr int AW = 4;    // ... of the adjoint layer with its weight gradient
constexpr int FWD_SMEM = NET_NDIR * 32 * 16 + FW * (int)sizeof(WarpStage);  // two blocks per SM
constexpr int DWF = NET_NDIR * 256;  // floats of one weight gradient
// shared memory of the adjoint kernel: weights, and per warp the gradient sums and the site operand
constexpr int ADJ_SMEM = NET_NDIR * 32 * 16 + AW * (DWF * 4 + 36 * 32 * 4);

}  // namespace nm

// The forward layer: hout = pre * sigmoid(|pre|^2 - b_c).  TRAIN: pre is stored
// and the sums are rounded.  A warp takes every nwarps-th group of 8 sites.
template <bool TRAIN>
__global__ void __launch_bounds__(32 * nm::FW, 2)
    k_net_layer_mma(NetGeom ng, const float2* __restrict__ hin, float2* __restrict__ pre, float2* __restrict__ hout,
                    const __nv_bfloat16* __restrict__ W, const float* __restrict__ bias) {
  using namespace nm;
  extern __shared__ __align__(16) unsigned char nm_fwd[];
  uint4* sB = (uint4*)nm_fwd;
  const int Vh = ng.g.Vh, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  WarpStage* st = (WarpStage*)(nm_fwd + NET_NDIR * 32 * 16) + (threadIdx.x >> 5);
  const int per = (Vh + 7) / 8, nwarps = gridDim.x * FW, first = blockIdx.x * FW + (threadIdx.x >> 5);
  Gather ahead(ng, hin, st, first, nwarps);
#pragma unroll
  for (int k = 0; k < STAGES; ++k) ahead.issue();
  stage_weights(sB, W, 0);
  __syncthreads();
  int stage = 0, slot = 0;
  for (int grp = first; grp < 2 * per; grp += nwarps) {
    const int p = grp >= per, s = (grp - p * per) * 8 + g;
    const bool in = s < Vh;
    float acc[3][2][4];
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int nt = 0; nt < 2; ++nt)
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[i][nt][e] = 0.f;
    auto mix = [&](int i, const float4& x0, const float4& x1, const uint4& b) {
      uint32_t h[4], l[4];
      tc::split2(x0.x, x0.y, h[0], l[0]);
      tc::split2(x0.z, x0.w, h[1], l[1]);
      tc::split2(x1.x, x1.y, h[2], l[2]);
      tc::split2(x1.z, x1.w, h[3], l[3]);
      if constexpr (TRAIN) {
        float s[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
        mma(s[0], l[0], l[1], l[2], l[3], b.x, b.y);
        mma(s[1], l[0], l[1], l[2], l[3], b.z, b.w);
        mma(s[0], h[0], h[1], h[2], h[3], b.x, b.y);
        mma(s[1], h[0], h[1], h[2], h[3], b.z, b.w);
        add(acc[i], s);
      } else {
        mma(acc[i][0], h[0], h[1], h[2], h[3], b.x, b.y);
        mma(acc[i][1], h[0], h[1], h[2], h[3], b.z, b.w);
        mma(acc[i][0], l[0], l[1], l[2], l[3], b.x, b.y);
        mma(acc[i][1], l[0], l[1], l[2], l[3], b.z, b.w);
      }
    };
    auto done = [&]() {  // the stage has been read by its lane, the slot by the warp: the next direction may come
      __syncwarp();
      ahead.issue();
      stage = stage == STAGES - 1 ? 0 : stage + 1;
    };
    {
      Gather::wait();
      const Pairs v = staged_pairs(st, stage, lane);
      const uint4 b = sB[lane];
#pragma unroll
      for (int i = 0; i < 3; ++i)
        mix(i, make_float4(v.v[0][0][i].x, v.v[0][1][i].x, v.v[0][0][i].y, v.v[0][1][i].y),
            make_float4(v.v[1][0][i].x, v.v[1][1][i].x, v.v[1][0][i].y, v.v[1][1][i].y), b);
      done();
    }
#pragma unroll 1
    for (int mu = 0; mu < 4; ++mu) {
      {
        Gather::wait();
        float2 w[9];
        staged_hop<0>(st, slot, g, w);
        const Pairs v = staged_pairs(st, stage, lane);
        const uint4 b = sB[(1 + 2 * mu) * 32 + lane];
#pragma unroll
        for (int i = 0; i < 3; ++i) mix(i, transported(v, w, 0, i), transported(v, w, 1, i), b);
        done();
      }
      {
        Gather::wait();
        float2 w[9];
        staged_hop<1>(st, slot, g, w);
        const Pairs v = staged_pairs(st, stage, lane);
        const uint4 b = sB[(2 + 2 * mu) * 32 + lane];
#pragma unroll
        for (int i = 0; i < 3; ++i) mix(i, transported(v, w, 0, i), transported(v, w, 1, i), b);
        done();
      }
      slot ^= 1;
    }
    // pair q of the output = accumulator nt = q
    Pairs o, h;
#pragma unroll
    for (int q = 0; q < 2; ++q)
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        float2 v[3];
#pragma unroll
        for (int i = 0; i < 3; ++i) v[i] = o.v[q][e][i] = make_float2(acc[i][q][e], acc[i][q][2 + e]);
        const float n2 = v[0].x * v[0].x + v[0].y * v[0].y + v[1].x * v[1].x + v[1].y * v[1].y + v[2].x * v[2].x +
                         v[2].y * v[2].y;
        const float sg = 1.f / (1.f + __expf(-(n2 - bias[2 * t + 8 * q + e])));
#pragma unroll
        for (int i = 0; i < 3; ++i) h.v[q][e][i] = make_float2(v[i].x * sg, v[i].y * sg);
      }
    if (in) {
      if (TRAIN) store_pairs(act_ptr(pre, 16, Vh, p, s), t, o);
      store_pairs(act_ptr(hout, 16, Vh, p, s), t, h);
    }
  }
  Gather::drain();
}

// Layers with one input and 16 output channels, on the CUDA cores: the first
// layer (GATE; its input is zero on odd sites, so an even site has only
// direction 0 and an odd site the eight hops), and the adjoint of the last
// (W' = sign(d) W[partner(d)]; its input, the output gradient, is zero on odd
// sites as well).  Lane 4 g + t computes site g's transports (the four lanes
// of a site all do: their loads are the same words) and takes the channel
// pairs t and t + 4, so that its sums are 24 registers and its stores whole
// 48-byte runs.
template <bool GATE>
__global__ void __launch_bounds__(256, 3)
    k_net_layer_1to16(NetGeom ng, const float2* __restrict__ hin, float2* __restrict__ pre, float2* __restrict__ hout,
                      const __nv_bfloat16* __restrict__ W, const float* __restrict__ bias) {
  using namespace nm;
  __shared__ float2 sw[NET_NDIR * 8];  // [d][pair]
  for (int i = threadIdx.x; i < NET_NDIR * 16; i += blockDim.x) {
    const int d = i >> 4, c = i & 15, dd = GATE || d == 0 ? d : ((d & 1) ? d + 1 : d - 1);
    const float w = __bfloat162float(W[dd * 16 + c]);
    ((float*)sw)[i] = GATE || d == 0 ? w : -w;
  }
  __syncthreads();
  const int Vh = ng.g.Vh, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3, per = (Vh + 7) / 8;
  const int grp = blockIdx.x * 8 + (threadIdx.x >> 5);
  if (grp >= 2 * per) return;
  const int p = grp >= per, s = (grp - p * per) * 8 + g;
  if (s >= Vh) return;
  Pairs o;
#pragma unroll
  for (int q = 0; q < 12; ++q) o.v[q / 6][q / 3 % 2][q % 3] = make_float2(0.f, 0.f);
  auto add = [&](int d, const float2 (&x)[3]) {
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const float2 w = sw[d * 8 + t + 4 * q];
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        o.v[q][0][i].x = fmaf(w.x, x[i].x, o.v[q][0][i].x);
        o.v[q][0][i].y = fmaf(w.x, x[i].y, o.v[q][0][i].y);
        o.v[q][1][i].x = fmaf(w.y, x[i].x, o.v[q][1][i].x);
        o.v[q][1][i].y = fmaf(w.y, x[i].y, o.v[q][1][i].y);
      }
    }
  };
  if (p == 0) {
    float2 v[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) v[i] = __ldg(hin + (size_t)s * 3 + i);
    add(0, v);
  } else {
    const Coord c = cb_coords(ng.g, s, p);
#pragma unroll 1
    for (int mu = 0; mu < 4; ++mu) {
      float2 w[2][9];
      load_hops(ng, p, s, mu, w);
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const float2* src = hin + (size_t)cb_neighbour(ng.g, s, c, mu, k ? -1 : 1) * 3;
        float2 v[3], x[3];
#pragma unroll
        for (int i = 0; i < 3; ++i) v[i] = __ldg(src + i);
#pragma unroll
        for (int i = 0; i < 3; ++i) {
          x[i] = make_float2(0.f, 0.f);
#pragma unroll
          for (int j = 0; j < 3; ++j) cmac(x[i], w[k][3 * i + j], v[j]);
        }
        add(1 + 2 * mu + k, x);
      }
    }
  }
  if (GATE) {
    if (pre) store_pairs(act_ptr(pre, 16, Vh, p, s), t, o);
#pragma unroll
    for (int q = 0; q < 2; ++q)
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const float2(&v)[3] = o.v[q][e];
        const float n2 = v[0].x * v[0].x + v[0].y * v[0].y + v[1].x * v[1].x + v[1].y * v[1].y + v[2].x * v[2].x +
                         v[2].y * v[2].y;
        const float sg = 1.f / (1.f + __expf(-(n2 - bias[2 * t + 8 * q + e])));
#pragma unroll
        for (int i = 0; i < 3; ++i) o.v[q][e][i] = make_float2(v[i].x * sg, v[i].y * sg);
      }
  }
  store_pairs(act_ptr(hout, 16, Vh, p, s), t, o);
}

// The adjoint layer gin = sum_d W'[d] T_d g and, from the same transports, the
// layer's weight gradient: since T_d^dag = -T_partner(d) (T_0 = 1),
//   dW[partner(d)][c][c'] = -sum_x Re <(T_d g_c)(x), h_c'(x)>   (d >= 1; + for d = 0),
// a product over sites whose operands are the transposed fragments.  hin is g,
// h the layer's input.  Each warp sums its groups' gradients in shared memory;
// part[block][9][16][16] gets the block's sum, warps in order.
__global__ void __launch_bounds__(32 * nm::AW, 3)
    k_net_adjoint_mma(NetGeom ng, const float2* __restrict__ hin, const float2* __restrict__ hsite,
                      float2* __restrict__ gout, const __nv_bfloat16* __restrict__ W, float* __restrict__ part) {
  using namespace nm;
  extern __shared__ __align__(16) unsigned char nm_sm[];
  uint4* sB = (uint4*)nm_sm;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  float4* dw = (float4*)(nm_sm + NET_NDIR * 32 * 16) + warp * (DWF / 4);  // [d][nt][lane] of four
  uint32_t* op = (uint32_t*)(nm_sm + NET_NDIR * 32 * 16 + AW * DWF * 4) + warp * 36 * 32;  // [word][lane]
  stage_weights(sB, W, 1);
  for (int i = lane; i < DWF / 4; i += 32) dw[i] = make_float4(0.f, 0.f, 0.f, 0.f);
  __syncthreads();
  const int Vh = ng.g.Vh, per = (Vh + 7) / 8, nwarps = gridDim.x * AW;
  for (int grp = blockIdx.x * AW + warp; grp < 2 * per; grp += nwarps) {
    const int p = grp >= per, s_raw = (grp - p * per) * 8 + g;
    const bool in = s_raw < Vh;
    const int s = in ? s_raw : Vh - 1;
    const Coord c = cb_coords(ng.g, s, p);
    {
      Pairs h = load_pairs(act_ptr(hsite, 16, Vh, p, s), t);
      if (!in) {
#pragma unroll
        for (int q = 0; q < 12; ++q) h.v[q / 6][q / 3 % 2][q % 3] = make_float2(0.f, 0.f);
      }
      uint32_t o[36];
      site_operand(h, o);
#pragma unroll
      for (int k = 0; k < 36; ++k) op[k * 32 + lane] = o[k];
    }
    float acc[3][2][4];
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int nt = 0; nt < 2; ++nt)
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[i][nt][e] = 0.f;
    auto direction = [&](int d, auto colour) {
      const uint4 b = sB[d * 32 + lane];
      float s4[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        const float4 x0 = colour(0, i), x1 = colour(1, i);
        uint32_t r0[3], i0[3], r1[3], i1[3];
        split3(x0.x, x0.y, r0);
        split3(x0.z, x0.w, i0);
        split3(x1.x, x1.y, r1);
        split3(x1.z, x1.w, i1);
        {
          float s[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
#pragma unroll
          for (int k = 1; k >= 0; --k) {
            mma(s[0], r0[k], i0[k], r1[k], i1[k], b.x, b.y);
            mma(s[1], r0[k], i0[k], r1[k], i1[k], b.z, b.w);
          }
          add(acc[i], s);
        }
        uint32_t a[3][4];
        uint2 q[3][2];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          a[k][0] = trans(r0[k]);
          a[k][1] = trans(r1[k]);
          a[k][2] = trans(i0[k]);
          a[k][3] = trans(i1[k]);
#pragma unroll
          for (int nt = 0; nt < 2; ++nt)
            q[k][nt] = make_uint2(op[(((k * 3 + i) * 2 + nt) * 2) * 32 + lane], op[(((k * 3 + i) * 2 + nt) * 2 + 1) * 32 + lane]);
        }
        outer(s4, a, q);
      }
#pragma unroll
      for (int nt = 0; nt < 2; ++nt) {
        float4 f = dw[(d * 2 + nt) * 32 + lane];
        f.x += s4[nt][0], f.y += s4[nt][1], f.z += s4[nt][2], f.w += s4[nt][3];
        dw[(d * 2 + nt) * 32 + lane] = f;
      }
    };
    {
      const Pairs v = load_pairs(act_ptr(hin, 16, Vh, p, s), t);
      direction(0, [&](int q, int i) {
        return make_float4(v.v[q][0][i].x, v.v[q][1][i].x, v.v[q][0][i].y, v.v[q][1][i].y);
      });
    }
#pragma unroll 1
    for (int mu = 0; mu < 4; ++mu) {
      float2 w[2][9];
      load_hops(ng, p, s, mu, w);
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const Pairs v = load_pairs(act_ptr(hin, 16, Vh, 1 - p, cb_neighbour(ng.g, s, c, mu, k ? -1 : 1)), t);
        direction(1 + 2 * mu + k, [&](int q, int i) { return transported(v, w[k], q, i); });
      }
    }
    if (in) {
      Pairs o;
#pragma unroll
      for (int q = 0; q < 2; ++q)
#pragma unroll
        for (int e = 0; e < 2; ++e)
#pragma unroll
          for (int i = 0; i < 3; ++i) o.v[q][e][i] = make_float2(acc[i][q][e], acc[i][q][2 + e]);
      store_pairs(act_ptr(gout, 16, Vh, p, s), t, o);
    }
  }
  __syncthreads();
  // accumulator (d, nt, lane, e): c = lane / 4 + 8 (e / 2), c' = 8 nt + 2 (lane % 4) + e % 2
  const float* all = (const float*)(nm_sm + NET_NDIR * 32 * 16);
  for (int i = threadIdx.x; i < DWF; i += blockDim.x) {
    const int e = i & 3, l = (i >> 2) & 31, nt = (i >> 7) & 1, d = i >> 8;
    float v = 0.f;
    for (int k = 0; k < AW; ++k) v += all[k * DWF + i];
    const int dd = d == 0 ? 0 : ((d & 1) ? d + 1 : d - 1);
    const int cc = (l >> 2) + 8 * (e >> 1), cp = 8 * nt + 2 * (l & 3) + (e & 1);
    part[(size_t)blockIdx.x * DWF + (dd * 16 + cc) * 16 + cp] = d ? -v : v;
  }
}

// Weight gradient of a layer between one channel u and sixteen channels f:
// sum_x Re <(T_d u)(x), f_c(x)>, [9][16].  1 -> 16: u the layer's input, f the
// output gradient.  16 -> 1 (adj): u the output gradient, f the input, and the
// sum for d belongs to partner(d) with the sign of T_d^dag = -T_partner(d).
// The nine directions take the place of the channels of the other operand:
// lane 4 g + t transports u to site g along 2t, 2t + 1 and (t = 0) 8.
// Bound by the latency of a group's loads: 33 us at 16 x 20 x 12 x 24 with
// twelve warps per SM (three blocks of four), 28 us with sixteen.
__global__ void __launch_bounds__(32 * nm::TW, 2)
    k_net_dw_thin(NetGeom ng, const float2* __restrict__ u, const float2* __restrict__ f, int adj,
                  float* __restrict__ part) {
  using namespace nm;
  const int Vh = ng.g.Vh, warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const int per = (Vh + 7) / 8, nwarps = gridDim.x * TW;
  float sum[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
  for (int grp = blockIdx.x * TW + warp; grp < 2 * per; grp += nwarps) {
    const int p = grp >= per, s_raw = (grp - p * per) * 8 + g;
    const bool in = s_raw < Vh;
    const int s = in ? s_raw : Vh - 1;
    const Coord c = cb_coords(ng.g, s, p);
    Pairs h = load_pairs(act_ptr(f, 16, Vh, p, s), t);
    if (!in) {
#pragma unroll
      for (int q = 0; q < 12; ++q) h.v[q / 6][q / 3 % 2][q % 3] = make_float2(0.f, 0.f);
    }
    uint32_t o[36];
    site_operand(h, o);
    float2 x[3][3];  // directions 2t, 2t + 1, 8
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const int d = k == 2 ? 8 : 2 * t + k, mu = (d + 3) / 2 - 2;  // d = 0 has no mu
      if (k == 2 && t) {
#pragma unroll
        for (int i = 0; i < 3; ++i) x[k][i] = make_float2(0.f, 0.f);
        continue;
      }
      const int ns = d ? cb_neighbour(ng.g, s, c, mu, (d & 1) ? 1 : -1) : s;
      const float2* src = u + ((size_t)(d ? 1 - p : p) * Vh + ns) * 3;
      float2 v[3], w[9];
#pragma unroll
      for (int i = 0; i < 3; ++i) v[i] = __ldg(src + i);
      if (d) {
        load_hop_matrix(ng, p, s, d, w);
#pragma unroll
        for (int i = 0; i < 3; ++i) {
          x[k][i] = make_float2(0.f, 0.f);
#pragma unroll
          for (int j = 0; j < 3; ++j) cmac(x[k][i], w[3 * i + j], v[j]);
        }
      } else {
#pragma unroll
        for (int i = 0; i < 3; ++i) x[k][i] = v[i];
      }
    }
    __syncwarp();
    float s4[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      uint32_t r0[3], i0[3], r1[3], i1[3], a[3][4];
      uint2 q[3][2];
      split3(x[0][i].x, x[1][i].x, r0);
      split3(x[0][i].y, x[1][i].y, i0);
      split3(x[2][i].x, 0.f, r1);
      split3(x[2][i].y, 0.f, i1);
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        a[k][0] = trans(r0[k]);
        a[k][1] = trans(r1[k]);
        a[k][2] = trans(i0[k]);
        a[k][3] = trans(i1[k]);
#pragma unroll
        for (int nt = 0; nt < 2; ++nt) q[k][nt] = make_uint2(o[((k * 3 + i) * 2 + nt) * 2], o[((k * 3 + i) * 2 + nt) * 2 + 1]);
      }
      outer(s4, a, q);
    }
#pragma unroll
    for (int nt = 0; nt < 2; ++nt)
#pragma unroll
      for (int e = 0; e < 4; ++e) sum[nt][e] += s4[nt][e];
  }
  // accumulator (nt, lane, e): d = lane / 4 + 8 (e / 2), c = 8 nt + 2 (lane % 4) + e % 2
  __shared__ float sm[TW][2][32][4];
#pragma unroll
  for (int nt = 0; nt < 2; ++nt)
#pragma unroll
    for (int e = 0; e < 4; ++e) sm[warp][nt][lane][e] = sum[nt][e];
  __syncthreads();
  for (int i = threadIdx.x; i < 256; i += 32 * TW) {
    const int e = i & 3, l = (i >> 2) & 31, nt = i >> 7, d = (l >> 2) + 8 * (e >> 1), cc = 8 * nt + 2 * (l & 3) + (e & 1);
    if (d >= NET_NDIR) continue;
    float v = 0.f;
    for (int k = 0; k < TW; ++k) v += sm[k][nt][l][e];
    const int dd = !adj || d == 0 ? d : ((d & 1) ? d + 1 : d - 1);
    part[(size_t)blockIdx.x * NET_NDIR * 16 + dd * 16 + cc] = adj && d ? -v : v;
  }
}

// The fragments above (weights, splits, products, transposes, outer products),
// one warp, on values whose sums are exact in FP32, against the CUDA cores:
// out = {max |difference|, max |reference|}.
__global__ void __launch_bounds__(32) k_mma_selftest(const __nv_bfloat16* __restrict__ W, float* out) {
  using namespace nm;
  __shared__ uint4 sB[2][NET_NDIR * 32];
  stage_weights(sB[0], W, 0);
  stage_weights(sB[1], W, 1);
  __syncthreads();
  const int lane = threadIdx.x, g = lane >> 2, t = lane & 3;
  // multiples of 2^-12 below 1 (fine) or of 1/8
  auto val = [](int d, int site, int c, int i, int im, bool fine) {
    const int h = (d * 7 + site * 13 + c * 5 + i * 3 + im) % 15 - 7;
    return (float)h * 0.125f + (fine ? (float)((site + c + d + im) % 5 - 2) * (1.f / 4096.f) : 0.f);
  };
  auto pairs = [&](int d, bool fine) {
    Pairs v;
#pragma unroll
    for (int q = 0; q < 2; ++q)
#pragma unroll
      for (int e = 0; e < 2; ++e)
#pragma unroll
        for (int i = 0; i < 3; ++i)
          v.v[q][e][i] = make_float2(val(d, g, 2 * t + 8 * q + e, i, 0, fine), val(d, g, 2 * t + 8 * q + e, i, 1, fine));
    return v;
  };
  float err = 0.f, most = 0.f;
  auto meet = [&](float got, float want) {
    err = fmaxf(err, fabsf(got - want));
    most = fmaxf(most, fabsf(want));
  };
  for (int tr = 0; tr < 2; ++tr) {
    float acc[3][2][4] = {};
    for (int d = 0; d < NET_NDIR; ++d) {
      const Pairs v = pairs(d, true);
      const uint4 b = sB[tr][d * 32 + lane];
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        uint32_t h[4], l[4];
        tc::split2(v.v[0][0][i].x, v.v[0][1][i].x, h[0], l[0]);
        tc::split2(v.v[0][0][i].y, v.v[0][1][i].y, h[1], l[1]);
        tc::split2(v.v[1][0][i].x, v.v[1][1][i].x, h[2], l[2]);
        tc::split2(v.v[1][0][i].y, v.v[1][1][i].y, h[3], l[3]);
        float s[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
        mma(s[0], l[0], l[1], l[2], l[3], b.x, b.y);
        mma(s[1], l[0], l[1], l[2], l[3], b.z, b.w);
        mma(s[0], h[0], h[1], h[2], h[3], b.x, b.y);
        mma(s[1], h[0], h[1], h[2], h[3], b.z, b.w);
        add(acc[i], s);
      }
    }
    for (int i = 0; i < 3; ++i)
      for (int q = 0; q < 2; ++q)
        for (int k = 0; k < 4; ++k) {
          const int c = 2 * t + 8 * q + (k & 1), im = k >> 1;
          float ref = 0.f;
          for (int d = 0; d < NET_NDIR; ++d) {
            const int dd = d == 0 ? 0 : ((d & 1) ? d + 1 : d - 1);
            for (int cp = 0; cp < 16; ++cp) {
              const float w = !tr ? __bfloat162float(W[(d * 16 + c) * 16 + cp])
                                  : (d ? -1.f : 1.f) * __bfloat162float(W[(dd * 16 + cp) * 16 + c]);
              ref += w * val(d, g, cp, i, im, true);
            }
          }
          meet(acc[i][q][k], ref);
        }
  }
  // sum over the eight sites, colours and (re, im) of a_c h_c'
  const Pairs a = pairs(2, true);
  uint32_t o[36];
  site_operand(pairs(5, false), o);
  float sum[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    uint32_t r0[3], i0[3], r1[3], i1[3], f[3][4];
    uint2 q[3][2];
    split3(a.v[0][0][i].x, a.v[0][1][i].x, r0);
    split3(a.v[0][0][i].y, a.v[0][1][i].y, i0);
    split3(a.v[1][0][i].x, a.v[1][1][i].x, r1);
    split3(a.v[1][0][i].y, a.v[1][1][i].y, i1);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      f[k][0] = trans(r0[k]);
      f[k][1] = trans(r1[k]);
      f[k][2] = trans(i0[k]);
      f[k][3] = trans(i1[k]);
#pragma unroll
      for (int nt = 0; nt < 2; ++nt) q[k][nt] = make_uint2(o[((k * 3 + i) * 2 + nt) * 2], o[((k * 3 + i) * 2 + nt) * 2 + 1]);
    }
    outer(sum, f, q);
  }
  for (int nt = 0; nt < 2; ++nt)
    for (int k = 0; k < 4; ++k) {
      const int c = (lane >> 2) + 8 * (k >> 1), cp = 8 * nt + 2 * (lane & 3) + (k & 1);
      float ref = 0.f;
      for (int site = 0; site < 8; ++site)
        for (int i = 0; i < 3; ++i)
          for (int im = 0; im < 2; ++im) ref += val(2, site, c, i, im, true) * val(5, site, cp, i, im, false);
      meet(sum[nt][k], ref);
    }
  for (int w = 16; w > 0; w >>= 1) {
    err = fmaxf(err, __shfl_xor_sync(0xffffffffu, err, w));
    most = fmaxf(most, __shfl_xor_sync(0xffffffffu, most, w));
  }
  if (lane == 0) {
    out[0] = err;
    out[1] = most;
  }
}

}  // namespace stag
