// net_kernels.cuh -- forward and backward kernels of the gauge-covariant
// preconditioner network (definition in include/stag.h, stag_net_create).
//
// Activations are full-lattice fields stored per parity: [2][Vh][C][3]
// complex FP32, a site's channels contiguous (16 channels: in the word order
// of net_mma.cuh).  A layer reads, for each
// of its 9 directions d, the fat-link hop of the staggered operator (the
// library's FP32 link copy: entries mu*CPM + 0..17 of the output parity's
// chunk list hold the +mu and -mu hop matrices with eta and 1/2 folded in)
// and the neighbour's channels, transports them, and mixes channels with the
// layer's real weights (stored as bfloat16, held in shared memory as FP32,
// FP32 accumulation).
#pragma once
#include <cuda_bf16.h>

#include "dslash_impl.cuh"

namespace stag {

constexpr int NET_NDIR = 9;
template <int V> struct IntC {
  static constexpr int value = V;
};

struct NetGeom {
  Geom g;
  const uint4* links[2];  // FP32 link chunks for output parity 0 and 1
  int cpm;                // complex entries per direction in the chunk list
};

__device__ __forceinline__ float2* act_ptr(float2* a, int C, int Vh, int p, int s) {
  return a + (((size_t)p * Vh + s) * C) * 3;
}
__device__ __forceinline__ const float2* act_ptr(const float2* a, int C, int Vh, int p, int s) {
  return a + (((size_t)p * Vh + s) * C) * 3;
}

// The 3x3 hop matrix of direction d (1..8) at site s of parity p.
__device__ __forceinline__ void load_hop_matrix(const NetGeom& ng, int p, int s, int d, float2 w[9]) {
  const int mu = (d - 1) >> 1;
  const int k0 = mu * ng.cpm + ((d & 1) ? 0 : 9);  // FP32: 2 complex per chunk
  const uint4* L = p ? ng.links[1] : ng.links[0];
  const int Vh = ng.g.Vh;
  // chunks c0 .. c0 + 4 hold entries 2 c0 .. 2 c0 + 9; the matrix starts at
  // the first entry (k0 even) or the second (k0 odd).  Indices into w stay
  // compile-time constants so that w lives in registers.
  const bool odd = k0 & 1;
  const uint4* src = L + (size_t)(k0 >> 1) * Vh + s;
#pragma unroll
  for (int j = 0; j < 5; ++j) {
    const uint4 c = __ldg(src + (size_t)j * Vh);
    const float2 a = make_float2(__uint_as_float(c.x), __uint_as_float(c.y));
    const float2 b = make_float2(__uint_as_float(c.z), __uint_as_float(c.w));
    if (j > 0) w[2 * j - 1] = odd ? a : w[2 * j - 1];
    if (j < 4) w[2 * j + 1] = odd ? w[2 * j + 1] : b;
    w[2 * j] = odd ? b : a;
  }
}

// Neighbour (parity, index) of (p, s) for direction d (0: itself).
__device__ __forceinline__ void net_neighbour(const NetGeom& ng, int p, int s, int d, int& np, int& ns) {
  if (d == 0) {
    np = p;
    ns = s;
    return;
  }
  const int mu = (d - 1) >> 1;
  Coord c = cb_coords(ng.g, s, p);
  ns = cb_neighbour(ng.g, s, c, mu, (d & 1) ? 1 : -1);
  np = 1 - p;
}

// The single layer of a network without hidden channels: out(x) = sum_d W[d] (T_d h)(x).
__global__ void __launch_bounds__(256) k_net_layer_1to1(NetGeom ng, const float2* __restrict__ hin, float2* __restrict__ hout,
                                                       const __nv_bfloat16* __restrict__ W) {
  const int Vh = ng.g.Vh;
  for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < 2 * Vh; idx += gridDim.x * blockDim.x) {
    const int p = idx / Vh, s = idx - p * Vh;
    float2 acc[3] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
#pragma unroll 1
    for (int d = 0; d < NET_NDIR; ++d) {
      int np, ns;
      net_neighbour(ng, p, s, d, np, ns);
      const float k = __bfloat162float(W[d]);
      const float2* src = hin + ((size_t)np * Vh + ns) * 3;
      float2 v[3], t[3], w[9];
      if (d) load_hop_matrix(ng, p, s, d, w);
#pragma unroll
      for (int i = 0; i < 3; ++i) v[i] = __ldg(src + i);
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        if (d) {
          t[i] = make_float2(0.f, 0.f);
#pragma unroll
          for (int j = 0; j < 3; ++j) cmac(t[i], w[3 * i + j], v[j]);
        } else {
          t[i] = v[i];
        }
        acc[i].x = fmaf(k, t[i].x, acc[i].x);
        acc[i].y = fmaf(k, t[i].y, acc[i].y);
      }
    }
#pragma unroll
    for (int i = 0; i < 3; ++i) hout[(size_t)idx * 3 + i] = acc[i];
  }
}

// Its weight gradient dW[d] = sum_x Re <g(x), (T_d h)(x)>: per-block sums, threads in order.
__global__ void __launch_bounds__(256) k_net_dw_1to1(NetGeom ng, const float2* __restrict__ hin, const float2* __restrict__ g,
                                                    float* __restrict__ part) {
  __shared__ float sm[256];
  const int Vh = ng.g.Vh;
  for (int d = 0; d < NET_NDIR; ++d) {
    float acc = 0.f;
    for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < 2 * Vh; idx += gridDim.x * blockDim.x) {
      const int p = idx / Vh, s = idx - p * Vh;
      int np, ns;
      net_neighbour(ng, p, s, d, np, ns);
      const float2* src = hin + ((size_t)np * Vh + ns) * 3;
      float2 v[3], w[9];
      if (d) load_hop_matrix(ng, p, s, d, w);
#pragma unroll
      for (int i = 0; i < 3; ++i) v[i] = __ldg(src + i);
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        float2 t = v[i];
        if (d) {
          t = make_float2(0.f, 0.f);
#pragma unroll
          for (int j = 0; j < 3; ++j) cmac(t, w[3 * i + j], v[j]);
        }
        const float2 q = __ldg(g + (size_t)idx * 3 + i);
        acc = fmaf(q.x, t.x, acc);
        acc = fmaf(q.y, t.y, acc);
      }
    }
    sm[threadIdx.x] = acc;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
      if ((int)threadIdx.x < o) sm[threadIdx.x] += sm[threadIdx.x + o];
      __syncthreads();
    }
    if (threadIdx.x == 0) part[(size_t)blockIdx.x * NET_NDIR + d] = sm[0];
    __syncthreads();
  }
}

// Gate backward: G_pre = s G_out + 2 s(1-s) Re<G_out, pre> pre  (in place on g)
// and per-block partial sums of db_c = -sum s(1-s) Re<G_out, pre>.  One
// thread per (site, channel pair), three 16-byte words of each field (their
// place in the record: net_mma.cuh); a thread's pair stays fixed over the
// grid-stride loop.
__global__ void __launch_bounds__(256) k_net_gate_bwd16(int n2vh, const float2* __restrict__ pre, float2* g,
                                                       const float* __restrict__ bias, float* __restrict__ db_part) {
  __shared__ float sdb[8][16];
  const int stride = gridDim.x * blockDim.x, q0 = blockIdx.x * blockDim.x + threadIdx.x, pair = q0 & 7;
  const float2 bc = make_float2(bias[2 * pair], bias[2 * pair + 1]);
  float db[2] = {0.f, 0.f};
  for (int q = q0; q < n2vh * 8; q += stride) {
    const size_t at = (size_t)(q >> 3) * 24 + 12 * (pair >> 2) + (pair & 3);
    const float4* pv = (const float4*)pre + at;
    float4* gv = (float4*)g + at;
    float2 v[2][3], o[2][3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const float4 a = __ldg(pv + 4 * k), b = gv[4 * k];
      v[(2 * k) / 3][(2 * k) % 3] = make_float2(a.x, a.y);
      v[(2 * k + 1) / 3][(2 * k + 1) % 3] = make_float2(a.z, a.w);
      o[(2 * k) / 3][(2 * k) % 3] = make_float2(b.x, b.y);
      o[(2 * k + 1) / 3][(2 * k + 1) % 3] = make_float2(b.z, b.w);
    }
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      float n2 = 0.f, pr = 0.f;
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        n2 += v[e][i].x * v[e][i].x + v[e][i].y * v[e][i].y;
        pr += o[e][i].x * v[e][i].x + o[e][i].y * v[e][i].y;
      }
      const float sg = 1.f / (1.f + __expf(-(n2 - (e ? bc.y : bc.x))));
      const float sp = sg * (1.f - sg);
      db[e] -= sp * pr;
#pragma unroll
      for (int i = 0; i < 3; ++i)
        o[e][i] = make_float2(sg * o[e][i].x + 2.f * sp * pr * v[e][i].x, sg * o[e][i].y + 2.f * sp * pr * v[e][i].y);
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const float2 a = o[(2 * k) / 3][(2 * k) % 3], b = o[(2 * k + 1) / 3][(2 * k + 1) % 3];
      gv[4 * k] = make_float4(a.x, a.y, b.x, b.y);
    }
  }
  // lanes l, l + 8, ... hold the same pair; then warps in order
#pragma unroll
  for (int e = 0; e < 2; ++e)
#pragma unroll
    for (int o = 8; o < 32; o <<= 1) db[e] += __shfl_xor_sync(0xffffffffu, db[e], o);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (lane < 8) {
    sdb[warp][2 * lane] = db[0];
    sdb[warp][2 * lane + 1] = db[1];
  }
  __syncthreads();
  if (threadIdx.x < 16) {
    float v = 0.f;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) v += sdb[w][threadIdx.x];
    db_part[(size_t)blockIdx.x * 16 + threadIdx.x] = v;
  }
}

// Output layer with one channel, for even output sites x (the prediction is
// read nowhere else).  Mix first: u_d(y) = sum_c' W[d][0][c'] h_c'(y),
// site-local, for the directions that lead from y to an even site (y even:
// d = 0, y odd: 1..8); then (k_net_transport_sum) out(x) = u_0(x) + sum_d
// (T_d u_d)(x).  U: [9][Vh][3].
// A warp takes 32 sites of one parity, whose records (one contiguous piece)
// pass through shared memory with whole-warp accesses; there a record takes
// 25 words (odd: no bank conflicts between sites).
__global__ void __launch_bounds__(128) k_net_mix_local16(int Vh, const float2* __restrict__ hin,
                                                        const __nv_bfloat16* __restrict__ W, float2* __restrict__ U) {
  __shared__ float sw[NET_NDIR * 16];
  __shared__ float4 rec[4][16 * 25];
  for (int i = threadIdx.x; i < NET_NDIR * 16; i += blockDim.x) sw[i] = __bfloat162float(W[i]);
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, per = (Vh + 31) / 32;
  float4* r = rec[warp];
  auto mix = [&](int p, int s0, auto first, auto count) {
    constexpr int D0 = decltype(first)::value, ND = decltype(count)::value;
    const int n = Vh - s0 < 32 ? Vh - s0 : 32;
    const float4* src = (const float4*)hin + ((size_t)p * Vh + s0) * 24;
    float2 u[ND][3];
#pragma unroll
    for (int d = 0; d < ND; ++d)
#pragma unroll
      for (int i = 0; i < 3; ++i) u[d][i] = make_float2(0.f, 0.f);
    // channels 0..7, then 8..15 (the halves of every record), 12 words per site each
#pragma unroll 1
    for (int q = 0; q < 2; ++q) {
      __syncwarp();
#pragma unroll
      for (int k = 0; k < 12; ++k) {
        const int w = k * 32 + lane, site = w / 12;
        if (site < n) r[(site & 15) * 25 + (site >> 4) * 12 + w % 12] = __ldg(src + (size_t)site * 24 + 12 * q + w % 12);
      }
      __syncwarp();
      const float4* me = r + (lane & 15) * 25 + (lane >> 4) * 12;
#pragma unroll
      for (int t = 0; t < 4; ++t)
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          const float4 f = me[4 * k + t];
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const int e = 2 * k + h, c = 2 * t + e / 3, i = e % 3;  // channel 8 q + c, colour i
            const float vx = h ? f.z : f.x, vy = h ? f.w : f.y;
#pragma unroll
            for (int d = 0; d < ND; ++d) {
              const float w = sw[(D0 + d) * 16 + 8 * q + c];
              u[d][i].x = fmaf(w, vx, u[d][i].x);
              u[d][i].y = fmaf(w, vy, u[d][i].y);
            }
          }
        }
    }
    if (lane < n) {
#pragma unroll
      for (int d = 0; d < ND; ++d)
#pragma unroll
        for (int i = 0; i < 3; ++i) U[((size_t)(D0 + d) * Vh + s0 + lane) * 3 + i] = u[d][i];
    }
  };
  for (int g = blockIdx.x * 4 + warp; g < 2 * per; g += gridDim.x * 4) {
    if (g < per)
      mix(0, g * 32, IntC<0>{}, IntC<1>{});
    else
      mix(1, (g - per) * 32, IntC<1>{}, IntC<NET_NDIR - 1>{});
  }
}

// out(x) = u_0(x) + sum_{d >= 1} hop_d(x) u_d(neighbour_d(x)), x even.
__global__ void __launch_bounds__(256) k_net_transport_sum(NetGeom ng, const float2* __restrict__ U,
                                                          float2* __restrict__ hout) {
  const int Vh = ng.g.Vh;
  for (int s = blockIdx.x * blockDim.x + threadIdx.x; s < Vh; s += gridDim.x * blockDim.x) {
    float2 acc[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) acc[i] = __ldg(U + (size_t)s * 3 + i);
#pragma unroll 2
    for (int d = 1; d < NET_NDIR; ++d) {
      int np, ns;
      net_neighbour(ng, 0, s, d, np, ns);
      float2 w[9], v[3];
      load_hop_matrix(ng, 0, s, d, w);
      const float2* src = U + ((size_t)d * Vh + ns) * 3;
#pragma unroll
      for (int j = 0; j < 3; ++j) v[j] = __ldg(src + j);
#pragma unroll
      for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) cmac(acc[i], w[3 * i + j], v[j]);
    }
#pragma unroll
    for (int i = 0; i < 3; ++i) hout[(size_t)s * 3 + i] = acc[i];
  }
}

// grad[i] += sum over blocks of part[block][i], in a fixed order: a block takes
// 32 entries, 32 threads each every 32nd partial, then the 32 in order.  (With
// eight threads the chain of loads took 10 to 12 us.)
__global__ void __launch_bounds__(1024) k_net_sum_parts(const float* __restrict__ part, int nblocks, int n, float* grad) {
  __shared__ float sm[32][33];
  const int x = threadIdx.x & 31, y = threadIdx.x >> 5, i = blockIdx.x * 32 + x;
  float s = 0.f;
  if (i < n) {
#pragma unroll 8
    for (int b = y; b < nblocks; b += 32) s += part[(size_t)b * n + i];
  }
  sm[y][x] = s;
  __syncthreads();
  if (y == 0 && i < n) {
#pragma unroll
    for (int k = 1; k < 32; ++k) s += sm[k][x];
    grad[i] += s;
  }
}

}  // namespace stag
