// fx.cu -- thin links to fixed point (see fx.cuh), with the check that decides
// whether the integer kernels may be used on them.
#include "fx.cuh"

namespace stag {
namespace fx {

// Reads each link once (576 B per site) and writes it once: bound by HBM.
// (With the doubles converted on the FP64 pipe it took 132 us at 24^4, 90 %
// of that pipe.)  The unitarity check is in FP32 on the high parts (rounding
// below 2^-20, tolerance 2^-12).
__global__ void __launch_bounds__(128) k_fx_links(long long V, const double2* __restrict__ U, int4* __restrict__ out,
                                                  int slots, int slot0, Header* hd) {
  __shared__ double2 sm[TS * SITE_W];
  __shared__ int count[2];
  if (threadIdx.x < 2) count[threadIdx.x] = 0;
  const long long x0 = (long long)blockIdx.x * TS;
  const int ns = (int)(V - x0 < TS ? V - x0 : TS);
  for (int i = threadIdx.x; i < ns * 36; i += 128) sm[(i / 36) * SITE_W + i % 36] = __ldg(U + x0 * 36 + i);
  __syncthreads();
  const int mu = threadIdx.x >> 5, s = threadIdx.x & 31;
  int flags = 0;
  float diag = 1.f;  // the distance from the diagonal matrices of 1, -1, i, -i
  if (s < ns) {
    float2 f[9];
    int4* o = out + row0(slots, (int)(x0 + s), slot0 + mu);
#pragma unroll
    for (int e = 0; e < 9; ++e) {
      const double2 u = sm[s * SITE_W + mu * 9 + e];
      // exponents of 2 and above (infinity and NaN among them) are out of range
      const int ex = max(__double2hiint(u.x) & 0x7fffffff, __double2hiint(u.y) & 0x7fffffff);
      if (ex >= 0x40000000) flags |= FX_NOT_UNITARY;
      int4 q;
      fxd::fixed_entry(u.x, 0, q.x, q.y);
      fxd::fixed_entry(u.y, 0, q.z, q.w);
      o[e * 32] = q;
      f[e] = make_float2((float)q.x * 0x1p-30f, (float)q.z * 0x1p-30f);
    }
    // sum of |(U U^dag - 1)_ij|, and the distance of U from 1
    float dev = 0.f, away = 0.f;
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = i; j < 3; ++j) {
        float re = i == j ? -1.f : 0.f, im = 0.f;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          const float2 a = f[3 * i + k], b = f[3 * j + k];
          re += a.x * b.x + a.y * b.y;
          im += a.y * b.x - a.x * b.y;
        }
        dev += fabsf(re) + fabsf(im);
      }
#pragma unroll
    for (int e = 0; e < 9; ++e)
      diag = fmaxf(e == 0 ? 0.f : diag, e % 4 == 0 ? fminf(fabsf(f[e].x), fabsf(f[e].y)) : fmaxf(fabsf(f[e].x), fabsf(f[e].y)));
#pragma unroll
    for (int e = 0; e < 9; ++e)
      away = fmaxf(away, fmaxf(fabsf(f[e].x - (e % 4 == 0 ? 1.f : 0.f)), fabsf(f[e].y)));
    if (!(dev <= 0x1p-12f)) flags |= FX_NOT_UNITARY;
    if (away >= 0x1p-5f) flags |= FX_AWAY;
  }
  // one atomic per warp, and none once the bits are set
  flags = (int)__reduce_or_sync(0xffffffffu, (unsigned)flags);
  if (s == 0 && (__ldcg(&hd->status) & flags) != flags) atomicOr(&hd->status, flags);
  // one atomic per block that holds such a link
  const int n6 = __popc(__ballot_sync(0xffffffffu, diag < 3 * 0x1p-6f)), n5 = __popc(__ballot_sync(0xffffffffu, diag < 3 * 0x1p-5f));
  if (__syncthreads_or(n5)) {
    if (s == 0) {
      atomicAdd(&count[NEAR_6], n6);
      atomicAdd(&count[NEAR_5], n5);
    }
    __syncthreads();
    if (threadIdx.x < 2 && count[threadIdx.x]) atomicAdd(&hd->near[threadIdx.x], (unsigned long long)count[threadIdx.x]);
  }
}

int launch_fx_links(long long V, const double2* U, int4* out, int slots, int slot0, Header* hd, cudaStream_t st) {
  if (cudaMemsetAsync(hd, 0, sizeof(Header), st) != cudaSuccess) {
    cudaGetLastError();
    return STAG_ECUDA;
  }
  k_fx_links<<<(unsigned)((V + TS - 1) / TS), 128, 0, st>>>(V, U, out, slots, slot0, hd);
  return last_launch_status();
}

}  // namespace fx
}  // namespace stag
