// net_tc.cuh -- tcgen05 helpers and the check of the fifth-generation tensor
// cores on this GPU (stag_tc_selftest): 384 x 16 rows of bfloat16 operands,
// nine accumulated K = 16 steps into tensor memory, against the CUDA cores.
// The network's layers once ran in this form; they now take mma.sync straight
// from registers (net_mma.cuh says why).
//
// Shared-memory operand layout (no swizzle, K-major): 8-row x 16-byte core
// matrices stored as 128 contiguous bytes; the two 16-byte K halves of a row
// group are 128 bytes apart (leading byte offset) and consecutive row groups
// 256 bytes apart (stride byte offset).
#pragma once
#include <cuda_bf16.h>
#include <stdint.h>

#include "net_kernels.cuh"

namespace stag {
namespace tc {

constexpr int ROWS = 384;                   // MMA rows
constexpr int A_BYTES = ROWS * 16 * 2;      // one operand part of one direction: 12288 B
constexpr int B_BYTES = 16 * 16 * 2;        // weights of one direction: 512 B
constexpr int TMEM_COLS = 64;               // 3 x 16 accumulator columns, allocated as 64
constexpr int SMEM_BYTES = 4 * A_BYTES + NET_NDIR * B_BYTES + 64;

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// UMMA shared-memory descriptor: start address, leading / stride byte
// offsets (all >> 4), descriptor version 1 (bits 46-47), no swizzle.
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
  uint64_t d = (uint64_t)((addr & 0x3FFFFu) >> 4);
  d |= (uint64_t)((lbo >> 4) & 0x3FFFu) << 16;
  d |= (uint64_t)((sbo >> 4) & 0x3FFFu) << 32;
  d |= (uint64_t)1 << 46;
  return d;
}

// Instruction descriptor of kind::f16: D FP32, A and B bfloat16, both K-major.
__host__ __device__ constexpr uint32_t idesc_bf16(int M, int N) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}

// Bounded wait for the completion of the phase with the given parity:
// gives up after about `cycles` SM clocks and returns false.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, long long cycles) {
  const long long t0 = clock64();
  while (!mbar_try_wait(bar, parity))
    if (clock64() - t0 > cycles) return false;
  return true;
}

__device__ __forceinline__ void fence_barrier_init() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// Whole warp: allocate `ncols` tensor-memory columns; the address lands in *dst.
__device__ __forceinline__ void tmem_alloc(uint32_t* dst, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(dst)), "r"(ncols)
               : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}

// Whole warp: release the columns.
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}

// One thread: D[tmem] (+)= A[adesc] x B[bdesc]^T.
__device__ __forceinline__ void mma_bf16(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                         uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}

// One thread: arrive on *bar once every tcgen05 operation it issued so far has completed.
__device__ __forceinline__ void mma_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
               : "memory");
}

// Whole warp: 16 consecutive FP32 columns of the warp's 32 lanes (lane field of taddr = 32 * (warp % 4)).
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float (&v)[16]) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

// Byte offset of element (row, k) in a K-major no-swizzle operand with
// 16-element (32-byte) rows: core matrix (row / 8, k / 8).
__host__ __device__ __forceinline__ int op_offset(int row, int k) {
  return (row >> 3) * 256 + (k >> 3) * 128 + (row & 7) * 16 + (k & 7) * 2;
}

// hi = bf16(x), lo = bf16(x - hi), two values packed per 32-bit word (a in
// the low half): one packing conversion for each part, the hi values
// widened back by a shift.
__device__ __forceinline__ void split2(float a, float b, uint32_t& hi, uint32_t& lo) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
  const __nv_bfloat162 l = __floats2bfloat162_rn(a - __low2float(h), b - __high2float(h));
  hi = *reinterpret_cast<const uint32_t*>(&h);
  lo = *reinterpret_cast<const uint32_t*>(&l);
}

constexpr long long WAIT_CYCLES = 4000000000LL;  // about two seconds at GB300 clocks

}  // namespace tc

// Check of the tensor-core path on this GPU: one tile (384 x 16 rows of
// bfloat16 hi/lo operands from a fixed integer pattern, 9 accumulated
// K = 16 steps) against the same products summed by the CUDA cores in FP32.
// out[0] = max |D_tc - D_ref| / max |D_ref|, out[1] = 1 if every wait ended.
__global__ void __launch_bounds__(128, 1) k_tc_selftest(float* out) {
  using namespace tc;
  extern __shared__ __align__(1024) unsigned char tc_smem[];
  unsigned char* A = tc_smem;
  unsigned char* Bw = tc_smem + 4 * A_BYTES;
  uint64_t* bar = (uint64_t*)(Bw + NET_NDIR * B_BYTES);
  uint32_t* tmem_slot = (uint32_t*)(bar + 2);
  int* s_ok = (int*)(tmem_slot + 1);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  auto aval = [](int d, int row, int k, int part) {  // exactly representable values
    const int h = (d * 7 + row * 13 + k * 5) % 17 - 8;
    return part == 0 ? (float)h * 0.125f : (float)((row + k + d) % 5 - 2) * (1.f / 4096.f);
  };
  auto bval = [](int d, int n, int k) { return (float)((d * 3 + n * 11 + k * 7) % 13 - 6) * 0.0625f; };
  for (int i = tid; i < NET_NDIR * 256; i += blockDim.x) {
    const int d = i >> 8, n = (i >> 4) & 15, k = i & 15;
    *(__nv_bfloat16*)(Bw + d * B_BYTES + op_offset(n, k)) = __float2bfloat16_rn(bval(d, n, k));
  }
  if (tid == 0) {
    mbar_init(&bar[0], 1);
    mbar_init(&bar[1], 1);
    *s_ok = 1;
    fence_barrier_init();
  }
  if (warp == 0) tmem_alloc(tmem_slot, TMEM_COLS);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  constexpr uint32_t IDESC = idesc_bf16(128, 16);
  const uint32_t a_base = smem_u32(A);
#pragma unroll 1
  for (int d = 0; d < NET_NDIR; ++d) {
    const int buf = d & 1;
    if (d >= 2) {
      if (tid == 0 && *s_ok && !mbar_wait(&bar[buf], (uint32_t)(((d - 2) >> 1) & 1), WAIT_CYCLES)) *s_ok = 0;
      __syncthreads();
    }
    for (int i = tid; i < ROWS * 16; i += blockDim.x) {
      const int row = i >> 4, k = i & 15;
      for (int part = 0; part < 2; ++part)
        *(__nv_bfloat16*)(A + (buf * 2 + part) * A_BYTES + op_offset(row, k)) =
            __float2bfloat16_rn(aval(d, row, k, part));
    }
    fence_async_smem();
    __syncthreads();
    if (tid == 0 && *s_ok) {
      tc_fence_after();
      const uint64_t bdesc = smem_desc(smem_u32(Bw + d * B_BYTES), 128, 256);
      for (int b = 0; b < 3; ++b) {
        mma_bf16(tmem + 16 * b, smem_desc(a_base + (buf * 2) * A_BYTES + b * 4096, 128, 256), bdesc, IDESC,
                 d > 0 ? 1u : 0u);
        mma_bf16(tmem + 16 * b, smem_desc(a_base + (buf * 2 + 1) * A_BYTES + b * 4096, 128, 256), bdesc, IDESC, 1u);
      }
      mma_commit(&bar[buf]);
    }
  }
  if (tid == 0 && *s_ok && !mbar_wait(&bar[0], 0u, WAIT_CYCLES)) *s_ok = 0;
  __syncthreads();
  tc_fence_after();
  float err = 0.f, ref_max = 0.f;
  if (*s_ok) {
    for (int b = 0; b < 3; ++b) {
      float v[16];
      tmem_ld16(tmem + ((uint32_t)(32 * warp) << 16) + 16 * b, v);
      const int row = 128 * b + 32 * warp + lane;
      for (int n = 0; n < 16; ++n) {
        float ref = 0.f;
        for (int d = 0; d < NET_NDIR; ++d)
          for (int k = 0; k < 16; ++k) ref += (aval(d, row, k, 0) + aval(d, row, k, 1)) * bval(d, n, k);
        err = fmaxf(err, fabsf(v[n] - ref));
        ref_max = fmaxf(ref_max, fabsf(ref));
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    tmem_dealloc(tmem, TMEM_COLS);
  }
  for (int o = 16; o > 0; o >>= 1) {
    err = fmaxf(err, __shfl_xor_sync(0xffffffffu, err, o));
    ref_max = fmaxf(ref_max, __shfl_xor_sync(0xffffffffu, ref_max, o));
  }
  __shared__ float red[2][4];
  if (lane == 0) {
    red[0][warp] = err;
    red[1][warp] = ref_max;
  }
  __syncthreads();
  if (tid == 0) {
    float e = 0.f, m = 0.f;
    for (int w = 0; w < 4; ++w) {
      e = fmaxf(e, red[0][w]);
      m = fmaxf(m, red[1][w]);
    }
    out[0] = m > 0.f ? e / m : e;
    out[1] = *s_ok ? 1.f : 0.f;
  }
}

}  // namespace stag
