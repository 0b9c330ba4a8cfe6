// cg_loop.cu -- the CG iterations between two reliable updates as one
// cooperative kernel, for lattices so small that an iteration's launches cost
// more than its work.
//
// On 8^4 the four kernels of an iteration (direction update, two operator
// halves, vector update) take about 6 us each, nearly all of it launch,
// drain and reduction latency, and a chunk of queued iterations runs on after
// the one that asked for a reliable update.  Here every block keeps its own
// copy of the solver state and the whole loop runs on the GPU with three
// grid barriers per iteration (four for 16-bit vectors):
//   A  t = D p on odd sites, with p = rh + beta p_old formed from the two
//      fields for every neighbour as it is read, and stored for its own site
//      in a second direction field (a 16-bit direction is rounded when
//      stored, so there it is stored first, behind a barrier of its own);
//   B  Ap = shift p - D t on even sites, <p, Ap>;
//   C  xh += alpha p, rh -= alpha Ap, ||rh||^2.
// Several threads share a site, each with the hops of one direction (two for
// the 16-bit links, whose 16-byte chunks hold entries of two directions), so
// that a site's loads are in flight together.  The sums are double-float per
// block; after the barrier every block adds the blocks' partials in block
// order, so all blocks follow the same scalars, bit for bit.
// Fields that the loop writes are read through L2 (__ldcg): L1 is not
// coherent between SMs.
// What bounds it is latency: an iteration at 8^4 takes 9.7 us, of which
// the three barriers with their sums some 5 and the two gathers (one trip to
// L2 each) 2 to 3.
#include "dslash_impl.cuh"

namespace stag {
namespace {

constexpr int LB = 128;                    // threads per block
constexpr unsigned SPIN_LIMIT = 1u << 22;  // polls of a barrier, about a second

struct LoopSync {
  unsigned* arrived;  // zero at the start
  unsigned* gave_up;  // set when a wait ran out
  unsigned limit;     // polls of one wait
};

// The two halves of a grid barrier, called by all threads.  arrive: what the
// block has written is visible to every block that has seen it arrive.  wait:
// false when the wait ran out (every block then gives up by itself).
__device__ __forceinline__ void grid_arrive(const LoopSync& sy, unsigned& target) {
  target += gridDim.x;
  __syncthreads();
  if (threadIdx.x == 0) asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(sy.arrived) : "memory");
}
__device__ __forceinline__ bool grid_wait(const LoopSync& sy, unsigned target) {
  __shared__ int ok;
  if (threadIdx.x == 0) {
    unsigned n = 0, seen;
    do {
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(sy.arrived) : "memory");
    } while ((int)(seen - target) < 0 && ++n < sy.limit);
    ok = (int)(seen - target) >= 0;
    if (!ok) atomicExch(sy.gave_up, 1u);
  }
  __syncthreads();
  return ok != 0;
}

// Reads of fields that other blocks write.
template <int P> struct Fresh {
  static __device__ __forceinline__ void ld(const Spinor<P>& f, int s, float2 o[3]) {
    s = STAG_BOUND(s, f.Vh, BOUND_VECTOR);
    if constexpr (P == 32 || P == 31) {
      const float2* p = (const float2*)f.v;
#pragma unroll
      for (int c = 0; c < 3; ++c) o[c] = __ldcg(p + c * (size_t)f.Vh + s);
    } else {
      SpinorLoad16<P>::unpack(__ldcg((const uint4*)f.v + s), o);
    }
  }
};

// The hops of directions [mu0, mu0 + NMU) of output site s, whose links are
// in buf; `load` gives a neighbour's vector.  All vectors are loaded before
// the first is used.
template <int P, int NL, int NMU, int NCH, class Load>
__device__ __forceinline__ void hops_part(const DslashArgs<P>& a, int s, const Coord& c, int mu0, const uint4 (&buf)[NCH],
                                          Load load, float2 out[3]) {
  constexpr int CPM = 18 + 2 * NL;
  const Geom& g = a.g;
  float2 F[3], L[3], psi[4 * NMU][3];
#pragma unroll
  for (int h = 0; h < 4 * NMU; ++h)
    load(cb_neighbour(g, s, c, mu0 + h / 4, (h & 2 ? 3 : 1) * (h & 1 ? -1 : 1)), psi[h]);
#pragma unroll
  for (int i = 0; i < 3; ++i) F[i] = L[i] = make_float2(0.f, 0.f);
#pragma unroll
  for (int m = 0; m < NMU; ++m) {
    const int k0 = m * CPM;
    hop_full<P>(F, buf, k0, psi[4 * m]);
    hop_full<P>(F, buf, k0 + 9, psi[4 * m + 1]);
    if (NL == 9) {
      hop_full<P>(L, buf, k0 + 18, psi[4 * m + 2]);
      hop_full<P>(L, buf, k0 + 27, psi[4 * m + 3]);
    } else {
      const bool neg = eta_bit(c, mu0 + m);
      hop_recon12<P>(L, buf, k0 + 18, psi[4 * m + 2], neg);
      hop_recon12<P>(L, buf, k0 + 18 + NL, psi[4 * m + 3], !neg);
    }
  }
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    out[i].x = a.fat_scale * F[i].x + a.long_scale * L[i].x;
    out[i].y = a.fat_scale * F[i].y + a.long_scale * L[i].y;
  }
}

// Stores the block's partial sum and arrives at the barrier; after the wait,
// adds the blocks' partials and finalises on the block's own state.  In the
// first `width` lanes of each warp: their sum, then the warps' in order.
__device__ __forceinline__ void reduce_arrive(const Acc1<float>& acc, int width, float2* partials, const LoopSync& sy,
                                              unsigned& target) {
  __shared__ float2 sm[LB / 32];
  DF v = acc.v;
  for (int o = width >> 1; o > 0; o >>= 1) {
    DF w;
    w.hi = __shfl_xor_sync(0xffffffffu, v.hi, o);
    w.lo = __shfl_xor_sync(0xffffffffu, v.lo, o);
    df_add_df(v, w);
  }
  if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = make_float2(v.hi, v.lo);
  __syncthreads();
  if (threadIdx.x == 0) {
#pragma unroll
    for (int i = 1; i < LB / 32; ++i) df_add_df(v, DF{sm[i].x, sm[i].y});
    __stcg(partials + blockIdx.x, make_float2(v.hi, v.lo));
  }
  grid_arrive(sy, target);
}
__device__ __forceinline__ bool reduce_wait(int op, CgState* S, const float2* partials, const LoopSync& sy,
                                            unsigned target) {
  if (!grid_wait(sy, target)) return false;
  if (threadIdx.x < 32) {
    DF w[1] = {DF{0.f, 0.f}};
#pragma unroll 5
    for (int b = threadIdx.x; b < (int)gridDim.x; b += 32) {
      const float2 q = __ldcg(partials + b);
      df_add_df(w[0], DF{q.x, q.y});
    }
    warp_sum_df<1>(w);
    if (threadIdx.x == 0) {
      const double t = df_value(w[0]);
      finalize(RedTarget{op, S, nullptr}, &t, 1);
    }
  }
  __syncthreads();
  return true;
}

// ONE: every warp has at most one group of sites, so each site's own p, rh,
// xh and Ap stay in the registers of one thread through the whole loop, and
// only what other blocks read is stored.
template <int P, int NL, bool ONE>
__global__ void __launch_bounds__(LB)
    k_cg_loop(DslashArgs<P> odd, DslashArgs<P> even, Spinor<P> p, Spinor<P> p2, Spinor<P> t, Spinor<32> Ap, Spinor<32> xh,
              Spinor<32> rh, CgState* st, float2* partials, LoopSync sy, int pending, int most) {
  constexpr bool FUSE = P == 32 || P == 31;
  constexpr int NMU = Chunk<P>::PER / 2, SPLIT = 4 / NMU, SPW = 32 / SPLIT;  // directions per thread; sites per warp
  __shared__ CgState S;
  if (threadIdx.x == 0) S = *st;
  __syncthreads();
  const int Vh = p.Vh, warp = (blockIdx.x * LB + threadIdx.x) >> 5, nwarps = gridDim.x * (LB / 32);
  const int lane = threadIdx.x & 31, part = lane / SPW, ls = lane - part * SPW;
  // the links of the warp's first sites are loaded ahead of the barrier before their use
  constexpr int NCH = NMU * (18 + 2 * NL) / Chunk<P>::PER;
  const int mine = warp * SPW + ls, first = mine < Vh ? mine : Vh - 1;
  const bool own = part == 0 && mine < Vh;
  uint4 links[NCH];
  load_chunks<NCH>(links, odd.links, part * NCH, NCH, Vh, first);
  unsigned target = 0;
  Spinor<P> cur = p, nxt = p2;
  float2 ro[3], po[3], xo[3], ao[3];  // ONE: the own site's rh, p, xh, Ap
#pragma unroll
  for (int c = 0; c < 3; ++c) ro[c] = po[c] = xo[c] = ao[c] = make_float2(0.f, 0.f);
  if (ONE && own) {
    Fresh<32>::ld(rh, mine, ro);
    Fresh<P>::ld(p, mine, po);
    Fresh<32>::ld(xh, mine, xo);
  }
  bool alive = true;
  auto sum_parts = [&](float2(&d)[3]) {
#pragma unroll
    for (int o = SPW; o < 32; o <<= 1)
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        d[i].x += __shfl_xor_sync(0xffffffffu, d[i].x, o);
        d[i].y += __shfl_xor_sync(0xffffffffu, d[i].y, o);
      }
  };
  auto axpy = [](float2(&v)[3], const float2(&r)[3], float beta) {  // v = r + beta v
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      v[c].x = r[c].x + beta * v[c].x;
      v[c].y = r[c].y + beta * v[c].y;
    }
  };
#pragma unroll 1
  for (int it = 0; it < most && alive && !(S.flags & F_STOP); ++it) {
    const float beta = (float)S.beta;
    const bool upd = pending != 0;
    // ---- A
    auto direction = [&](int n, float2(&v)[3]) {
      Fresh<P>::ld(cur, n, v);
      if (FUSE && upd) {
        float2 r[3];
        Fresh<32>::ld(rh, n, r);
        axpy(v, r, beta);
      }
    };
    if (ONE) {
      if (upd && own) {
        axpy(po, ro, beta);
        SpinorLoad<P>::st(FUSE ? nxt : cur, mine, po);
        if (!FUSE) Fresh<P>::ld(cur, mine, po);  // as stored
      }
    } else if (!FUSE && upd) {
      for (int s = blockIdx.x * LB + threadIdx.x; s < Vh; s += gridDim.x * LB) {
        float2 v[3], r[3];
        Fresh<P>::ld(cur, s, v);
        Fresh<32>::ld(rh, s, r);
        axpy(v, r, beta);
        SpinorLoad<P>::st(cur, s, v);
      }
    }
    if (!FUSE && upd) {
      grid_arrive(sy, target);
      if (!(alive = grid_wait(sy, target))) break;
    }
    for (int s0 = warp * SPW; s0 < Vh; s0 += nwarps * SPW) {
      const bool in = s0 + ls < Vh;
      const int s = in ? s0 + ls : Vh - 1;
      float2 d[3], o[3];
      if (!ONE && s0 != warp * SPW) load_chunks<NCH>(links, odd.links, part * NCH, NCH, Vh, s);
      if (!ONE && FUSE && upd && part == SPLIT - 1) direction(s, o);
      hops_part<P, NL, NMU>(odd, s, cb_coords(odd.g, s, 1), part * NMU, links,
                            [&](int n, float2(&v)[3]) { direction(n, v); }, d);
      sum_parts(d);
      if (in && part == 0) SpinorLoad<P>::st(t, s, d);
      if (!ONE && FUSE && upd && in && part == SPLIT - 1) SpinorLoad<P>::st(nxt, s, o);
      if (ONE) break;
    }
    if (FUSE && upd) {
      const Spinor<P> q = cur;
      cur = nxt;
      nxt = q;
    }
    pending = 1;
    grid_arrive(sy, target);
    load_chunks<NCH>(links, even.links, part * NCH, NCH, Vh, first);
    if (!(alive = grid_wait(sy, target))) break;
    // ---- B
    Acc1<float> acc;
    const float cx = (float)S.shift;
    for (int s0 = warp * SPW; s0 < Vh; s0 += nwarps * SPW) {
      const bool in = s0 + ls < Vh;
      const int s = in ? s0 + ls : Vh - 1;
      float2 d[3], x[3];
      if (ONE) {
#pragma unroll
        for (int i = 0; i < 3; ++i) x[i] = po[i];
      } else {
        if (s0 != warp * SPW) load_chunks<NCH>(links, even.links, part * NCH, NCH, Vh, s);
        Fresh<P>::ld(cur, s, x);
      }
      hops_part<P, NL, NMU>(even, s, cb_coords(even.g, s, 0), part * NMU, links,
                            [&](int n, float2(&v)[3]) { Fresh<P>::ld(t, n, v); }, d);
      sum_parts(d);
      if (in && part == 0) {
#pragma unroll
        for (int i = 0; i < 3; ++i) {
          d[i].x = cx * x[i].x - d[i].x;
          d[i].y = cx * x[i].y - d[i].y;
          acc.add_prod(x[i].x, d[i].x);
          acc.add_prod(x[i].y, d[i].y);
        }
        if (!ONE) SpinorLoad<32>::st(Ap, s, d);
      }
      if (ONE) {
#pragma unroll
        for (int i = 0; i < 3; ++i) ao[i] = d[i];
        break;
      }
    }
    reduce_arrive(acc, SPW, partials, sy, target);
    load_chunks<NCH>(links, odd.links, part * NCH, NCH, Vh, first);
    if (!(alive = reduce_wait(RED_CG_ALPHA, &S, partials, sy, target))) break;
    if (S.flags & F_BREAKDOWN) break;
    // ---- C
    const float alpha = (float)S.alpha;
    Acc1<float> rr;
    auto residual = [&](float2(&r)[3], const float2(&ap)[3]) {
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        r[c].x -= alpha * ap[c].x;
        r[c].y -= alpha * ap[c].y;
        rr.add_prod(r[c].x, r[c].x);
        rr.add_prod(r[c].y, r[c].y);
      }
    };
    if (ONE) {
      if (own) {
        residual(ro, ao);
        SpinorLoad<32>::st(rh, mine, ro);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          xo[c].x += alpha * po[c].x;
          xo[c].y += alpha * po[c].y;
        }
      }
    } else {
      for (int s = blockIdx.x * LB + threadIdx.x; s < Vh; s += gridDim.x * LB) {
        float2 r[3], ap[3];
        Fresh<32>::ld(rh, s, r);
        Fresh<32>::ld(Ap, s, ap);
        residual(r, ap);
        SpinorLoad<32>::st(rh, s, r);
      }
    }
    reduce_arrive(rr, ONE ? SPW : 32, partials + gridDim.x, sy, target);
    if (!ONE) {
      // xh is this thread's alone: updated while the others arrive
      for (int s = blockIdx.x * LB + threadIdx.x; s < Vh; s += gridDim.x * LB) {
        float2 x[3], pv[3];
        Fresh<32>::ld(xh, s, x);
        Fresh<P>::ld(cur, s, pv);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          x[c].x += alpha * pv[c].x;
          x[c].y += alpha * pv[c].y;
        }
        SpinorLoad<32>::st(xh, s, x);
      }
    }
    if (!(alive = reduce_wait(RED_CG_BETA, &S, partials + gridDim.x, sy, target))) break;
  }
  if (!alive) return;
  // xh, and the current direction back to p (no block reads p any more: the last barrier came after phase A)
  if (ONE) {
    if (own) {
      SpinorLoad<32>::st(xh, mine, xo);
      if (FUSE) SpinorLoad<P>::st(p, mine, po);
    }
  } else if (cur.v != p.v) {
    for (int s = blockIdx.x * LB + threadIdx.x; s < Vh; s += gridDim.x * LB) {
      float2 v[3];
      Fresh<P>::ld(cur, s, v);
      SpinorLoad<P>::st(p, s, v);
    }
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) *st = S;
}

}  // namespace

// Iterations until a stop flag is raised or `most` have run.  `gave_up`
// (device, beside the barrier's counter) is set if a wait ran out: the fields
// are then not usable, and the state is as it was or the loop's (the caller
// solves again with queued launches).  STAG_EINVAL where the form does not apply or the grid
// cannot be resident at once (the caller queues the iterations instead).
template <int P>
int launch_cg_loop(stag_lattice_s* lat, Spinor<P> p, Spinor<P> p2, Spinor<P> t, Spinor<32> Ap, Spinor<32> xh,
                   Spinor<32> rh, CgState* state, int pending, int most, RedScratch rs, unsigned* sync, cudaStream_t st) {
  const LinkCopy& L = lat->links[prec_index<P>()];
  if (!L.present) return STAG_EINVAL;
  DslashArgs<P> odd = make_args<P>(lat, p, 1), even = make_args<P>(lat, t, 0);
  constexpr int SPLIT = 8 / Chunk<P>::PER;
  const int want = (p.Vh * SPLIT + LB - 1) / LB;
  auto kernel = [&](bool one) {
    return L.nl == 6 ? one ? (const void*)k_cg_loop<P, 6, true> : (const void*)k_cg_loop<P, 6, false>
                     : one ? (const void*)k_cg_loop<P, 9, true> : (const void*)k_cg_loop<P, 9, false>;
  };
  int dev = 0, sms = 0, coop = 0, occ = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) != cudaSuccess || !coop ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kernel(want <= sms), LB, 0) != cudaSuccess || occ < 1) {
    cudaGetLastError();
    return STAG_EINVAL;
  }
  // one block per SM at most: more make the barrier dearer than they save
  const int G = want < sms ? want : sms;
  const void* k = kernel(want <= sms);
  if (2 * G > rs.max_grid * 3) return STAG_EINVAL;  // (the caller's partials hold three per block of max_grid)
  float2* partials = (float2*)rs.partials;
  LoopSync sy{sync, sync + 1, lat->loop_polls ? lat->loop_polls : SPIN_LIMIT};
  int s = cuda_status(cudaMemsetAsync(sync, 0, 2 * sizeof(unsigned), st));
  if (!s && lat->loop_test == 1) s = cuda_status(cudaMemsetAsync(sync, 0xc0, sizeof(unsigned), st));
  if (s) return s;
  void* args[] = {&odd, &even, &p, &p2, &t, &Ap, &xh, &rh, &state, &partials, &sy, &pending, &most};
  ProfScope ps("cg_loop", st);
  if (cudaLaunchCooperativeKernel(k, dim3(G), dim3(LB), args, 0, st) != cudaSuccess) {
    cudaGetLastError();
    return STAG_EINVAL;
  }
  return STAG_OK;
}

#define STAG_CG_LOOP(P)                                                                                             \
  template int launch_cg_loop<P>(stag_lattice_s*, Spinor<P>, Spinor<P>, Spinor<P>, Spinor<32>, Spinor<32>, Spinor<32>, \
                                 CgState*, int, int, RedScratch, unsigned*, cudaStream_t);
STAG_CG_LOOP(32)
STAG_CG_LOOP(31)
STAG_CG_LOOP(16)
STAG_CG_LOOP(15)

}  // namespace stag
