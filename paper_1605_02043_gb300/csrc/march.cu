// march.cu -- resident kernels for runs of several explicit steps (sm_103a).
//
// The step kernels (flux_tma.cu) stream the whole mesh through every SM on
// every step: state, slots and weights come from the L2 or from HBM, and the
// launch, the first fills and the last blocks cost about 5 us a step.  When a
// run makes several steps and every part of the mesh (march.h) fits an SM, the
// state stays in shared memory from the first step to the last, with the slots
// and weights beside it where they fit too (otherwise they are read from the
// L2, coalesced, once a step), and only boundary values travel: each part
// stores the new values of its boundary vertices to an exchange buffer and
// gathers its halo from there.
//
// One CUDA block per part, one per SM, launched cooperatively (all parts are
// resident, so a wait for a neighbour's value ends).  A value says by itself
// which step it belongs to: it travels in 16-byte chunks of three components
// and a step tag, stored and loaded whole (128-bit accesses, single-copy
// atomic), and the reader loads a chunk again until its tag is the step's.
// No fence, counter or grid barrier stands between a store and its use: with
// a counter per part (stores, fence, counter up, neighbours poll, gather) a
// step of the 65,521-point mesh took 6.2 us, 4.8 of them in the fence and the
// poll.  Two buffers take turns; a part overwrites a value two steps later,
// after it has received the next value of every part that reads it, so the
// old one has been used (neighbourhood is symmetric).
//
// Boundary slices come first, so their values travel while the interior is
// computed.  A position's new value must not replace the old one before every
// slice that reads it is done: it is held in tensor memory (256 KB per SM,
// read and written lane by lane, otherwise idle here), which leaves the
// registers to the slots in flight and the shared memory to one copy of the
// state.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "flux_common.cuh"
#include "kernels.h"
#include "tma_sync.cuh"

namespace ep {
namespace dev {
namespace {

constexpr int kErrTimeoutNeighbour = 4;

// Exchange chunk: three components and the step's tag, one 128-bit access.
__device__ __forceinline__ void chunk_store(float* p, const float* v, uint32_t tag) {
  asm volatile(
      "{\n\t.reg .b64 lo, hi;\n\t.reg .b128 q;\n\t"
      "mov.b64 lo, {%1, %2};\n\tmov.b64 hi, {%3, %4};\n\tmov.b128 q, {lo, hi};\n\t"
      "st.relaxed.gpu.global.b128 [%0], q;\n\t}" ::"l"(p),
      "r"(__float_as_uint(v[0])), "r"(__float_as_uint(v[1])), "r"(__float_as_uint(v[2])), "r"(tag)
      : "memory");
}
__device__ __forceinline__ uint32_t chunk_load(const float* p, float* v) {
  uint32_t a, b, c, tag;
  asm volatile(
      "{\n\t.reg .b64 lo, hi;\n\t.reg .b128 q;\n\t"
      "ld.relaxed.gpu.global.b128 q, [%4];\n\tmov.b128 {lo, hi}, q;\n\t"
      "mov.b64 {%0, %1}, lo;\n\tmov.b64 {%2, %3}, hi;\n\t}"
      : "=r"(a), "=r"(b), "=r"(c), "=r"(tag)
      : "l"(p)
      : "memory");
  v[0] = __uint_as_float(a), v[1] = __uint_as_float(b), v[2] = __uint_as_float(c);
  return tag;
}

// ---------------------------------------------------------- tensor memory

__device__ __forceinline__ void tmem_alloc(uint32_t* where, uint32_t cols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(saddr(where)), "r"(cols)
               : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_free(uint32_t base, uint32_t cols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(base), "r"(cols) : "memory");
}
// columns of one held record: every access is aligned to its width
__host__ __device__ constexpr int hold_stride(int D) { return D <= 2 ? D : D <= 4 ? 4 : 8; }
// D values of every lane of the warp <-> D columns at `at`
template <int D, int K = 0>
__device__ __forceinline__ void tmem_put(uint32_t at, const float* v) {
  if constexpr (K < Planes<D>::NP) {
    constexpr int W = Planes<D>::width(K), F = Planes<D>::first(K);
    if constexpr (W == 4)
      asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1, %2, %3, %4};" ::"r"(at + F), "f"(v[F]),
                   "f"(v[F + 1]), "f"(v[F + 2]), "f"(v[F + 3])
                   : "memory");
    else if constexpr (W == 2)
      asm volatile("tcgen05.st.sync.aligned.32x32b.x2.b32 [%0], {%1, %2};" ::"r"(at + F), "f"(v[F]), "f"(v[F + 1])
                   : "memory");
    else
      asm volatile("tcgen05.st.sync.aligned.32x32b.x1.b32 [%0], {%1};" ::"r"(at + F), "f"(v[F]) : "memory");
    tmem_put<D, K + 1>(at, v);
  }
}
__device__ __forceinline__ void tmem_put_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
template <int D, int K = 0>
__device__ __forceinline__ void tmem_get_issue(uint32_t at, float* v) {
  if constexpr (K < Planes<D>::NP) {
    constexpr int W = Planes<D>::width(K), F = Planes<D>::first(K);
    if constexpr (W == 4)
      asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
                   : "=f"(v[F]), "=f"(v[F + 1]), "=f"(v[F + 2]), "=f"(v[F + 3])
                   : "r"(at + F)
                   : "memory");
    else if constexpr (W == 2)
      asm volatile("tcgen05.ld.sync.aligned.32x32b.x2.b32 {%0, %1}, [%2];"
                   : "=f"(v[F]), "=f"(v[F + 1])
                   : "r"(at + F)
                   : "memory");
    else
      asm volatile("tcgen05.ld.sync.aligned.32x32b.x1.b32 {%0}, [%1];" : "=f"(v[F]) : "r"(at + F) : "memory");
    tmem_get_issue<D, K + 1>(at, v);
  }
}
template <int D>
__device__ __forceinline__ void tmem_get(uint32_t at, float* v) {
  tmem_get_issue<D>(at, v);
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int c = 0; c < D; ++c) asm volatile("" : "+f"(v[c]));  // not used before the wait
}

// ----------------------------------------------------------------- pieces

// one bulk copy per plane of the records [lo, lo + n) (lo a multiple of 4)
template <int D, int K = 0>
__device__ __forceinline__ uint32_t load_planes(const float* g, int64_t n_rec, int lo, int n, float* s, int npos,
                                                uint64_t* bar, bool issue) {
  if constexpr (K < Planes<D>::NP) {
    constexpr int W = Planes<D>::width(K), F = Planes<D>::first(K);
    const uint32_t bytes = ((uint32_t)n * W * 4u + 15u) & ~15u;
    if (issue && bytes) bulk_load(s + F * npos, g + F * n_rec + (int64_t)lo * W, bytes, bar);
    return bytes + load_planes<D, K + 1>(g, n_rec, lo, n, s, npos, bar, issue);
  }
  return 0;
}

// Halo values of the state before the first step, four records in flight
template <int D>
__device__ __forceinline__ void first_halo(const MarchArgs& a, const MarchPart& d, float* xs) {
  for (int j0 = threadIdx.x; j0 < d.nh; j0 += 4 * blockDim.x) {
    int32_t r[4];
    float v[4][D];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int j = j0 + u * blockDim.x;
      r[u] = j < d.nh ? __ldg(a.halo + d.h0 + j) : -1;
    }
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (r[u] >= 0) rec_load<D>(a.x_in, a.n_rec, r[u], v[u]);
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (r[u] >= 0) rec_store<D>(xs, a.npos, d.hbase + j0 + u * blockDim.x, v[u]);
  }
}

// kHaloBatch halo records per thread: receive() loads each until all of its
// chunks carry the tag (false when the wait runs out), store() puts them into
// their positions.
constexpr int kHaloBatch = 3;
template <int D>
struct HaloBatch {
  static constexpr int NC = ex_chunks(D);
  float v[kHaloBatch][3 * NC];
  __device__ __forceinline__ bool receive(const MarchArgs& a, const MarchPart& d, const float* ex, uint32_t tag,
                                          int j0) {
    int32_t r[kHaloBatch];
    uint32_t todo = 0;
#pragma unroll
    for (int u = 0; u < kHaloBatch; ++u) {
      const int j = j0 + u * blockDim.x;
      r[u] = j < d.nh ? __ldg(a.halo + d.h0 + j) : 0;
      todo |= (uint32_t)(j < d.nh) << u;
    }
    long long t0 = 0;
    for (int tries = 0; todo; ++tries) {
#pragma unroll
      for (int u = 0; u < kHaloBatch; ++u)
        if (todo >> u & 1u) {
          bool here = true;
#pragma unroll
          for (int k = 0; k < NC; ++k)
            here &= chunk_load(ex + ((int64_t)r[u] * NC + k) * 4, v[u] + 3 * k) == tag;
          if (here) todo &= ~(1u << u);
        }
      if (todo && tries >= 64) {
        if (t0 == 0) t0 = clock64();
        if (clock64() - t0 > kWaitCycles) return false;
      }
    }
    return true;
  }
  __device__ __forceinline__ void store(const MarchArgs& a, const MarchPart& d, float* xs, int j0) const {
#pragma unroll
    for (int u = 0; u < kHaloBatch; ++u) {
      const int j = j0 + u * blockDim.x;
      if (j < d.nh) rec_store<D>(xs, a.npos, d.hbase + j, v[u]);
    }
  }
};

// One entry of the pull: acc += w (x_o - x_p) / (1 + |x_o - x_p|^2).  The
// denominator is at least 1, so the approximate reciprocal (1 ulp, no scaling
// steps for denominators near the ends of the range) is as accurate here as
// __fdividef, which it replaces; past 2^126 both give 0.
__device__ __forceinline__ float rcp_approx(float v) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
  return r;
}
template <int D>
__device__ __forceinline__ void pull(const float* xs, int npos, uint32_t o, float w, const float* xp, float* acc) {
  float d[D], q = 1.f;
  rec_load<D>(xs, npos, o, d);
#pragma unroll
  for (int c = 0; c < D; ++c) {
    d[c] -= xp[c];
    q = fmaf(d[c], d[c], q);
  }
  const float f = w * rcp_approx(q);
#pragma unroll
  for (int c = 0; c < D; ++c) acc[c] = fmaf(f, d[c], acc[c]);
}

// ------------------------------------------------------------------ forward

template <int D, bool RES>
__global__ void __launch_bounds__(1024, 1) march_fwd_kernel(const MarchArgs a) {
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ __align__(8) uint64_t bar;
  __shared__ uint32_t tmem_at;
  __shared__ int fail;
  constexpr int NC = ex_chunks(D);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nt = blockDim.x, nw = nt >> 5;
  const MarchPart d = a.part[blockIdx.x];
  const int npos = a.npos;
  float* xs = reinterpret_cast<float*>(smem);
  uint32_t* s_ent = reinterpret_cast<uint32_t*>(smem + a.off_ent);
  float2* s_w = reinterpret_cast<float2*>(smem + a.off_w);
  uint16_t* moff = reinterpret_cast<uint16_t*>(smem + a.off_moff);
  if (threadIdx.x == 0) {
    mbar_init(&bar, 1);
    fail = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) tmem_alloc(&tmem_at, a.tmem_cols);
  __syncthreads();
  const uint32_t tmem = tmem_at;
  if (threadIdx.x == 0) {
    const uint32_t b_off = ((uint32_t)(d.nsl + 1) * 2u + 15u) & ~15u;
    uint32_t bytes = b_off + load_planes<D>(a.x_in, a.n_rec, d.lo, d.own, xs, npos, &bar, false);
    if (RES) bytes += (uint32_t)d.ncol * 384u;
    mbar_arrive_tx(&bar, bytes);
    load_planes<D>(a.x_in, a.n_rec, d.lo, d.own, xs, npos, &bar, true);
    bulk_load(moff, a.moff + d.q0, b_off, &bar);
    if (RES && d.ncol) {
      bulk_load(s_ent, a.ent + 32 * (int64_t)d.s0, (uint32_t)d.ncol * 128u, &bar);
      bulk_load(s_w, a.w + 64 * (int64_t)d.s0, (uint32_t)d.ncol * 256u, &bar);
    }
  }
  // tags go on from the part's own count of published steps, which is the
  // same for all parts at the start of a launch
  const uint32_t base = *(volatile const uint32_t*)(a.flag + blockIdx.x);
  first_halo<D>(a, d, xs);
  if (!mbar_wait(&bar, 0)) fail = 1;
  __syncthreads();
  // this warp's columns of tensor memory: the 32 lanes of its quadrant
  const uint32_t hold = tmem + ((uint32_t)(warp & 3) << 21) + (uint32_t)(warp >> 2) * a.hold_cols;
  const uint32_t* pe = (RES ? s_ent : a.ent + 32 * (int64_t)d.s0) + lane;
  const float2* pw = (RES ? s_w : reinterpret_cast<const float2*>(a.w) + 32 * (int64_t)d.s0) + lane;
  for (int t = 0; fail == 0; ++t) {
    const bool last = t == a.steps - 1;
    const uint32_t tag = base + (uint32_t)t + 1u;
    float* ex = a.ex + (size_t)((t + 1) & 1) * a.n_rec * (4 * NC);
    if (a.ckpt && t % a.every == 0) {  // the state before step t, kept for the reverse sweep
      float* g = a.ckpt + (size_t)(t / a.every) * a.n_rec * D;
      for (int p = threadIdx.x; p < d.own; p += nt) {
        float v[D];
        rec_load<D>(xs, npos, p, v);
        rec_store<D>(g, a.n_rec, (int64_t)d.lo + p, v);
      }
    }
    uint32_t at = hold;
    for (int j = warp; j < d.nsl; j += nw, at += hold_stride(D)) {
      const int p = 32 * j + lane;
      float xp[D], acc[D];
      rec_load<D>(xs, npos, p, xp);
#pragma unroll
      for (int c = 0; c < D; ++c) acc[c] = 0.f;
      const int c1 = moff[j + 1];
      int c = moff[j];
      uint32_t e = 0;
      float2 w = make_float2(0.f, 0.f);
      if (c < c1) {
        e = RES ? pe[32 * c] : __ldg(pe + 32 * c);
        w = RES ? pw[32 * c] : __ldg(pw + 32 * c);
      }
      while (c < c1) {
        const uint32_t e0 = e;
        const float2 w0 = w;
        if (++c < c1) {  // the next pair of slots in flight
          e = RES ? pe[32 * c] : __ldg(pe + 32 * c);
          w = RES ? pw[32 * c] : __ldg(pw + 32 * c);
        }
        pull<D>(xs, npos, e0 & kSlotPos, w0.x, xp, acc);
        pull<D>(xs, npos, (e0 >> 16) & kSlotPos, w0.y, xp, acc);
      }
      float xn[3 * NC];
#pragma unroll
      for (int k = 0; k < 3 * NC; ++k) xn[k] = k < D ? fmaf(a.tau, acc[k < D ? k : 0], xp[k < D ? k : 0]) : 0.f;
      if (last) {
        if (p < d.own) {
          rec_store<D>(a.x_out, a.n_rec, (int64_t)d.lo + p, xn);
          if (a.out) rec_store<D>(a.out, a.n_rec, (int64_t)d.lo + p, acc);
        }
      } else {
        if (p < d.nb) {
#pragma unroll
          for (int k = 0; k < NC; ++k) chunk_store(ex + ((int64_t)(d.lo + p) * NC + k) * 4, xn + 3 * k, tag);
        }
        __syncwarp();
        tmem_put<D>(at, xn);
      }
    }
    if (last) break;
    tmem_put_wait();
    // the first batch of the halo arrives while other warps still compute
    HaloBatch<D> hb;
    bool here = hb.receive(a, d, ex, tag, threadIdx.x);
    __syncthreads();  // every slice has read its positions
    hb.store(a, d, xs, threadIdx.x);
    for (int j0 = threadIdx.x + kHaloBatch * nt; j0 < d.nh; j0 += kHaloBatch * nt) {
      here &= hb.receive(a, d, ex, tag, j0);
      hb.store(a, d, xs, j0);
    }
    if (!here) {
      fail = 1;
      atomicOr(a.err, kErrTimeoutNeighbour);
    }
    __syncwarp();
    at = hold;
    for (int j = warp; j < d.nsl; j += nw, at += hold_stride(D)) {
      float xn[D];
      tmem_get<D>(at, xn);
      if (32 * j + lane < d.own) rec_store<D>(xs, npos, 32 * j + lane, xn);
      __syncwarp();
    }
    __syncthreads();
    if (a.stall >= 0 && t + 1 >= a.stall && blockIdx.x == 0) break;  // test hook: part 0 leaves
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    if (fail) atomicOr(a.err, 1);
    a.flag[blockIdx.x] = base + (uint32_t)(a.steps - 1);
  }
  if (warp == 0) tmem_free(tmem, a.tmem_cols);
}

template <int D, bool RES>
cudaError_t march_launch_t(const MarchArgs& a, const MarchPlan& P, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(P.parts);
  cfg.blockDim = dim3(P.threads);
  cfg.dynamicSmemBytes = P.smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, march_fwd_kernel<D, RES>, a);
}

template <int D>
const void* march_ptr_t(bool res) {
  return res ? (const void*)march_fwd_kernel<D, true> : (const void*)march_fwd_kernel<D, false>;
}

}  // namespace

const void* march_kernel_ptr(int D, bool res) {
  switch (D) {
    case 1: return march_ptr_t<1>(res);
    case 2: return march_ptr_t<2>(res);
    case 3: return march_ptr_t<3>(res);
    case 4: return march_ptr_t<4>(res);
    case 5: return march_ptr_t<5>(res);
    case 6: return march_ptr_t<6>(res);
    case 7: return march_ptr_t<7>(res);
    case 8: return march_ptr_t<8>(res);
  }
  return nullptr;
}

// Shared-memory layout of a part and the launch shape, from the largest part's
// sizes.  smem_max: what a block may ask for.  parts = 0 when it does not fit.
MarchPlan march_plan(const MarchSizes& z, int D, int smem_max) {
  auto up = [](int64_t x, int64_t m) { return (x + m - 1) / m * m; };
  MarchPlan P = {};
  P.npos = (int)up(z.max_pos, 4);
  P.off_moff = (int)up((int64_t)D * P.npos * 4, 16);
  const int64_t base = P.off_moff + up((int64_t)(z.max_nsl + 1) * 2, 128);
  if (base > smem_max) return P;
  P.resident = base + (int64_t)z.max_col * 384 <= smem_max;
  P.off_ent = (int)base;
  P.off_w = (int)(base + (P.resident ? (int64_t)z.max_col * 128 : 0));
  P.smem = (size_t)(base + (P.resident ? (int64_t)z.max_col * 384 : 0));
  // one warp per slice up to 32; whole quadrants of four warps keep the
  // tensor-memory split even
  const int warps = (std::max(8, std::min(32, z.max_nsl)) + 3) / 4 * 4;
  P.threads = 32 * warps;
  const int iters = (z.max_nsl + warps - 1) / warps;
  P.hold_cols = iters * hold_stride(D);
  int cols = 32;
  while (cols < P.hold_cols * (warps / 4)) cols <<= 1;
  if (cols > 512) return P;  // more new values than tensor memory holds
  P.tmem_cols = cols;
  P.parts = z.parts;
  return P;
}

cudaError_t march_fwd(const MarchArgs& a0, const MarchPlan& P, int D, cudaStream_t st) {
  MarchArgs a = a0;
  a.npos = P.npos;
  a.off_moff = P.off_moff;
  a.off_ent = P.off_ent;
  a.off_w = P.off_w;
  a.hold_cols = (uint32_t)P.hold_cols;
  a.tmem_cols = (uint32_t)P.tmem_cols;
#define EP_M(DD) \
  case DD: return P.resident ? march_launch_t<DD, true>(a, P, st) : march_launch_t<DD, false>(a, P, st);
  switch (D) {
    EP_M(1) EP_M(2) EP_M(3) EP_M(4) EP_M(5) EP_M(6) EP_M(7) EP_M(8)
  }
#undef EP_M
  return cudaErrorInvalidValue;
}

}  // namespace dev
}  // namespace ep
