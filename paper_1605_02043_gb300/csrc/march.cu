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
// Threads of a block, which set the registers a thread has for slot pairs in
// flight (65,536 per SM).  Widths above 5 (the reverse sweep: above 2) spill
// with 1024 threads: 150,001 points, D = 8, ten steps 103 us, 81 with 512.
// Widths 3 to 5 (WIDE: 1024) need the warps only where a warp has many slices,
// and otherwise fewer threads meet sooner at a step's two barriers: 2^20 points
// (223 slices a part) 1228 us with 1024, 1285 with 512; 2^18 in input order (57
// slices, a large halo) 143 and 130; 4096 points, 50 steps 105 and 101.
constexpr int kWideSlices = 128;
constexpr int march_threads(int D, bool grad, bool wide) {
  return D <= 2 || (!grad && D <= 5 && wide) ? 1024 : 512;
}
constexpr bool march_wide(int D, bool grad, int slices) { return grad || D < 3 || D > 5 || slices > kWideSlices; }

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

// One bulk copy per plane between the records [lo, lo + n) of a planar state
// (lo a multiple of 4) and the positions [0, n) in shared memory.
template <int D, int K = 0>
__device__ __forceinline__ uint32_t plane_bytes(int n) {
  if constexpr (K < Planes<D>::NP) return (((uint32_t)n * Planes<D>::width(K) * 4u + 15u) & ~15u) + plane_bytes<D, K + 1>(n);
  return 0;
}
template <int D, int K = 0>
__device__ __forceinline__ void load_planes(const float* g, int64_t n_rec, int lo, int n, float* s, int npos,
                                            uint64_t* bar) {
  if constexpr (K < Planes<D>::NP) {
    constexpr int W = Planes<D>::width(K), F = Planes<D>::first(K);
    const uint32_t bytes = ((uint32_t)n * W * 4u + 15u) & ~15u;
    if (bytes) bulk_load(s + F * npos, g + F * n_rec + (int64_t)lo * W, bytes, bar);
    load_planes<D, K + 1>(g, n_rec, lo, n, s, npos, bar);
  }
}
template <int D, int K = 0>
__device__ __forceinline__ void store_planes(float* g, int64_t n_rec, int lo, int n, const float* s, int npos) {
  if constexpr (K < Planes<D>::NP) {
    constexpr int W = Planes<D>::width(K), F = Planes<D>::first(K);
    const uint32_t bytes = ((uint32_t)n * W * 4u + 15u) & ~15u;
    if (bytes)
      asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(g + F * n_rec + (int64_t)lo * W),
                   "r"(saddr(s + F * npos)), "r"(bytes)
                   : "memory");
    store_planes<D, K + 1>(g, n_rec, lo, n, s, npos);
  }
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_read() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_done() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }
// this thread's shared-memory stores before a later bulk copy of them
__device__ __forceinline__ void fence_bulk() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// Halo values of a state of which only the owners' records are written, four
// records in flight per thread
template <int D>
__device__ __forceinline__ void first_halo(const MarchArgs& a, const MarchPart& d, const float* state, float* xs) {
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
      if (r[u] >= 0) rec_load<D>(state, a.n_rec, r[u], v[u]);
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

// A warp's slices as one stream of pair columns: begin(slice) starts a slice,
// take(entries, weights, column) handles one pair column of it, end(slice)
// finishes it.  Entries and weights are read ahead across the slices' ends into
// a ring of registers whose places are fixed by the unrolling (a slice's end is
// a branch inside it).  One column ahead is enough: three (9 more registers)
// cost 4% on the 1M-point mesh, whose slots come from the L2, and 5% where
// they are in shared memory.
template <bool RES, typename Begin, typename Take, typename End>
__device__ __forceinline__ void march_slices(const MarchPart& d, const uint16_t* tab, int v, int W, const uint32_t* pe,
                                             const float2* pw, Begin begin, Take take, End end) {
  int j = v;
  if (j >= d.nsl) return;
  int i = tab[v];
  uint32_t e[kMarchAhead];
  float2 w[kMarchAhead];
#pragma unroll
  for (int u = 0; u < kMarchAhead - 1; ++u) {
    e[u] = RES ? pe[32 * (i + u)] : __ldg(pe + 32 * (i + u));
    w[u] = RES ? pw[32 * (i + u)] : __ldg(pw + 32 * (i + u));
  }
  int left = tab[W + j];
  begin(j);
  for (;;) {
#pragma unroll
    for (int u = 0; u < kMarchAhead; ++u) {
      constexpr int A = kMarchAhead - 1;
      e[(u + A) % kMarchAhead] = RES ? pe[32 * (i + A)] : __ldg(pe + 32 * (i + A));
      w[(u + A) % kMarchAhead] = RES ? pw[32 * (i + A)] : __ldg(pw + 32 * (i + A));
      take(e[u], w[u], i);
      ++i;
      if (--left == 0) {
        end(j);
        if ((j += W) >= d.nsl) return;
        left = tab[W + j];
        begin(j);
      }
    }
  }
}

// Start of a kernel: barrier, tensor memory, the part's tables, slots and
// weights (RES) and the own records of `state` (whole images where `image`).
struct MarchSmem {
  float* x;
  float* lam;
  uint16_t* tab;
  const uint32_t* pe;  // this lane's entries and weights
  const float2* pw;
};
template <int D, bool RES>
__device__ __forceinline__ MarchSmem march_smem(const MarchArgs& a, const MarchPart& d, unsigned char* smem) {
  const int lane = threadIdx.x & 31;
  MarchSmem S;
  S.x = reinterpret_cast<float*>(smem);
  S.lam = reinterpret_cast<float*>(smem + a.off_lam);
  S.tab = reinterpret_cast<uint16_t*>(smem + a.off_tab);
  S.pe = (RES ? reinterpret_cast<const uint32_t*>(smem + a.off_ent) : a.ent + 32 * (int64_t)d.s0) + lane;
  S.pw = (RES ? reinterpret_cast<const float2*>(smem + a.off_w) : reinterpret_cast<const float2*>(a.w) + 32 * (int64_t)d.s0) +
         lane;
  return S;
}
template <bool RES>
__device__ __forceinline__ uint32_t table_bytes(const MarchArgs& a, const MarchPart& d) {
  return (((uint32_t)(a.warps + d.nsl) * 2u + 15u) & ~15u) + (RES ? (uint32_t)(d.ncol + kMarchAhead) * 384u : 0u);
}
template <bool RES>
__device__ __forceinline__ void load_tables(const MarchArgs& a, const MarchPart& d, unsigned char* smem, uint64_t* bar) {
  bulk_load(smem + a.off_tab, a.tab + d.q0, ((uint32_t)(a.warps + d.nsl) * 2u + 15u) & ~15u, bar);
  if (RES) {  // with the columns the read-ahead touches
    bulk_load(smem + a.off_ent, a.ent + 32 * (int64_t)d.s0, (uint32_t)(d.ncol + kMarchAhead) * 128u, bar);
    bulk_load(smem + a.off_w, a.w + 64 * (int64_t)d.s0, (uint32_t)(d.ncol + kMarchAhead) * 256u, bar);
  }
}

// One forward step of this warp's slices: new values of boundary positions
// published with `tag` and every new value held in tensor memory from `hold`
// on; the last step of a run goes to memory instead (x_out, out).
template <int D, bool RES>
__device__ __forceinline__ void forward_slices(const MarchArgs& a, const MarchPart& d, const MarchSmem& S, uint32_t hold,
                                               float* ex, uint32_t tag, bool last) {
  constexpr int NC = ex_chunks(D);
  const int lane = threadIdx.x & 31, nw = blockDim.x >> 5, npos = a.npos;
  const float* xs = S.x;
  uint32_t at = hold;
  float xp[D], acc[D];
  auto begin = [&](int j) {
    rec_load<D>(xs, npos, 32 * j + lane, xp);
#pragma unroll
    for (int c = 0; c < D; ++c) acc[c] = 0.f;
  };
  auto take = [&](uint32_t e, float2 w, int) {  // acc += w (x_o - x_p) / (1 + |x_o - x_p|^2), two slots
    float d0[D], d1[D], q0 = kDenStart<D>, q1 = kDenStart<D>;
    rec_load<D>(xs, npos, e & kSlotPos, d0);
    rec_load<D>(xs, npos, (e >> 16) & kSlotPos, d1);
#pragma unroll
    for (int c = 0; c < D; ++c) {
      d0[c] -= xp[c], d1[c] -= xp[c];
      q0 = fmaf(d0[c], d0[c], q0), q1 = fmaf(d1[c], d1[c], q1);
    }
    const float f0 = w.x * rcp_den<D>(q0), f1 = w.y * rcp_den<D>(q1);
#pragma unroll
    for (int c = 0; c < D; ++c) acc[c] = fmaf(f1, d1[c], fmaf(f0, d0[c], acc[c]));
  };
  auto end = [&](int j) {
    const int p = 32 * j + lane;
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
      at += hold_stride(D);
    }
  };
  for (int v = threadIdx.x >> 5; v < a.warps; v += nw)
    march_slices<RES>(d, S.tab, v, a.warps, S.pe, S.pw, begin, take, end);
  tmem_put_wait();
}

// The rest of a step: the halo of the planes `xs`, and the held values into
// their positions.  `between` runs in thread 0 once every slice has read its
// positions.  False when a neighbour's value did not come.
template <int D, typename Between>
__device__ __forceinline__ bool settle(const MarchArgs& a, const MarchPart& d, float* xs, uint32_t hold, const float* ex,
                                       uint32_t tag, Between between) {
  const int lane = threadIdx.x & 31, nt = blockDim.x, nw = nt >> 5;
  // the first batch arrives while other warps still compute
  HaloBatch<D> hb;
  bool here = hb.receive(a, d, ex, tag, threadIdx.x);
  __syncthreads();  // every slice has read its positions
  if (threadIdx.x == 0) between();
  hb.store(a, d, xs, threadIdx.x);
  for (int j0 = threadIdx.x + kHaloBatch * nt; j0 < d.nh; j0 += kHaloBatch * nt) {
    here &= hb.receive(a, d, ex, tag, j0);
    hb.store(a, d, xs, j0);
  }
  __syncwarp();
  uint32_t at = hold;
  for (int v = threadIdx.x >> 5; v < a.warps; v += nw)
    for (int j = v; j < d.nsl; j += a.warps, at += hold_stride(D)) {
      float xn[D];
      tmem_get<D>(at, xn);
      if (32 * j + lane < d.own) rec_store<D>(xs, a.npos, 32 * j + lane, xn);
      __syncwarp();
    }
  return here;
}

// ------------------------------------------------------------------ forward

template <int D, bool RES, bool WIDE>
__global__ void __launch_bounds__(march_threads(D, false, WIDE), 1) march_fwd_kernel(const MarchArgs a) {
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ __align__(8) uint64_t bar;
  __shared__ uint32_t tmem_at;
  __shared__ int fail;
  constexpr int NC = ex_chunks(D);
  const int warp = threadIdx.x >> 5;
  const MarchPart d = a.part[blockIdx.x];
  const MarchSmem S = march_smem<D, RES>(a, d, smem);
  if (threadIdx.x == 0) {
    mbar_init(&bar, 1);
    fail = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) tmem_alloc(&tmem_at, a.tmem_cols);
  __syncthreads();
  const uint32_t tmem = tmem_at;
  if (threadIdx.x == 0) {
    mbar_arrive_tx(&bar, table_bytes<RES>(a, d) + plane_bytes<D>(d.own));
    load_planes<D>(a.x_in, a.n_rec, d.lo, d.own, S.x, a.npos, &bar);
    load_tables<RES>(a, d, smem, &bar);
  }
  // tags go on from the part's own count of published steps, which is the
  // same for all parts at the start of a launch
  const uint32_t base = *(volatile const uint32_t*)(a.flag + blockIdx.x);
  first_halo<D>(a, d, a.x_in, S.x);
  if (!mbar_wait(&bar, 0)) fail = 1;
  if (a.ckpt) fence_bulk();
  __syncthreads();
  // this warp's columns of tensor memory: the 32 lanes of its quadrant
  const uint32_t hold = tmem + ((uint32_t)(warp & 3) << 21) + (uint32_t)(warp >> 2) * a.hold_cols;
  for (int t = 0; fail == 0; ++t) {
    const bool last = t == a.steps - 1;
    const uint32_t tag = base + (uint32_t)t + 1u;
    float* ex = a.ex + (size_t)((t + 1) & 1) * a.n_rec * (4 * NC);
    if (a.ckpt && t % a.every == 0 && threadIdx.x == 0) {  // the state before step t, halo and all
      store_planes<D>(a.ckpt + (size_t)(t / a.every) * a.n_rec * D, a.n_rec, d.lo, d.hbase + d.nh, S.x, a.npos);
      bulk_commit();
    }
    forward_slices<D, RES>(a, d, S, hold, ex, tag, last);
    if (last) break;
    // the checkpoint's copy out of S.x is over before settle()'s barrier lets
    // S.x change (usually it is by now: the slices take longer)
    if (a.ckpt && threadIdx.x == 0) bulk_wait_read();
    const bool here = settle<D>(a, d, S.x, hold, ex, tag, [] {});
    if (!here) {
      fail = 1;
      atomicOr(a.err, kErrTimeoutNeighbour);
    }
    if (a.ckpt) fence_bulk();
    __syncthreads();
    if (a.stall >= 0 && t + 1 >= a.stall && blockIdx.x == 0) break;  // test hook: part 0 leaves
  }
  if (threadIdx.x == 0 && a.ckpt) bulk_wait_done();
  __syncthreads();
  if (threadIdx.x == 0) {
    if (fail) atomicOr(a.err, 1);
    a.flag[blockIdx.x] = base + (uint32_t)(a.steps - 1);
  }
  if (warp == 0) tmem_free(tmem, a.tmem_cols);
}

// ----------------------------------------------------------------- gradient

// One reverse step of this warp's slices at the state S.x, cotangent S.lam
// (flux_common.cuh adj_slice): new cotangents published and held like the
// forward's values (the last one to memory), weight gradients added to (by the
// first reverse step: stored in) their task's slot at its first endpoint.
template <int D, bool RES>
__device__ __forceinline__ void adjoint_slices(const MarchArgs& a, const MarchPart& d, const MarchSmem& S, uint32_t hold,
                                               float* ex, uint32_t tag, bool first, bool last) {
  constexpr int NC = ex_chunks(D);
  const int lane = threadIdx.x & 31, nw = blockDim.x >> 5, npos = a.npos;
  uint32_t at = hold;
  float xp[D], lp[D], acc[D];
  float* gw = a.gw + 64 * (int64_t)d.s0 + 2 * lane;
  auto begin = [&](int j) {
    rec_load<D>(S.x, npos, 32 * j + lane, xp);
    rec_load<D>(S.lam, npos, 32 * j + lane, lp);
#pragma unroll
    for (int c = 0; c < D; ++c) acc[c] = 0.f;
  };
  auto one = [&](uint32_t e, float w, float* g) {
    float dx[D], dl[D], q = kDenStart<D>, dg = 0.f;
    rec_load<D>(S.x, npos, e & kSlotPos, dx);
    rec_load<D>(S.lam, npos, e & kSlotPos, dl);
#pragma unroll
    for (int c = 0; c < D; ++c) {
      dx[c] -= xp[c];
      dl[c] = lp[c] - dl[c];
      q = fmaf(dx[c], dx[c], q);
      dg = fmaf(dx[c], dl[c], dg);
    }
    const float inv = rcp_den<D>(q), s = dg * inv, two = 2.f * s * inv;
#pragma unroll
    for (int c = 0; c < D; ++c) acc[c] -= w * (dl[c] * inv - two * dx[c]);
    if (e & kSlotSrc) {  // one lane's slot throughout: no reader before the next launch
      if (first)
        *g = a.tau * s;
      else
        atomicAdd(g, a.tau * s);  // fire-and-forget reduction
    }
  };
  auto take = [&](uint32_t e, float2 w, int i) {
    one(e & 0xffffu, w.x, gw + 64 * (int64_t)i);
    one(e >> 16, w.y, gw + 64 * (int64_t)i + 1);
  };
  auto end = [&](int j) {
    const int p = 32 * j + lane;
    float ln[3 * NC];
#pragma unroll
    for (int k = 0; k < 3 * NC; ++k) ln[k] = k < D ? fmaf(a.tau, acc[k < D ? k : 0], lp[k < D ? k : 0]) : 0.f;
    if (last) {
      if (p < d.own) rec_store<D>(a.lam_out, a.n_rec, (int64_t)d.lo + p, ln);
    } else {
      if (p < d.nb) {
#pragma unroll
        for (int k = 0; k < NC; ++k) chunk_store(ex + ((int64_t)(d.lo + p) * NC + k) * 4, ln + 3 * k, tag);
      }
      __syncwarp();
      tmem_put<D>(at, ln);
      at += hold_stride(D);
    }
  };
  for (int v = threadIdx.x >> 5; v < a.warps; v += nw)
    march_slices<RES>(d, S.tab, v, a.warps, S.pe, S.pw, begin, take, end);
  tmem_put_wait();
}

// The whole reverse sweep of a run of `steps` steps in one launch: segment by
// segment from the last, the states between two checkpoints are recomputed
// (and kept as images in `hist`, which only their own part reads again) and the
// reverse steps walk back over them.  Segment g starts from image g of `ckpt`;
// with one segment `x_in` may give its state instead (owners' records, `ckpt`
// then receives the image).
template <int D, bool RES>
__global__ void __launch_bounds__(march_threads(D, true, true), 1) march_grad_kernel(const MarchArgs a) {
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ __align__(8) uint64_t bar;
  __shared__ uint32_t tmem_at;
  __shared__ int fail;
  constexpr int NC = ex_chunks(D);
  const int warp = threadIdx.x >> 5;
  const MarchPart d = a.part[blockIdx.x];
  const MarchSmem S = march_smem<D, RES>(a, d, smem);
  const int image = d.hbase + d.nh;
  const size_t state = (size_t)a.n_rec * D;
  if (threadIdx.x == 0) {
    mbar_init(&bar, 1);
    fail = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) tmem_alloc(&tmem_at, a.tmem_cols);
  __syncthreads();
  const uint32_t tmem = tmem_at;
  int seg = (a.steps - 1) / a.every;
  if (threadIdx.x == 0) {
    const int n = a.x_in ? d.own : image;
    mbar_arrive_tx(&bar, table_bytes<RES>(a, d) + plane_bytes<D>(n) + plane_bytes<D>(d.own));
    load_planes<D>(a.x_in ? a.x_in : a.ckpt + seg * state, a.n_rec, d.lo, n, S.x, a.npos, &bar);
    load_planes<D>(a.lam_in, a.n_rec, d.lo, d.own, S.lam, a.npos, &bar);
    load_tables<RES>(a, d, smem, &bar);
  }
  const uint32_t base = *(volatile const uint32_t*)(a.flag + blockIdx.x);
  first_halo<D>(a, d, a.lam_in, S.lam);
  if (a.x_in) first_halo<D>(a, d, a.x_in, S.x);
  uint32_t ph = 0;  // loads done
  if (!mbar_wait(&bar, ph++ & 1u)) fail = 1;
  fence_bulk();
  __syncthreads();
  if (a.x_in && threadIdx.x == 0) {  // the only checkpoint, made here
    store_planes<D>(a.ckpt, a.n_rec, d.lo, image, S.x, a.npos);
    bulk_commit();
  }
  const uint32_t hold = tmem + ((uint32_t)(warp & 3) << 21) + (uint32_t)(warp >> 2) * a.hold_cols;
  uint32_t sent = 0;  // exchanges so far, states and cotangents
  bool first = true;  // the first reverse step sets the weight gradients, the others add
  auto ex_of = [&](uint32_t s) { return a.ex + (size_t)((s + 1) & 1) * a.n_rec * (4 * NC); };
  for (; seg >= 0 && fail == 0; --seg) {
    const int T = min(a.every, a.steps - seg * a.every);
    for (int t = 1; t < T && fail == 0; ++t) {  // x_t of the segment into S.x
      float* ex = ex_of(sent);
      const uint32_t tag = base + ++sent;
      forward_slices<D, RES>(a, d, S, hold, ex, tag, false);
      // the copy of x_{t-1} out of S.x is over before S.x changes
      if (threadIdx.x == 0) bulk_wait_read();
      if (!settle<D>(a, d, S.x, hold, ex, tag, [] {})) {
        fail = 1;
        atomicOr(a.err, kErrTimeoutNeighbour);
      }
      fence_bulk();
      __syncthreads();
      if (t < T - 1 && threadIdx.x == 0) {
        store_planes<D>(a.hist + (size_t)(t - 1) * state, a.n_rec, d.lo, image, S.x, a.npos);
        bulk_commit();
      }
      if (a.stall >= 0 && (int)sent >= a.stall && blockIdx.x == 0) {  // test hook: part 0 leaves
        seg = -1;
        break;
      }
    }
    for (int t = T - 1; t >= 0 && seg >= 0 && fail == 0; --t) {
      const bool last = t == 0 && seg == 0;
      float* ex = ex_of(sent);
      const uint32_t tag = base + sent + 1u;
      adjoint_slices<D, RES>(a, d, S, hold, ex, tag, first, last);
      first = false;
      if (last) break;
      ++sent;
      // the state before this one, or the checkpoint before this segment's
      const float* prev = t > 1 ? a.hist + (size_t)(t - 2) * state : a.ckpt + (size_t)(t == 1 ? seg : seg - 1) * state;
      if (!settle<D>(a, d, S.lam, hold, ex, tag, [&] {
            bulk_wait_done();
            mbar_arrive_tx(&bar, plane_bytes<D>(image));
            load_planes<D>(prev, a.n_rec, d.lo, image, S.x, a.npos, &bar);
          })) {
        fail = 1;
        atomicOr(a.err, kErrTimeoutNeighbour);
      }
      if (!mbar_wait(&bar, ph++ & 1u)) fail = 1;
      __syncthreads();
      if (a.stall >= 0 && (int)sent >= a.stall && blockIdx.x == 0) seg = -1;  // test hook: part 0 leaves
    }
  }
  if (threadIdx.x == 0) bulk_wait_done();
  __syncthreads();
  if (threadIdx.x == 0) {
    if (fail) atomicOr(a.err, 1);
    // every part sends the same number: T - 1 states and T cotangents a segment, less the last cotangent
    const int segs = (a.steps - 1) / a.every + 1;
    a.flag[blockIdx.x] = base + (uint32_t)(2 * a.steps - segs - 1);
  }
  if (warp == 0) tmem_free(tmem, a.tmem_cols);
}

template <typename K>
cudaError_t march_launch_t(K kernel, const MarchArgs& a, const MarchPlan& P, cudaStream_t st) {
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
  return cudaLaunchKernelEx(&cfg, kernel, a);
}

using MarchKernel = void (*)(const MarchArgs);
template <int D, bool WIDE>
MarchKernel march_fwd_t(bool res) {
  return res ? march_fwd_kernel<D, true, WIDE> : march_fwd_kernel<D, false, WIDE>;
}
template <int D>
MarchKernel march_kernel_t(bool grad, bool res, bool wide) {
  if (grad) return res ? march_grad_kernel<D, true> : march_grad_kernel<D, false>;
  if constexpr (D >= 3 && D <= 5)
    if (!wide) return march_fwd_t<D, false>(res);
  return march_fwd_t<D, true>(res);
}
MarchKernel march_kernel(int D, bool grad, bool res, bool wide) {
  switch (D) {
    case 1: return march_kernel_t<1>(grad, res, wide);
    case 2: return march_kernel_t<2>(grad, res, wide);
    case 3: return march_kernel_t<3>(grad, res, wide);
    case 4: return march_kernel_t<4>(grad, res, wide);
    case 5: return march_kernel_t<5>(grad, res, wide);
    case 6: return march_kernel_t<6>(grad, res, wide);
    case 7: return march_kernel_t<7>(grad, res, wide);
    case 8: return march_kernel_t<8>(grad, res, wide);
  }
  return nullptr;
}

}  // namespace

const void* march_kernel_ptr(const MarchPlan& P, int D, bool grad) {
  return reinterpret_cast<const void*>(march_kernel(D, grad, P.resident, P.wide));
}

// Shared-memory layout of a part and the launch shape, from the largest part's
// sizes.  smem_max: what a block may ask for.  parts = 0 when it does not fit.
MarchPlan march_plan(const MarchSizes& z, int D, bool grad, int smem_max) {
  auto up = [](int64_t x, int64_t m) { return (x + m - 1) / m * m; };
  MarchPlan P = {};
  P.npos = (int)up(z.max_pos, 4);
  const int64_t planes = up((int64_t)D * P.npos * 4, 16);
  P.off_lam = grad ? (int)planes : 0;
  P.off_tab = (int)(grad ? 2 * planes : planes);
  const int64_t base = P.off_tab + up((int64_t)(z.max_nsl + z.warps) * 2, 128), cols = z.max_col + kMarchAhead;
  if (base > smem_max) return P;
  P.resident = base + cols * 384 <= smem_max;
  P.off_ent = (int)base;
  P.off_w = (int)(base + (P.resident ? cols * 128 : 0));
  P.smem = (size_t)(base + (P.resident ? cols * 384 : 0));
  // a warp per stream of slices (march.h), in whole groups of four: one per
  // quadrant of the tensor memory
  P.wide = march_wide(D, grad, z.max_nsl);
  P.threads = std::min(32 * z.warps, march_threads(D, grad, P.wide));
  P.warps = z.warps;
  const int per_warp = (z.warps * 32 + P.threads - 1) / P.threads;  // streams of one warp
  const int iters = (z.max_nsl + z.warps - 1) / z.warps * per_warp;
  P.hold_cols = iters * hold_stride(D);
  int tc = 32;
  while (tc < P.hold_cols * (P.threads / 128)) tc <<= 1;
  if (tc > 512) return P;  // more new values than tensor memory holds
  P.tmem_cols = tc;
  P.parts = z.parts;
  return P;
}

cudaError_t march_run(const MarchArgs& a0, const MarchPlan& P, int D, bool grad, cudaStream_t st) {
  MarchArgs a = a0;
  a.warps = P.warps;
  a.npos = P.npos;
  a.off_lam = P.off_lam;
  a.off_tab = P.off_tab;
  a.off_ent = P.off_ent;
  a.off_w = P.off_w;
  a.hold_cols = (uint32_t)P.hold_cols;
  a.tmem_cols = (uint32_t)P.tmem_cols;
  const MarchKernel k = march_kernel(D, grad, P.resident, P.wide);
  return k ? march_launch_t(k, a, P, st) : cudaErrorInvalidValue;
}

}  // namespace dev
}  // namespace ep
