// kernels.cu -- device code of libepcache (sm_103a).
//
// The software-cache kernel of Section 4 (Fig. 7(d)), restated for GB300:
// every CUDA block takes one schedule block, copies the distinct vertices of
// that block (the vertex set the cost model of Eq. 1 counts once per block)
// from HBM into shared memory, runs its tasks out of shared memory, and
// writes back once per vertex: vertices no other block uses are updated in
// place with plain stores, shared vertices get one vector atomic add into an
// accumulator, applied to every copy by the next step's fix-up or by the
// finish (bnd_update_kernel).  Also here: the SpMV kernel, the cost kernels,
// the layout conversions and the shard-halo moves.
#include <cuda_runtime.h>

#include <climits>
#include <cstddef>
#include <cstdint>
#include <mutex>
#include <unordered_set>

#include "block_distinct.cuh"
#include "flux_common.cuh"
#include "kernels.h"
#include "tma_sync.cuh"

namespace ep {
namespace dev {
namespace {

// Shared-memory carve-up of one kernel block (the stage layout of the
// pipelined kernels, one stage): state planes, cotangent planes (adjoint),
// slots, slot weights, shared ids, slice offsets.
struct BlockSmem {
  float* x;
  float* lam;
  uint16_t* sidx;
  float* w;
  int32_t* sid;
  uint16_t* soff;
};
__device__ __forceinline__ BlockSmem block_smem(unsigned char* base, const TmaLayout& L) {
  BlockSmem r;
  r.x = reinterpret_cast<float*>(base);
  r.lam = reinterpret_cast<float*>(base + L.off_lam);
  r.sidx = reinterpret_cast<uint16_t*>(base + L.off_sidx);
  r.w = reinterpret_cast<float*>(base + L.off_w);
  r.sid = reinterpret_cast<int32_t*>(base + L.off_sid);
  r.soff = reinterpret_cast<uint16_t*>(base + L.off_soff);
  return r;
}

// copy `bytes` (a multiple of 16) as 16-byte vectors, the whole CUDA block
__device__ __forceinline__ void copy16(void* dst, const void* src, uint32_t bytes) {
  uint4* d = reinterpret_cast<uint4*>(dst);
  const uint4* s = reinterpret_cast<const uint4*>(src);
  for (uint32_t i = threadIdx.x; i < bytes / 16u; i += blockDim.x) d[i] = __ldg(s + i);
}
__device__ __forceinline__ uint32_t up16(uint32_t b) { return (b + 15u) & ~15u; }

template <int D, int K = 0>
__device__ __forceinline__ void copy_run(float* sx, int npos, const float* gx, int64_t n, int lo, int nv) {
  if constexpr (K < Planes<D>::NP) {
    constexpr int W = Planes<D>::width(K), F = Planes<D>::first(K);
    copy16(sx + F * npos, gx + F * n + (int64_t)lo * W, up16((uint32_t)nv * W * 4u));
    copy_run<D, K + 1>(sx, npos, gx, n, lo, nv);
  }
}

// The same pieces the pipelined kernels bulk-copy, moved by the CUDA block's
// threads as 16-byte vectors (every piece is 16-byte aligned and padded).
template <int D>
__device__ __forceinline__ void stage_block(const FluxDesc& d, const FluxArgs& a, const float* lam,
                                            const BlockSmem& S, const TmaLayout& L) {
  copy16(S.sidx, a.sidx + d.s0, (uint32_t)d.nslot * 2u);
  copy16(S.w, a.w + d.s0, (uint32_t)d.nslot * 4u);
  copy16(S.soff, a.soff + d.q0, up16((uint32_t)(d.nsl + 1) * 2u));
  copy16(S.sid, a.sid + d.h0, up16((uint32_t)(d.nv - d.ni) * 4u));
  copy_run<D>(S.x, L.npos, a.x_in, a.n_rec, d.rec_lo, d.nv);
  if (lam) copy_run<D>(S.lam, L.npos, lam, a.n_rec, d.rec_lo, d.nv);
}

// ------------------------------------------------------------- flux forward

// One CUDA block per kernel block: stage, bring the pending shared copies up
// to date, then every warp takes slices of 32 positions (pull form,
// flux_common.cuh).  Only the staged copy is read, so the in-place update of
// the interior records cannot overtake a read.
template <int D>
__global__ void __launch_bounds__(1024) flux_fwd_kernel(const FluxArgs a, TmaLayout L) {
  extern __shared__ __align__(128) unsigned char smem[];
  const FluxDesc d = a.desc[blockIdx.x];
  const BlockSmem S = block_smem(smem, L);
  const int q = *a.phase;
  stage_block<D>(d, a, nullptr, S, L);
  __syncthreads();
  fixup_copies<D>(d, S.x, L.npos, S.sid, acc_buffer<D>(a, q + 2), acc_buffer<D>(a, q + 1), a.tau,
                  threadIdx.x, blockDim.x);
  __syncthreads();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  for (int sl = warp; sl < d.nsl; sl += nw)
    fwd_block_slice<D>(a, acc_buffer<D>(a, q), d, S.x, L.npos, S.sidx, S.w, S.soff, S.sid, sl, lane);
  advance_phase(a, q);
}

// Read-only-cache variant: the texture-cache kernel of Section 5 (Fig. 7(c)),
// with the read-only data cache (ld.global.nc) in place of texture binding.
// No staging: slots, weights and states are read from global memory through
// that cache, so it runs on a finished state (no pending copies: the previous
// step's accumulator is zero).  Warp w takes slices w, w + W, ..., up to R of
// them, and keeps their sums in registers; writes wait for a block barrier,
// because interior records are updated in place and other warps may still be
// reading them.
template <int D, int R>
__global__ void __launch_bounds__(1024) flux_fwd_ldg_kernel(const FluxArgs a) {
  const FluxDesc d = a.desc[blockIdx.x];
  const int q = *a.phase;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  float xp[R][D], acc[R][D];
#pragma unroll
  for (int i = 0; i < R; ++i) {
    const int sl = warp + i * nw, p = 32 * sl + lane;
#pragma unroll
    for (int c = 0; c < D; ++c) xp[i][c] = acc[i][c] = 0.f;
    if (sl >= d.nsl) continue;
    const int c0 = __ldg(a.soff + d.q0 + sl), K = __ldg(a.soff + d.q0 + sl + 1) - c0;
    if (p < d.nv) rec_load<D, true>(a.x_in, a.n_rec, (int64_t)d.rec_lo + p, xp[i]);
    const int64_t s = (int64_t)d.s0 + 32 * c0 + lane;
    fwd_slice<D, true>(a.x_in, a.n_rec, d.rec_lo, a.sidx + s, a.w + s, K, xp[i], acc[i]);
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < R; ++i) {
    const int sl = warp + i * nw, p = 32 * sl + lane;
    if (sl >= d.nsl || p >= d.nv) continue;
    if (p < d.ni) {
      float xn[D];
#pragma unroll
      for (int c = 0; c < D; ++c) xn[c] = fmaf(a.tau, acc[i][c], xp[i][c]);
      rec_store<D>(a.x_out, a.n_rec, (int64_t)d.rec_lo + p, xn);
      if (a.out) rec_store<D>(a.out, a.n_rec, (int64_t)d.rec_lo + p, acc[i]);
    } else {  // this step's sum, the clearing, and the copy (x_out may be another buffer)
      const int32_t raw = __ldg(a.sid + d.h0 + p - d.ni);
      acc_red<D>(acc_buffer<D>(a, q), raw & kSidMask, acc[i]);
      if (raw < 0) acc_zero<D>(acc_buffer<D>(a, q + 1), raw & kSidMask);
      rec_store<D>(a.x_out, a.n_rec, (int64_t)d.rec_lo + p, xp[i]);
    }
  }
  advance_phase(a, q);
}

// The finish of a pending state, one thread per copy (fold_rec / fold_sid in
// record order: coalesced record accesses, one dependent round trip;
// flux_common.cuh fold_copies and the accumulator rotation).
template <int D>
__global__ void bnd_update_kernel(const FluxArgs a, const float* x_in, float* x_out, float* out) {
  // launched with programmatic serialisation after the edge kernel: wait for
  // it (the accumulators and records it wrote) before reading
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const int q = *a.phase;
  fold_copies<D>(a, x_in, x_out, out, acc_buffer<D>(a, q + 2), acc_buffer<D>(a, q + 1),
                 blockIdx.x * (int64_t)blockDim.x + threadIdx.x, a.n_copies,
                 (int64_t)gridDim.x * blockDim.x);
  advance_phase(a, q);
}

// ------------------------------------------------------------- flux adjoint

// One CUDA block per kernel block, the adjoint step (flux_common.cuh adj_*):
// stage the state (finished) and the cotangent (copies pending), bring the
// cotangent copies up to date, compute.
template <int D>
__global__ void __launch_bounds__(1024) flux_adj_kernel(const FluxArgs a, float* lam, float* gw,
                                                        TmaLayout L) {
  extern __shared__ __align__(128) unsigned char smem[];
  const FluxDesc d = a.desc[blockIdx.x];
  const BlockSmem S = block_smem(smem, L);
  const int q = *a.phase;
  stage_block<D>(d, a, lam, S, L);
  __syncthreads();
  fixup_copies<D>(d, S.lam, L.npos, S.sid, acc_buffer<D>(a, q + 2), acc_buffer<D>(a, q + 1), a.tau,
                  threadIdx.x, blockDim.x);
  __syncthreads();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  for (int sl = warp; sl < d.nsl; sl += nw)
    adj_block_slice<D>(a, acc_buffer<D>(a, q), d, S.x, S.lam, L.npos, S.sidx, S.w, S.soff, S.sid, lam,
                       gw, sl, lane);
  advance_phase(a, q);
}

// --------------------------------------------------------------------- SpMV

// SpMV over the edge partition (Section 5.2), one warp per schedule block at
// a time.  The block's entries are ranked by row position and cut into 32
// equal chunks, one per lane, so every lane does the same work whatever the
// row lengths: a lane walks its chunk in order, summing runs of equal rows in a
// register.  A run that neither starts nor ends the chunk is a whole row and is
// stored at once; the first and last runs of the chunks are joined across lanes
// by a segmented scan over the warp.  Row totals go to a shared array and leave
// it in row order (plain stores for rows of this block alone, atomics for
// shared rows).
//
// The software cache (HOT): x records are ordered by how many blocks use the
// column, and one persistent CUDA block per SM keeps the kSpmvHot most used ones
// beside the row totals.  On power-law matrices most entries name one of those;
// the others are read at the entry, through the L1 that is left: all of shared
// memory for columns (about 45,000) leaves none, and R-MAT scale 20 in CSR order
// takes 51.5 us instead of 44.0 (1,024 columns: 49.7; 8,192: 47.9), scale 18
// partitioned 53 instead of 31.5.  Staging each block's own distinct columns, as
// before, read an id and a 32-byte sector per column and block, with next to no
// reuse inside a block of 512 tasks: 73.7 us at scale 20, of which staging was
// 39.  Bound now by latency (the join and the write-out of one block follow its
// entries; 24 warps per SM, 80 registers), at 2.2 times the time its 143 MB
// take at 6.8 TB/s.
constexpr int kSpmvBatch = 4;  // 16-byte chunks of entries (and weights) in flight per lane
constexpr int kSpmvMaxThreads = 768;
constexpr int64_t kSpmvHotBlocks = 24;
constexpr int64_t kSpmvHot = 24576;

__host__ __device__ constexpr int spmv_up4(int v) { return (v + 3) & ~3; }

// x at byte offset `off` of the records: from the kept prefix or from memory.
// The two loads go to registers of their own (one register for both makes the
// second wait for the first), each lane making the one it needs; set to 0
// first, or a register that some lanes leave alone stays live around the loop.
template <bool HOT>
__device__ __forceinline__ float spmv_x(const float* __restrict__ x, uint32_t hot_at, uint32_t hot4, uint32_t off) {
  const float* p = reinterpret_cast<const float*>(reinterpret_cast<const char*>(x) + off);
  if (!HOT) return __ldg(p);
  float kept, cold;
  asm volatile("{\n\t.reg .pred p;\n\tmov.f32 %0, 0f00000000;\n\tsetp.lt.u32 p, %1, %2;\n\t@p ld.shared.f32 %0, [%3];\n\t}"
      : "=&f"(kept)
      : "r"(off), "r"(hot4), "r"(hot_at + off));
  asm volatile("{\n\t.reg .pred p;\n\tmov.f32 %0, 0f00000000;\n\tsetp.ge.u32 p, %1, %2;\n\t@p ld.global.nc.f32 %0, [%3];\n\t}"
      : "=&f"(cold)
      : "r"(off), "r"(hot4), "l"(p));
  return off < hot4 ? kept : cold;
}

__device__ __forceinline__ uint32_t word(const uint4& v, int i) { return i == 0 ? v.x : i == 1 ? v.y : i == 2 ? v.z : v.w; }

// chunks c of this lane, c0 <= c < c0 + kSpmvBatch: entries and weights (or the
// tasks whose weights they are), read once and not kept in the caches
template <bool MAP>
__device__ __forceinline__ void spmv_load(const SpmvArgs& a, int64_t i0, int lane, int c0, uint4* ev, uint4* wv) {
  const uint4* ep = reinterpret_cast<const uint4*>(a.ent + i0) + lane;
  const uint4* wp = (MAP ? reinterpret_cast<const uint4*>(a.wmap + i0) : reinterpret_cast<const uint4*>(a.w + i0)) + lane;
#pragma unroll
  for (int c = 0; c < kSpmvBatch; ++c)
    if (4 * (c0 + c) < a.u) {
      ev[c] = __ldcs(ep + 32 * (c0 + c));
      wv[c] = __ldcs(wp + 32 * (c0 + c));
    }
}

// Row totals out: four rows in flight per lane
struct SpmvRows {
  int yi_lo, n_yi, yb_lo, n_yob, fy0, n_yf;
};
__device__ __forceinline__ void spmv_write_out(const SpmvRows& d, const SpmvArgs& a, const float* ys, int lane) {
  const int ny = d.n_yi + d.n_yob + d.n_yf, own = d.n_yi + d.n_yob;
  for (int p0 = lane; p0 < ny; p0 += 4 * 32) {
    int32_t r[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int p = p0 + 32 * u;
      r[u] = p >= ny ? -1
                     : (p < d.n_yi ? d.yi_lo + p
                                   : (p < own ? d.yb_lo + (p - d.n_yi)
                                              : __ldg(a.ylist + d.fy0 + (p - own))));
    }
    if (a.yrow) {
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (r[u] >= 0) r[u] = __ldg(a.yrow + r[u]);
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int p = p0 + 32 * u;
      if (r[u] < 0) continue;
      if (p < d.n_yi)
        a.y[r[u]] = ys[p];
      else
        atomicAdd(a.y + r[u], ys[p]);
    }
  }
}

template <bool HOT, bool MAP>
__global__ void __launch_bounds__(HOT ? kSpmvMaxThreads : 256, HOT ? 1 : 3) spmv_kernel(const SpmvArgs a, int cap, int hot) {
  extern __shared__ float4 smem4[];
  __shared__ __align__(8) uint64_t bar;
  const int wi = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  float* xs = reinterpret_cast<float*>(smem4);
  float* ys = xs + (HOT ? hot : 0) + (size_t)wi * cap;
  if (HOT) {
    if (threadIdx.x == 0) {
      mbar_init(&bar, 1);
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
      mbar_arrive_tx(&bar, 4u * hot);
      bulk_load(xs, a.x, 4u * hot, &bar);
    }
    __syncthreads();
  }
  const uint32_t hot_at = HOT ? saddr(xs) : 0;
  uint32_t hot4 = 4u * hot;
  const int64_t stride = (int64_t)gridDim.x * nw;
  int64_t b = (int64_t)blockIdx.x * nw + wi;
  if (b >= a.k) return;  // warp-uniform; the warps do not synchronise from here on
  uint4 ev[kSpmvBatch], wv[kSpmvBatch];
  spmv_load<MAP>(a, 32 * (int64_t)a.u * b, lane, 0, ev, wv);
  if (HOT) {  // the entries are in flight; a copy that does not land costs speed only
    if (!mbar_wait(&bar, 0)) hot4 = 0;
  }
  // the descriptor as one word per lane (lane f holds word f), read a block
  // ahead like the row positions of the lanes' first entries
  const unsigned full = 0xffffffffu;
  auto word_of = [&](int64_t blk) { return __ldg(reinterpret_cast<const int*>(a.desc + blk) + (lane & 15)); };
  int next_word = word_of(b), next_row = __ldg(a.row0 + 32 * b + lane);
  for (; b < a.k; b += stride) {
    const int dw = next_word, row = next_row;
    if (b + stride < a.k) {
      next_word = word_of(b + stride);
      next_row = __ldg(a.row0 + 32 * (b + stride) + lane);
    }
    const int ne = __shfl_sync(full, dw, offsetof(SpmvDesc, ne) / 4);
    SpmvRows d;
    d.fy0 = __shfl_sync(full, dw, offsetof(SpmvDesc, fy0) / 4);
    d.n_yf = __shfl_sync(full, dw, offsetof(SpmvDesc, n_yf) / 4);
    if (32 * lane < d.n_yf) asm volatile("prefetch.global.L2 [%0];" ::"l"(a.ylist + d.fy0 + 32 * lane));
    const int64_t i0 = 32 * (int64_t)a.u * b;
    const int nj = min(max(ne - lane * a.u, 0), a.u);  // this lane's real entries
    const bool cont = lane > 0 && nj > 0 && !(ev[0].x & kEntRow);  // which the lane before began
    ev[0].x &= ~kEntRow;
    // the next block's lines into the L2: the loads below then miss only the L1
    if (b + stride < a.k && a.u == 4 * kSpmvBatch) {
      const char* next = lane < 16 ? reinterpret_cast<const char*>(a.ent + i0 + 32 * (int64_t)a.u * stride)
                                   : (MAP ? reinterpret_cast<const char*>(a.wmap + i0 + 32 * (int64_t)a.u * stride)
                                          : reinterpret_cast<const char*>(a.w + i0 + 32 * (int64_t)a.u * stride));
      asm volatile("prefetch.global.L2 [%0];" ::"l"(next + 128 * (lane & 15)));
    }
    // A run that ends inside the chunk goes to its row's total as it stands
    // (the first one may still lack what the lanes before summed).
    float acc = 0.f;
    float* at = ys + row;
    auto batch = [&](int c0, bool whole) {
#pragma unroll
      for (int h = 0; h < kSpmvBatch; h += 2) {  // eight entries' loads in flight, then their sums
        float v[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const uint32_t e = word(ev[h + (i >> 2)], i & 3), w = word(wv[h + (i >> 2)], i & 3);
          if (whole || 4 * (c0 + h) + i < nj) {
            const float wt = MAP ? __ldg(a.w + w) : __uint_as_float(w);
            v[i] = wt * spmv_x<HOT>(a.x, hot_at, hot4, e & ~kEntRow);
          }
        }
#pragma unroll
        for (int i = 0; i < 8; ++i)
          if (whole || 4 * (c0 + h) + i < nj) {
            if (word(ev[h + (i >> 2)], i & 3) & kEntRow) {
              *at++ = acc;
              acc = 0.f;
            }
            acc += v[i];
          }
      }
    };
    for (int c0 = 0; 4 * c0 < a.u; c0 += kSpmvBatch) {
      if (c0 > 0) spmv_load<MAP>(a, i0, lane, c0, ev, wv);
      if (ne - 31 * a.u >= 4 * (c0 + kSpmvBatch))  // every lane's batch is full
        batch(c0, true);
      else
        batch(c0, false);
    }
    const bool whole = at == ys + row;  // the chunk is one run
    // the next block's entries, in flight during the join and the write-out
    if (b + stride < a.k) spmv_load<MAP>(a, i0 + 32 * (int64_t)a.u * stride, lane, 0, ev, wv);
    // Joins the chunks' end runs: a lane's first run continues the lane
    // before's last run (cont), and a lane whose chunk is one run passes the
    // sum on (segmented inclusive scan of the last-run sums over the lanes).
    // Afterwards every row of the block has its total in ys, stored once.
    float S = acc;
    int F = !(whole && cont);  // a segment starts here
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const float Sp = __shfl_up_sync(full, S, o);
      const int Fp = __shfl_up_sync(full, F, o);
      if (lane >= o && !F) {
        S += Sp;
        F = Fp;
      }
    }
    const float S_prev = __shfl_up_sync(full, S, 1);
    const int cont_next = __shfl_down_sync(full, (int)cont, 1);
    if (!whole && cont) ys[row] += S_prev;
    if (nj > 0 && !(lane < 31 && cont_next)) *at = S;
    __syncwarp();
    d.yi_lo = __shfl_sync(full, dw, offsetof(SpmvDesc, yi_lo) / 4);
    d.n_yi = __shfl_sync(full, dw, offsetof(SpmvDesc, n_yi) / 4);
    d.yb_lo = __shfl_sync(full, dw, offsetof(SpmvDesc, yb_lo) / 4);
    d.n_yob = __shfl_sync(full, dw, offsetof(SpmvDesc, n_yob) / 4);
    spmv_write_out(d, a, ys, lane);
    __syncwarp();
  }
}

// Device entries of a schedule: one warp per block
__global__ void spmv_entries_kernel(const SpmvDesc* __restrict__ desc, int64_t k, const uint32_t* __restrict__ sent,
                                    const int32_t* __restrict__ xlist, uint32_t* __restrict__ ent,
                                    uint16_t* __restrict__ row0) {
  const int lane = threadIdx.x & 31;
  const int64_t b = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  if (b >= k) return;
  const SpmvDesc d = desc[b];
  const uint32_t* src = sent + d.i0;
  uint32_t* dst = ent + d.i0;
  for (int t = lane; t < 32 * d.u; t += 32) {
    const int j = spmv_slot(t, d.u);
    uint32_t v = 0;
    if (t < d.ne) {
      const uint32_t e = src[j], row = e >> kRowShift;
      v = 4u * (uint32_t)xlist[d.fx0 + (int)(e & kColMask)];
      if (t == 0 || src[spmv_slot(t - 1, d.u)] >> kRowShift != row) v |= kEntRow;
      if (t % d.u == 0) row0[32 * b + t / d.u] = (uint16_t)row;
    } else if (t % d.u == 0) {
      row0[32 * b + t / d.u] = 0;
    }
    dst[j] = v;
  }
}

// ------------------------------------------------------------- shard halo

// Halo sums of a shard schedule (one of several that split a schedule's
// blocks): hmap[i] is the shared id of halo vertex i here, or -1 where this
// shard does not touch it.  Pack copies the sums of the last forward edge
// kernel (the accumulator buffer before the current phase) into buf[i][D]
// (zeros for -1); unpack writes buf back after the sum over shards.
template <int D>
__global__ void halo_kernel(const FluxArgs a, const int32_t* __restrict__ hmap, int64_t nh,
                            float* __restrict__ buf, bool pack) {
  float* last = acc_buffer<D>(a, *a.phase + 2);
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < nh;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int32_t h = __ldg(hmap + i);
    float v[D];
    if (pack) {
#pragma unroll
      for (int c = 0; c < D; ++c) v[c] = 0.f;
      if (h >= 0) acc_load<D>(last, h, v);
#pragma unroll
      for (int c = 0; c < D; ++c) buf[i * D + c] = v[c];
    } else if (h >= 0) {
#pragma unroll
      for (int c = 0; c < D; ++c) v[c] = buf[i * D + c];
      acc_store<D>(last, h, v);
    }
  }
}

// ------------------------------------------------------------------- layout

// Every element of these conversions costs two dependent loads (a map entry,
// then a record or value somewhere else), so a thread takes several elements,
// a block's width apart, and has all of their loads in flight together.
constexpr int kLayoutThreads = 256;
__host__ __device__ constexpr int layout_batch(int D) { return D <= 4 ? 4 : 2; }  // vertices per thread
constexpr int kWeightBatch = 8;                               // weights per thread

// caller layout [D][n] (by data vertex) -> planar records: x read in vertex
// order (coalesced; in host memory the GPU reads it over the host link); CSR:
// every record of vertex v is written (its record and the copies of a shared
// vertex, recs[ptr[v] .. ptr[v + 1])), else the one record map[v]
template <int D, bool CSR>
__device__ __forceinline__ void state_in(int64_t tile, const int32_t* __restrict__ map, const int32_t* __restrict__ recs,
                                         int64_t n, int64_t n_rec, const float* __restrict__ x,
                                         float* __restrict__ x_lay) {
  constexpr int B = layout_batch(D);
  const int64_t v0 = tile * (B * kLayoutThreads) + threadIdx.x;
  float t[B][D];
  int32_t lo[B], hi[B];
#pragma unroll
  for (int u = 0; u < B; ++u) {
    const int64_t v = v0 + u * kLayoutThreads;
    lo[u] = v < n ? __ldg(map + v) : 0;
    hi[u] = v < n ? (CSR ? __ldg(map + v + 1) : lo[u] + 1) : 0;
#pragma unroll
    for (int c = 0; c < D; ++c) t[u][c] = v < n ? x[(size_t)c * n + v] : 0.f;
  }
#pragma unroll
  for (int u = 0; u < B; ++u)
    for (int32_t i = lo[u]; i < hi[u]; ++i) rec_store<D>(x_lay, n_rec, CSR ? __ldg(recs + i) : i, t[u]);
}

// weights: gathered into slots (perm: slot -> task, -1 unused), or read in task
// order and written to the task's two slots (-1 for none; w in host memory)
__device__ __forceinline__ void weights_gather(int64_t tile, const int32_t* __restrict__ perm, int64_t m,
                                               const float* __restrict__ w, float* __restrict__ w_lay) {
  const int64_t i0 = tile * (kWeightBatch * kLayoutThreads) + threadIdx.x;
  int32_t t[kWeightBatch];
  float v[kWeightBatch];
#pragma unroll
  for (int u = 0; u < kWeightBatch; ++u) t[u] = i0 + u * kLayoutThreads < m ? __ldg(perm + i0 + u * kLayoutThreads) : -1;
#pragma unroll
  for (int u = 0; u < kWeightBatch; ++u) v[u] = t[u] >= 0 ? __ldg(w + t[u]) : 0.f;
#pragma unroll
  for (int u = 0; u < kWeightBatch; ++u)
    if (i0 + u * kLayoutThreads < m) w_lay[i0 + u * kLayoutThreads] = v[u];
}
__device__ __forceinline__ void weights_scatter(int64_t tile, const int2* __restrict__ slots, int64_t m,
                                                const float* __restrict__ w, float* __restrict__ w_lay) {
  const int64_t i0 = tile * (kWeightBatch * kLayoutThreads) + threadIdx.x;
  int2 sl[kWeightBatch];
  float v[kWeightBatch];
#pragma unroll
  for (int u = 0; u < kWeightBatch; ++u) {
    const int64_t t = i0 + u * kLayoutThreads;
    v[u] = t < m ? w[t] : 0.f;
    sl[u] = t < m ? __ldg(slots + t) : make_int2(-1, -1);
  }
#pragma unroll
  for (int u = 0; u < kWeightBatch; ++u) {
    if (sl[u].x >= 0) w_lay[sl[u].x] = v[u];
    if (sl[u].y >= 0) w_lay[sl[u].y] = v[u];
  }
}

// A state and (W: 1 gathered, 2 scattered) the weights in one launch: the first
// `state_tiles` blocks do the state, the others the weights.
struct InputArgs {
  const int32_t *map, *recs, *wmap;
  const float *x, *w;
  float *x_lay, *w_lay;
  int64_t n, n_rec, nw, state_tiles;
};
template <int D, bool CSR, int W>
__global__ void __launch_bounds__(kLayoutThreads) inputs_kernel(const InputArgs a) {
  if (W == 0 || blockIdx.x < a.state_tiles)
    state_in<D, CSR>(blockIdx.x, a.map, a.recs, a.n, a.n_rec, a.x, a.x_lay);
  else if (W == 1)
    weights_gather(blockIdx.x - a.state_tiles, a.wmap, a.nw, a.w, a.w_lay);
  else
    weights_scatter(blockIdx.x - a.state_tiles, reinterpret_cast<const int2*>(a.wmap), a.nw, a.w, a.w_lay);
}
__global__ void __launch_bounds__(kLayoutThreads) gather_kernel(const int32_t* __restrict__ perm, int64_t m,
                                                               const float* __restrict__ w, float* __restrict__ w_lay) {
  weights_gather(blockIdx.x, perm, m, w, w_lay);
}

// planar records -> caller layout, one state or two (TWO) over the same map
template <int D, bool TWO>
__global__ void __launch_bounds__(kLayoutThreads) layout_out_kernel(const int32_t* __restrict__ rec_of, int64_t n,
                                                                   int64_t n_rec, const float* __restrict__ x_lay,
                                                                   float* __restrict__ x,
                                                                   const float* __restrict__ y_lay,
                                                                   float* __restrict__ y) {
  constexpr int B = layout_batch(D);
  const int64_t v0 = blockIdx.x * (int64_t)(B * kLayoutThreads) + threadIdx.x;
  int32_t r[B];
  float t[B][D], q[B][D];
#pragma unroll
  for (int u = 0; u < B; ++u) r[u] = v0 + u * kLayoutThreads < n ? __ldg(rec_of + v0 + u * kLayoutThreads) : -1;
#pragma unroll
  for (int u = 0; u < B; ++u)
    if (r[u] >= 0) {
      rec_load<D, true>(x_lay, n_rec, r[u], t[u]);
      if (TWO) rec_load<D, true>(y_lay, n_rec, r[u], q[u]);
    }
#pragma unroll
  for (int u = 0; u < B; ++u)
    if (r[u] >= 0) {
#pragma unroll
      for (int c = 0; c < D; ++c) {
        x[(size_t)c * n + v0 + u * kLayoutThreads] = t[u][c];
        if (TWO) y[(size_t)c * n + v0 + u * kLayoutThreads] = q[u][c];
      }
    }
}

__global__ void scatter_add_kernel(const int32_t* __restrict__ perm, int64_t m,
                                   const float* __restrict__ w_lay, float* __restrict__ w) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < m;
       i += (int64_t)gridDim.x * blockDim.x)
  {
    const int32_t t = perm[i];
    if (t >= 0) w[t] += w_lay[i];
  }
}

__global__ void gather_add_kernel(const int32_t* __restrict__ slot, int64_t m,
                                  const float* __restrict__ w_lay, float* __restrict__ w) {
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < m;
       t += (int64_t)gridDim.x * blockDim.x)
    w[t] += __ldg(w_lay + __ldg(slot + t));
}

// --------------------------------------------------------------------- cost

// One CUDA block per schedule block: bitonic sort of the block's endpoint ids
// in shared memory, then count distinct ids and mark them touched.
__global__ void cost_block_kernel(const int64_t* __restrict__ block_ptr, const int32_t* __restrict__ eu,
                                  const int32_t* __restrict__ ev, int P, uint8_t* __restrict__ touched,
                                  unsigned long long* __restrict__ loads) {
  extern __shared__ float4 smem4[];
  int32_t* key = reinterpret_cast<int32_t*>(smem4);
  const int64_t e0 = block_ptr[blockIdx.x];
  const int ne = (int)(block_ptr[blockIdx.x + 1] - e0);
  const int nk = 2 * ne;
  for (int i = threadIdx.x; i < P; i += blockDim.x)
    key[i] = i < ne ? eu[e0 + i] : i < nk ? ev[e0 + i - ne] : INT_MAX;
  __syncthreads();
  block_bitonic_sort(key, P);
  const unsigned int cnt = count_distinct_sorted(key, nk, [&](int32_t v) { touched[v] = 1; });
  block_sum_add(cnt, loads);
}

__global__ void count_flags_kernel(const uint8_t* __restrict__ f, int64_t nd,
                                   unsigned long long* __restrict__ total) {
  sum_flags(f, nd, total);
}

int grid_for(int64_t work, int tpb) {
  int64_t g = (work + tpb - 1) / tpb;
  if (g < 1) g = 1;
  if (g > 152 * 32) g = 152 * 32;
  return (int)g;
}

// Opens a kernel's dynamic shared-memory limit to the device maximum once
// (a per-kernel attribute shared by all callers); launches above 48 KB need it.
std::mutex g_smem_mu;
std::unordered_set<const void*> g_smem_opened;  // kernels whose limit is open

template <typename K>
cudaError_t allow_smem(K kernel, size_t bytes) {
  if (bytes <= 48 * 1024) return cudaSuccess;
  int dev = 0, optin = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (e != cudaSuccess) return e;
  cudaFuncAttributes fa;
  e = cudaFuncGetAttributes(&fa, kernel);
  if (e != cudaSuccess) return e;
  const int dyn_max = optin - (int)fa.sharedSizeBytes;  // minus the kernel's static shared memory
  if (bytes > (size_t)dyn_max) return cudaErrorInvalidValue;
  std::lock_guard<std::mutex> lock(g_smem_mu);
  const void* key = reinterpret_cast<const void*>(kernel);
  if (g_smem_opened.count(key)) return cudaSuccess;
  e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, dyn_max);
  if (e == cudaSuccess) g_smem_opened.insert(key);
  return e;
}

struct Scope {
  Timer* t;
  int cls;
  cudaStream_t st;
  Scope(Timer* t_, int c, cudaStream_t s) : t(t_), cls(c), st(s) {
    if (t) t->begin(cls, st);
  }
  ~Scope() {
    if (t) t->end(cls, st);
  }
};

// PDL launch of the finish (the edge kernel before it may still be draining)
template <int D>
cudaError_t fold_launch(const FluxArgs& a, float* x_out, const float* x_in, float* out, cudaStream_t st) {
  if (a.n_sh <= 0) return cudaSuccess;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid_for((a.n_copies + kFoldUnroll - 1) / kFoldUnroll, 256));
  cfg.blockDim = dim3(256);
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, bnd_update_kernel<D>, a, x_in, x_out, out);
}

template <int D>
cudaError_t flux_step_t(const FluxArgs& a, cudaStream_t st) {
  const TmaLayout L = tma_layout(a, D, false);
  const size_t smem = (size_t)L.stage_bytes;
  cudaError_t e = allow_smem(flux_fwd_kernel<D>, smem);
  if (e != cudaSuccess) return e;
  if (a.k > 0) {
    Scope sc(a.timer, T_EDGE_FWD, st);
    flux_fwd_kernel<D><<<(unsigned)a.k, a.tpb, smem, st>>>(a, L);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  return cudaSuccess;
}

template <int D, int R>
void flux_ldg_launch(const FluxArgs& a, int threads, cudaStream_t st) {
  flux_fwd_ldg_kernel<D, R><<<(unsigned)a.k, threads, 0, st>>>(a);
}

template <int D>
cudaError_t flux_step_ldg_t(const FluxArgs& a, cudaStream_t st) {
  const int R = (a.max_nsl + 31) / 32;  // slices per warp
  const int threads = 32 * std::max(1, (a.max_nsl + R - 1) / std::max(R, 1));
  if (a.k > 0) {
    Scope sc(a.timer, T_EDGE_FWD, st);
    switch (R) {
      case 0:
      case 1: flux_ldg_launch<D, 1>(a, threads, st); break;
      case 2: flux_ldg_launch<D, 2>(a, threads, st); break;
      case 3: flux_ldg_launch<D, 3>(a, threads, st); break;
      case 4: flux_ldg_launch<D, 4>(a, threads, st); break;
      default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
  }
  return cudaSuccess;
}

template <int D>
cudaError_t flux_adj_t(const FluxArgs& a, float* lam, float* gw, cudaStream_t st) {
  const TmaLayout L = tma_layout(a, D, true);
  const size_t smem = (size_t)L.stage_bytes;
  cudaError_t e = allow_smem(flux_adj_kernel<D>, smem);
  if (e != cudaSuccess) return e;
  if (a.k > 0) {
    Scope sc(a.timer, T_EDGE_ADJ, st);
    flux_adj_kernel<D><<<(unsigned)a.k, a.tpb, smem, st>>>(a, lam, gw, L);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace

cudaError_t flux_step(const FluxArgs& a, int D, cudaStream_t st) {
  switch (D) {
    case 1: return flux_step_t<1>(a, st);
    case 2: return flux_step_t<2>(a, st);
    case 3: return flux_step_t<3>(a, st);
    case 4: return flux_step_t<4>(a, st);
    case 5: return flux_step_t<5>(a, st);
    case 6: return flux_step_t<6>(a, st);
    case 7: return flux_step_t<7>(a, st);
    case 8: return flux_step_t<8>(a, st);
  }
  return cudaErrorInvalidValue;
}

cudaError_t flux_step_ldg(const FluxArgs& a, int D, cudaStream_t st) {
  switch (D) {
    case 1: return flux_step_ldg_t<1>(a, st);
    case 2: return flux_step_ldg_t<2>(a, st);
    case 3: return flux_step_ldg_t<3>(a, st);
    case 4: return flux_step_ldg_t<4>(a, st);
    case 5: return flux_step_ldg_t<5>(a, st);
    case 6: return flux_step_ldg_t<6>(a, st);
    case 7: return flux_step_ldg_t<7>(a, st);
    case 8: return flux_step_ldg_t<8>(a, st);
  }
  return cudaErrorInvalidValue;
}

#define EP_DISPATCH_D(D, CALL) \
  switch (D) {                    \
    case 1: CALL(1); break;       \
    case 2: CALL(2); break;       \
    case 3: CALL(3); break;       \
    case 4: CALL(4); break;       \
    case 5: CALL(5); break;       \
    case 6: CALL(6); break;       \
    case 7: CALL(7); break;       \
    case 8: CALL(8); break;       \
    default: return cudaErrorInvalidValue; \
  }

// shared-vertex fold after a pipelined edge kernel
cudaError_t bnd_update(const FluxArgs& a, int D, float* x_out, const float* x_in, float* out,
                       cudaStream_t st) {
  if (a.n_sh <= 0) return cudaSuccess;
  Scope sc(a.timer, T_BND, st);
#define EP_BU(DD) return fold_launch<DD>(a, x_out, x_in, out, st)
  switch (D) {
    case 1: EP_BU(1);
    case 2: EP_BU(2);
    case 3: EP_BU(3);
    case 4: EP_BU(4);
    case 5: EP_BU(5);
    case 6: EP_BU(6);
    case 7: EP_BU(7);
    case 8: EP_BU(8);
  }
#undef EP_BU
  return cudaErrorInvalidValue;
}

TmaLayout tma_layout(const FluxArgs& a, int D, bool adjoint) {
  auto up = [](int64_t x, int64_t m) { return (x + m - 1) / m * m; };
  TmaLayout L = {};
  L.npos = (int)up(a.max_nv, 4);
  const int64_t xb = (int64_t)D * L.npos * 4;
  L.off_lam = (int)xb;
  L.off_sidx = (int)(L.off_lam + (adjoint ? xb : 0));
  L.off_w = (int)(L.off_sidx + up((int64_t)a.max_nslot * 2, 16));
  L.off_sid = (int)(L.off_w + (int64_t)a.max_nslot * 4);
  L.off_soff = (int)(L.off_sid + up((int64_t)a.max_nsh * 4, 16));
  L.off_desc = (int)(L.off_soff + up((int64_t)(a.max_nsl + 1) * 2, 16));
  L.stage_bytes = (int)up(L.off_desc + (int64_t)sizeof(FluxDesc), 128);
  L.stages = 1;
  L.stall = -1;
  return L;
}

cudaError_t flux_adjoint_step(const FluxArgs& a, int D, float* lam, float* gw, cudaStream_t st) {
  switch (D) {
    case 1: return flux_adj_t<1>(a, lam, gw, st);
    case 2: return flux_adj_t<2>(a, lam, gw, st);
    case 3: return flux_adj_t<3>(a, lam, gw, st);
    case 4: return flux_adj_t<4>(a, lam, gw, st);
    case 5: return flux_adj_t<5>(a, lam, gw, st);
    case 6: return flux_adj_t<6>(a, lam, gw, st);
    case 7: return flux_adj_t<7>(a, lam, gw, st);
    case 8: return flux_adj_t<8>(a, lam, gw, st);
  }
  return cudaErrorInvalidValue;
}

size_t flux_block_smem(const FluxArgs& a, int D, bool adjoint) {
  return (size_t)tma_layout(a, D, adjoint).stage_bytes;
}

SpmvPlan spmv_plan(const SpmvArgs& a, int smem_optin, int sms) {
  SpmvPlan P = {};
  P.cap = spmv_up4(a.max_ny);
  const size_t per_warp = (size_t)P.cap * sizeof(float), limit = (size_t)smem_optin - 1024;
  if (per_warp > limit) return P;
  // Columns are kept where an SM has at least kSpmvHotBlocks blocks of 512
  // entries to share them.  Kept against not, us: scale 17 (25 blocks an SM)
  // partitioned 15.5 / 16.1, CSR 13.9 / 13.6; scale 16 (12) 11.3 / 11.3 and
  // 10.1 / 9.5; scale 15 (6) 9.6 / 9.2 and 10.3 / 9.1; scale 18 31.5 / 39.
  // The SM's blocks are dealt to up to 24 warps in rounds of equal size.
  const int64_t per_sm = (a.k + sms - 1) / sms;
  if (!a.readonly && per_sm * a.u >= 16 * kSpmvHotBlocks) {
    const int most = (int)std::min<int64_t>(kSpmvMaxThreads / 32, std::max<int64_t>(1, (int64_t)(limit / 2 / per_warp)));
    const int64_t rounds = (per_sm + most - 1) / most;
    P.wpb = (int)((per_sm + rounds - 1) / rounds);
    P.grid = std::min<int64_t>(sms, (a.k + P.wpb - 1) / P.wpb);
    // whole 16-byte pieces of x: none of a vector of fewer than 4 elements
    P.hot = (int)std::min<int64_t>(std::min<int64_t>(a.n, kSpmvHot) / 4 * 4, (int64_t)((limit - P.wpb * per_warp) / 16 * 4));
    P.smem = P.wpb * per_warp + (size_t)P.hot * sizeof(float);
    if (P.hot > 0) return P;
  }
  int wpb = std::max(1, std::min(8, a.tpb / 32));
  while (wpb > 1 && per_warp * wpb > (size_t)48 * 1024) --wpb;  // room for several CUDA blocks per SM
  P.wpb = wpb;
  P.grid = (a.k + wpb - 1) / wpb;
  P.smem = per_warp * wpb;
  return P;
}

cudaError_t spmv(const SpmvArgs& a, cudaStream_t st) {
  int dev = 0, optin = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  const SpmvPlan P = spmv_plan(a, optin, sms);
  if (P.wpb == 0) return cudaErrorInvalidValue;
  using Kernel = void (*)(const SpmvArgs, int, int);
  const Kernel kern = P.hot ? (a.wmap ? (Kernel)spmv_kernel<true, true> : (Kernel)spmv_kernel<true, false>)
                            : (a.wmap ? (Kernel)spmv_kernel<false, true> : (Kernel)spmv_kernel<false, false>);
  if ((e = allow_smem(kern, P.smem)) != cudaSuccess) return e;
  // rows that several blocks add to (all rows, where records are not in order)
  if (a.yrow)
    e = cudaMemsetAsync(a.y, 0, (size_t)a.n * sizeof(float), st);
  else if (a.ny_zero > 0)
    e = cudaMemsetAsync(a.y + a.ny_int, 0, (size_t)a.ny_zero * sizeof(float), st);
  if (e != cudaSuccess) return e;
  if (a.k <= 0) return cudaSuccess;
  Scope sc(a.timer, T_SPMV, st);
  kern<<<(unsigned)P.grid, 32 * P.wpb, P.smem, st>>>(a, P.cap, P.hot);
  return cudaGetLastError();
}

cudaError_t spmv_entries(const SpmvDesc* desc, int64_t k, const uint32_t* sent, const int32_t* xlist, uint32_t* ent,
                         uint16_t* row0, cudaStream_t st) {
  spmv_entries_kernel<<<(unsigned)((k + 7) / 8), 256, 0, st>>>(desc, k, sent, xlist, ent, row0);
  return cudaGetLastError();
}

cudaError_t halo_move(const FluxArgs& a, int D, const int32_t* hmap, int64_t nh, float* buf, bool pack,
                      cudaStream_t st) {
  if (nh <= 0) return cudaSuccess;
  const int g = grid_for(nh, 256);
#define EP_HALO(DD) halo_kernel<DD><<<g, 256, 0, st>>>(a, hmap, nh, buf, pack)
  EP_DISPATCH_D(D, EP_HALO)
#undef EP_HALO
  return cudaGetLastError();
}

namespace {
template <int D>
void inputs_launch(const InputArgs& a, bool csr, int w, unsigned grid, cudaStream_t st) {
  using Kernel = void (*)(const InputArgs);
  const Kernel k = csr ? (w == 0 ? (Kernel)inputs_kernel<D, true, 0> : w == 1 ? (Kernel)inputs_kernel<D, true, 1>
                                                                              : (Kernel)inputs_kernel<D, true, 2>)
                       : (w == 0 ? (Kernel)inputs_kernel<D, false, 0> : w == 1 ? (Kernel)inputs_kernel<D, false, 1>
                                                                               : (Kernel)inputs_kernel<D, false, 2>);
  k<<<grid, kLayoutThreads, 0, st>>>(a);
}
int64_t tiles(int64_t n, int per_thread) {
  return std::max<int64_t>(1, (n + (int64_t)per_thread * kLayoutThreads - 1) / ((int64_t)per_thread * kLayoutThreads));
}
}  // namespace

cudaError_t inputs(const LayoutIn& in, int D, cudaStream_t st, Timer* t) {
  Scope sc(t, T_LAYOUT, st);
  InputArgs a;
  a.map = in.map, a.recs = in.recs, a.x = in.x, a.x_lay = in.x_lay, a.n = in.n, a.n_rec = in.n_rec;
  a.wmap = in.wmap, a.w = in.w, a.w_lay = in.w_lay, a.nw = in.nw;
  a.state_tiles = tiles(in.n, layout_batch(D));
  const int w = in.w_lay == nullptr ? 0 : in.scatter ? 2 : 1;
  const unsigned g = (unsigned)(a.state_tiles + (w ? tiles(in.nw, kWeightBatch) : 0));
#define EP_LIN(DD) inputs_launch<DD>(a, in.recs != nullptr, w, g, st)
  EP_DISPATCH_D(D, EP_LIN)
#undef EP_LIN
  return cudaGetLastError();
}

cudaError_t layout_out(const int32_t* rec_of, int64_t n, int64_t n_rec, int D, const float* x_lay, float* x,
                       const float* y_lay, float* y, cudaStream_t st, Timer* t) {
  Scope sc(t, T_LAYOUT, st);
  const unsigned g = (unsigned)tiles(n, layout_batch(D));
  if (y) {
#define EP_LOUT(DD) layout_out_kernel<DD, true><<<g, kLayoutThreads, 0, st>>>(rec_of, n, n_rec, x_lay, x, y_lay, y)
    EP_DISPATCH_D(D, EP_LOUT)
#undef EP_LOUT
  } else {
#define EP_LOUT(DD) layout_out_kernel<DD, false><<<g, kLayoutThreads, 0, st>>>(rec_of, n, n_rec, x_lay, x, nullptr, nullptr)
    EP_DISPATCH_D(D, EP_LOUT)
#undef EP_LOUT
  }
  return cudaGetLastError();
}

cudaError_t gather(const int32_t* perm, int64_t m, const float* w, float* w_lay, cudaStream_t st,
                   Timer* t) {
  Scope sc(t, T_LAYOUT, st);
  gather_kernel<<<(unsigned)tiles(m, kWeightBatch), kLayoutThreads, 0, st>>>(perm, m, w, w_lay);
  return cudaGetLastError();
}

cudaError_t scatter_add(const int32_t* perm, int64_t m, const float* w_lay, float* w, cudaStream_t st,
                        Timer* t) {
  Scope sc(t, T_LAYOUT, st);
  scatter_add_kernel<<<grid_for(m, 256), 256, 0, st>>>(perm, m, w_lay, w);
  return cudaGetLastError();
}

cudaError_t gather_add(const int32_t* slot, int64_t m, const float* w_lay, float* w, cudaStream_t st,
                       Timer* t) {
  Scope sc(t, T_LAYOUT, st);
  gather_add_kernel<<<grid_for(m, 256), 256, 0, st>>>(slot, m, w_lay, w);
  return cudaGetLastError();
}

cudaError_t cost(const CostArgs& a, cudaStream_t st) {
  int P = 2;
  while (P < 2 * a.max_ne) P <<= 1;
  const size_t smem = (size_t)P * sizeof(int32_t);
  cudaError_t e = allow_smem(cost_block_kernel, smem);
  if (e != cudaSuccess) return e;
  e = cudaMemsetAsync(a.touched, 0, (size_t)a.nd, st);
  if (e != cudaSuccess) return e;
  e = cudaMemsetAsync(a.counters, 0, 2 * sizeof(unsigned long long), st);
  if (e != cudaSuccess) return e;
  const int tpb = P >= 1024 ? 1024 : (P < 32 ? 32 : P);  // whole warps for the shuffles
  Scope sc(a.timer, T_COST, st);
  cost_block_kernel<<<(unsigned)a.k, tpb, smem, st>>>(a.block_ptr, a.eu, a.ev, P, a.touched, a.counters);
  count_flags_kernel<<<grid_for(a.nd, 256), 256, 0, st>>>(a.touched, a.nd, a.counters + 1);
  return cudaGetLastError();
}

}  // namespace dev
}  // namespace ep
