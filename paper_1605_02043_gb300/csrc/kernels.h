// kernels.h -- launchers of the device code (internal to libepcache).
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

#include "internal.h"
#include "march.h"

namespace ep {
namespace dev {

// Optional per-launch timing hook (events recorded on the launch stream).
struct Timer {
  virtual void begin(int cls, cudaStream_t st) = 0;
  virtual void end(int cls, cudaStream_t st) = 0;
  virtual ~Timer() = default;
};
enum { T_EDGE_FWD = 0, T_BND = 1, T_EDGE_ADJ = 2, T_SPMV = 3, T_LAYOUT = 4, T_COST = 5 };

struct FluxArgs {
  const FluxDesc* desc;
  int64_t k;             // kernel blocks
  const uint16_t* sidx;  // slots
  const uint16_t* soff;  // slice offsets
  const int32_t* sid;    // shared ids of the shared positions
  const float* w;        // task weights in slot layout
  const float* x_in;     // state in schedule layout (planar, n_rec records)
  float* x_out;          // may equal x_in
  float* bacc;           // 3 x n_sh accumulator records (acc_stride(D) floats each) of this kind
  int* phase;            // accumulator phase of this kind (0..2)
  int* done;             // CUDA blocks finished (the last one advances the phase)
  float* out;            // flux in schedule layout or nullptr
  const int32_t* fold_rec;  // every copy of a shared vertex: its record and shared id
  const int32_t* fold_sid;
  int64_t n_copies;
  int64_t n_rec, n_sh;
  float tau;
  int32_t max_nv, max_nslot, max_nsh, max_nsl;
  int tpb;
  Timer* timer;
};

struct SpmvArgs {
  const SpmvDesc* desc;
  int64_t k;
  const int32_t* ylist;
  const uint32_t* ent;     // device entries (kEntRow | x record)
  const uint16_t* row0;    // row position of every lane's first entry, 32 per block
  const float* w;          // weight layout (one weight per entry, same index), or
  const int32_t* wmap;     // task weights read through this map (slot -> task)
  const float* x;          // x records, the most used first
  float* y;                // y records; the shared ones are zeroed first
  const int32_t* yrow;     // y record -> row: results straight to the caller's rows, or nullptr
  int64_t n, ny_int, ny_zero;
  int32_t max_ny;
  int32_t u;               // entries per lane (every block's runs: 32 u slots)
  int tpb;                 // threads per CUDA block where no columns are kept
  bool readonly = false;   // no columns kept: x read through the read-only cache
  Timer* timer;
};

struct CostArgs {
  const int64_t* block_ptr;
  int64_t k;
  const int32_t* eu;  // endpoint ids in schedule order
  const int32_t* ev;
  int32_t max_ne;
  uint8_t* touched;   // nd bytes of workspace
  int64_t nd;
  unsigned long long* counters;  // [0] loads, [1] touched
  Timer* timer;
};

// Persistent pipelined kernels (flux_tma.cu): per-stage shared-memory layout
// (byte offsets, all multiples of 16) and launch plan.
constexpr int kMaxStages = 8;
// fix-up warps of the pipelined flux kernels (warps 1..kFixupWarps; one
// producer warp and the consumer warps besides)
constexpr int kFixupWarps = 2;
struct TmaLayout {
  int npos;  // positions per state plane (multiple of 4)
  int off_lam, off_sidx, off_w, off_sid, off_soff, off_desc;
  int stage_bytes;
  int stages;
  int stall;  // test hook: leave the stage of this block index unfilled (-1: off)
};
struct TmaPlan {
  TmaLayout L;
  int grid, threads, per_sm;
  size_t smem;
  int* err;  // error word (bit 0: a "full" wait expired, bit 1: an "empty" wait expired)
  bool fits = true;  // false: two stages exceed shared memory; use the one-block kernel
};
// bytes of one stage (state copies: 1 forward, 2 adjoint) and its layout
TmaLayout tma_layout(const FluxArgs& a, int D, bool adjoint);
cudaError_t flux_fwd_tma(const FluxArgs& a, const TmaPlan& P, int D, cudaStream_t st);
cudaError_t flux_adj_tma(const FluxArgs& a, const TmaPlan& P, int D, float* lam, float* gw,
                         cudaStream_t st);
const void* flux_tma_kernel_ptr(int D, bool adjoint);

// Resident runs of several steps (march.cu): one CUDA block per part.
struct MarchArgs {
  const MarchPart* part;
  const int32_t* halo;
  const uint16_t* tab;
  const uint32_t* ent;
  const float* w;      // weights in the layout's slots
  const float* x_in;   // planar state of n_rec records, the owners' ones written
  float* x_out;        // may equal x_in when steps > 1
  float* out;          // flux of the last step, or nullptr
  float* ckpt;         // images of the states before steps 0, every, 2 every, ...; or nullptr
  const float* lam_in; // gradient: cotangent in and out, images between two
  float* lam_out;      // checkpoints (every - 1), weight gradient slots (tasks' first endpoints)
  float* hist;
  float* gw;
  float* ex;           // 2 x n_rec exchange records (ex_chunks(D) chunks)
  uint32_t* flag;      // steps published so far by every part
  int* err;
  int64_t n_rec;
  int every, steps;
  float tau;
  int stall;           // test hook: part 0 leaves after publishing this many steps (-1: off)
  int warps, npos, off_lam, off_tab, off_ent, off_w;
  uint32_t hold_cols, tmem_cols;
};
// 16-byte chunks of one exchange record: three components and a tag each
__host__ __device__ constexpr int ex_chunks(int D) { return (D + 2) / 3; }
struct MarchSizes {
  int32_t parts, warps, max_pos, max_col, max_nsl;
};
struct MarchPlan {
  int parts;  // 0: does not fit
  int threads, warps, npos, off_lam, off_tab, off_ent, off_w, hold_cols, tmem_cols;
  bool resident;  // slots and weights stay in shared memory too
  bool wide;      // the variant with more threads and fewer registers
  size_t smem;
};
// grad: the reverse sweep (state and cotangent on the chip), else the forward run
MarchPlan march_plan(const MarchSizes& z, int D, bool grad, int smem_max);
const void* march_kernel_ptr(const MarchPlan& P, int D, bool grad);
cudaError_t march_run(const MarchArgs& a, const MarchPlan& P, int D, bool grad, cudaStream_t st);

cudaError_t flux_step(const FluxArgs& a, int D, cudaStream_t st);
// read-only-cache variant (no staging); needs max_np <= 4096
cudaError_t flux_step_ldg(const FluxArgs& a, int D, cudaStream_t st);
// finish of a pending state: every copy r of shared vertex h becomes
// x_out[r] = x_in[r] + tau * prev[h]; out[r] (if not null) = prev[h]
// (flux_common.cuh: the accumulator rotation)
cudaError_t bnd_update(const FluxArgs& a, int D, float* x_out, const float* x_in, float* out,
                       cudaStream_t st);
cudaError_t flux_adjoint_step(const FluxArgs& a, int D, float* lam, float* gw, cudaStream_t st);
cudaError_t spmv(const SpmvArgs& a, cudaStream_t st);
// shared memory the one-block kernels stage for the schedule's largest block
size_t flux_block_smem(const FluxArgs& a, int D, bool adjoint);
// SpMV launch shape; 0 warps when one warp's row totals do not fit
struct SpmvPlan {
  int wpb;       // warps per CUDA block (0: does not fit)
  int cap;       // floats of a warp's row totals
  int hot;       // x records kept in shared memory
  int64_t grid;
  size_t smem;   // dynamic shared memory per CUDA block
};
SpmvPlan spmv_plan(const SpmvArgs& a, int smem_optin, int sms);
// device entries of a schedule from its host entries and x lists
cudaError_t spmv_entries(const SpmvDesc* desc, int64_t k, const uint32_t* sent, const int32_t* xlist, uint32_t* ent,
                         uint16_t* row0, cudaStream_t st);
// planar records -> caller layout, one state (y null) or two over the same map
cudaError_t layout_out(const int32_t* rec_of, int64_t n, int64_t n_rec, int D, const float* x_lay, float* x,
                       const float* y_lay, float* y, cudaStream_t st, Timer* t);
// halo sums of a shard schedule (forward kind): pack the last edge kernel's
// sums of halo vertices i (shared id hmap[i], -1: not here) into buf[i][D], or
// unpack buf into them
cudaError_t halo_move(const FluxArgs& a, int D, const int32_t* hmap, int64_t nh, float* buf, bool pack,
                      cudaStream_t st);
// Inputs into a layout, a state and (w_lay not null) the weights in one launch.
// State, in vertex order: into the record map[v], or with recs into every record
// recs[map[v] .. map[v + 1]).  Weights: w_lay[i] = w[wmap[i]] for i < nw (0
// where negative), or with scatter w read in task order and written
// to the slots wmap[2 t] and wmap[2 t + 1] (-1 for none; w in host memory).
struct LayoutIn {
  const int32_t* map = nullptr;
  const int32_t* recs = nullptr;
  int64_t n = 0, n_rec = 0;
  const float* x = nullptr;
  float* x_lay = nullptr;
  const int32_t* wmap = nullptr;
  int64_t nw = 0;
  const float* w = nullptr;
  float* w_lay = nullptr;
  bool scatter = false;
};
cudaError_t inputs(const LayoutIn& in, int D, cudaStream_t st, Timer* t);
cudaError_t gather(const int32_t* perm, int64_t m, const float* w, float* w_lay, cudaStream_t st,
                   Timer* t);
cudaError_t scatter_add(const int32_t* perm, int64_t m, const float* w_lay, float* w, cudaStream_t st,
                        Timer* t);
// w[t] += w_lay[slot[t]] for t < m
cudaError_t gather_add(const int32_t* slot, int64_t m, const float* w_lay, float* w, cudaStream_t st,
                       Timer* t);
cudaError_t cost(const CostArgs& a, cudaStream_t st);

}  // namespace dev
}  // namespace ep
