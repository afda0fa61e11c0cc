// march.h -- layout of the resident run kernels (internal to libepcache).
//
// A run of several explicit steps keeps the whole mesh on the chip: the data
// vertices, in the order of first appearance over the schedule's blocks
// (cpack, Section 4.1, the locality the partition made), are cut into one
// part per CUDA block, and vertices that have most of their neighbours in
// another part then move there (march.cpp, smooth_parts).  A part owns its
// vertices: it computes the whole flux of each of them (pull form, every task at
// both endpoints, as the step kernels do), so nothing is accumulated across
// parts; what a part needs from the others is the value of the neighbours it
// does not own (its halo).
#pragma once

#include <cstdint>
#include <string>
#include <vector>

#include "internal.h"

namespace ep {

// One part.  Positions [0, own): its vertices, the boundary ones (in some
// other part's halo) first, each class by descending degree; positions
// [hbase, hbase + nh): the halo, ascending by record; both but for swaps inside
// the octets of eight positions, which even out the banks (banks.h).  Position p
// is the state record lo + p, own or halo, so a part's image is one run of
// records; halo[h0 + j] is the record where halo position j is its owner's.
// Slices of 32 positions are dealt to `warps` warps, slice j to warp j % warps;
// the pair columns (32 lanes of two slots each) of one warp's slices follow each
// other, so that a warp reads its columns as one stream: warp v's start at
// column s0 + tab[q0 + v], and slice j has tab[q0 + warps + j] of them.  Entry
// pair 32 * column + lane holds two 16-bit entries (position of the other endpoint,
// kSlotSrc on the task's first endpoint) and two weights.  An unused slot has
// weight 0 and names the lane's own position or one of its neighbours, whichever
// costs the fewest bank conflicts: its term is zero whenever the lane's used
// slots are finite.  A lane of no vertex names what another lane reads.
struct MarchPart {
  int32_t lo, own, nb, nsl;
  int32_t hbase, nh, h0, q0;
  int32_t s0, ncol;  // pair columns [s0, s0 + ncol)
  int32_t pad[6];
};
static_assert(sizeof(MarchPart) == 64, "MarchPart layout");

// Columns past the last one that a stream's read-ahead may touch.
constexpr int kMarchAhead = 2;

struct MarchLayout {
  int32_t parts = 0, warps = 0;
  int64_t n_rec = 0;               // records per plane of a state (multiple of 4)
  int64_t n_run = 0;               // records [0, n_run) are the parts' images
  int64_t n_col = 0;               // pair columns in all, kMarchAhead unused ones included
  std::vector<MarchPart> part;
  std::vector<int32_t> rec_of;     // data vertex -> its own record (untouched vertices after the parts)
  std::vector<int32_t> halo;       // owners' records
  std::vector<uint16_t> tab;       // stream starts and slice columns, each part's padded to 8
  std::vector<uint32_t> ent;       // entry pairs
  std::vector<int32_t> wmap;       // weight slot (64 column + 2 lane + which) -> task, -1 unused
  std::vector<int32_t> gslot;      // task -> weight slot at its first endpoint
  int32_t max_pos = 0, max_col = 0, max_nsl = 0;
};

// Builds the layout for at most `max_parts` parts.  False when the graph does
// not suit it (a vertex of very large degree, whose slots one lane would walk
// alone, or more positions in a part than an entry can name).
bool build_march(const HostSchedule& s, int32_t max_parts, int threads, MarchLayout& out);

}  // namespace ep
