// banks.h -- placing the slots of a slice by shared-memory bank (host side;
// used by the layouts of the step kernels and of the resident runs).
#pragma once

#include <algorithm>
#include <atomic>
#include <cstdint>
#include <new>
#include <system_error>
#include <thread>
#include <utility>
#include <vector>

namespace ep {

// f(i) for i < n on up to `threads` host threads (fewer where no more can be
// started).  Memory running out in one of them is thrown here.
template <typename F>
void parallel_for(int64_t n, int threads, F f) {
  threads = (int)std::max<int64_t>(1, std::min<int64_t>(threads, n));
  std::atomic<int64_t> next{0};
  std::atomic<bool> failed{false};
  auto work = [&] {
    try {
      for (int64_t i; !failed && (i = next.fetch_add(1)) < n;) f(i);
    } catch (const std::bad_alloc&) {
      failed = true;
    }
  };
  std::vector<std::thread> pool;
  pool.reserve(threads);
  try {
    for (int t = 1; t < threads; ++t) pool.emplace_back(work);
  } catch (const std::system_error&) {
  }
  work();
  for (auto& th : pool) th.join();
  if (failed) throw std::bad_alloc();
}

struct SlotEntry {
  int32_t o;  // position of the other endpoint
  int32_t e;  // task
  bool src;   // source side of the task (owns its weight-gradient element)
};

// Shared-memory banks.  A column of a slice is one load per plane: a 16-byte
// load is served 8 lanes at a time, each record covering the 4 banks of its
// position mod 8; a 4-byte load 32 lanes at a time, position mod 32.  Two
// things are free: the order of the 8 vertices of an octet of positions (the
// residues its neighbours see), and which column a slot goes to.  Both are
// chosen here; greedy columns alone left 8.3 wavefronts per 16-byte column on
// the 1M-point mesh (4 is the least), 5.4 now; the gathers were what a step of
// a resident run waited for (11 us of 14, 8.4 now), and a third of the step
// kernels' shared-memory wavefronts were conflicts.

// Residues: swaps inside the octets of [lo, hi) (lo aligned to 8; positions
// below `keep` and those from it on do not mix) that even out, for every reading
// octet, how many of its slots fall on each residue (sum of squares).  who[p -
// lo]: the vertex at position p (negative: none); its slots' octets are oct[ptr[v]
// .. ptr[v + 1]); cnt: [octet][8].
inline void even_residues(int32_t lo, int32_t hi, int32_t keep, const std::vector<int32_t>& ptr, const std::vector<int32_t>& oct,
                   std::vector<int32_t>& cnt, std::vector<int32_t>& who) {
  auto cost = [&](int32_t v, int from, int to) {  // half the change when v's residue moves
    int32_t c = 0;
    for (int32_t i = ptr[v]; i < ptr[v + 1]; ++i) {
      const int32_t* n = &cnt[8 * (size_t)oct[i]];
      c += 1 + n[to] - n[from];
    }
    return c;
  };
  auto move = [&](int32_t v, int from, int to) {
    for (int32_t i = ptr[v]; i < ptr[v + 1]; ++i) {
      int32_t* n = &cnt[8 * (size_t)oct[i]];
      --n[from], ++n[to];
    }
  };
  bool moved = true;
  for (int pass = 0; pass < 2 && moved; ++pass) {
    moved = false;
    for (int32_t o = lo; o < hi; o += 8)
      for (int32_t i = o; i < std::min(hi, o + 8); ++i)
        for (int32_t j = i + 1; j < std::min(hi, o + 8); ++j) {
          int32_t &a = who[i - lo], &b = who[j - lo];
          if ((i < keep) != (j < keep) || a < 0 || b < 0) continue;
          // (an octet that reads both counts as worse than it is)
          if (cost(a, i & 7, j & 7) + cost(b, j & 7, i & 7) >= 0) continue;
          move(a, i & 7, j & 7);
          move(b, j & 7, i & 7);
          std::swap(a, b);
          moved = true;
        }
  }
}

// Columns of one octet: lane l's entries (n[l] <= K of them, residues in
// res[l]) get different columns, and entries of one residue different columns
// too as far as there are no more than K of them: an edge colouring of the
// bipartite lane-residue graph, by alternating paths (Koenig).  col[l][i]
// receives the column of entry i.
// The search is quadratic in K: past kColourMost columns (a vertex in that many
// tasks of one block) entries keep their order.
constexpr int32_t kColourMost = 96;
struct OctetColumns {
  std::vector<int16_t> lane_at, res_at;  // [8][K]: entry of a lane / lane of a residue in a column
  std::vector<uint32_t> used, mine;      // spread_slice's scratch
  std::vector<uint8_t> res[8], taken;
  std::vector<int16_t> col[8];
  std::vector<int32_t> to;
  void in_order(const int32_t* n, int32_t K, int16_t* const* col) {
    lane_at.assign(8 * (size_t)K, -1);
    for (int l = 0; l < 8; ++l)
      for (int32_t i = 0; i < n[l]; ++i) lane_at[l * K + i] = col[l][i] = (int16_t)i;
  }
  void run(const int32_t* n, const uint8_t* const* res, int32_t K, int16_t* const* col) {
    lane_at.assign(8 * (size_t)K, -1);
    res_at.assign(8 * (size_t)K, -1);
    for (int l = 0; l < 8; ++l)
      for (int32_t i = 0; i < n[l]; ++i) {
        const int r = res[l][i];
        int32_t a = -1, b = -1, both = -1;
        for (int32_t c = 0; c < K && both < 0; ++c) {
          const bool fl = lane_at[l * K + c] < 0, fr = res_at[r * K + c] < 0;
          if (fl && fr) both = c;
          if (fl && a < 0) a = c;
          if (fr && b < 0) b = c;
        }
        if (both < 0 && b >= 0) {  // a is free at the lane, b at the residue: swap a and b along the path from r
          int rr = r;
          const int32_t x = a, y = b;
          int path_l[8], n_path = 0;  // residue -x- lane -y- residue -x- ...
          while (n_path < 8) {
            const int ll = res_at[rr * K + x];
            if (ll < 0) break;
            path_l[n_path++] = ll;
            const int16_t e2 = lane_at[ll * K + y];
            if (e2 < 0) break;
            rr = res[ll][e2];
            if (res_at[rr * K + y] != ll) break;  // an overflowing entry ends the path
          }
          auto mark = [&](int k, bool on) {
            const int ll = path_l[k];
            for (int32_t c : {x, y}) {
              const int16_t e2 = lane_at[ll * K + c];
              if (e2 < 0) continue;
              int16_t& at = res_at[res[ll][e2] * K + c];
              if (on ? at < 0 : at == ll) at = on ? (int16_t)ll : (int16_t)-1;
            }
          };
          for (int k = 0; k < n_path; ++k) mark(k, false);
          for (int k = 0; k < n_path; ++k) std::swap(lane_at[path_l[k] * K + x], lane_at[path_l[k] * K + y]);
          for (int k = 0; k < n_path; ++k) mark(k, true);
          both = a;
        }
        const int32_t c = both >= 0 ? both : a;
        lane_at[l * K + c] = (int16_t)i;
        if (res_at[r * K + c] < 0) res_at[r * K + c] = (int16_t)l;
      }
    for (int l = 0; l < 8; ++l)
      for (int32_t c = 0; c < K; ++c)
        if (lane_at[l * K + c] >= 0) col[l][lane_at[l * K + c]] = (int16_t)c;
  }
};

// The slots of one slice: lane l's entries ents[lo[l] .. hi[l]) over K columns,
// octet by octet; an octet's columns are then ordered so that the four octets'
// positions mod 32 differ where they can.  pad(lane, read, score) names the
// position of an unused slot: read is a position that a lane of the octet reads
// in this column (-1: none), score(o) is 0 where o costs no extra wavefront.
// put(column, lane, position, entry or null).
template <typename Pad, typename Put>
void spread_slice(const std::vector<SlotEntry>& ents, const int32_t* lo, const int32_t* hi, int32_t K, OctetColumns& oc,
                  Pad pad, Put put) {
  std::vector<uint32_t>&used = oc.used, &mine = oc.mine;
  used.assign(K, 0);  // residues mod 32 per final column
  std::vector<uint8_t>* res = oc.res;
  std::vector<int16_t>* col = oc.col;
  for (int g = 0; g < 4; ++g) {
    int32_t n[8];
    const uint8_t* rp[8];
    int16_t* cp[8];
    mine.assign(K, 0);
    for (int l = 0; l < 8; ++l) {
      const int L = 8 * g + l;
      n[l] = hi[L] - lo[L];
      res[l].resize(n[l]);
      col[l].resize(n[l]);
      for (int32_t i = 0; i < n[l]; ++i) res[l][i] = (uint8_t)(ents[lo[L] + i].o & 7);
      rp[l] = res[l].data();
      cp[l] = col[l].data();
    }
    if (K <= kColourMost)
      oc.run(n, rp, K, cp);
    else
      oc.in_order(n, K, cp);
    for (int l = 0; l < 8; ++l)
      for (int32_t i = 0; i < n[l]; ++i) mine[col[l][i]] |= 1u << (ents[lo[8 * g + l] + i].o & 31);
    // each of this octet's columns to the final column it clashes least with
    std::vector<int32_t>& to = oc.to;
    std::vector<uint8_t>& taken = oc.taken;
    to.assign(K, -1);
    taken.assign(K, 0);
    for (int32_t c = 0; c < K; ++c) {
      if (K > kColourMost) {
        to[c] = c;
        continue;
      }
      int32_t best = -1, bs = 64;
      for (int32_t f = 0; f < K; ++f) {
        if (taken[f]) continue;
        const int sc = __builtin_popcount(used[f] & mine[c]);
        if (sc < bs) best = f, bs = sc;
      }
      to[c] = best;
      taken[best] = 1;
    }
    for (int32_t c = 0; c < K; ++c) {
      const int32_t f = to[c];
      uint32_t used8 = 0;
      int32_t named[8], read = -1;
      int16_t at[8];
      for (int l = 0; l < 8; ++l) {
        at[l] = oc.lane_at[l * K + c];
        if (at[l] < 0) continue;
        read = named[l] = ents[lo[8 * g + l] + at[l]].o;
        used8 |= 1u << (read & 7);
        used[f] |= 1u << (read & 31);
      }
      for (int l = 0; l < 8; ++l) {
        const int L = 8 * g + l;
        if (at[l] >= 0) {
          put(f, L, named[l], &ents[lo[L] + at[l]]);
          continue;
        }
        named[l] = pad(L, read, [&](int32_t o) {
          const int sc = 2 * (int)(used8 >> (o & 7) & 1u) + (int)(used[f] >> (o & 31) & 1u);
          for (int k = 0; k < 8 && sc > 0; ++k)
            if (at[k] >= 0 && named[k] == o) return 0;  // read there anyway
          return sc;
        });
        used8 |= 1u << (named[l] & 7);
        used[f] |= 1u << (named[l] & 31);
        put(f, L, named[l], (const SlotEntry*)nullptr);
      }
    }
  }
}

}  // namespace ep
