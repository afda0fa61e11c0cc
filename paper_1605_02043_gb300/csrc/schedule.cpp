// schedule.cpp -- from a task partition to the arrays the kernels use.
//
//   reconstruction   tasks grouped by block, ascending id inside a block
//                    (Definition 4);
//   vertex lists     distinct data vertices of each block in first-touch
//                    order (the block's share of the data, Section 4 Fig. 7);
//   cpack            ids in order of first appearance over blocks (Section
//                    4.1, after Ding and Kennedy), untouched vertices last;
//   cost             loads = sum_b |V_b|, vertex cut = loads - touched (Eq. 1);
//   kernel layout    flux: one contiguous record run per kernel block with
//                    the vertices only that block uses (updated in place)
//                    followed by its own copies of the shared vertices
//                    (accumulated by atomics, refreshed by the fold), the
//                    incidence in sliced-ELL slots with one weight per slot,
//                    and the copy lists of the shared vertices; SpMV: row-
//                    ranked entries over x records ordered by use.
#include <algorithm>
#include <atomic>
#include <climits>
#include <thread>

#include "banks.h"
#include "internal.h"

namespace ep {
namespace {

// Endpoint pair of task e as data-vertex ids (bipartite: y_i -> n + i).
inline void task_ends(const HostSchedule& s, int64_t e, int32_t& u, int32_t& v) {
  const bool bip = (s.flags & 1u) != 0;
  u = bip ? (int32_t)(s.n + s.src[e]) : s.src[e];
  v = s.dst[e];
}

// Per-block first-touch vertex lists, computed block-parallel with one stamp
// array per worker, then concatenated.
void vertex_lists(HostSchedule& s, int threads) {
  const int64_t k = s.k;
  std::vector<int64_t> count(k, 0);
  std::vector<std::vector<int32_t>> chunks(threads);
  std::vector<int64_t> lo(threads + 1);
  for (int t = 0; t <= threads; ++t) lo[t] = k * t / threads;
  auto work = [&](int t) {
    std::vector<int32_t> stamp(s.nd, -1);
    auto& out = chunks[t];
    for (int64_t b = lo[t]; b < lo[t + 1]; ++b) {
      const int64_t before = (int64_t)out.size();
      for (int64_t i = s.block_ptr[b]; i < s.block_ptr[b + 1]; ++i) {
        int32_t u, v;
        task_ends(s, s.edge_perm[i], u, v);
        if (stamp[u] != (int32_t)b) {
          stamp[u] = (int32_t)b;
          out.push_back(u);
        }
        if (stamp[v] != (int32_t)b) {
          stamp[v] = (int32_t)b;
          out.push_back(v);
        }
      }
      count[b] = (int64_t)out.size() - before;
    }
  };
  if (threads == 1) {
    work(0);
  } else {
    std::vector<std::thread> pool;
    for (int t = 0; t < threads; ++t) pool.emplace_back(work, t);
    for (auto& th : pool) th.join();
  }
  s.vert_ptr.assign(k + 1, 0);
  for (int64_t b = 0; b < k; ++b) s.vert_ptr[b + 1] = s.vert_ptr[b] + count[b];
  s.vert_list.clear();
  s.vert_list.reserve(s.vert_ptr[k]);
  for (auto& c : chunks) s.vert_list.insert(s.vert_list.end(), c.begin(), c.end());
  s.loads = s.vert_ptr[k];
}

void cpack(HostSchedule& s) {
  s.relabel.assign(s.nd, -1);
  int32_t next = 0;
  for (int32_t v : s.vert_list)
    if (s.relabel[v] < 0) s.relabel[v] = next++;
  s.touched = next;
  for (int64_t v = 0; v < s.nd; ++v)
    if (s.relabel[v] < 0) s.relabel[v] = next++;
}

// Number of blocks using each vertex (p_v) and the first such block.
void usage(const HostSchedule& s, std::vector<int32_t>& p, std::vector<int32_t>& owner) {
  p.assign(s.nd, 0);
  owner.assign(s.nd, -1);
  for (int64_t b = 0; b < s.k; ++b)
    for (int64_t i = s.vert_ptr[b]; i < s.vert_ptr[b + 1]; ++i) {
      const int32_t v = s.vert_list[i];
      if (p[v]++ == 0) owner[v] = (int32_t)b;
    }
}

// In-block degree of every vertex of block b (tasks of b touching it).
void block_degrees(const HostSchedule& s, int64_t b, std::vector<int32_t>& deg) {
  for (int64_t i = s.block_ptr[b]; i < s.block_ptr[b + 1]; ++i) {
    int32_t u, v;
    task_ends(s, s.edge_perm[i], u, v);
    ++deg[u];
    if (v != u) ++deg[v];
  }
}

// The vertices of V_b satisfying `pick`, first-touch order, then stably
// sorted by descending in-block degree (so warps see similar list lengths).
template <typename Pick>
void class_order(const HostSchedule& s, int64_t b, const std::vector<int32_t>& deg, Pick pick,
                 std::vector<int32_t>& out) {
  out.clear();
  for (int64_t i = s.vert_ptr[b]; i < s.vert_ptr[b + 1]; ++i)
    if (pick(s.vert_list[i])) out.push_back(s.vert_list[i]);
  std::stable_sort(out.begin(), out.end(), [&](int32_t a, int32_t c) { return deg[a] > deg[c]; });
}

// Places the entries of slice j (positions 32 j + l, l < 32) in its columns
// (banks.h).  An unused slot has weight 0, so its term is exactly zero whatever
// position it names: the one of the first 32 that falls on a free bank.
void place_slice(HostSchedule& s, const FluxDesc& d, int32_t j, const std::vector<int32_t>& ent_ptr,
                 const std::vector<SlotEntry>& ents, OctetColumns& oc) {
  const int32_t c0 = s.soff[d.q0 + j], K = s.soff[d.q0 + j + 1] - c0;
  int32_t lo[32], hi[32];
  for (int l = 0; l < 32; ++l) {
    const int32_t p = 32 * j + l;
    lo[l] = p < d.nv ? ent_ptr[p] : 0;
    hi[l] = p < d.nv ? ent_ptr[p + 1] : 0;
  }
  const int32_t npad = std::min(d.nv, 32);
  auto pad = [&](int, int32_t read_there, auto score) {
    if (read_there >= 0 && read_there < npad) return read_there;
    int32_t best = 0, bs = 4;
    for (int32_t o = 0; o < npad && bs > 0; ++o)
      if (const int sc = score(o); sc < bs) best = o, bs = sc;
    return best;
  };
  spread_slice(ents, lo, hi, K, oc, pad, [&](int32_t c, int l, int32_t o, const SlotEntry* x) {
    const int64_t slot = (int64_t)d.s0 + 32 * ((int64_t)c0 + c) + l;
    s.sidx[slot] = (uint16_t)((uint32_t)o | (x && x->src ? kSlotSrc : 0u));
    if (!x) return;  // weight slot stays -1: weight 0
    s.wmap[slot] = x->e;
    if (x->src) s.gslot[x->e] = (int32_t)slot;
  });
}

// f(lo, hi) over contiguous ranges of [0, n), one per host thread
template <typename F>
void parallel_blocks(int64_t n, int threads, F f) {
  threads = (int)std::max<int64_t>(1, std::min<int64_t>(threads, n / 16));
  parallel_for(threads, threads, [&](int64_t t) { f(n * t / threads, n * (t + 1) / threads); });
}

std::string flux_layout_blocks(HostSchedule& s, int threads) {
  std::vector<int32_t> p, owner;
  usage(s, p, owner);
  // halo vertices of a shard (touched by other shards' tasks too) take the
  // shared path even when one block here uses them: their sums must go
  // through an accumulator that the exchange can reach
  for (int32_t v : s.halo)
    if (v >= 0 && v < s.nd && p[v] == 1) p[v] = 2;
  auto align4 = [](int64_t v) { return (v + 3) & ~(int64_t)3; };
  // shared ids in order of first appearance over the kernel blocks
  std::vector<int32_t> sid(s.nd, -1);
  int64_t n_sh = 0;
  for (int64_t b = 0; b < s.k; ++b)
    for (int64_t i = s.vert_ptr[b]; i < s.vert_ptr[b + 1]; ++i) {
      const int32_t v = s.vert_list[i];
      if (p[v] > 1 && sid[v] < 0) sid[v] = (int32_t)n_sh++;
    }
  s.n_sh = n_sh;
  s.fdesc.assign(s.k, FluxDesc{});
  s.rec_of.assign(s.nd, -1);
  s.gslot.assign(s.m, -1);
  s.max_nv = s.max_nslot = s.max_nsh = s.max_nsl = 0;
  std::vector<int32_t> order(s.vert_list.size());     // positions of every block, vert_ptr offsets
  std::vector<uint16_t> cols(s.vert_list.size() + s.k);  // slice offsets, vert_ptr[b] + b
  std::atomic<const char*> err{nullptr};
  // every block by itself: its positions (interior vertices, then shared
  // ones, each by descending degree) and its slices' columns
  parallel_blocks(s.k, threads, [&](int64_t lo, int64_t hi) {
    std::vector<int32_t> deg(s.nd, 0), pos(s.nd), ord, cls, rp, ro, cnt, who;
    for (int64_t b = lo; b < hi; ++b) {
      FluxDesc& d = s.fdesc[b];
      d.ne = (int32_t)(s.block_ptr[b + 1] - s.block_ptr[b]);
      block_degrees(s, b, deg);
      class_order(s, b, deg, [&](int32_t v) { return p[v] == 1; }, ord);
      d.ni = (int32_t)ord.size();
      class_order(s, b, deg, [&](int32_t v) { return p[v] > 1; }, cls);
      ord.insert(ord.end(), cls.begin(), cls.end());
      d.nv = (int32_t)ord.size();
      // the order inside an octet of positions, by bank
      for (int32_t q = 0; q < d.nv; ++q) pos[ord[q]] = q;
      rp.assign(d.nv + 1, 0);
      auto ends = [&](auto f) {  // f(position, the other endpoint's) for every slot of the block
        for (int64_t i = s.block_ptr[b]; i < s.block_ptr[b + 1]; ++i) {
          int32_t u, v;
          task_ends(s, s.edge_perm[i], u, v);
          f(pos[u], pos[v]);
          if (v != u) f(pos[v], pos[u]);
        }
      };
      ends([&](int32_t, int32_t o) { ++rp[o + 1]; });
      for (int32_t q = 0; q < d.nv; ++q) rp[q + 1] += rp[q];
      ro.resize(rp[d.nv]);
      cnt.assign(((size_t)d.nv + 7) / 8 * 8, 0);
      who.assign(rp.begin(), rp.end() - 1);  // fill positions first
      ends([&](int32_t p_, int32_t o) {
        ro[who[o]++] = p_ >> 3;
        ++cnt[8 * (p_ >> 3) + (o & 7)];
      });
      for (int32_t q = 0; q < d.nv; ++q) who[q] = q;
      even_residues(0, d.nv, d.ni, rp, ro, cnt, who);
      for (int32_t q = 0; q < d.nv; ++q) order[s.vert_ptr[b] + q] = ord[who[q]];
      // slices of 32 positions; columns = largest degree in the slice
      d.nsl = (d.nv + 31) / 32;
      uint16_t* off = &cols[s.vert_ptr[b] + b];
      int32_t c = off[0] = 0;
      for (int32_t j = 0; j < d.nsl; ++j) {
        int32_t K = 0;
        for (int32_t q = 32 * j; q < std::min(d.nv, 32 * j + 32); ++q) K = std::max(K, deg[ord[q]]);
        c += K;
        if (c > 0xffff) {
          err = "block has too many incidence entries";
          break;
        }
        off[j + 1] = (uint16_t)c;
      }
      if (d.nv > (int32_t)kSlotPos) err = "block touches too many vertices";
      d.nslot = 32 * c;
      for (int64_t i = s.vert_ptr[b]; i < s.vert_ptr[b + 1]; ++i) deg[s.vert_list[i]] = 0;
      if (err.load()) return;
    }
  });
  if (err.load()) return err.load();
  // where every block's segments start (16-byte boundaries)
  int64_t next = 0, n_sid = 0, n_off = 0, n_slot = 0;
  for (int64_t b = 0; b < s.k; ++b) {
    FluxDesc& d = s.fdesc[b];
    next = align4(next);
    d.rec_lo = (int32_t)next;
    d.h0 = (int32_t)n_sid;
    d.q0 = (int32_t)n_off;
    d.s0 = (int32_t)n_slot;  // a multiple of 32
    next += d.nv;
    n_sid += align4(d.nv - d.ni);
    n_off += (d.nsl + 1 + 7) & ~7;
    n_slot += d.nslot;
    s.max_nv = std::max(s.max_nv, d.nv);
    s.max_nslot = std::max(s.max_nslot, d.nslot);
    s.max_nsh = std::max(s.max_nsh, d.nv - d.ni);
    s.max_nsl = std::max(s.max_nsl, d.nsl);
    if (n_slot >= INT32_MAX || next >= INT32_MAX / 2) return "schedule too large";
  }
  s.sid_list.assign(n_sid, 0);
  s.soff.assign(n_off, 0);
  s.sidx.assign(n_slot, 0);
  s.wmap.assign(n_slot, -1);
  parallel_blocks(s.k, threads, [&](int64_t blo, int64_t bhi) {
    std::vector<int32_t> pos(s.nd), ent_ptr, col;
    std::vector<SlotEntry> ents;
    OctetColumns oc;
    for (int64_t b = blo; b < bhi; ++b) {
      const FluxDesc& d = s.fdesc[b];
      const int32_t* ord = order.data() + s.vert_ptr[b];
      // shared ids of positions [ni, nv); the first copy of each shared vertex
      // (in its first block) carries kSidFirst and is the vertex's record
      for (int32_t q = 0; q < d.nv; ++q) {
        const int32_t v = ord[q];
        pos[v] = q;
        if (owner[v] == b) s.rec_of[v] = d.rec_lo + q;
        if (q >= d.ni) s.sid_list[d.h0 + q - d.ni] = sid[v] | (owner[v] == b ? kSidFirst : 0);
      }
      std::copy_n(&cols[s.vert_ptr[b] + b], d.nsl + 1, s.soff.begin() + d.q0);
      // the entries of every position: each task at both endpoints (a self
      // loop once), the source side flagged
      ent_ptr.assign(d.nv + 1, 0);
      for (int64_t i = s.block_ptr[b]; i < s.block_ptr[b + 1]; ++i) {
        int32_t u, v;
        task_ends(s, s.edge_perm[i], u, v);
        ++ent_ptr[pos[u] + 1];
        if (v != u) ++ent_ptr[pos[v] + 1];
      }
      for (int32_t q = 0; q < d.nv; ++q) ent_ptr[q + 1] += ent_ptr[q];
      ents.resize(ent_ptr[d.nv]);
      col.assign(ent_ptr.begin(), ent_ptr.end() - 1);
      for (int64_t i = s.block_ptr[b]; i < s.block_ptr[b + 1]; ++i) {
        const int32_t e = s.edge_perm[i];
        int32_t u, v;
        task_ends(s, e, u, v);
        const int32_t pu = pos[u], pv = pos[v];
        ents[col[pu]++] = SlotEntry{pv, e, true};
        if (v != u) ents[col[pv]++] = SlotEntry{pu, e, false};
      }
      for (int32_t j = 0; j < d.nsl; ++j) place_slice(s, d, j, ent_ptr, ents, oc);
    }
  });
  s.n_run = align4(next);
  next = s.n_run;
  for (int64_t v = 0; v < s.nd; ++v)
    if (s.rec_of[v] < 0) s.rec_of[v] = (int32_t)next++;  // untouched vertices
  s.n_rec = align4(next);  // keeps every plane of a state buffer 16-byte aligned
  s.vrec.assign(s.n_rec, -1);
  for (int64_t v = 0; v < s.nd; ++v) s.vrec[s.rec_of[v]] = (int32_t)v;
  // the fold's work list: every copy in record order (block runs in order)
  s.fold_rec.clear();
  s.fold_sid.clear();
  for (int64_t b = 0; b < s.k; ++b) {
    const FluxDesc& d = s.fdesc[b];
    for (int32_t q = d.ni; q < d.nv; ++q) {
      s.fold_rec.push_back(d.rec_lo + q);
      s.fold_sid.push_back(s.sid_list[d.h0 + q - d.ni]);
    }
  }
  // the copies of every shared vertex, in block order (fold_rec is)
  s.cptr.assign(n_sh + 1, 0);
  for (int32_t h : s.fold_sid) ++s.cptr[(h & kSidMask) + 1];
  for (int64_t h = 0; h < n_sh; ++h) s.cptr[h + 1] += s.cptr[h];
  s.crec.resize(s.fold_rec.size());
  {
    std::vector<int32_t> cur(s.cptr.begin(), s.cptr.end() - 1);
    for (size_t i = 0; i < s.fold_sid.size(); ++i) s.crec[cur[s.fold_sid[i] & kSidMask]++] = s.fold_rec[i];
  }
  for (int64_t v = 0; v < s.nd; ++v)  // every copy of a shared vertex maps back to it
    if (sid[v] >= 0)
      for (int32_t c = s.cptr[sid[v]]; c < s.cptr[sid[v] + 1]; ++c) s.vrec[s.crec[c]] = (int32_t)v;
  s.w_pad = (int64_t)s.wmap.size();
  return "";
}

// Kernel blocks of the flux layout.  A schedule block whose vertex set is
// far above the typical one (more than 3/2 of the median |V_b|) is cut in
// task order into halves, recursively, until every piece is within that
// size; each piece is then laid out as a block of its own (vertices shared
// by the pieces become shared vertices).  The schedule and its cost are
// unchanged; the kernels' shared-memory stages, sized for the largest kernel
// block, get smaller.  Returns false when no block needs cutting.
struct Pieces {
  int64_t k = 0;
  std::vector<int64_t> block_ptr, vert_ptr;
  std::vector<int32_t> vert_list;
};

bool cut_large_blocks(const HostSchedule& s, Pieces& out) {
  if (s.k < 2) return false;
  std::vector<int64_t> sz(s.k);
  for (int64_t b = 0; b < s.k; ++b) sz[b] = s.vert_ptr[b + 1] - s.vert_ptr[b];
  const int64_t biggest = *std::max_element(sz.begin(), sz.end());
  std::nth_element(sz.begin(), sz.begin() + s.k / 2, sz.end());
  const int64_t limit = std::max<int64_t>(64, sz[s.k / 2] * 3 / 2);
  if (biggest <= limit) return false;
  std::vector<int32_t> stamp(s.nd, -1);
  int32_t piece = 0;
  out.block_ptr.assign(1, 0);
  out.vert_ptr.assign(1, 0);
  out.vert_list.clear();
  // first-touch vertex list of tasks [lo, hi) appended to out.vert_list
  auto touch = [&](int64_t lo, int64_t hi) {
    const size_t before = out.vert_list.size();
    for (int64_t i = lo; i < hi; ++i) {
      int32_t u, v;
      task_ends(s, s.edge_perm[i], u, v);
      if (stamp[u] != piece) {
        stamp[u] = piece;
        out.vert_list.push_back(u);
      }
      if (stamp[v] != piece) {
        stamp[v] = piece;
        out.vert_list.push_back(v);
      }
    }
    return (int64_t)(out.vert_list.size() - before);
  };
  std::vector<std::pair<int64_t, int64_t>> todo;
  for (int64_t b = 0; b < s.k; ++b) {
    todo.assign(1, {s.block_ptr[b], s.block_ptr[b + 1]});
    while (!todo.empty()) {  // depth first, left half first: pieces stay in task order
      const auto [lo, hi] = todo.back();
      todo.pop_back();
      const size_t mark = out.vert_list.size();
      const int64_t nv = touch(lo, hi);
      if (nv > limit && hi - lo > 1) {
        out.vert_list.resize(mark);
        ++piece;  // fresh stamps for the halves
        const int64_t mid = lo + (hi - lo + 1) / 2;
        todo.push_back({mid, hi});
        todo.push_back({lo, mid});
        continue;
      }
      ++piece;
      out.block_ptr.push_back(hi);
      out.vert_ptr.push_back((int64_t)out.vert_list.size());
    }
  }
  out.k = (int64_t)out.block_ptr.size() - 1;
  return true;
}

std::string flux_layout(HostSchedule& s, int threads) {
  Pieces pc;
  const bool cut = cut_large_blocks(s, pc);
  if (cut) {
    std::swap(s.k, pc.k);
    s.block_ptr.swap(pc.block_ptr);
    s.vert_ptr.swap(pc.vert_ptr);
    s.vert_list.swap(pc.vert_list);
  }
  std::string err = flux_layout_blocks(s, threads);
  if (cut) {  // the schedule itself is the uncut one
    std::swap(s.k, pc.k);
    s.block_ptr.swap(pc.block_ptr);
    s.vert_ptr.swap(pc.vert_ptr);
    s.vert_list.swap(pc.vert_list);
  }
  return err;
}

std::string spmv_layout(HostSchedule& s) {
  std::vector<int32_t> p, owner;
  usage(s, p, owner);
  const int32_t n = (int32_t)s.n;
  s.xrec_of.assign(n, -1);
  s.yrec_of.assign(n, -1);
  s.sdesc.assign(s.k, SpmvDesc{});
  std::vector<int32_t> deg(s.nd, 0), cls;
  // x records: the columns that most blocks use first (the kernel keeps a
  // prefix of them in shared memory), columns of equal use in cpack order
  {
    int32_t most = 0;
    for (int32_t v = 0; v < n; ++v) most = std::max(most, p[v]);
    std::vector<int32_t> at(most + 2, 0), by_rank(s.nd, -1);
    for (int32_t v = 0; v < n; ++v) ++at[most - p[v] + 1];
    for (int32_t q = 0; q <= most; ++q) at[q + 1] += at[q];
    for (int32_t v = 0; v < n; ++v) by_rank[s.relabel[v]] = v;
    for (int32_t v : by_rank)
      if (v >= 0) s.xrec_of[v] = at[most - p[v]]++;
  }
  // y records: single-block rows first, then shared rows; longest lists first
  int32_t ny = 0;
  for (int64_t b = 0; b < s.k; ++b) {
    SpmvDesc& d = s.sdesc[b];
    block_degrees(s, b, deg);
    d.yi_lo = ny;
    class_order(s, b, deg, [&](int32_t v) { return v >= n && owner[v] == b && p[v] == 1; }, cls);
    for (int32_t v : cls) s.yrec_of[v - n] = ny++;
    d.n_yi = ny - d.yi_lo;
    for (int64_t i = s.vert_ptr[b]; i < s.vert_ptr[b + 1]; ++i) deg[s.vert_list[i]] = 0;
  }
  s.ny_int = ny;
  for (int64_t b = 0; b < s.k; ++b) {
    SpmvDesc& d = s.sdesc[b];
    block_degrees(s, b, deg);
    d.yb_lo = ny;
    class_order(s, b, deg, [&](int32_t v) { return v >= n && owner[v] == b && p[v] > 1; }, cls);
    for (int32_t v : cls) s.yrec_of[v - n] = ny++;
    d.n_yob = ny - d.yb_lo;
    for (int64_t i = s.vert_ptr[b]; i < s.vert_ptr[b + 1]; ++i) deg[s.vert_list[i]] = 0;
  }
  s.ny_bnd = ny - s.ny_int;
  for (int32_t i = 0; i < n; ++i)
    if (s.yrec_of[i] < 0) s.yrec_of[i] = ny++;
  s.xlist.clear();
  s.ylist.clear();
  s.sent.clear();
  s.wmap.clear();
  s.max_ny = 0;
  std::vector<int32_t> pos(s.nd, -1), cnt;
  // one entry run of 32 * u slots per block (u from the largest block), so
  // that block b's run starts at slot 32 * u * b
  int64_t big = 0;
  for (int64_t b = 0; b < s.k; ++b) big = std::max(big, s.block_ptr[b + 1] - s.block_ptr[b]);
  s.spmv_u = (int32_t)(((big + 31) / 32 + 3) / 4 * 4);
  for (int64_t b = 0; b < s.k; ++b) {
    SpmvDesc& d = s.sdesc[b];
    d.ne = (int32_t)(s.block_ptr[b + 1] - s.block_ptr[b]);
    d.fx0 = (int32_t)s.xlist.size();
    d.fy0 = (int32_t)s.ylist.size();
    int32_t nxf = 0;
    for (int64_t i = s.vert_ptr[b]; i < s.vert_ptr[b + 1]; ++i) {
      const int32_t v = s.vert_list[i];
      if (v >= n) continue;
      pos[v] = nxf++;
      s.xlist.push_back(s.xrec_of[v]);
    }
    d.n_xf = nxf;
    block_degrees(s, b, deg);
    for (int64_t i = s.vert_ptr[b]; i < s.vert_ptr[b + 1]; ++i) {
      const int32_t v = s.vert_list[i];
      if (v < n || owner[v] != b) continue;
      const int32_t r = s.yrec_of[v - n];
      pos[v] = r < s.ny_int ? r - d.yi_lo : d.n_yi + (r - d.yb_lo);
    }
    class_order(s, b, deg, [&](int32_t v) { return v >= n && owner[v] != b; }, cls);
    int32_t nyf = 0;
    for (int32_t v : cls) {
      pos[v] = d.n_yi + d.n_yob + nyf++;
      s.ylist.push_back(s.yrec_of[v - n]);
    }
    d.n_yf = nyf;
    for (int64_t i = s.vert_ptr[b]; i < s.vert_ptr[b + 1]; ++i) deg[s.vert_list[i]] = 0;
    const int32_t nys = d.n_yi + d.n_yob + nyf;
    if (nxf > (int32_t)kColMask + 1 || nys > (int32_t)kColMask + 1)
      return "block touches too many vertices";
    s.max_ny = std::max(s.max_ny, nys);
    // entries sorted by row position (a counting sort; schedule order within
    // a row), each lane of the kernel's warp taking u consecutive ones
    cnt.assign(nys + 1, 0);
    for (int64_t i = s.block_ptr[b]; i < s.block_ptr[b + 1]; ++i) {
      int32_t u, v;
      task_ends(s, s.edge_perm[i], u, v);
      ++cnt[pos[u] + 1];
    }
    for (int32_t q = 0; q < nys; ++q) cnt[q + 1] += cnt[q];
    d.u = s.spmv_u;
    d.i0 = (int32_t)s.sent.size();
    const size_t run = (size_t)32 * d.u;
    s.sent.resize(d.i0 + run, 0u);
    s.wmap.resize(d.i0 + run, -1);
    for (int64_t i = s.block_ptr[b]; i < s.block_ptr[b + 1]; ++i) {
      int32_t u, v;
      task_ends(s, s.edge_perm[i], u, v);
      const int32_t t = cnt[pos[u]]++;  // rank in row order
      const int32_t j = d.i0 + spmv_slot(t, d.u);
      s.sent[j] = ((uint32_t)pos[u] << kRowShift) | (uint32_t)pos[v];
      s.wmap[j] = s.edge_perm[i];
    }
    if (s.sent.size() >= (size_t)INT32_MAX) return "schedule too large";
  }
  s.w_pad = (int64_t)s.wmap.size();
  return "";
}

}  // namespace

std::string rebuild_flux_layout(HostSchedule& s) {
  return flux_layout(s, (int)std::max(1u, std::thread::hardware_concurrency()));
}

std::string build_schedule(HostSchedule& s, int threads) {
  if (threads <= 0) threads = (int)std::max(1u, std::thread::hardware_concurrency());
  threads = (int)std::max<int64_t>(1, std::min<int64_t>(threads, s.k));
  // reconstruction (Definition 4): counting sort by block keeps ascending ids
  s.block_ptr.assign(s.k + 1, 0);
  for (int64_t e = 0; e < s.m; ++e) ++s.block_ptr[s.part[e] + 1];
  s.max_ne = 0;
  for (int64_t b = 0; b < s.k; ++b) {
    s.max_ne = std::max<int32_t>(s.max_ne, (int32_t)s.block_ptr[b + 1]);
    s.block_ptr[b + 1] += s.block_ptr[b];
  }
  s.edge_perm.assign(s.m, 0);
  {
    std::vector<int64_t> cur(s.block_ptr.begin(), s.block_ptr.end() - 1);
    for (int64_t e = 0; e < s.m; ++e) s.edge_perm[cur[s.part[e]]++] = (int32_t)e;
  }
  vertex_lists(s, threads);
  cpack(s);
  return (s.flags & 1u) ? spmv_layout(s) : flux_layout(s, threads);
}

}  // namespace ep
