// march.cpp -- host side of the resident run kernels' layout (march.h).
#include "march.h"

#include "banks.h"

#include <algorithm>
#include <atomic>
#include <thread>

namespace ep {
namespace {

// A vertex's slots are walked by one lane: past this degree the lane would be
// on its own for longer than a whole step of an ordinary part takes (about
// 3 us), and every other lane of its slice would carry as many unused slots.
constexpr int32_t kMarchMaxDegree = 192;
// Vertices per part below which more parts only add neighbours to wait for.
constexpr int64_t kMarchMinPart = 64;

// The first block that touches a vertex is not always the part most of its
// neighbours are in, and the parts' cuts fall anywhere: passes over the
// vertices move each one to the part that most of its neighbours are in, as
// long as no part gets more than 3% above equal work (a step takes as long as
// its largest part) or a third below it (which lets the few parts that hold
// the partition's scattered remainders dissolve: they have the largest halo,
// and it sets the shared memory).  1M-point mesh, 152 parts: mean halo 2478 ->
// 1607 records, largest 5147 -> 2396.
constexpr int kSmoothPasses = 2;
void smooth_parts(const std::vector<int32_t>& ptr, const std::vector<int32_t>& nb, int32_t P, int64_t total,
                  std::vector<int32_t>& part_of) {
  if (P < 2) return;
  const int64_t n = (int64_t)part_of.size();
  std::vector<int64_t> load(P, 0);
  for (int64_t v = 0; v < n; ++v) load[part_of[v]] += 4 + ptr[v + 1] - ptr[v];
  const int64_t hi = total / P + total / P / 33 + 16, lo = total / P - total / P / 3 - 16;
  for (int pass = 0; pass < kSmoothPasses; ++pass)
    for (int64_t v = 0; v < n; ++v) {
      const int32_t q = part_of[v], deg = ptr[v + 1] - ptr[v];
      int32_t cand[8], cnt[8], nc = 0, mine = 0;
      for (int32_t j = ptr[v]; j < ptr[v + 1]; ++j) {
        const int32_t po = part_of[nb[j]];
        if (po == q) {
          mine += nb[j] != v;
          continue;
        }
        int32_t i = 0;
        while (i < nc && cand[i] != po) ++i;
        if (i == nc) {
          if (nc == 8) continue;
          cand[nc] = po, cnt[nc++] = 0;
        }
        ++cnt[i];
      }
      int32_t best = -1, bc = mine;
      for (int32_t i = 0; i < nc; ++i)
        if (cnt[i] > bc && load[cand[i]] + 4 + deg <= hi) best = cand[i], bc = cnt[i];
      if (best < 0 || load[q] - 4 - deg < lo) continue;
      load[q] -= 4 + deg, load[best] += 4 + deg, part_of[v] = best;
    }
}

}  // namespace

// Vertices go by their cpack rank throughout (neighbours are near each other
// in it), tasks in schedule order.
bool build_march(const HostSchedule& s, int32_t max_parts, int threads, MarchLayout& L) {
  if (s.flags & 1u) return false;
  if (threads <= 0) threads = (int)std::max(1u, std::thread::hardware_concurrency());
  const int64_t nd = s.nd, m = s.m, n = s.touched;
  if (n > (int64_t)max_parts * kSlotPos) return false;  // more positions a part than an entry can name
  threads = (int)std::max<int64_t>(1, std::min<int64_t>(threads, m / 1024));  // a thread costs about 50 us
  std::vector<int32_t> ru(m), rv(m);  // endpoint ranks in schedule order
  constexpr int64_t kChunk = 1 << 14;
  parallel_for((m + kChunk - 1) / kChunk, threads, [&](int64_t c) {
    for (int64_t i = c * kChunk; i < std::min(m, (c + 1) * kChunk); ++i) {
      const int32_t e = s.edge_perm[i];
      ru[i] = s.relabel[s.src[e]];
      rv[i] = s.relabel[s.dst[e]];
    }
  });
  // incidence lists: the neighbour and the task's place in schedule order,
  // negative (~i) where the vertex is the task's second endpoint
  std::vector<int32_t> ptr(n + 1, 0);
  for (int64_t i = 0; i < m; ++i) {
    ++ptr[ru[i] + 1];
    if (rv[i] != ru[i]) ++ptr[rv[i] + 1];
  }
  for (int64_t v = 0; v < n; ++v) {
    if (ptr[v + 1] > kMarchMaxDegree) return false;
    ptr[v + 1] += ptr[v];
  }
  std::vector<int32_t> nb(ptr[n]), inc(ptr[n]);
  {
    std::vector<int32_t> cur(ptr.begin(), ptr.end() - 1);
    for (int64_t i = 0; i < m; ++i) {
      const int32_t u = ru[i], v = rv[i];
      nb[cur[u]] = v, inc[cur[u]++] = (int32_t)i;
      if (v != u) nb[cur[v]] = u, inc[cur[v]++] = ~(int32_t)i;
    }
  }
  // contiguous parts of equal slot work (a position costs about as much as
  // four slots: its own load, its store, its share of the exchange)
  const int32_t P = (int32_t)std::max<int64_t>(1, std::min<int64_t>(max_parts, n / kMarchMinPart));
  const int64_t total = (int64_t)ptr[n] + 4 * n;
  std::vector<int32_t> part_of(n, 0), rec(n, -1), order(n);  // order: the ranks part by part
  std::vector<int64_t> cut(P + 1, 0);
  {
    int64_t sum = 0;
    int32_t q = 0;
    for (int64_t v = 0; v < n; ++v) {
      while (q + 1 < P && sum * P >= total * (q + 1)) ++q;
      part_of[v] = q;
      sum += 4 + ptr[v + 1] - ptr[v];
    }
  }
  smooth_parts(ptr, nb, P, total, part_of);
  {
    for (int64_t v = 0; v < n; ++v) ++cut[part_of[v] + 1];
    for (int32_t q = 0; q < P; ++q) cut[q + 1] += cut[q];
    std::vector<int64_t> at(cut.begin(), cut.end() - 1);
    for (int64_t v = 0; v < n; ++v) order[at[part_of[v]]++] = (int32_t)v;
  }
  L = MarchLayout();
  L.parts = P;
  L.part.assign(P, MarchPart{});
  for (int32_t q = 0; q < P; ++q) {
    MarchPart& d = L.part[q];
    d.own = (int32_t)(cut[q + 1] - cut[q]);
    d.nsl = (d.own + 31) / 32;
    d.hbase = (d.own + 3) & ~3;
    L.max_nsl = std::max(L.max_nsl, d.nsl);
  }
  L.warps = std::max(4, std::min(32, (L.max_nsl + 3) / 4 * 4));
  // positions: boundary vertices first, then by descending degree
  parallel_for(P, threads, [&](int64_t q) {
    MarchPart& d = L.part[q];
    std::vector<std::pair<int32_t, int32_t>> key(d.own);  // (class and degree, place)
    for (int32_t i = 0; i < d.own; ++i) {
      const int32_t v = order[cut[q] + i];
      bool bnd = false;
      for (int32_t j = ptr[v]; j < ptr[v + 1] && !bnd; ++j) bnd = part_of[nb[j]] != q;
      d.nb += bnd;
      key[i] = {-((bnd ? 2 * kMarchMaxDegree : 0) + ptr[v + 1] - ptr[v]), i};
    }
    std::sort(key.begin(), key.end());
    for (int32_t p = 0; p < d.own; ++p) rec[order[cut[q] + key[p].second]] = p;
    std::vector<int32_t> cnt(((size_t)d.own + 7) / 8 * 8, 0), who(d.own), rp(d.own + 1, 0), ro;
    for (int32_t i = 0; i < d.own; ++i) {
      const int32_t v = order[cut[q] + i];
      who[rec[v]] = i;
      for (int32_t j = ptr[v]; j < ptr[v + 1]; ++j)
        if (part_of[nb[j]] == q) {
          const int32_t o = rec[nb[j]] >> 3;
          ro.push_back(o);
          ++cnt[8 * o + (rec[v] & 7)];
        }
      rp[i + 1] = (int32_t)ro.size();
    }
    even_residues(0, d.own, d.nb, rp, ro, cnt, who);
    for (int32_t p = 0; p < d.own; ++p) rec[order[cut[q] + who[p]]] = p;
    // (rec: position so far; its part's first record is added below)
  });
  // halo lists (by vertex, then sorted by record once the runs have a place)
  struct Piece {
    std::vector<int32_t> halo, wmap;
    std::vector<uint16_t> tab;
    std::vector<uint32_t> ent;
  };
  std::vector<Piece> piece(P);
  parallel_for(P, threads, [&](int64_t q) {
    std::vector<int32_t>& halo = piece[q].halo;
    for (int64_t i = cut[q]; i < cut[q + 1]; ++i)
      for (int32_t j = ptr[order[i]]; j < ptr[order[i] + 1]; ++j)
        if (part_of[nb[j]] != q) halo.push_back(nb[j]);
    std::sort(halo.begin(), halo.end());
    halo.erase(std::unique(halo.begin(), halo.end()), halo.end());
    L.part[q].nh = (int32_t)halo.size();
  });
  int64_t next = 0;
  for (MarchPart& d : L.part) {
    if (d.hbase + d.nh > (int32_t)kSlotPos) return false;
    d.lo = (int32_t)next;
    next += d.hbase + ((d.nh + 3) & ~3);
    if (next > INT32_MAX / 2) return false;
  }
  for (int64_t v = 0; v < n; ++v) rec[v] += L.part[part_of[v]].lo;
  // the slots
  L.gslot.assign(m, -1);
  std::atomic<bool> ok{true};
  parallel_for(P, threads, [&](int64_t q) {
    MarchPart& d = L.part[q];
    Piece& t = piece[q];
    for (int32_t& v : t.halo) v = rec[v];
    std::sort(t.halo.begin(), t.halo.end());  // the owners' order, but for the swaps inside octets
    std::vector<int32_t> vert(d.own);
    for (int64_t r = cut[q]; r < cut[q + 1]; ++r) vert[rec[order[r]] - d.lo] = order[r];
    // positions of the other endpoints, slot by slot; then the halo's residues,
    // the own positions standing
    std::vector<int32_t> ip(d.own + 1, 0), pos;
    pos.reserve(8 * (size_t)d.own);
    for (int32_t p = 0; p < d.own; ++p) {
      for (int32_t j = ptr[vert[p]]; j < ptr[vert[p] + 1]; ++j)
        pos.push_back(part_of[nb[j]] == q ? rec[nb[j]] - d.lo
                                          : d.hbase + (int32_t)(std::lower_bound(t.halo.begin(), t.halo.end(), rec[nb[j]]) -
                                                                t.halo.begin()));
      ip[p + 1] = (int32_t)pos.size();
    }
    if (d.nh > 0) {
      std::vector<int32_t> cnt(((size_t)d.own + 7) / 8 * 8, 0), rp(d.nh + 1, 0), ro, at, moved(d.nh);
      for (int32_t x : pos)
        if (x >= d.hbase) ++rp[x - d.hbase + 1];
      for (int32_t i = 0; i < d.nh; ++i) rp[i + 1] += rp[i];
      ro.resize(rp[d.nh]);
      at.assign(rp.begin(), rp.end() - 1);
      for (int32_t p = 0; p < d.own; ++p)
        for (int32_t i = ip[p]; i < ip[p + 1]; ++i) {
          ++cnt[8 * (p >> 3) + (pos[i] & 7)];
          if (pos[i] >= d.hbase) ro[at[pos[i] - d.hbase]++] = p >> 3;
        }
      const int32_t lo8 = d.hbase & ~7;
      std::vector<int32_t> who(d.hbase + d.nh - lo8, -1), rec_at(t.halo);
      for (int32_t i = 0; i < d.nh; ++i) who[d.hbase - lo8 + i] = i;
      even_residues(lo8, d.hbase + d.nh, 0, rp, ro, cnt, who);
      for (int32_t i = 0; i < d.nh; ++i) {
        const int32_t h = who[d.hbase - lo8 + i];
        t.halo[i] = rec_at[h];
        moved[h] = d.hbase + i;
      }
      for (int32_t& x : pos)
        if (x >= d.hbase) x = moved[x - d.hbase];
    }
    const int32_t W = L.warps;
    std::vector<int32_t> kcol(d.nsl), c0(d.nsl);
    for (int32_t j = 0; j < d.nsl; ++j)
      for (int32_t p = 32 * j; p < std::min(d.own, 32 * j + 32); ++p)
        kcol[j] = std::max(kcol[j], (ptr[vert[p] + 1] - ptr[vert[p]] + 1) / 2);
    int32_t cols = 0;
    t.tab.resize(W + d.nsl);
    for (int32_t v = 0; v < W; ++v) {
      t.tab[v] = (uint16_t)cols;
      for (int32_t j = v; j < d.nsl; j += W) c0[j] = cols, cols += kcol[j], t.tab[W + j] = (uint16_t)kcol[j];
    }
    if (cols > 0xffff) {
      ok = false;
      return;
    }
    d.ncol = cols;
    t.ent.assign((size_t)cols * 32, 0);
    t.wmap.assign((size_t)cols * 64, -1);
    std::vector<SlotEntry> ents;
    OctetColumns oc;
    for (int32_t j = 0; j < d.nsl; ++j) {
      int32_t lo[32], hi[32];
      ents.clear();
      for (int l = 0; l < 32; ++l) {
        lo[l] = (int32_t)ents.size();
        const int32_t p = 32 * j + l;
        if (p < d.own)
          for (int32_t i = ptr[vert[p]], k = ip[p]; i < ptr[vert[p] + 1]; ++i, ++k)
            ents.push_back(SlotEntry{pos[k], s.edge_perm[inc[i] < 0 ? ~inc[i] : inc[i]], inc[i] >= 0});
        hi[l] = (int32_t)ents.size();
      }
      // An unused slot names the lane's own position or one of its neighbours:
      // its weight is 0, and its term zero whenever the lane's used slots are
      // finite.  A lane of no vertex names what another lane reads.
      auto pad = [&](int l, int32_t read_there, auto score) {
        int32_t best = 32 * j + l;
        if (lo[l] == hi[l] && read_there >= 0) return read_there;
        int bs = score(best);
        for (int32_t i = lo[l]; i < hi[l] && bs > 0; ++i)
          if (const int sc = score(ents[i].o); sc < bs) best = ents[i].o, bs = sc;
        return best;
      };
      spread_slice(ents, lo, hi, 2 * kcol[j], oc, pad, [&](int32_t c, int l, int32_t o, const SlotEntry* x) {
        const size_t at = (size_t)32 * (c0[j] + c / 2) + l;
        const uint32_t v = (uint32_t)o | (x && x->src ? kSlotSrc : 0u);
        t.ent[at] |= v << (16 * (c & 1));
        if (x) t.wmap[2 * at + (c & 1)] = x->e;
      });
    }
    while (t.tab.size() % 8) t.tab.push_back(0);
  });
  if (!ok) return false;
  int64_t nh = 0, nq = 0, nc = 0;
  for (int32_t q = 0; q < P; ++q) {
    MarchPart& d = L.part[q];
    d.h0 = (int32_t)nh, d.q0 = (int32_t)nq, d.s0 = (int32_t)nc;
    nh += d.nh, nq += (int64_t)piece[q].tab.size(), nc += d.ncol;
    L.max_pos = std::max(L.max_pos, std::max(d.hbase + ((d.nh + 3) & ~3), 32 * d.nsl));
    L.max_col = std::max(L.max_col, d.ncol);
  }
  nc += kMarchAhead;
  if (nc > INT32_MAX / 64) return false;
  L.n_col = nc;
  L.halo.resize(nh), L.tab.resize(nq), L.ent.resize(32 * nc, 0), L.wmap.resize(64 * nc, -1);
  parallel_for(P, threads, [&](int64_t q) {
    const MarchPart& d = L.part[q];
    const Piece& t = piece[q];
    std::copy(t.halo.begin(), t.halo.end(), L.halo.begin() + d.h0);
    std::copy(t.tab.begin(), t.tab.end(), L.tab.begin() + d.q0);
    std::copy(t.ent.begin(), t.ent.end(), L.ent.begin() + 32 * (int64_t)d.s0);
    std::copy(t.wmap.begin(), t.wmap.end(), L.wmap.begin() + 64 * (int64_t)d.s0);
    for (int64_t i = 0; i < 64 * (int64_t)d.ncol; ++i)
      if (t.wmap[i] >= 0 && ((t.ent[i / 2] >> (16 * (i & 1))) & kSlotSrc))
        L.gslot[t.wmap[i]] = (int32_t)(64 * (int64_t)d.s0 + i);
  });
  L.n_run = next;
  L.rec_of.resize(nd);
  for (int64_t v = 0; v < nd; ++v)  // untouched vertices after the parts
    L.rec_of[v] = s.relabel[v] < n ? rec[s.relabel[v]] : (int32_t)next++;
  L.n_rec = (next + 3) & ~(int64_t)3;
  return true;
}

}  // namespace ep
