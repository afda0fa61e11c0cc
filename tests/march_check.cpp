// Host-only check of the resident runs' layout (test code): invariants of the
// parts, halos and slots, then several explicit steps emulated in FP64 the way
// the kernels compute them (every part from its own image: own records and halo
// gathered from the owners) against the plain edge-list steps.
// Prints "total fails N"; exit status 1 on any failure.
#include <cmath>
#include <cstdio>
#include <random>
#include <vector>

#include "march.h"

using namespace ep;

static int fails = 0;
#define CHECK(c, what)                                          \
  do {                                                          \
    if (!(c)) {                                                 \
      if (fails++ < 20) printf("FAIL line %d: %s\n", __LINE__, what); \
    }                                                           \
  } while (0)

static bool build(HostSchedule& h, int n, const std::vector<int32_t>& src, const std::vector<int32_t>& dst, int C,
                  bool dflt) {
  h.m = (int64_t)src.size();
  h.n = h.nd = n;
  h.C = C;
  h.flags = dflt ? 2u : 0u;
  h.k = (h.m + C - 1) / C;
  h.src = src;
  h.dst = dst;
  h.part.resize(h.m);
  if (dflt)
    for (int64_t e = 0; e < h.m; ++e) h.part[e] = (int32_t)(e / C);
  else
    partition_edges(src.data(), dst.data(), h.m, n, C, 0, 4, h.part.data());
  return build_schedule(h, 4).empty();
}

static void check(int n, const std::vector<int32_t>& src, const std::vector<int32_t>& dst, int C, bool dflt, int parts,
                  int threads) {
  HostSchedule h;
  CHECK(build(h, n, src, dst, C, dflt), "schedule");
  MarchLayout L;
  const bool ok = build_march(h, parts, threads, L);
  CHECK(ok, "layout built");
  if (!ok) return;
  const int64_t m = h.m;
  CHECK(L.parts <= parts && L.n_rec % 4 == 0 && L.n_run <= L.n_rec, "sizes");
  CHECK(L.warps >= 4 && L.warps <= 32 && L.warps % 4 == 0, "warps");
  std::vector<int> vert(L.n_rec, -1), part_of(n, -1), slots(m, 0);
  for (int v = 0; v < n; ++v) vert[L.rec_of[v]] = v;
  int64_t own = 0;
  for (int q = 0; q < L.parts; ++q) {
    const MarchPart& d = L.part[q];
    own += d.own;
    for (int p = 0; p < d.own; ++p) {
      CHECK(vert[d.lo + p] >= 0, "own record of a vertex");
      part_of[vert[d.lo + p]] = q;
    }
  }
  CHECK(own == h.touched, "every touched vertex owned once");
  auto record = [&](const MarchPart& d, int p) { return p < d.hbase ? d.lo + p : L.halo[d.h0 + p - d.hbase]; };
  for (int q = 0; q < L.parts; ++q) {
    const MarchPart& d = L.part[q];
    CHECK(d.lo % 4 == 0 && d.hbase % 4 == 0 && d.hbase >= d.own && d.q0 % 8 == 0, "alignment");
    CHECK(d.hbase + d.nh <= L.max_pos && 32 * d.nsl <= L.max_pos && d.ncol <= L.max_col && d.nsl <= L.max_nsl, "maxima");
    CHECK(d.nsl == (d.own + 31) / 32, "slices");
    for (int j = 0; j < d.nh; ++j) {
      const int r = L.halo[d.h0 + j], v = vert[r];
      CHECK(v >= 0 && part_of[v] >= 0 && part_of[v] != q, "halo record owned elsewhere");
      CHECK(r - L.part[part_of[v]].lo < L.part[part_of[v]].nb, "halo record is a boundary one of its owner");
    }
    int cols = 0;
    for (int w = 0; w < L.warps; ++w) {
      CHECK(L.tab[d.q0 + w] == cols, "stream start");
      for (int j = w; j < d.nsl; j += L.warps) {
        const int K = L.tab[d.q0 + L.warps + j];
        CHECK(K > 0, "columns of a slice");
        for (int c = cols; c < cols + K; ++c)
          for (int l = 0; l < 32; ++l)
            for (int u = 0; u < 2; ++u) {
              const int64_t at = 32 * ((int64_t)d.s0 + c) + l;
              const int e = (L.ent[at] >> (16 * u)) & 0xffff, o = e & kSlotPos, t = L.wmap[2 * at + u], p = 32 * j + l;
              if (p >= d.own) {
                CHECK(t < 0 && !(e & kSlotSrc) && o < L.max_pos, "slot of no vertex");
                continue;
              }
              CHECK(o < d.own || (o >= d.hbase && o < d.hbase + d.nh), "slot position");
              const int vp = vert[d.lo + p], vo = vert[record(d, o)];
              if (t >= 0) {
                ++slots[t];
                const bool s = e & kSlotSrc;
                CHECK(vp == (s ? src[t] : dst[t]) && vo == (s ? dst[t] : src[t]), "slot endpoints");
                if (s) CHECK(L.gslot[t] == 2 * at + u, "source slot of the task");
                continue;
              }
              bool near = vo == vp;  // unused: itself or a neighbour, so no other vertex's infinity gets in
              for (int64_t i = 0; i < m && !near && m < 3000; ++i)
                near = (src[i] == vp && dst[i] == vo) || (dst[i] == vp && src[i] == vo);
              CHECK(near || m >= 3000, "unused slot names a neighbour");
            }
        cols += K;
      }
    }
    CHECK(cols == d.ncol, "columns of a part");
  }
  CHECK(L.n_col >= L.part.back().s0 + L.part.back().ncol + kMarchAhead, "room for the read-ahead");
  for (int64_t t = 0; t < m; ++t) CHECK(slots[t] == (src[t] == dst[t] ? 1 : 2), "slots per task");

  const int D = 2, T = 3;
  const double tau = 0.01;
  std::mt19937 rng(7);
  std::normal_distribution<double> nd(0, 1);
  std::vector<double> x((size_t)n * D), w(m), g((size_t)L.n_rec * D, 0.0), wl(64 * (size_t)L.n_col, 0.0);
  for (auto& v : x) v = nd(rng);
  for (auto& v : w) v = 0.5 + (rng() % 1000) / 1000.0;
  for (int v = 0; v < n; ++v)
    for (int c = 0; c < D; ++c) g[(size_t)L.rec_of[v] * D + c] = x[(size_t)v * D + c];
  for (size_t i = 0; i < wl.size(); ++i)
    if (L.wmap[i] >= 0) wl[i] = w[L.wmap[i]];
  auto term = [&](const double* xo, const double* xp, double wt, double* a, double sign) {
    double d[D], q = 1;
    for (int c = 0; c < D; ++c) d[c] = xo[c] - xp[c], q += d[c] * d[c];
    for (int c = 0; c < D; ++c) a[c] += sign * wt * d[c] / q;
  };
  for (int s = 0; s < T; ++s) {
    std::vector<double> f((size_t)n * D, 0.0), g2 = g;
    for (int64_t t = 0; t < m; ++t) {
      term(&x[(size_t)dst[t] * D], &x[(size_t)src[t] * D], w[t], &f[(size_t)src[t] * D], 1);
      term(&x[(size_t)dst[t] * D], &x[(size_t)src[t] * D], w[t], &f[(size_t)dst[t] * D], -1);
    }
    for (size_t i = 0; i < x.size(); ++i) x[i] += tau * f[i];
    for (const MarchPart& d : L.part)
      for (int v = 0; v < L.warps; ++v) {
        int c = L.tab[d.q0 + v];
        for (int j = v; j < d.nsl; j += L.warps) {
          const int end = c + L.tab[d.q0 + L.warps + j];
          for (; c < end; ++c)
            for (int l = 0; l < 32; ++l) {
              const int p = 32 * j + l;
              if (p >= d.own) continue;
              double a[D] = {0, 0};
              for (int u = 0; u < 2; ++u) {
                const int64_t at = 32 * ((int64_t)d.s0 + c) + l;
                const int o = (L.ent[at] >> (16 * u)) & kSlotPos;
                term(&g[(size_t)record(d, o) * D], &g[(size_t)(d.lo + p) * D], wl[2 * at + u], a, 1);
              }
              for (int k = 0; k < D; ++k) g2[(size_t)(d.lo + p) * D + k] += tau * a[k];
            }
        }
      }
    g.swap(g2);
  }
  double err = 0, nrm = 0;
  for (int v = 0; v < n; ++v)
    for (int c = 0; c < D; ++c) {
      const double want = x[(size_t)v * D + c], got = g[(size_t)L.rec_of[v] * D + c];
      err += (got - want) * (got - want);
      nrm += want * want;
    }
  CHECK(std::sqrt(err / nrm) < 1e-13, "emulated steps against the edge list");
  printf("n %d m %lld C %d %s: parts %d, rel %.2e\n", n, (long long)m, C, dflt ? "default" : "partitioned", L.parts,
         std::sqrt(err / nrm));
}

int main() {
  std::mt19937 rng(3);
  auto graph = [&](int n, int m, int reach, int touched, std::vector<int32_t>& s, std::vector<int32_t>& d) {
    s.clear(), d.clear();
    for (int i = 0; i < m; ++i) {
      s.push_back((int32_t)(rng() % touched));
      d.push_back((int32_t)((s.back() + 1 + rng() % reach) % touched));
    }
    for (int i = 0; i < m / 50; ++i) s[i] = d[i];                             // self loops
    for (int i = m / 50; i < m / 25; ++i) s[i] = s[i + m / 25], d[i] = d[i + m / 25];  // repeated pairs
    (void)n;
  };
  std::vector<int32_t> s, d;
  graph(40, 90, 5, 40, s, d);
  check(40, s, d, 16, false, 152, 1);  // one part
  graph(900, 2500, 30, 800, s, d);     // isolated vertices
  for (bool dflt : {false, true}) check(900, s, d, 64, dflt, 152, 2);
  graph(9000, 25000, 40, 9000, s, d);
  for (int parts : {1, 3, 152})
    for (bool dflt : {false, true}) check(9000, s, d, 256, dflt, parts, 4);
  // the same for any number of threads
  HostSchedule h;
  CHECK(build(h, 9000, s, d, 256, false), "schedule");
  MarchLayout a, b;
  CHECK(build_march(h, 152, 1, a) && build_march(h, 152, 7, b), "layouts");
  CHECK(a.ent == b.ent && a.wmap == b.wmap && a.halo == b.halo && a.rec_of == b.rec_of && a.gslot == b.gslot, "threads");
  // a vertex in more tasks than one lane should walk
  s.assign(500, 0);
  d.resize(500);
  for (int i = 0; i < 500; ++i) d[i] = i + 1;
  HostSchedule star;
  CHECK(build(star, 501, s, d, 64, false), "schedule");
  CHECK(!build_march(star, 152, 2, a), "a hub is refused");
  printf("total fails %d\n", fails);
  return fails != 0;
}
