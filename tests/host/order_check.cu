// Host check of the sweeps' order on a coarsest level: the passes of the
// one-block bottom kernels and of the fused V-cycle tail (the maps the kernels
// themselves walk, both the indexed and the register-slot form, for every slab
// of every cluster size).  In each
//  * a sweep visits every point of the level once,
//  * no two points of one pass are neighbours, also through a periodic wrap (a
//    pass updates in place without a barrier, so they would race); in the slot
//    form, which stores a pass's values behind a barrier where the level is odd
//    along a periodic axis, none but those that the wrap of such an axis makes
//    neighbours,
//  * on a periodic axis node n, the copy of node 0, is in node 0's pass.
// Driven by tests/test_host_sweep_order.py.
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <vector>

#include "hb_internal.h"
#include "hb_vcycle_tail.cuh"

using namespace hb;
using namespace hb::batch;

static Geom make(int d, const int* n, const int* per) {
  Geom g;
  std::memset(&g, 0, sizeof g);
  for (int a = 0; a < 3; ++a) {
    g.n[a] = a < d ? n[a] : 1;
    g.per[a] = a < d ? per[a] : 0;
  }
  g.h = 1.0 / 16;
  g.ncell = g.n[0] * g.n[1] * g.n[2];
  g.nnode = (g.n[0] + 1) * (g.n[1] + 1) * (d == 3 ? g.n[2] + 1 : 1);
  g.nface[0] = (g.n[0] + 1) * g.n[1] * g.n[2];
  g.nface[1] = g.n[0] * (g.n[1] + 1) * g.n[2];
  g.nface[2] = d == 3 ? g.n[0] * g.n[1] * (g.n[2] + 1) : 0;
  geom_finish(g);
  return g;
}

// the pass of every point, by coordinates
template <int D, bool NODE>
struct Passes {
  const Geom& g;
  int e[3];
  std::vector<int> pass;
  bool ok = true;
  explicit Passes(const Geom& g_) : g(g_) {
    for (int a = 0; a < 3; ++a) e[a] = a < D ? g.n[a] + (NODE ? 1 : 0) : 1;
    pass.assign((size_t)e[0] * e[1] * e[2], -1);
  }
  int& at(const int* p) { return pass[p[0] + e[0] * (p[1] + (D == 3 ? e[1] * p[2] : 0))]; }
  void visit(const int* p, int q) {
    for (int a = 0; a < D; ++a) ok = ok && p[a] >= 0 && p[a] < e[a];
    if (!ok) return;
    ok = at(p) == -1;
    at(p) = q;
  }
  // the wrap of an odd axis makes p and q neighbours: among 0, n - 1 and (nodes) n
  bool odd_pair(const int* p, const int* q) const {
    for (int a = 0; a < D; ++a) {
      const int n = g.n[a];
      auto end = [&](int v) { return v == 0 || v == n - 1 || v == n; };
      if (odd_wrap(g, a) && p[a] != q[a] && end(p[a]) && end(q[a])) return true;
    }
    return false;
  }
  bool check(const char* what, bool slots = false) {
    bool good = ok;
    for (int t = 0; t < (int)pass.size() && good; ++t) {
      int p[3] = {t % e[0], t / e[0] % e[1], t / e[0] / e[1]};
      good = pass[t] >= 0;
      for (int o = 0; o < 27 && good; ++o) {
        int q[3], d[3] = {o % 3 - 1, o / 3 % 3 - 1, o / 9 - 1}, nz = 0;
        bool in = true;
        for (int a = 0; a < 3; ++a) {
          nz += d[a] != 0;
          q[a] = p[a] + d[a];
          if (a >= D) in = in && d[a] == 0;
          if (a < D && (q[a] < 0 || q[a] >= e[a])) {
            // node n repeats node 0
            if (g.per[a])
              q[a] = q[a] < 0 ? g.n[a] - 1 : (NODE ? 1 : 0);
            else
              in = false;
          }
        }
        if (!in || nz == 0 || (!NODE && nz > 1)) continue;
        if (q[0] == p[0] && q[1] == p[1] && q[2] == p[2]) continue;
        good = at(q) != pass[t] || (slots && odd_pair(p, q));
      }
      for (int a = 0; a < D && good && NODE; ++a)
        if (g.per[a] && p[a] == g.n[a]) {
          int q[3] = {p[0], p[1], p[2]};
          q[a] = 0;
          good = at(q) == pass[t];
        }
    }
    if (!good)
      std::fprintf(stderr, "%s: D %d n %d %d %d per %d%d%d\n", what, D, g.n[0], g.n[1], g.n[2], g.per[0], g.per[1], g.per[2]);
    return good;
  }
};

// the kernels of one block
template <int D>
static bool bottoms(const Geom& g) {
  Passes<D, false> c(g);
  for (int q = 0; q < rb_passes(g); ++q)
    for (int t = 0; t < rb_count<D>(g); ++t) {
      int p[3];
      if (rb_pass_cell<D>(g, t, q, p)) c.visit(p, q);
    }
  Passes<D, true> n(g);
  for (int q = 0; q < nd_passes<D>(g); ++q)
    for (int t = 0; t < nd_pass_count<D>(g, q); ++t) {
      int p[3];
      nd_pass_node<D>(g, t, q, p);
      n.visit(p, q);
    }
  return c.check("bottom, cells") && n.check("bottom, nodes");
}

// the tail's passes of the first component over the slabs of a cluster of nblk blocks
template <int D, typename T, int KIND, bool PER>
static bool tail(const Geom& g, int nblk, bool solo) {
  constexpr bool NODE = KIND == kNodal;
  Passes<D, NODE> a(g), b(g);
  const int np = tail_passes<D, KIND, PER>(g) / (KIND == kVisc ? D : 1);
  for (int r = 0; r < nblk; ++r) {
    TailLevel<T> w;
    unsigned at = 0;
    tail_level_init<D, T, KIND>(w, g, nblk, r, solo, at);
    if (w.k0 >= w.k1) continue;
    for (int q = 0; q < np; ++q)
      for (int t = 0; t < tail_pass_count<D, T, KIND, PER>(w, g, q); ++t) {
        int p[3];
        if (tail_pass_point<D, T, KIND, PER>(w, g, q, t, p)) a.visit(p, q);
      }
    for (int u = 0; u < 4 * w.ps * w.rp + 64; ++u) {
      TailSlot<D, T> s;
      tail_slot_init<D, T, KIND, PER, PER>(s, w, g, u);
      if (s.col < 0) continue;
      const int ex = g.n[0] + (NODE ? 1 : 0), p[3] = {s.q % ex, D == 3 ? s.q / ex : s.k, D == 3 ? s.k : 0};
      b.visit(p, s.col);
    }
  }
  return a.check("tail, indexed") && b.check("tail, slots", true) && (rb_parts(g) == 2 || a.pass == b.pass);
}

template <int D, bool PER>
static bool all(const Geom& g) {
  if (!bottoms<D>(g)) return false;
  for (int nblk = 1; nblk <= 16; nblk *= 2)
    if (!tail<D, double, kVisc, PER>(g, nblk, false) || !tail<D, double, kVisc, PER>(g, nblk, true) ||
        !tail<D, double, kMac, PER>(g, nblk, true) || !tail<D, double, kNodal, PER>(g, nblk, true))
      return false;
  return true;
}

int main(int argc, char** argv) {
  if (argc != 6) return 1;
  const int d = std::atoi(argv[1]);
  int n[3], per[3];
  for (int a = 0; a < 3; ++a) {
    n[a] = std::atoi(argv[2 + a]);
    per[a] = argv[5][a] == '1';
  }
  const Geom g = make(d, n, per);
  bool ok = d == 3 ? all<3, true>(g) : all<2, true>(g);
  if (!per[0] && !per[1] && !per[2]) ok = ok && (d == 3 ? all<3, false>(g) : all<2, false>(g));
  return ok ? 0 : 3;
}
