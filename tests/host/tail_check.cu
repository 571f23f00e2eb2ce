// Host check of the fused V-cycle tail's plan (hb_vcycle_tail.cuh): over a
// range of hierarchies, arithmetics, problems and cluster sizes,
//  * every block of the cluster arrives at the same cluster barriers (the
//    kernel's visit loop restated with counters),
//  * the slabs of a level cover its planes once, and a swept coarsest level is
//    never split when the level above it is not,
//  * the shared-memory arrays of a block neither overlap nor pass the size
//    that the launch asks for,
//  * every halo plane of every slab is written by exactly one point's update
//    (tail_put's rules restated) and holds the plane its neighbour offsets
//    mean.
// Driven by tests/test_host_tail.py.
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
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

#define NEED(x)                                                                             \
  do {                                                                                      \
    if (!(x)) {                                                                             \
      std::fprintf(stderr, "line %d: %s (D %d kind %d T %d lf %d L %d nblk %d swept %d)\n", __LINE__, #x, D, KIND, \
                   (int)sizeof(T), lf, L, nblk, (int)swept);                                \
      return false;                                                                         \
    }                                                                                       \
  } while (0)

// who writes which plane into the halos of the slabs, by tail_put's rules
template <int D, typename T, typename U, int KIND>
static bool halos(const Geom& g, const std::vector<TailLevel<U>>& w, int lf, int L, int nblk, bool swept) {
  const bool per = g.per[D - 1];
  std::map<std::pair<int, int>, std::vector<int>> got;  // (block, halo index) -> planes
  for (int r = 0; r < w[0].np; ++r) {
    const TailLevel<U>& v = w[r];
    for (int k = v.k0; k < v.k1; ++k) {
      const int kl = k - v.k0;
      if (v.np > 1) {
        if (kl == 0 && k > 0) got[{r - 1, v.rp + 1}].push_back(k);
        if (k == v.k1 - 1 && k < v.N - 1) got[{r + 1, 0}].push_back(k);
      }
      if (per) {
        const int lr = (v.N - 1) / v.rp, lc = v.N - lr * v.rp;
        const int lo = KIND == kNodal ? v.N - 2 : v.N - 1, hi = KIND == kNodal ? 1 : 0;
        if (k == lo) got[{0, 0}].push_back(k);
        if (k == hi) got[{lr, lc + 1}].push_back(k);
      }
    }
  }
  for (int r = 0; r < w[0].np; ++r) {
    const TailLevel<U>& v = w[r];
    const int nk = v.k1 - v.k0;
    NEED(nk > 0);
    int below = v.k0 - 1, above = v.k1;
    if (below < 0) below = per ? (KIND == kNodal ? v.N - 2 : v.N - 1) : -1;
    if (above >= v.N) above = per ? (KIND == kNodal ? 1 : 0) : -1;
    const std::vector<int> lo = got[{r, 0}], hi = got[{r, nk + 1}];
    NEED(below < 0 ? lo.empty() : lo == std::vector<int>{below});
    NEED(above < 0 ? hi.empty() : hi == std::vector<int>{above});
  }
  return true;
}

template <int D, typename T, int KIND>
static bool check(const std::vector<Geom>& hs, int lf, int nblk, bool swept) {
  const int L = (int)hs.size() - 1;
  std::vector<const Geom*> gs;
  for (const Geom& g : hs) gs.push_back(&g);
  const size_t smem = tail_smem<D, T, KIND>(gs.data(), lf, L, nblk, swept);
  const bool has_wide = tail_has_wide<D, T, KIND>(gs.data(), lf, L, swept);
  std::vector<std::vector<TailLevel<T>>> lev(L + 1);
  std::vector<TailLevel<double>> bot(nblk);
  std::vector<unsigned> top(nblk);
  for (int l = 0; l <= L; ++l) lev[l].resize(nblk);
  for (int r = 0; r < nblk; ++r) {
    unsigned at = 0;
    for (int l = lf; l <= L; ++l) {
      TailLevel<T>& w = lev[l][r];
      if (l < L) {
        tail_level_init<D, T, KIND>(w, hs[l], nblk, r, false, at);
      } else if (swept) {
        tail_level_init<D, double, KIND>(bot[r], hs[l], nblk, r,
                                         tail_swept_solo<D, T, KIND>(l > lf ? &hs[l - 1] : nullptr, nblk), at);
        w.np = bot[r].np;
      } else {
        tail_level_init<D, T, KIND>(w, hs[l], 1, r, true, at);
      }
    }
    top[r] = at;
    NEED(at <= smem);
  }
  for (int l = lf; l <= L; ++l) {
    if (l < L && !halos<D, T, T, KIND>(hs[l], lev[l], lf, L, nblk, swept)) return false;
    if (l == L && swept && !halos<D, T, double, KIND>(hs[l], bot, lf, L, nblk, swept)) return false;
    if (l > lf) NEED(lev[l][0].np <= 1 || lev[l - 1][0].np > 1);  // no wide level below a one-slab one
    NEED(lev[l][0].np <= nblk);
    NEED(lev[l][0].np == 1 || has_wide);
  }
  // scratch of the one-slab levels
  for (int l = lf; l < L; ++l)
    if (lev[l][0].np == 1) {
      NEED(top[0] + (size_t)(KIND == kVisc ? D : 1) * lev[l][0].N * lev[l][0].ps * sizeof(T) <= smem);
      break;
    }
  // cluster barriers of each block in the visit loop, as (visit, place) marks
  std::vector<std::vector<int>> marks(nblk);
  const int nd = L - lf, nu = 2, sweeps = 3;
  for (int r = 0; r < nblk; ++r) {
    auto& m = marks[r];
    for (int visit = 0; visit <= 2 * nd; ++visit) {
      const bool down = visit < nd;
      const int l = visit <= nd ? lf + visit : lf + 2 * nd - visit;
      const bool wide = lev[l][0].np > 1;
      if (!wide && r) continue;
      auto sync = [&](int place) {
        if (wide) m.push_back(visit * 16 + place);
      };
      if (visit == nd) {
        if (swept)
          for (int s = 0; s < sweeps; ++s) sync(0);
      } else {
        if (!down) {
          sync(1);
          sync(2);
        }
        for (int s = 0; s < nu; ++s) sync(3);
        if (down) {
          sync(4);
          const bool cwide = lev[l + 1][0].np > 1;
          if (cwide || r == 0)
            if (cwide) m.push_back(visit * 16 + 5);
        }
      }
    }
    NEED(m == marks[0]);
  }
  return true;
}

template <int D>
static bool all(const std::vector<Geom>& hs, int nblk) {
  const int L = (int)hs.size() - 1;
  for (int lf = 0; lf <= L; ++lf)
    for (int swept = 0; swept < 2; ++swept)
      if (!check<D, float, kVisc>(hs, lf, nblk, swept) || !check<D, float, kMac>(hs, lf, nblk, swept) ||
          !check<D, float, kNodal>(hs, lf, nblk, swept) || !check<D, double, kVisc>(hs, lf, nblk, swept) ||
          !check<D, double, kMac>(hs, lf, nblk, swept) || !check<D, double, kNodal>(hs, lf, nblk, swept))
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
  std::vector<Geom> hs{make(d, n, per)};
  for (;;) {
    const Geom& g = hs.back();
    bool can = true;
    for (int a = 0; a < d; ++a) can = can && g.n[a] % 2 == 0 && g.n[a] / 2 >= 2;
    if (!can) break;
    hs.push_back(d == 3 ? coarse_of<3>(g) : coarse_of<2>(g));
  }
  for (int nblk = 1; nblk <= 16; nblk *= 2)
    if (!(d == 3 ? all<3>(hs, nblk) : all<2>(hs, nblk))) return 3;
  return 0;
}
