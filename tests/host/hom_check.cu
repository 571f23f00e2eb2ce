// Host build of the branch-free homogeneous-wall viscous sweep and residual
// (hb_visc_hom.cuh) against the general forms (visc_gs_point, mg_tensor_point)
// on seeded fields: every cell of boxes with walls and periodic axes, down to
// two cells per axis, FP64 and FP32.  Driven by tests/test_host_hom.py.
//
// The two forms sum the same terms in another order, so they differ by
// rounding: at most kOps operations of relative error eps on terms whose
// magnitudes add up to `scale` (the update is a weighted mean of neighbours
// with weights up to 3 in all, plus b over the diagonal; the residual's terms
// are at most 4 bs diag max|u|, with wall faces counted twice).
#include <cmath>
#include <cstdio>
#include <cstring>
#include <limits>
#include <vector>

#include "hb_internal.h"
#include "hb_visc_hom.cuh"

using namespace hb;

static unsigned long long seed_;
static double rnd() {
  seed_ = seed_ * 6364136223846793005ull + 1442695040888963407ull;
  return (double)(seed_ >> 11) / 4503599627370496.0 - 1.0;
}

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

template <int D, typename T, int C, bool PER>
static bool check_comp(const Geom& g, const std::vector<T>& u, const std::vector<T>& b, const T* const* ef, T beta) {
  const T bs = beta * g_ihh<T>(g);
  const double eps = std::numeric_limits<T>::epsilon(), kOps = 64;
  double umax = 0.0;
  for (T v : u) umax = std::fmax(umax, std::fabs((double)v));
  for (int t = 0; t < g.ncell; ++t) {
    int p[3];
    cell_coords<D>(g, t, p[0], p[1], p[2]);
    const T bc = b[(size_t)C * g.ncell + t], u0 = u[(size_t)C * g.ncell + t];
    const T inv = visc_inv_point<D, T, PER>(ef, g, C, p, bs);
    const double w = (double)visc_gs_point<D, T, PER>(u.data(), b.data(), FaceEta<T>{ef}, g, C, p, beta, true);
    const double v = (double)visc_gs_hom<D, T, PER>(u.data(), bc, inv, ef, g, C, p, t, bs);
    const double s1 = 3 * umax + std::fabs((double)bc);
    const T Lu = mg_tensor_point<D, T, PER>(u.data(), FaceEta<T>{ef}, g, C, p, true);
    const double rw = (double)op_out<T>(u0, Lu, beta, b.data(), (size_t)C * g.ncell + t);
    const double r = (double)visc_res_hom<D, T, PER>(u.data(), bc, ef, g, C, p, t, beta);
    const double s2 = std::fabs((double)bc) + umax * (1 + 4 / (double)inv);
    if (!(std::fabs(v - w) <= kOps * eps * s1) || !(std::fabs(r - rw) <= kOps * eps * s2)) {
      std::fprintf(stderr, "D %d C %d PER %d n %d %d %d cell %d %d %d: sweep %.17g %.17g, residual %.17g %.17g\n", D, C,
                   (int)PER, g.n[0], g.n[1], g.n[2], p[0], p[1], p[2], v, w, r, rw);
      return false;
    }
  }
  return true;
}

template <int D, typename T>
static bool check(const Geom& g, double bb) {
  std::vector<T> u((size_t)D * g.ncell), b(u.size()), e[3];
  const T* ef[3] = {nullptr, nullptr, nullptr};
  for (T& v : u) v = (T)rnd();
  for (T& v : b) v = (T)rnd();
  for (int a = 0; a < D; ++a) {
    e[a].resize(g.nface[a]);
    for (T& v : e[a]) v = (T)std::exp(3.0 * rnd());
    if (g.per[a])  // the last face along a periodic axis repeats the first
      for (int t = 0; t < g.nface[a]; ++t) {
        int p[3];
        face_coords(g, a, t, p[0], p[1], p[2]);
        if (p[a] != g.n[a]) continue;
        p[a] = 0;
        e[a][t] = e[a][fidx(g, a, p[0], p[1], p[2])];
      }
    ef[a] = e[a].data();
  }
  const T beta = (T)bb;
  bool ok = check_comp<D, T, 0, true>(g, u, b, ef, beta) && check_comp<D, T, 1, true>(g, u, b, ef, beta) &&
            check_comp<D, T, D - 1, true>(g, u, b, ef, beta);
  if (!g.per[0] && !g.per[1] && !g.per[2])
    ok = ok && check_comp<D, T, 0, false>(g, u, b, ef, beta) && check_comp<D, T, 1, false>(g, u, b, ef, beta) &&
         check_comp<D, T, D - 1, false>(g, u, b, ef, beta);
  return ok;
}

int main(int argc, char** argv) {
  if (argc != 8) return 1;
  const int d = std::atoi(argv[1]);
  int n[3], per[3];
  for (int a = 0; a < 3; ++a) {
    n[a] = std::atoi(argv[2 + a]);
    per[a] = argv[5][a] == '1';
  }
  const double beta = std::atof(argv[6]);
  seed_ = std::strtoull(argv[7], nullptr, 10);
  const Geom g = make(d, n, per);
  const bool ok = d == 3 ? check<3, double>(g, beta) && check<3, float>(g, beta)
                         : check<2, double>(g, beta) && check<2, float>(g, beta);
  return ok ? 0 : 3;
}
