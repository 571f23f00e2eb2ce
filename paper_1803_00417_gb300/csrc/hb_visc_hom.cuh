// The viscous smoothing and residual of the V-cycles on levels with stored
// face viscosities (every level of the FP64 V-cycles, the coarse levels of
// the FP32 ones): the operator with homogeneous walls, as the error equation
// has them, in one branch-free form for interior, wall and periodic cells,
// with the Gauss-Seidel diagonal's reciprocal precomputed.
//
// Why: GB300 issues two FP64 operations per SM and cycle, so the FP64 sweeps
// are bound by their count of FP64 operations: the update took about 31
// operations for the off-diagonal and cross terms, 9 for the diagonal and a
// division (a reciprocal iteration of FP64 operations) per cell, and a warp
// with a wall cell issued the wall stencil besides.  The diagonal depends on
// the viscosity and dt only, so k_visc_inv forms 1 / (1 + bs diag) once per
// solve (each solve runs 8 to 22 V-cycles of four sweeps), and the wall forms
// become a zeroed face coefficient and a flipped sign bit, which cost no
// floating-point operation.
#pragma once
#include "hb_mg_kernels.cuh"

namespace hb {

// One axis seen from a cell: the offsets om / op of the neighbours below and
// above (wrapped on a periodic axis; 0 past a wall, where the homogeneous
// ghost is minus the cell's own value: fm / fp hold the sign bit there and 0
// elsewhere).
struct HomAxis {
  int om, op;
  unsigned fm, fp;
  __host__ __device__ __forceinline__ HomAxis() {}
  // position q of n along an axis of stride s
  __host__ __device__ __forceinline__ HomAxis(int q, int n, int s, bool per) {
    const bool lo = q == 0, hi = q == n - 1;
    om = lo ? (per ? (n - 1) * s : 0) : -s;
    op = hi ? (per ? -(n - 1) * s : 0) : s;
    fm = lo && !per ? 0x80000000u : 0u;
    fp = hi && !per ? 0x80000000u : 0u;
  }
  // the slowest axis of a slab with a halo plane on either side: a periodic
  // neighbour is in the halo
  __host__ __device__ __forceinline__ HomAxis(int q, int n, int s, bool per, bool /*halo*/) {
    const bool lo = q == 0 && !per, hi = q == n - 1 && !per;
    om = lo ? 0 : -s;
    op = hi ? 0 : s;
    fm = lo ? 0x80000000u : 0u;
    fp = hi ? 0x80000000u : 0u;
  }
};

// the component's axis comes first, then the others in cyclic order
template <int D>
__host__ __device__ __forceinline__ int hom_next(int a) {
  return a + 1 == D ? 0 : a + 1;
}

// The stencil of component c at a cell, by role r = 0 (the component's own
// axis), 1, .. (the other axes in cyclic order): the axis as the cell sees it,
// the component of that axis at the cell, and the face viscosities below and
// above the cell on that axis.  c may be a run-time value.
template <int D, typename T>
struct HomCell {
  HomAxis ax[D];
  const T* u[D];
  T elo[D], ehi[D];
};

// 1 / (1 + bs diag), diag = sum_a k_a (e_lo + e_hi) with wall faces counted
// twice (their ghost is minus the cell), k = 2 on the component's own axis and
// 1 on the others, bs = beta / h^2
template <int D, typename T>
__host__ __device__ __forceinline__ T hom_inv(const HomCell<D, T>& s, T bs) {
  T diag = T(0);
#pragma unroll
  for (int r = 0; r < D; ++r) {
    T lo = s.elo[r], hi = s.ehi[r];
    if (s.ax[r].fm) lo = rn_mul(T(2), lo);
    if (s.ax[r].fp) hi = rn_mul(T(2), hi);
    const T w = rn_add(lo, hi);
    diag = r == 0 ? rn_mul(T(2), w) : rn_add(diag, w);
  }
  return T(1) / rn_fma(bs, diag, T(1));
}

// the differences of q's component along c at the cell and at its two
// neighbours along a (homogeneous ghosts past a wall normal to c), summed over
// the two cells of the face above (xhi) and below (xlo)
template <typename T>
__host__ __device__ __forceinline__ void hom_cross(const T* q, const HomAxis& a, const HomAxis& c, T& xhi, T& xlo) {
  const T mid = rn_add(sgn_flip(q[c.op], c.fp), -sgn_flip(q[c.om], c.fm));
  const T* qp = q + a.op;
  const T* qm = q + a.om;
  xhi = rn_add(mid, rn_add(sgn_flip(qp[c.op], c.fp), -sgn_flip(qp[c.om], c.fm)));
  xlo = rn_add(rn_add(sgn_flip(qm[c.op], c.fp), -sgn_flip(qm[c.om], c.fm)), mid);
}

// Gauss-Seidel value: visc_gs_core's sums with zero coefficients at wall faces
// (a wall face has no cross term, and its normal term is in the diagonal),
// times the diagonal's reciprocal.  Explicitly rounded in FP32: the launches
// and the fused tail get the same bits.
template <int D, typename T>
__host__ __device__ __forceinline__ T hom_gs(const HomCell<D, T>& s, T bc, T inv, T bs) {
  T offd = T(0), cross = T(0);
#pragma unroll
  for (int r = 0; r < D; ++r) {
    const HomAxis& a = s.ax[r];
    const T elo = a.fm ? T(0) : s.elo[r], ehi = a.fp ? T(0) : s.ehi[r];
    const T f = rn_fma(elo, s.u[0][a.om], rn_mul(ehi, s.u[0][a.op]));
    offd = r == 0 ? rn_mul(T(2), f) : rn_add(offd, f);
    if (r > 0) {
      T xhi, xlo;
      hom_cross(s.u[r], a, s.ax[0], xhi, xlo);
      cross = rn_add(cross, rn_fma(ehi, xhi, -rn_mul(elo, xlo)));
    }
  }
  return rn_mul(rn_fma(bs, rn_fma(T(0.25), cross, offd), bc), inv);
}

// u - beta L u: tensor_core's terms, with the normal flux of a wall face
// e (u - (-u)) and no cross term there
template <int D, typename T>
__host__ __device__ __forceinline__ T hom_op(const HomCell<D, T>& s, T beta, T ihh) {
  const T u0 = s.u[0][0];
  T acc = T(0);
#pragma unroll
  for (int r = 0; r < D; ++r) {
    const HomAxis& a = s.ax[r];
    T dlo = rn_add(u0, -sgn_flip(s.u[0][a.om], a.fm)), dhi = rn_add(sgn_flip(s.u[0][a.op], a.fp), -u0);
    if (r > 0) {
      T xhi, xlo;
      hom_cross(s.u[r], a, s.ax[0], xhi, xlo);
      dlo = rn_fma(T(0.25), a.fm ? T(0) : xlo, dlo);
      dhi = rn_fma(T(0.25), a.fp ? T(0) : xhi, dhi);
    }
    const T f = rn_fma(s.ehi[r], dhi, -rn_mul(s.elo[r], dlo));
    acc = r == 0 ? rn_mul(T(2), f) : rn_add(acc, f);
  }
  return rn_fma(-beta, rn_mul(acc, ihh), u0);
}
template <int D, typename T>
__host__ __device__ __forceinline__ T hom_res(const HomCell<D, T>& s, T bc, T beta, T ihh) {
  return rn_add(bc, -hom_op<D, T>(s, beta, ihh));
}

// the stencil of component c at cell p of a whole level (flat index id)
template <int D, typename T, bool PER>
__host__ __device__ __forceinline__ HomCell<D, T> hom_cell(const T* u, const T* const* ef, const Geom& g, int c,
                                                           const int* p, int id) {
  auto axis = [&](int a) {
    return HomAxis(p[a], g.n[a], a == 0 ? 1 : (a == 1 ? g.n[0] : g.n[0] * g.n[1]), PER && g.per[a]);
  };
  auto comp = [&](int a) { return u + (size_t)a * g.ncell + id; };
  auto face = [&](int a) { return ef[a] + fidx(g, a, p[0], p[1], p[2]); };
  auto step = [&](int a) { return a == 0 ? 1 : (a == 1 ? g.n[0] : g.n[0] * g.n[1]); };
  const int a1 = hom_next<D>(c), a2 = hom_next<D>(a1);
  if constexpr (D == 3)
    return {{axis(c), axis(a1), axis(a2)},
            {comp(c), comp(a1), comp(a2)},
            {*face(c), *face(a1), *face(a2)},
            {face(c)[step(c)], face(a1)[step(a1)], face(a2)[step(a2)]}};
  else
    return {{axis(c), axis(a1)},
            {comp(c), comp(a1)},
            {*face(c), *face(a1)},
            {face(c)[step(c)], face(a1)[step(a1)]}};
}

template <int D, typename T, bool PER>
__host__ __device__ __forceinline__ T visc_inv_point(const T* const* ef, const Geom& g, int c, const int* p, T bs) {
  return hom_inv<D, T>(hom_cell<D, T, PER>(nullptr, ef, g, c, p, 0), bs);
}
template <int D, typename T, bool PER>
__host__ __device__ __forceinline__ T visc_gs_hom(const T* u, T bc, T inv, const T* const* ef, const Geom& g, int c,
                                                  const int* p, int id, T bs) {
  return hom_gs<D, T>(hom_cell<D, T, PER>(u, ef, g, c, p, id), bc, inv, bs);
}
template <int D, typename T, bool PER>
__host__ __device__ __forceinline__ T visc_res_hom(const T* u, T bc, const T* const* ef, const Geom& g, int c,
                                                   const int* p, int id, T beta) {
  return hom_res<D, T>(hom_cell<D, T, PER>(u, ef, g, c, p, id), bc, beta, g_ihh<T>(g));
}

// thread t of a sweep of component c, colour col (rb_cell's map)
template <int D, typename T, bool PER>
__host__ __device__ __forceinline__ void visc_smooth_hom_at(T* u, const T* b, const T* inv, const T* const* ef,
                                                            const Geom& g, int c, int col, T bs, int t) {
  int p[3];
  if (!rb_cell<D>(g, t, col, p)) return;
  const int id = cidx<D>(g, p[0], p[1], p[2]);
  const size_t o = (size_t)c * g.ncell + id;
  u[o] = visc_gs_hom<D, T, PER>(u, b[o], inv[o], ef, g, c, p, id, bs);
}

template <int D, typename T, int C, bool PER>
__global__ void __launch_bounds__(256) k_visc_smooth_hom(T* u, const T* __restrict__ b, const T* __restrict__ inv,
                                                         const T* __restrict__ ef0, const T* __restrict__ ef1,
                                                         const T* __restrict__ ef2, const __grid_constant__ Geom g,
                                                         int col, T bs) {
  pdl_wait();
  const T* ef[3] = {ef0, ef1, ef2};
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t < rb_count<D>(g)) visc_smooth_hom_at<D, T, PER>(u, b, inv, ef, g, C, col, bs, t);
}

// r = b - (u - beta L u) of every component, or u - beta L u when b is null
// (thread t: cell t)
template <int D, typename T, bool PER>
__host__ __device__ __forceinline__ void visc_res_hom_at(const T* u, const T* b, T* r, const T* const* ef,
                                                         const Geom& g, T beta, int t) {
  int p[3];
  cell_coords<D>(g, t, p[0], p[1], p[2]);
#pragma unroll
  for (int c = 0; c < D; ++c) {
    const size_t o = (size_t)c * g.ncell + t;
    const T Au = hom_op<D, T>(hom_cell<D, T, PER>(u, ef, g, c, p, t), beta, g_ihh<T>(g));
    r[o] = b ? rn_add(b[o], -Au) : Au;
  }
}

template <int D, typename T, bool PER>
__global__ void __launch_bounds__(256) k_visc_res_hom(const T* __restrict__ u, const T* __restrict__ b,
                                                      T* __restrict__ r, const T* __restrict__ ef0,
                                                      const T* __restrict__ ef1, const T* __restrict__ ef2,
                                                      const __grid_constant__ Geom g, T beta) {
  pdl_wait();
  const T* ef[3] = {ef0, ef1, ef2};
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t < g.ncell) visc_res_hom_at<D, T, PER>(u, b, r, ef, g, beta, t);
}

// inv[c] = visc_inv_point of every cell and component (thread t: cell t)
template <int D, typename T, bool PER>
__host__ __device__ __forceinline__ void visc_inv_at(T* inv, const T* const* ef, const Geom& g, T bs, int t) {
  int p[3];
  cell_coords<D>(g, t, p[0], p[1], p[2]);
#pragma unroll
  for (int c = 0; c < D; ++c) inv[(size_t)c * g.ncell + t] = visc_inv_point<D, T, PER>(ef, g, c, p, bs);
}

template <int D, typename T>
__global__ void __launch_bounds__(256) k_visc_inv(T* inv, const T* __restrict__ ef0, const T* __restrict__ ef1,
                                                  const T* __restrict__ ef2, const __grid_constant__ Geom g, T bs) {
  pdl_wait();
  const T* ef[3] = {ef0, ef1, ef2};
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t < g.ncell) visc_inv_at<D, T, true>(inv, ef, g, bs, t);
}

// Block size of a one-thread-per-element launch: 256, or smaller while the
// launch would leave SMs without a block (the level then is bound by the
// latency of its few warps, and for FP64 by the two FP64 operations an SM
// issues per cycle, so the work is spread over as many SMs as it can fill)
inline int spread_threads(long long work) {
  int t = 256;
  while (t > 32 && work < 152LL * t) t >>= 1;
  return t;
}

}  // namespace hb
