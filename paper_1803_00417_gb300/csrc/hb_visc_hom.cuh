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

// v, or -v when m has the sign bit set (on the integer pipe)
__host__ __device__ __forceinline__ float sgn_flip(float v, unsigned m) {
#ifdef __CUDA_ARCH__
  return __uint_as_float(__float_as_uint(v) ^ m);
#else
  return m ? -v : v;
#endif
}
__host__ __device__ __forceinline__ double sgn_flip(double v, unsigned m) {
#ifdef __CUDA_ARCH__
  return __hiloint2double(__double2hiint(v) ^ (int)m, __double2loint(v));
#else
  return m ? -v : v;
#endif
}

// Where the neighbours of cell p along each axis sit: the offsets om / op
// below and above it (wrapped on a periodic axis; 0 past a wall, where the
// homogeneous ghost is minus the cell's own value: fm / fp hold the sign bit
// there and 0 elsewhere).
template <int D, bool PER>
struct HomNbr {
  int om[D], op[D];
  unsigned fm[D], fp[D];
  __host__ __device__ __forceinline__ HomNbr(const Geom& g, const int* p) {
    int s = 1;
#pragma unroll
    for (int a = 0; a < D; ++a) {
      const bool lo = p[a] == 0, hi = p[a] == g.n[a] - 1;
      if (PER && g.per[a]) {
        om[a] = lo ? (g.n[a] - 1) * s : -s;
        op[a] = hi ? -(g.n[a] - 1) * s : s;
        fm[a] = fp[a] = 0u;
      } else {
        om[a] = lo ? 0 : -s;
        op[a] = hi ? 0 : s;
        fm[a] = lo ? 0x80000000u : 0u;
        fp[a] = hi ? 0x80000000u : 0u;
      }
      s *= g.n[a];
    }
  }
};

// the faces of axis a below and above cell p in the face array ef[a] (from
// face f on, the next one fs further): both values
template <int D>
__host__ __device__ __forceinline__ int face_step(const Geom& g, int a) {
  return a == 0 ? 1 : (a == 1 ? g.n[0] : g.n[0] * g.n[1]);
}

// 1 / (1 + bs diag) of component c at cell p, diag = sum_a k_a (e_lo + e_hi)
// with wall faces counted twice (their ghost is minus the cell), k_c = 2,
// k_a = 1 otherwise, bs = beta / h^2
template <int D, typename T, bool PER>
__host__ __device__ __forceinline__ T visc_inv_point(const T* const* ef, const Geom& g, int c, const int* p, T bs) {
  T diag = T(0);
#pragma unroll
  for (int a = 0; a < D; ++a) {
    const int f = fidx(g, a, p[0], p[1], p[2]);
    const bool wall = !(PER && g.per[a]);
    T lo = ef[a][f], hi = ef[a][f + face_step<D>(g, a)];
    if (wall && p[a] == 0) lo = rn_mul(T(2), lo);
    if (wall && p[a] == g.n[a] - 1) hi = rn_mul(T(2), hi);
    const T w = rn_add(lo, hi);
    diag = a == c ? rn_fma(T(2), w, diag) : rn_add(diag, w);
  }
  return T(1) / rn_fma(bs, diag, T(1));
}

// The differences of u_a along c at the cell id and at its two neighbours
// along a (homogeneous ghosts past a wall normal to c)
template <int D, typename T, bool PER>
__host__ __device__ __forceinline__ void hom_cross(const T* ua, const HomNbr<D, PER>& nb, int id, int a, int c, T& xhi,
                                                   T& xlo) {
  const T* q = ua + id;
  const T mid = rn_add(sgn_flip(q[nb.op[c]], nb.fp[c]), -sgn_flip(q[nb.om[c]], nb.fm[c]));
  const T* qp = q + nb.op[a];
  const T* qm = q + nb.om[a];
  xhi = rn_add(mid, rn_add(sgn_flip(qp[nb.op[c]], nb.fp[c]), -sgn_flip(qp[nb.om[c]], nb.fm[c])));
  xlo = rn_add(rn_add(sgn_flip(qm[nb.op[c]], nb.fp[c]), -sgn_flip(qm[nb.om[c]], nb.fm[c])), mid);
}

// Gauss-Seidel value of component C at cell p (flat index id): visc_gs_core's
// sums with zero coefficients at wall faces (a wall face has no cross term,
// and its normal term is in the diagonal), times the diagonal's reciprocal.
// Explicitly rounded in FP32: the launches and the fused tail get the same
// bits.
template <int D, typename T, int C, bool PER>
__host__ __device__ __forceinline__ T visc_gs_hom(const T* u, T bc, T inv, const T* const* ef, const Geom& g,
                                                  const int* p, int id, T bs) {
  const HomNbr<D, PER> nb(g, p);
  const T* uc = u + (size_t)C * g.ncell + id;
  T offd = T(0), cross = T(0);
#pragma unroll
  for (int a = 0; a < D; ++a) {
    const T* e = ef[a] + fidx(g, a, p[0], p[1], p[2]);
    const T elo = nb.fm[a] ? T(0) : e[0], ehi = nb.fp[a] ? T(0) : e[face_step<D>(g, a)];
    const T f = rn_fma(elo, uc[nb.om[a]], rn_mul(ehi, uc[nb.op[a]]));
    offd = a == C ? rn_fma(T(2), f, offd) : rn_add(offd, f);
    if (a != C) {
      T xhi, xlo;
      hom_cross<D, T, PER>(u + (size_t)a * g.ncell, nb, id, a, C, xhi, xlo);
      cross = rn_add(cross, rn_fma(ehi, xhi, -rn_mul(elo, xlo)));
    }
  }
  return rn_mul(rn_fma(bs, rn_fma(T(0.25), cross, offd), bc), inv);
}

// b - (u - beta L u) of component C at cell p, homogeneous walls: tensor_core's
// terms, with the normal flux of a wall face e (u - (-u)) and no cross term
// there
template <int D, typename T, int C, bool PER>
__host__ __device__ __forceinline__ T visc_res_hom(const T* u, T bc, const T* const* ef, const Geom& g, const int* p,
                                                   int id, T beta) {
  const HomNbr<D, PER> nb(g, p);
  const T* uc = u + (size_t)C * g.ncell + id;
  const T u0 = uc[0];
  T acc = T(0);
#pragma unroll
  for (int a = 0; a < D; ++a) {
    const T* e = ef[a] + fidx(g, a, p[0], p[1], p[2]);
    const T elo = e[0], ehi = e[face_step<D>(g, a)];
    const T dlo = rn_add(u0, -sgn_flip(uc[nb.om[a]], nb.fm[a]));
    const T dhi = rn_add(sgn_flip(uc[nb.op[a]], nb.fp[a]), -u0);
    T flo, fhi;
    if (a == C) {
      flo = rn_mul(elo, rn_mul(T(2), dlo));
      fhi = rn_mul(ehi, rn_mul(T(2), dhi));
    } else {
      T xhi, xlo;
      hom_cross<D, T, PER>(u + (size_t)a * g.ncell, nb, id, a, C, xhi, xlo);
      flo = rn_mul(elo, rn_fma(T(0.25), nb.fm[a] ? T(0) : xlo, dlo));
      fhi = rn_mul(ehi, rn_fma(T(0.25), nb.fp[a] ? T(0) : xhi, dhi));
    }
    acc = rn_add(acc, rn_add(fhi, -flo));
  }
  const T Lu = rn_mul(acc, g_ihh<T>(g));
  return rn_add(bc, -rn_fma(-beta, Lu, u0));
}

// thread t of a sweep of colour col (rb_cell's map)
template <int D, typename T, int C, bool PER>
__host__ __device__ __forceinline__ void visc_smooth_hom_at(T* u, const T* b, const T* inv, const T* const* ef,
                                                            const Geom& g, int col, T bs, int t) {
  int p[3];
  if (!rb_cell<D>(g, t, col, p)) return;
  const int id = cidx<D>(g, p[0], p[1], p[2]);
  const size_t o = (size_t)C * g.ncell + id;
  u[o] = visc_gs_hom<D, T, C, PER>(u, b[o], inv[o], ef, g, p, id, bs);
}

template <int D, typename T, int C, bool PER>
__global__ void __launch_bounds__(256) k_visc_smooth_hom(T* u, const T* __restrict__ b, const T* __restrict__ inv,
                                                         const T* __restrict__ ef0, const T* __restrict__ ef1,
                                                         const T* __restrict__ ef2, const __grid_constant__ Geom g,
                                                         int col, T bs) {
  const T* ef[3] = {ef0, ef1, ef2};
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t < rb_count<D>(g)) visc_smooth_hom_at<D, T, C, PER>(u, b, inv, ef, g, col, bs, t);
}

// r = b - (u - beta L u) of every component (thread t: cell t)
template <int D, typename T, bool PER>
__host__ __device__ __forceinline__ void visc_res_hom_at(const T* u, const T* b, T* r, const T* const* ef,
                                                         const Geom& g, T beta, int t) {
  int p[3];
  cell_coords<D>(g, t, p[0], p[1], p[2]);
  r[t] = visc_res_hom<D, T, 0, PER>(u, b[t], ef, g, p, t, beta);
  const size_t o1 = (size_t)g.ncell + t;
  r[o1] = visc_res_hom<D, T, 1, PER>(u, b[o1], ef, g, p, t, beta);
  if constexpr (D == 3) {
    const size_t o2 = 2 * (size_t)g.ncell + t;
    r[o2] = visc_res_hom<D, T, 2, PER>(u, b[o2], ef, g, p, t, beta);
  }
}

template <int D, typename T, bool PER>
__global__ void __launch_bounds__(256) k_visc_res_hom(const T* __restrict__ u, const T* __restrict__ b,
                                                      T* __restrict__ r, const T* __restrict__ ef0,
                                                      const T* __restrict__ ef1, const T* __restrict__ ef2,
                                                      const __grid_constant__ Geom g, T beta) {
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
