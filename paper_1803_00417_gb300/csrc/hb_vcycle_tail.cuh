// Argument records of the multigrid operations on one cavity's level, the
// block-level exact bottom solve, and the fused V-cycle tail: one launch walks
// a cavity's small levels (smoothing, residual, restriction, bottom solve,
// prolongation) with barriers between the phases.  Used by the batched sweep
// (one thread-block cluster per cavity) and by the single-cavity solves (one
// cluster).
#pragma once
#include "hb_batch.cuh"
#include "hb_mg_kernels.cuh"
#include "hb_visc_hom.cuh"

namespace hb {
namespace batch {

enum Kind { kVisc = 0, kMac = 1, kNodal = 2 };

template <typename T>
struct ViscArg {
  T* x;
  const T* b;
  T* out;
  T* inv;  // the Gauss-Seidel reciprocals (k_visc_inv)
  const T* ef[3];
  Geom g;
  T beta;
  int hom;
};

template <typename T>
struct PoisArg {
  T* x;
  T* b;
  T* r;
  Geom g;
};

// grid transfers: restriction writes the coarse right-hand side and zeroes
// the coarse iterate; prolongation adds the coarse correction
template <typename T>
struct XferArg {
  const T* src;
  T* dst;
  T* zero;
  Geom gf, gc;
  int ncomp;
  int sign;
};

template <typename T>
struct BottomArg {
  const double* Minv;  // the exact inverse; null: sweeps Gauss-Seidel sweeps in FP64
  int m;      // matrix size (n, or n + 1 when bordered)
  int n;      // unknowns
  T* x;
  T* b;
  Geom g;
  int kind;   // 0 viscous, 1 MAC, 2 nodal
  int level;  // the cavity's coarsest level
  int sweeps;
  const double* ef[3];  // FP64 face viscosities and reciprocals (sweeps, viscous)
  const double* inv;
  double beta;
};

// sum of v(i) over i < n by the whole block, in a fixed order; every thread
// gets it (sh: 33 doubles)
template <typename F>
__device__ __forceinline__ double block_sum(int n, double* sh, F v) {
  double s = 0.0;
  for (int i = threadIdx.x; i < n; i += blockDim.x) s += v(i);
  for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x < 32) {
    s = threadIdx.x < (blockDim.x >> 5) ? sh[threadIdx.x] : 0.0;
    for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    if (threadIdx.x == 0) sh[32] = s;
  }
  __syncthreads();
  const double r = sh[32];
  __syncthreads();
  return r;
}

// v -= its weighted mean over the unknowns of a singular problem
template <int D>
__device__ inline void bottom_sub_mean(double* v, int n, int kind, const Geom& g, double* sh) {
  const double s = block_sum(n, sh, [&](int i) { return (kind == kNodal ? node_weight(g, D, i) : 1.0) * v[i]; });
  const double wsum = kind == kNodal ? (double)g.n[0] * g.n[1] * (D == 3 ? g.n[2] : 1) : (double)n;
  const double mean = s * (1.0 / wsum);
  for (int i = threadIdx.x; i < n; i += blockDim.x) v[i] -= mean;
  __syncthreads();
}

// exact solve of one cavity's coarsest level by the whole block, from b into
// x (unknown i of its component's n at x[i + (cs - n) * component]): the rows
// of the inverse one per warp
template <int D, typename T>
__device__ void bottom_block(const BottomArg<T>& a, const T* b, T* x, int cs, int nc) {
  __shared__ double sb[kDenseMax + 1];
  __shared__ double sx[kDenseMax + 1];
  __shared__ double sh[33];
  for (int i = threadIdx.x; i < a.n; i += blockDim.x) sb[i] = (double)b[i];
  __syncthreads();
  if (a.kind != kVisc) bottom_sub_mean<D>(sb, a.n, a.kind, a.g, sh);
  const int lane = threadIdx.x & 31;
  for (int i = threadIdx.x >> 5; i < a.n; i += blockDim.x >> 5) {
    double acc = 0.0;
    for (int j = lane; j < a.n; j += 32) acc += a.Minv[(size_t)i * a.m + j] * sb[j];
    for (int off = 16; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
    if (lane == 0) sx[i] = acc;
  }
  __syncthreads();
  if (a.kind != kVisc) bottom_sub_mean<D>(sx, a.n, a.kind, a.g, sh);
  const int m = a.n / nc;
  for (int i = threadIdx.x; i < a.n; i += blockDim.x) x[i % m + (i / m) * cs] = (T)sx[i];
  __syncthreads();
}

// the argument tables of an instance, by level, for the fused tail kernel
struct TailTabs {
  const void* lv[kMaxLev];
  const void* bot;
};

// ---------------------------------------------------------------------------
// fused tail of the V-cycle
// ---------------------------------------------------------------------------
// One cluster per cavity runs every level from lf down to the cavity's
// coarsest and back in one launch.  A V(2,2) cycle is a chain of about 28
// dependent phases per level (11 to 35 by problem); launched one by one a
// phase of a small level costs 3 to 7 us (launch, drain, and in FP64 two
// operations per SM and cycle on the few SMs its blocks reach) for well under
// 1 us of work.  Each level is cut into slabs of whole planes along its
// slowest axis, one slab per block, held in that block's shared memory with a
// halo plane on either side (x, b, and for the viscous problem the
// reciprocals and the face viscosities).  A thread that updates a point of a
// slab's first or last plane also writes it into the neighbouring block's halo
// (distributed shared memory), so a sweep's loads are all local, and
// barrier.cluster ends the phase.  Levels with at most tail_solo_points points
// take one slab: block 0 alone, with __syncthreads.  Residuals and corrections
// that cross slabs between levels go through the levels' global arrays (L2).
// The operations and their order are those of the level-by-level launches.
constexpr int kTailThreads = 512;

// points of a level that one block takes alone: a phase is then one block
// barrier (about 40 cycles) instead of a cluster's, worth the wider split only
// when a phase has more work than the barrier costs; FP64 issues 2 operations
// per SM and cycle, so it splits early
template <int D, typename T>
constexpr int tail_solo_points() {
  return sizeof(T) == 4 ? (D == 3 ? 512 : 1024) : 64;
}

// A level as a block of the cluster holds it.  Slab r takes the planes [r rp,
// (r + 1) rp) of the N planes of ps points along the slowest axis; offsets are
// bytes of the dynamic shared memory.
template <typename T>
struct TailLevel {
  int N, ps, rp, np;  // np: slabs; 1: block 0 alone
  int k0, k1;         // this block's planes (empty past the last slab)
  int cs;             // x: component stride, (rp + 2) ps; plane k0 at ps
  unsigned x, b, inv, ef[3];
  T *gx, *gr;         // global arrays
  const T *gb, *ginv;
  const T* gef[3];
};

template <int D, int KIND>
__host__ __device__ inline void tail_planes(const Geom& g, int& N, int& ps) {
  const int e = KIND == kNodal ? 1 : 0;
  N = g.n[D - 1] + e;
  ps = (g.n[0] + e) * (D == 3 ? g.n[1] + e : 1);
}

// planes per slab of a level shared by nblk blocks (arithmetic T).  Points
// fall from level to level, so past the first one-slab level every level is
// one; a swept coarsest level, whose FP64 slabs would split earlier, is one
// too when the level above it is (solo), and always for a singular problem,
// whose means block 0 takes alone.
template <int D, typename T, int KIND>
__host__ __device__ inline int tail_rows(const Geom& g, int nblk, bool solo = false) {
  int N, ps;
  tail_planes<D, KIND>(g, N, ps);
  if (N * ps <= tail_solo_points<D, T>() || solo) return N;
  return (N + nblk - 1) / nblk;
}

// the swept coarsest level L is one slab (up: the level above it, null when
// the tail starts on L)
template <int D, typename T, int KIND>
__host__ __device__ inline bool tail_swept_solo(const Geom* up, int nblk) {
  if (KIND != kVisc) return true;
  if (!up) return false;
  int N, ps;
  tail_planes<D, KIND>(*up, N, ps);
  return tail_rows<D, T, KIND>(*up, nblk) == N;
}

// shared memory of a slab of rp planes: x with its halo, b, and for the
// viscous problem the reciprocals and the face viscosities (fills o when not
// null)
template <int D, typename T, int KIND>
__host__ __device__ inline unsigned tail_slab_bytes(const Geom& g, int rp, unsigned at, TailLevel<T>* o) {
  int N, ps;
  tail_planes<D, KIND>(g, N, ps);
  const unsigned NC = KIND == kVisc ? D : 1;
  unsigned q = at;
  auto take = [&](unsigned count) {
    const unsigned r = q;
    q += (count * (unsigned)sizeof(T) + 15) / 16 * 16;
    return r;
  };
  const unsigned ox = take(NC * (rp + 2) * ps), ob = take(NC * rp * ps);
  unsigned oi = 0, oe[3] = {0, 0, 0};
  if (KIND == kVisc) {
    oi = take(NC * rp * ps);
    oe[0] = take(rp * (g.n[0] + 1) * (D == 3 ? g.n[1] : 1));
    if (D == 3) oe[1] = take(rp * g.n[0] * (g.n[1] + 1));
    oe[D - 1] = take((rp + 1) * ps);
  }
  if (o) {
    o->x = ox;
    o->b = ob;
    o->inv = oi;
    for (int a = 0; a < 3; ++a) o->ef[a] = oe[a];
  }
  return q - at;
}

// v into block r's shared memory at p's place in this block's
__device__ __forceinline__ void st_block(float* p, unsigned r, float v) {
  unsigned a = (unsigned)__cvta_generic_to_shared(p), q;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(q) : "r"(a), "r"(r));
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(q), "f"(v) : "memory");
}
__device__ __forceinline__ void st_block(double* p, unsigned r, double v) {
  unsigned a = (unsigned)__cvta_generic_to_shared(p), q;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(q) : "r"(a), "r"(r));
  asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(q), "d"(v) : "memory");
}

// x of component c at point q of plane k = v, and the copies in the halos of
// the slabs that border on plane k.  lo / hi of a periodic slowest axis: the
// planes that wrap (cells: N - 1 and 0; nodes, whose last plane repeats the
// first: N - 2 and 1).
template <int D, typename T, int KIND, bool PER>
__device__ __forceinline__ void tail_put(T* x, const TailLevel<T>& w, bool per, int c, int k, int q, unsigned rank,
                                         T v) {
  const int kl = k - w.k0;
  T* xc = x + c * w.cs + q;
  xc[(kl + 1) * w.ps] = v;
  if (w.np > 1) {
    if (kl == 0 && k > 0) st_block(xc + (w.rp + 1) * w.ps, rank - 1, v);  // a full slab lies below
    if (k == w.k1 - 1 && k < w.N - 1) st_block(xc, rank + 1, v);
  }
  if (PER && per) {
    const int lr = (w.N - 1) / w.rp, lc = w.N - lr * w.rp;  // the last slab and its planes
    const int lo = KIND == kNodal ? w.N - 2 : w.N - 1, hi = KIND == kNodal ? 1 : 0;
    if (k == lo) {
      if (w.np > 1)
        st_block(xc, 0, v);
      else
        xc[0] = v;
    }
    if (k == hi) {
      if (w.np > 1)
        st_block(xc + (lc + 1) * w.ps, lr, v);
      else
        xc[(lc + 1) * w.ps] = v;
    }
  }
}

// the viscous stencil of component c at cell p of the slab
template <int D, typename T, bool PER>
__device__ __forceinline__ HomCell<D, T> tail_hom_cell(const char* mem, const TailLevel<T>& w, const Geom& g, int c,
                                                       const int* p) {
  const int kl = p[D - 1] - w.k0;
  const int q = D == 3 ? p[0] + g.n[0] * p[1] : p[0];
  const T* x = (const T*)(mem + w.x) + (kl + 1) * w.ps + q;
  auto axis = [&](int a) {
    const bool per = PER && g.per[a];
    if (a == D - 1) return HomAxis(p[D - 1], g.n[D - 1], w.ps, per, true);
    return HomAxis(a == 0 ? p[0] : p[1], g.n[a], a == 0 ? 1 : g.n[0], per);
  };
  auto comp = [&](int a) { return x + a * w.cs; };
  auto face = [&](int a) {
    const T* e = (const T*)(mem + w.ef[a]);
    if (a == D - 1) return e + kl * w.ps + q;
    if (a == 0) return e + p[0] + (g.n[0] + 1) * (D == 3 ? p[1] + g.n[1] * kl : kl);
    return e + p[0] + g.n[0] * (p[1] + (g.n[1] + 1) * kl);
  };
  auto step = [&](int a) { return a == D - 1 ? w.ps : (a == 0 ? 1 : g.n[0]); };
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

// neighbours of cell p of the slab for the cell Poisson problem
template <int D, bool PER>
struct SlabNbr {
  int om[D], op[D];
  bool lo[D], hi[D];
  __device__ __forceinline__ SlabNbr(const Geom& g, int ps, const int* p) {
    int s = 1;
#pragma unroll
    for (int a = 0; a < D; ++a) {
      const bool per = PER && g.per[a];
      const bool first = p[a] == 0, last = p[a] == g.n[a] - 1;
      lo[a] = per || !first;
      hi[a] = per || !last;
      om[a] = a == D - 1 || !first ? -s : (g.n[a] - 1) * s;
      op[a] = a == D - 1 || !last ? s : -(g.n[a] - 1) * s;
      s = a + 1 == D - 1 ? ps : s * g.n[a];
    }
  }
};

// neighbour offsets of node p of the slab
template <int D, bool PER>
__host__ __device__ __forceinline__ void slab_node_offsets(const Geom& g, int ps, const int* p, int* om, int* op) {
  node_offsets(p[0], g.n[0], 1, PER && g.per[0], om[0], op[0]);
  if (D == 3) node_offsets(p[1], g.n[1], g.n[0] + 1, PER && g.per[1], om[1], op[1]);
  const bool per = PER && g.per[D - 1];  // a periodic neighbour is in the halo
  om[D - 1] = p[D - 1] == 0 && !per ? ps : -ps;
  op[D - 1] = p[D - 1] == g.n[D - 1] && !per ? -ps : ps;
}

// passes of one sweep: (component, colour), or the colours.  ODD: the level may
// be odd along a periodic axis and then has more (rb_parts, nd_classes); only a
// swept coarsest level may, and in the others the code for it costs 5%.
template <int D, int KIND, bool ODD>
__host__ __device__ __forceinline__ int tail_passes(const Geom& g) {
  if (KIND == kNodal) return ODD ? nd_passes<D>(g) : 1 << D;
  return (KIND == kVisc ? 2 * D : 2) * (ODD ? rb_parts(g) : 1);
}

// threads of one pass over this block's points of a level, and the point p of
// thread t (false: none).  An odd periodic slowest axis of nodes is not cut
// (such a level is swept by block 0 alone).
template <int D, typename T, int KIND, bool ODD>
__host__ __device__ __forceinline__ int tail_pass_count(const TailLevel<T>& w, const Geom& g, int pass) {
  if (KIND != kNodal) return (g.n[0] + 1) / 2 * (D == 3 ? g.n[1] : 1) * (w.k1 - w.k0);
  int c[3] = {pass & 1, (pass >> 1) & 1, (pass >> 2) & 1};
  if (ODD) nd_classes<D>(g, pass, c);
  int nk;
  if (ODD && odd_wrap(g, D - 1)) {
    nk = nd_count(g, D - 1, c[D - 1]);
  } else {
    const int kf = w.k0 + ((w.k0 + c[D - 1]) & 1);  // the slab's first plane of the colour
    nk = kf < w.k1 ? (w.k1 - kf + 1) / 2 : 0;
  }
  const int c0 = ODD ? nd_count(g, 0, c[0]) : (g.n[0] + 2 - c[0]) / 2;
  const int c1 = D == 3 ? (ODD ? nd_count(g, 1, c[1]) : (g.n[1] + 2 - c[1]) / 2) : 1;
  return c0 * c1 * nk;
}
template <int D, typename T, int KIND, bool ODD>
__host__ __device__ __forceinline__ bool tail_pass_point(const TailLevel<T>& w, const Geom& g, int pass, int t, int* p) {
  p[1] = p[2] = 0;
  if constexpr (KIND != kNodal) {
    const int two = ODD ? rb_parts(g) - 1 : 0, col = (pass >> two) & 1;
    const int nh = (g.n[0] + 1) / 2;
    const int r = divm(t, nh, g.m_rb), ih = t - r * nh;
    const int kl = D == 3 ? divm(r, g.n[1], g.m_n1) : r, j = D == 3 ? r - kl * g.n[1] : 0;
    const int k = w.k0 + kl;
    p[0] = 2 * ih + ((j + k + col) & 1);
    p[1] = j;
    p[D - 1] = k;
    if (p[0] >= g.n[0]) return false;
    return !(ODD && two) || rb_part(g, p) == (pass & 1);
  } else {
    int c[3] = {pass & 1, (pass >> 1) & 1, (pass >> 2) & 1};
    if (ODD && rb_parts(g) == 2) {
      nd_classes<D>(g, pass, c);
      const int c0 = nd_count(g, 0, c[0]), c1 = D == 3 ? nd_count(g, 1, c[1]) : 1;
      const int r = t / c0, kk = r / c1;
      p[0] = nd_pos(g, 0, c[0], t - r * c0);
      if (D == 3) p[1] = nd_pos(g, 1, c[1], r - kk * c1);
      p[D - 1] = odd_wrap(g, D - 1) ? nd_pos(g, D - 1, c[D - 1], kk) : w.k0 + ((w.k0 + c[D - 1]) & 1) + 2 * kk;
      return true;
    }
    const int c0 = (g.n[0] + 2 - c[0]) / 2, c1 = D == 3 ? (g.n[1] + 2 - c[1]) / 2 : 1;
    const int r = divm(t, c0, g.m_mc0[c[0]]), kk = D == 3 ? divm(r, c1, g.m_mc1[c[1]]) : r;
    p[0] = 2 * (t - r * c0) + c[0];
    if (D == 3) p[1] = 2 * (r - kk * c1) + c[1];
    p[D - 1] = w.k0 + ((w.k0 + c[D - 1]) & 1) + 2 * kk;
    return true;
  }
}

// one pass over this block's points of a level
template <int D, typename T, int KIND, bool PER, bool ODD>
__device__ __forceinline__ void tail_pass(char* mem, const TailLevel<T>& w, const Geom& g, T bs, int pass,
                                          unsigned rank) {
  const bool per = PER && g.per[D - 1];
  T* x = (T*)(mem + w.x);
  const T* b = (const T*)(mem + w.b);
  const int n = tail_pass_count<D, T, KIND, ODD>(w, g, pass);
  for (int t = threadIdx.x; t < n; t += blockDim.x) {
    int p[3];
    if (!tail_pass_point<D, T, KIND, ODD>(w, g, pass, t, p)) continue;
    const int k = p[D - 1], q = p[0] + (KIND == kNodal ? g.n[0] + 1 : g.n[0]) * (D == 3 ? p[1] : 0);
    const int o = (k - w.k0) * w.ps + q;
    int c = 0;
    T v;
    if constexpr (KIND == kVisc) {
      c = pass >> (ODD ? rb_parts(g) : 1);
      const int oc = c * w.rp * w.ps + o;
      v = hom_gs<D, T>(tail_hom_cell<D, T, PER>(mem, w, g, c, p), b[oc], ((const T*)(mem + w.inv))[oc], bs);
    } else if constexpr (KIND == kMac) {
      const SlabNbr<D, PER> nb(g, w.ps, p);
      v = cell_gs_value<D, T>(x + o + w.ps, b[o], g_hh<T>(g), nb.om, nb.op, nb.lo, nb.hi);
    } else {
      int om[3], op[3];
      slab_node_offsets<D, PER>(g, w.ps, p, om, op);
      v = (g_hh<T>(g) * b[o] - nodal_nbr_sum<D, T>(x + o + w.ps, om, op)) * T(-3.0 / 8.0);
    }
    tail_put<D, T, KIND, PER>(x, w, per, c, k, q, rank, v);
  }
}

// the block's share of a level's residual, into r (the whole level's layout)
template <int D, typename T, int KIND, bool PER>
__device__ __forceinline__ void tail_resid(const char* mem, const TailLevel<T>& w, const Geom& g, T beta, T* r) {
  const T* x = (const T*)(mem + w.x);
  const T* b = (const T*)(mem + w.b);
  const int np = w.ps * (w.k1 - w.k0), n = (KIND == kVisc ? D : 1) * np;
  for (int t = threadIdx.x; t < n; t += blockDim.x) {
    const int c = KIND == kVisc && t >= np ? (t >= 2 * np ? 2 : 1) : 0;
    const int o = t - c * np, id = w.k0 * w.ps + o;
    int p[3];
    if constexpr (KIND == kNodal) {
      node_coords(g, id, p[0], p[1], p[2]);
      int om[3], op[3];
      slab_node_offsets<D, PER>(g, w.ps, p, om, op);
      const T* q = x + o + w.ps;
      r[id] = b[o] - (nodal_nbr_sum<D, T>(q, om, op) - T(8.0 / 3.0) * q[0]) * g_ihh<T>(g);
    } else {
      cell_coords<D>(g, id, p[0], p[1], p[2]);
      if constexpr (KIND == kVisc) {
        r[(size_t)c * g.ncell + id] = hom_res<D, T>(tail_hom_cell<D, T, PER>(mem, w, g, c, p),
                                                    b[c * w.rp * w.ps + o], beta, g_ihh<T>(g));
      } else {
        const SlabNbr<D, PER> nb(g, w.ps, p);
        r[id] = cell_res_value<D, T>(x + o + w.ps, b[o], g_ihh<T>(g), nb.om, nb.op, nb.lo, nb.hi);
      }
    }
  }
}

// Smoothing of a level whose block holds few points: each thread keeps up to
// NS points ("slots", the block's points in colour order, so that a warp's
// share one colour) with everything that stays fixed over a visit in
// registers: the neighbours' offsets, the wall flags, b, the reciprocals and
// the face viscosities.  A pass is then the loads of x, the update and the
// barrier.  Indexing every point anew (tail_pass) took most of a small level's
// phase: about 350 dependent instructions.
template <int D, int KIND>
constexpr int tail_slots() {
  return KIND == kNodal ? 3 : (KIND == kVisc && D == 3 ? 1 : 2);  // what 128 registers hold
}

template <int D, typename T>
struct TailSlot {
  int col = -1;       // colour; -1: no point
  int k, q, o;        // plane, point of the plane, offset in x
  int om[D], op[D];   // neighbours
  unsigned wall = 0;  // bit 2a: no neighbour below on axis a (a wall), bit 2a + 1: above
  __host__ __device__ __forceinline__ unsigned flip(int bit) const { return (wall << (31 - bit)) & 0x80000000u; }
};

// this thread's slot u of the block's points of the level
template <int D, typename T, int KIND, bool PER, bool ODD>
__host__ __device__ __forceinline__ void tail_slot_init(TailSlot<D, T>& s, const TailLevel<T>& w, const Geom& g, int u) {
  int p[3] = {0, 0, 0};
  s.col = -1;
  s.wall = 0;
  const int nk = w.k1 - w.k0;
  if constexpr (KIND != kNodal) {
    const int nh = (g.n[0] + 1) / 2, n = nh * (D == 3 ? g.n[1] : 1) * nk;
    const int col = u >= n ? 1 : 0, t = u - col * n;
    if (t >= n) return;
    const int r = divm(t, nh, g.m_rb), ih = t - r * nh;
    const int kl = D == 3 ? divm(r, g.n[1], g.m_n1) : r, j = D == 3 ? r - kl * g.n[1] : 0;
    s.k = w.k0 + kl;
    p[0] = 2 * ih + ((j + s.k + col) & 1);
    if (p[0] >= g.n[0]) return;
    p[1] = j;
    p[D - 1] = s.k;
    s.col = col;
    s.q = p[0] + g.n[0] * j;
    const HomAxis x(p[0], g.n[0], 1, PER && g.per[0]);
    s.om[0] = x.om;
    s.op[0] = x.op;
    s.wall = (x.fm >> 31) | ((x.fp >> 31) << 1);
    if (D == 3) {
      const HomAxis y(p[1], g.n[1], g.n[0], PER && g.per[1]);
      s.om[1] = y.om;
      s.op[1] = y.op;
      s.wall |= ((y.fm >> 31) << 2) | ((y.fp >> 31) << 3);
    }
    const HomAxis z(s.k, g.n[D - 1], w.ps, PER && g.per[D - 1], true);
    s.om[D - 1] = z.om;
    s.op[D - 1] = z.op;
    s.wall |= ((z.fm >> 31) << (2 * D - 2)) | ((z.fp >> 31) << (2 * D - 1));
  } else {
    int t = u;
    for (int col = 0; col < tail_passes<D, KIND, ODD>(g); ++col) {
      const int n = tail_pass_count<D, T, KIND, ODD>(w, g, col);
      if (t < n) {
        tail_pass_point<D, T, KIND, ODD>(w, g, col, t, p);
        s.k = p[D - 1];
        s.q = p[0] + (g.n[0] + 1) * (D == 3 ? p[1] : 0);
        s.col = col;
        if (ODD && rb_parts(g) == 2) {  // node n - 1 with the even ones
          int c[3] = {0, 0, 0};
          nd_classes<D>(g, col, c);
          s.col = (c[0] & 1) | ((c[1] & 1) << 1) | ((c[2] & 1) << 2);
        }
        break;
      }
      t -= n;
    }
    if (s.col < 0) return;
    slab_node_offsets<D, PER>(g, w.ps, p, s.om, s.op);
  }
  s.o = (s.k - w.k0 + 1) * w.ps + s.q;
}

// the block's points of a level fit in its threads' slots
template <int D, int KIND, typename T>
__device__ __forceinline__ bool tail_fits_slots(const TailLevel<T>& w, const Geom& g) {
  const int nk = w.rp, e = KIND == kNodal ? g.n[0] + 1 : (g.n[0] + 1) / 2 * 2;
  const int n = e * (D == 3 ? (KIND == kNodal ? g.n[1] + 1 : g.n[1]) : 1) * nk;
  return n <= tail_slots<D, KIND>() * kTailThreads;
}

// One colour of the slots: value(i) of each slot i of the colour, put(i, v), a
// barrier.  On a level that is odd along a periodic axis (wrap) some points of a
// colour are neighbours through the wrap: every value is formed before any is
// stored, with a barrier between, so that both read the other's old value.  A
// barrier costs less than the second pass that the indexed form and the one-block
// kernels take there (rb_parts: a pass of these small levels is one chain long).
template <bool ODD, typename T, int NS, class SL, class V, class P, class S>
__device__ __forceinline__ void tail_slot_pass(const SL* sl, int col, bool wrap, V value, P put, S sync) {
  if constexpr (ODD) {
    T v[NS];
#pragma unroll
    for (int i = 0; i < NS; ++i)
      if (sl[i].col == col) v[i] = value(i);
    if (wrap) sync();
#pragma unroll
    for (int i = 0; i < NS; ++i)
      if (sl[i].col == col) put(i, v[i]);
  } else {
#pragma unroll
    for (int i = 0; i < NS; ++i)
      if (sl[i].col == col) put(i, value(i));
  }
  sync();
}

// sweeps sweeps of the level, a barrier after each pass; then, when r is not
// null, the residual into r (the whole level's layout) and a barrier
template <int D, typename T, int KIND, bool PER, bool ODD, class S>
__device__ __forceinline__ void tail_visit(char* mem, const TailLevel<T>& w, const Geom& g, T beta, int sweeps, T* r,
                                           unsigned rank, S sync) {
  const T bs = KIND == kVisc ? rn_mul(beta, g_ihh<T>(g)) : T(0);
  constexpr int NS = tail_slots<D, KIND>();
  const bool per = PER && g.per[D - 1];
  T* const x = (T*)(mem + w.x);
  const T* const b = (const T*)(mem + w.b);
  if (!tail_fits_slots<D, KIND>(w, g)) {
    const int np = tail_passes<D, KIND, ODD>(g);
#pragma unroll 1
    for (int s = 0; s < sweeps; ++s)
#pragma unroll 1
      for (int q = 0; q < np; ++q) {
        tail_pass<D, T, KIND, PER, ODD>(mem, w, g, bs, q, rank);
        sync();
      }
    if (r) {
      tail_resid<D, T, KIND, PER>(mem, w, g, beta, r);
      sync();
    }
    return;
  }
  const bool wrap = ODD && rb_parts(g) == 2;
  TailSlot<D, T> sl[NS];
#pragma unroll
  for (int i = 0; i < NS; ++i) tail_slot_init<D, T, KIND, PER, ODD>(sl[i], w, g, (int)threadIdx.x + i * kTailThreads);
  const int bc = w.rp * w.ps;  // component stride of b and the reciprocals
  if constexpr (KIND == kVisc) {
    T e[NS][2 * D], bv[NS][D], iv[NS][D];
#pragma unroll
    for (int i = 0; i < NS; ++i) {
      if (sl[i].col < 0) continue;
      const int p0 = D == 3 ? sl[i].q % g.n[0] : sl[i].q;
      const int p[3] = {p0, D == 3 ? sl[i].q / g.n[0] : sl[i].k, sl[i].k};
      const HomCell<D, T> h = tail_hom_cell<D, T, PER>(mem, w, g, 0, p);
#pragma unroll
      for (int a = 0; a < D; ++a) {
        e[i][2 * a] = h.elo[a];
        e[i][2 * a + 1] = h.ehi[a];
        bv[i][a] = b[a * bc + sl[i].o - w.ps];
        iv[i][a] = ((const T*)(mem + w.inv))[a * bc + sl[i].o - w.ps];
      }
    }
    auto cell = [&](int i, int c) {
      HomCell<D, T> h;
#pragma unroll
      for (int q = 0; q < D; ++q) {
        const int a = c + q < D ? c + q : c + q - D;
        h.ax[q].om = sl[i].om[a];
        h.ax[q].op = sl[i].op[a];
        h.ax[q].fm = sl[i].flip(2 * a);
        h.ax[q].fp = sl[i].flip(2 * a + 1);
        h.u[q] = x + a * w.cs + sl[i].o;
        h.elo[q] = e[i][2 * a];
        h.ehi[q] = e[i][2 * a + 1];
      }
      return h;
    };
#pragma unroll 1
    for (int s = 0; s < sweeps; ++s)
#pragma unroll
      for (int c = 0; c < D; ++c)
#pragma unroll 1
        for (int col = 0; col < 2; ++col)
          tail_slot_pass<ODD, T, NS>(
              sl, col, wrap, [&](int i) { return hom_gs<D, T>(cell(i, c), bv[i][c], iv[i][c], bs); },
              [&](int i, T v) { tail_put<D, T, KIND, PER>(x, w, per, c, sl[i].k, sl[i].q, rank, v); }, sync);
    if (r) {
#pragma unroll
      for (int c = 0; c < D; ++c)
#pragma unroll
        for (int i = 0; i < NS; ++i)
          if (sl[i].col >= 0)
            r[(size_t)c * g.ncell + sl[i].k * w.ps + sl[i].q] = hom_res<D, T>(cell(i, c), bv[i][c], beta, g_ihh<T>(g));
      sync();
    }
  } else {
    T bv[NS];
#pragma unroll
    for (int i = 0; i < NS; ++i) bv[i] = sl[i].col >= 0 ? b[sl[i].o - w.ps] : T(0);
    auto flags = [&](int i, bool* lo, bool* hi) {
#pragma unroll
      for (int a = 0; a < D; ++a) {
        lo[a] = !((sl[i].wall >> (2 * a)) & 1);
        hi[a] = !((sl[i].wall >> (2 * a + 1)) & 1);
      }
    };
#pragma unroll 1
    for (int s = 0; s < sweeps; ++s)
#pragma unroll 1
      for (int col = 0; col < (KIND == kMac ? 2 : 1 << D); ++col)
        tail_slot_pass<ODD, T, NS>(
            sl, col, wrap,
            [&](int i) {
              const T* q = x + sl[i].o;
              if constexpr (KIND == kMac) {
                bool lo[D], hi[D];
                flags(i, lo, hi);
                return cell_gs_value<D, T>(q, bv[i], g_hh<T>(g), sl[i].om, sl[i].op, lo, hi);
              } else {
                return (g_hh<T>(g) * bv[i] - nodal_nbr_sum<D, T>(q, sl[i].om, sl[i].op)) * T(-3.0 / 8.0);
              }
            },
            [&](int i, T v) { tail_put<D, T, KIND, PER>(x, w, per, 0, sl[i].k, sl[i].q, rank, v); }, sync);
    if (r) {
#pragma unroll
      for (int i = 0; i < NS; ++i)
        if (sl[i].col >= 0) {
          const T* q = x + sl[i].o;
          T v;
          if constexpr (KIND == kMac) {
            bool lo[D], hi[D];
            flags(i, lo, hi);
            v = cell_res_value<D, T>(q, bv[i], g_ihh<T>(g), sl[i].om, sl[i].op, lo, hi);
          } else {
            v = bv[i] - (nodal_nbr_sum<D, T>(q, sl[i].om, sl[i].op) - T(8.0 / 3.0) * q[0]) * g_ihh<T>(g);
          }
          r[sl[i].k * w.ps + sl[i].q] = v;
        }
      sync();
    }
  }
}

// b of the block's coarse points from r of the fine level (TB: the coarse
// slab's arithmetic, FP64 on a swept coarsest level)
template <int D, typename T, int KIND, bool PER, typename TB>
__device__ __forceinline__ void tail_restrict(char* mem, const TailLevel<TB>& w, const T* r, const Geom& gf,
                                              const Geom& gc) {
  TB* b = (TB*)(mem + w.b);
  const int np = w.ps * (w.k1 - w.k0), n = (KIND == kVisc ? D : 1) * np;
  for (int t = threadIdx.x; t < n; t += blockDim.x) {
    const int c = KIND == kVisc && t >= np ? (t >= 2 * np ? 2 : 1) : 0;
    const int o = t - c * np, id = w.k0 * w.ps + o;
    int I, J, K;
    if constexpr (KIND == kNodal) {
      node_coords(gc, id, I, J, K);
      b[o] = (TB)restrict_node_value<D, T, PER>(r, gf, I, J, K);
    } else {
      cell_coords<D>(gc, id, I, J, K);
      b[c * w.rp * w.ps + o] = (TB)restrict_cell_value<D, T>(r + (size_t)c * gf.ncell, gf, I, J, K);
    }
  }
}

// x of the block's points += P e, e the coarse correction (component stride
// cs)
template <int D, typename T, int KIND, bool PER>
__device__ __forceinline__ void tail_prolong(char* mem, const TailLevel<T>& w, const T* e, int cs, const Geom& gf,
                                             const Geom& gc, unsigned rank) {
  T* x = (T*)(mem + w.x);
  const bool per = PER && gf.per[D - 1];
  const int np = w.ps * (w.k1 - w.k0), n = (KIND == kVisc ? D : 1) * np;
  for (int t = threadIdx.x; t < n; t += blockDim.x) {
    const int c = KIND == kVisc && t >= np ? (t >= 2 * np ? 2 : 1) : 0;
    const int o = t - c * np;
    int i, j, k;
    T v;
    if constexpr (KIND == kNodal) {
      node_coords(gf, w.k0 * w.ps + o, i, j, k);
      v = prolong_node_value<D, T>(e, gc, i, j, k);
    } else {
      cell_coords<D>(gf, w.k0 * w.ps + o, i, j, k);
      v = prolong_cell_value<D, T, PER>(e + c * cs, gc, i, j, k, KIND == kVisc ? T(-1) : T(1));
    }
    const int kp = D == 3 ? k : j, q = o - (kp - w.k0) * w.ps;
    v = x[c * w.cs + o + w.ps] + v;
    tail_put<D, T, KIND, PER>(x, w, per, c, kp, q, rank, v);
  }
}

template <typename T>
__device__ __forceinline__ void block_copy(T* dst, const T* src, int n) {
  for (int t = threadIdx.x; t < n; t += blockDim.x) dst[t] = src[t];
}

// the level's constants (viscous problem): the reciprocals and the face
// viscosities of the block's planes; every array is a run of whole planes
template <int D, typename T>
__device__ __forceinline__ void tail_load_const(char* mem, const TailLevel<T>& w, const Geom& g) {
  const int nk = w.k1 - w.k0;
  if (nk <= 0) return;
  for (int c = 0; c < D; ++c)
    block_copy((T*)(mem + w.inv) + c * w.rp * w.ps, w.ginv + (size_t)c * g.ncell + w.k0 * w.ps, nk * w.ps);
  const int f0 = (g.n[0] + 1) * (D == 3 ? g.n[1] : 1);
  block_copy((T*)(mem + w.ef[0]), w.gef[0] + (size_t)w.k0 * f0, nk * f0);
  if (D == 3) {
    const int f1 = g.n[0] * (g.n[1] + 1);
    block_copy((T*)(mem + w.ef[1]), w.gef[1] + (size_t)w.k0 * f1, nk * f1);
  }
  block_copy((T*)(mem + w.ef[D - 1]), w.gef[D - 1] + (size_t)w.k0 * w.ps, (nk + 1) * w.ps);
}

__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive;\n\tbarrier.cluster.wait;" ::: "memory");
}

// thread 0: the level record of this block
template <int D, typename T, int KIND>
__host__ __device__ inline void tail_level_init(TailLevel<T>& w, const Geom& g, int nblk, unsigned rank, bool solo,
                                                unsigned& at) {
  tail_planes<D, KIND>(g, w.N, w.ps);
  w.rp = tail_rows<D, T, KIND>(g, nblk, solo);
  w.np = (w.N + w.rp - 1) / w.rp;
  w.k0 = (int)rank * w.rp < w.N ? (int)rank * w.rp : w.N;
  w.k1 = w.k0 + w.rp < w.N ? w.k0 + w.rp : w.N;
  w.cs = (w.rp + 2) * w.ps;
  at += tail_slab_bytes<D, T, KIND>(g, w.rp, at, &w);
}

// PER = false: every level of every cavity has walls on every axis.  Grid:
// ncav clusters.  x_lf, b_lf: level lf's iterate and right-hand side in place
// of the record's (null: the record's).
template <int D, typename T, int KIND, bool PER = true>
__global__ void __launch_bounds__(kTailThreads, 1) k_vcycle_tail(TailTabs tb, int lf, int ncav,
                                                                  const int* __restrict__ mask, int nu1, int nu2,
                                                                  T* x_lf, const T* b_lf) {
  pdl_wait();
  extern __shared__ __align__(16) char mem[];
  __shared__ TailLevel<T> sw[kMaxLev];
  __shared__ TailLevel<double> sbw;  // the coarsest level, when it is swept
  __shared__ Geom sg[kMaxLev];
  __shared__ double sh[33];
  __shared__ T sbeta;
  __shared__ unsigned scratch;
  constexpr int NC = KIND == kVisc ? D : 1;
  unsigned rank, nblk;
  asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
  asm("mov.u32 %0, %%cluster_nctarank;" : "=r"(nblk));
  const int c = blockIdx.x / nblk;
  if (c >= ncav || (mask && !mask[c])) return;
  const BottomArg<T>& bot = ((const BottomArg<T>*)tb.bot)[c];
  const int L = bot.level;
  if (L < lf) return;
  const bool swept = bot.Minv == nullptr;
  for (int l = lf; l <= L; ++l) {
    const Geom* g;
    if constexpr (KIND == kVisc)
      g = &((const ViscArg<T>*)tb.lv[l])[c].g;
    else
      g = &((const PoisArg<T>*)tb.lv[l])[c].g;
    for (int q = threadIdx.x; q < (int)(sizeof(Geom) / 4); q += blockDim.x) ((int*)&sg[l])[q] = ((const int*)g)[q];
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned at = 0;
    for (int l = lf; l <= L; ++l) {
      TailLevel<T>& w = sw[l];
      if constexpr (KIND == kVisc) {
        const ViscArg<T>& a = ((const ViscArg<T>*)tb.lv[l])[c];
        w.gx = a.x;
        w.gr = a.out;
        w.gb = a.b;
        w.ginv = a.inv;
        for (int q = 0; q < 3; ++q) w.gef[q] = a.ef[q];
        sbeta = a.beta;
      } else {
        const PoisArg<T>& a = ((const PoisArg<T>*)tb.lv[l])[c];
        w.gx = a.x;
        w.gr = a.r;
        w.gb = a.b;
        sbeta = T(0);
      }
      if (l == lf && x_lf) {
        w.gx = x_lf;
        w.gb = b_lf;
      }
      if (l < L) {
        tail_level_init<D, T, KIND>(w, sg[l], (int)nblk, rank, false, at);
      } else if (swept) {
        sbw.ginv = bot.inv;
        for (int q = 0; q < 3; ++q) sbw.gef[q] = bot.ef[q];
        tail_level_init<D, double, KIND>(sbw, sg[l], (int)nblk, rank,
                                         tail_swept_solo<D, T, KIND>(l > lf ? &sg[l - 1] : nullptr, (int)nblk), at);
        w.np = sbw.np;
      } else {  // the exact solve: block 0
        tail_level_init<D, T, KIND>(w, sg[l], 1, rank, true, at);
      }
    }
    scratch = at;  // the one-slab levels' residuals
  }
  __syncthreads();
  const T beta = sbeta;
  // the constants of this block's planes, and the first level's b and x
  if (KIND == kVisc) {
    for (int l = lf; l < L; ++l) tail_load_const<D, T>(mem, sw[l], sg[l]);
    if (swept) tail_load_const<D, double>(mem, sbw, sg[L]);
  }
  auto zero_x = [&](auto& w) {
    auto* x = (decltype(w.gx))(mem + w.x);
    for (int t = threadIdx.x; t < NC * w.cs; t += blockDim.x) x[t] = 0;
  };
  if (L == lf && swept) {
    const int n = sbw.ps * (sbw.k1 - sbw.k0);
    for (int q = 0; q < NC; ++q)
      for (int t = threadIdx.x; t < n; t += blockDim.x)
        ((double*)(mem + sbw.b))[q * sbw.rp * sbw.ps + t] =
            (double)sw[L].gb[(size_t)q * sbw.N * sbw.ps + sbw.k0 * sbw.ps + t];
    zero_x(sbw);
  } else {
    const TailLevel<T>& w = sw[lf];
    const int n = w.ps * (w.k1 - w.k0);
    for (int q = 0; q < NC; ++q)
      block_copy((T*)(mem + w.b) + q * w.rp * w.ps, w.gb + (size_t)q * w.N * w.ps + w.k0 * w.ps, n);
    zero_x(w);
    __syncthreads();
    if (lf == 0 && n > 0) {
      // level 0 starts from the given iterate, its halos included
      const bool per = PER && sg[0].per[D - 1];
      const int lo = KIND == kNodal ? w.N - 2 : w.N - 1, hi = KIND == kNodal ? 1 : 0;
      T* x = (T*)(mem + w.x);
      for (int q = 0; q < NC; ++q) {
        const T* gx = w.gx + (size_t)q * w.N * w.ps;
        for (int t = threadIdx.x; t < (w.k1 - w.k0 + 2) * w.ps; t += blockDim.x) {
          const int kl = t / w.ps;
          int k = w.k0 + kl - 1;
          if (k < 0) k = per ? lo : -1;
          if (k >= w.N) k = per ? hi : -1;
          if (k >= 0) x[q * w.cs + t] = gx[(size_t)k * w.ps + t - kl * w.ps];
        }
      }
    }
  }
  if (nblk > 1)
    cluster_sync();
  else
    __syncthreads();
  // visit v: the levels lf .. L - 1 downwards, the coarsest, and back up
  const int nd = L - lf;
#pragma unroll 1
  for (int visit = 0; visit <= 2 * nd; ++visit) {
    const bool down = visit < nd;
    const int l = visit <= nd ? lf + visit : lf + 2 * nd - visit;
    const TailLevel<T>& w = sw[l];
    const Geom& g = sg[l];
    const bool wide = w.np > 1;
    if (!wide && rank) continue;  // block 0 alone; the others wait at the next wide barrier
    auto sync = [&] {
      if (wide)
        cluster_sync();
      else
        __syncthreads();
    };
    if (visit == nd) {
      if (!swept) {
        bottom_block<D, T>(bot, (const T*)(mem + w.b), (T*)(mem + w.x) + w.ps, w.cs, NC);
      } else {
        const int n = sbw.ps * (sbw.k1 - sbw.k0);
        double *xd = (double*)(mem + sbw.x) + sbw.ps, *bd = (double*)(mem + sbw.b);
        if (KIND != kVisc) bottom_sub_mean<D>(bd, n, KIND, g, sh);
        tail_visit<D, double, KIND, PER, PER>(mem, sbw, g, bot.beta, bot.sweeps, (double*)nullptr, rank, sync);
        if (KIND != kVisc) bottom_sub_mean<D>(xd, n, KIND, g, sh);
        for (int q = 0; q < NC; ++q)
          for (int t = threadIdx.x; t < n; t += blockDim.x)
            w.gx[(size_t)q * sbw.N * sbw.ps + sbw.k0 * sbw.ps + t] = (T)xd[q * sbw.cs + t];
        if (!wide) __syncthreads();
      }
    } else {
      T* const r = wide ? w.gr : (T*)(mem + scratch);
      if (!down) {
        if (wide) cluster_sync();  // the coarse level's result is in its global array
        const bool local = !wide && !(l + 1 == L && swept);
        const TailLevel<T>& wc = sw[l + 1];
        tail_prolong<D, T, KIND, PER>(mem, w, local ? (const T*)(mem + wc.x) + wc.ps : (const T*)wc.gx,
                                      local ? wc.cs : (KIND == kVisc ? sg[l + 1].ncell : 0), g, sg[l + 1], rank);
        sync();
      }
      tail_visit<D, T, KIND, PER, false>(mem, w, g, beta, down ? nu1 : nu2, down ? r : (T*)nullptr, rank, sync);
      if (down) {
        const bool cwide = sw[l + 1].np > 1;
        if (cwide || rank == 0) {
          if (l + 1 == L && swept) {
            tail_restrict<D, T, KIND, PER>(mem, sbw, r, g, sg[l + 1]);
            zero_x(sbw);
          } else {
            tail_restrict<D, T, KIND, PER>(mem, sw[l + 1], r, g, sg[l + 1]);
            zero_x(sw[l + 1]);
          }
          if (cwide)
            cluster_sync();
          else
            __syncthreads();
        }
      }
    }
    // a result that another block or the next launch reads
    if (visit >= nd && (l == lf || sw[l - 1].np > 1) && !(visit == nd && swept)) {
      const int n = w.ps * (w.k1 - w.k0);
      const T* x = (const T*)(mem + w.x) + w.ps;
      for (int q = 0; q < NC; ++q)
        block_copy(w.gx + (size_t)q * w.N * w.ps + w.k0 * w.ps, x + q * w.cs, n);
    }
  }
}

// ---------------------------------------------------------------------------
// host side of the tail
// ---------------------------------------------------------------------------
constexpr size_t kTailSmem = 200 * 1024;  // dynamic shared memory a block of the tail may take

// dynamic shared memory of block 0 of the tail (the largest) over the levels
// lf..L of the hierarchy gs with nblk blocks (swept: the coarsest level has no
// exact inverse)
template <int D, typename T, int KIND>
inline size_t tail_smem(const Geom* const* gs, int lf, int L, int nblk, bool swept) {
  size_t b = 0, r = 0;
  for (int l = lf; l < L; ++l) {
    int N, ps;
    tail_planes<D, KIND>(*gs[l], N, ps);
    const int rp = tail_rows<D, T, KIND>(*gs[l], nblk);
    b += tail_slab_bytes<D, T, KIND>(*gs[l], rp, 0, nullptr);
    if (rp == N && r == 0) r = (size_t)(KIND == kVisc ? D : 1) * N * ps * sizeof(T);  // the finest one-slab level
  }
  if (swept)
    b += tail_slab_bytes<D, double, KIND>(
        *gs[L], tail_rows<D, double, KIND>(*gs[L], nblk, tail_swept_solo<D, T, KIND>(L > lf ? gs[L - 1] : nullptr, nblk)),
        0, nullptr);
  else
    b += tail_slab_bytes<D, T, KIND>(*gs[L], tail_rows<D, T, KIND>(*gs[L], 1), 0, nullptr);
  return b + r;
}

// some level of lf..L is cut into several slabs
template <int D, typename T, int KIND>
inline bool tail_has_wide(const Geom* const* gs, int lf, int L, bool swept) {
  int N, ps;
  tail_planes<D, KIND>(*gs[lf], N, ps);
  if (lf < L) return tail_rows<D, T, KIND>(*gs[lf], 16) < N;
  return swept && tail_rows<D, double, KIND>(*gs[L], 16, tail_swept_solo<D, T, KIND>(nullptr, 16)) < N;
}

// Sets the tail kernel up on the current device and returns the blocks per
// cluster for ncav cavities with (wide) levels of several slabs: as many as
// share the SMs without a second wave of clusters, 16 at most (8 where the
// device cannot place 16); 0 when the set-up fails.
template <int D, typename T, int KIND, bool PER>
inline int tail_blocks(int ncav, bool wide) {
  auto kern = k_vcycle_tail<D, T, KIND, PER>;
  int nblk = wide ? 16 : 1;
  while (nblk > 1 && nblk * ncav > 152) nblk >>= 1;
  if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTailSmem) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  if (nblk > 8) {
    int n = 0;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)nblk);
    cfg.blockDim = dim3((unsigned)kTailThreads);
    cfg.dynamicSmemBytes = kTailSmem;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim = {(unsigned)nblk, 1, 1};
    cfg.attrs = at;
    cfg.numAttrs = 1;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess ||
        cudaOccupancyMaxActiveClusters(&n, kern, &cfg) != cudaSuccess || n < 1) {
      cudaGetLastError();
      nblk = 8;
    }
  }
  return nblk;
}

// Cells of the default first level of a single cavity's tail.  Measured per
// phase, a cluster of 16 against launches: FP32 128^2 1.2 against 2.9 us, 32^3
// 3.7 against 3 to 6 us; FP64, which is bound by the operations of 16 SMs, 64^2
// 1.4 against 3.1 us and 128^2 5.7 against 3.6 us (viscous; the cheaper MAC and
// nodal phases 3 against 3 us), 16^3 2.3 against 3 us.
template <int D, typename T, int KIND>
constexpr int tail_wide_cells() {
  return sizeof(T) == 4 ? (D == 3 ? 32768 : 16384) : (D == 3 || KIND == kVisc ? 4096 : 16384);
}

// launch on stream s: ncav clusters of nblk blocks (tail_blocks)
template <int D, typename T, int KIND, bool PER>
inline cudaError_t tail_launch(cudaStream_t s, const TailTabs& tb, int lf, int ncav, const int* mask, int nu1, int nu2,
                               int nblk, size_t smem, T* x_lf = nullptr, const T* b_lf = nullptr) {
  auto kern = k_vcycle_tail<D, T, KIND, PER>;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(nblk * ncav));
  cfg.blockDim = dim3((unsigned)kTailThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim = {(unsigned)nblk, 1, 1};
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;  // it begins with pdl_wait()
  at[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, kern, tb, lf, ncav, mask, nu1, nu2, x_lf, b_lf);
}

}  // namespace batch
}  // namespace hb
