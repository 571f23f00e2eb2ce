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
// x: the rows of the inverse one per warp
template <int D, typename T>
__device__ void bottom_block(const BottomArg<T>& a, const T* b, T* x) {
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
  for (int i = threadIdx.x; i < a.n; i += blockDim.x) x[i] = (T)sx[i];
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
// dependent phases per level; launched one by one a phase of a small level
// costs 3 to 7 us (launch, drain, and in FP64 two operations per SM and cycle
// on the few SMs its blocks reach) for well under 1 us of work.  Two forms of
// a phase, by level:
//   wide  (lf <= l < ls): every block of the cluster takes part, the arrays
//         stay in global memory (L2), barrier.cluster between the phases (its
//         release / acquire makes the blocks' writes visible to each other);
//         up to 16 SMs share a level's FP64 work.
//   solo  (l >= ls): block 0 alone, the level's arrays in shared memory,
//         __syncthreads between the phases.
// The operations and their order are those of the level-by-level launches.
template <typename T>
struct TailView {
  T *x, *r;
  const T *b, *inv;
  const T* ef[3];
};

template <typename T>
constexpr int tail_threads() {
  return sizeof(T) == 4 ? 1024 : 256;
}

struct SyncSolo {
  __device__ __forceinline__ void operator()() const { __syncthreads(); }
};
struct SyncWide {
  __device__ __forceinline__ void operator()() const {
    asm volatile("barrier.cluster.arrive;\n\tbarrier.cluster.wait;" ::: "memory");
  }
};

template <int D, typename T, int KIND>
__host__ __device__ __forceinline__ int tail_points(const Geom& g) {
  return KIND == kNodal ? g.nnode : g.ncell;
}

// shared memory of one solo level: x and b, for the viscous problem also the
// reciprocals and the face viscosities
template <int D, typename T, int KIND>
__host__ __device__ inline size_t tail_level_bytes(const Geom& g) {
  size_t e = 2 * (size_t)tail_points<D, T, KIND>(g);
  if (KIND == kVisc) e = 3 * (size_t)D * g.ncell + g.nface[0] + g.nface[1] + (D == 3 ? g.nface[2] : 0);
  return (e * sizeof(T) + 15) / 16 * 16;
}

// FP64 copies of the coarsest level for its Gauss-Seidel sweeps (no exact
// inverse): laid out as a solo level of FP64
template <int D, int KIND>
__host__ __device__ inline size_t tail_bottom_bytes(const Geom& g) {
  return tail_level_bytes<D, double, KIND>(g);
}

template <int D, typename T, int C, bool PER, class S>
__device__ __forceinline__ void tail_visc_colours(const TailView<T>& v, const Geom& g, T bs, int tid, int nth, S sync) {
  const int nt = rb_count<D>(g);
  for (int col = 0; col < 2; ++col) {
    for (int t = tid; t < nt; t += nth) visc_smooth_hom_at<D, T, C, PER>(v.x, v.b, v.inv, v.ef, g, col, bs, t);
    sync();
  }
}

template <int D, typename T, int KIND, bool PER, class S>
__device__ __forceinline__ void tail_smooth(const TailView<T>& v, const Geom& g, T beta, int tid, int nth, S sync) {
  if constexpr (KIND == kVisc) {
    const T bs = rn_mul(beta, g_ihh<T>(g));
    tail_visc_colours<D, T, 0, PER>(v, g, bs, tid, nth, sync);
    tail_visc_colours<D, T, 1, PER>(v, g, bs, tid, nth, sync);
    if constexpr (D == 3) tail_visc_colours<D, T, 2, PER>(v, g, bs, tid, nth, sync);
  } else if constexpr (KIND == kMac) {
    const int nt = rb_count<D>(g);
    for (int col = 0; col < 2; ++col) {
      for (int t = tid; t < nt; t += nth) k_cell_smooth_at<D, T, PER>(v.x, v.b, g, col, t);
      sync();
    }
  } else {
    for (int col = 0; col < (1 << D); ++col) {
      const int nt = mc_count<D>(g, col);
      for (int t = tid; t < nt; t += nth) k_nodal_smooth_at<D, T, PER>(v.x, v.b, g, col, t);
      sync();
    }
  }
}

template <int D, typename T, int KIND, bool PER>
__device__ __forceinline__ void tail_resid(const TailView<T>& v, const Geom& g, T beta, int tid, int nth) {
  if constexpr (KIND == kVisc) {
    for (int t = tid; t < D * g.ncell; t += nth) {
      const int c = t >= g.ncell ? (t >= 2 * g.ncell ? 2 : 1) : 0;
      const int id = t - c * g.ncell;
      int p[3];
      cell_coords<D>(g, id, p[0], p[1], p[2]);
      v.r[t] = c == 0   ? visc_res_hom<D, T, 0, PER>(v.x, v.b[t], v.ef, g, p, id, beta)
               : c == 1 ? visc_res_hom<D, T, 1, PER>(v.x, v.b[t], v.ef, g, p, id, beta)
                        : visc_res_hom<D, T, D - 1, PER>(v.x, v.b[t], v.ef, g, p, id, beta);
    }
  } else if constexpr (KIND == kMac) {
    for (int t = tid; t < g.ncell; t += nth) k_cell_resid_at<D, T, PER>(v.x, v.b, v.r, g, t);
  } else {
    for (int t = tid; t < g.nnode; t += nth) k_nodal_resid_at<D, T, PER>(v.x, v.b, v.r, g, t);
  }
}

// b of the coarse level from r of the fine one, and a zero coarse iterate
template <int D, typename T, int KIND, bool PER>
__device__ __forceinline__ void tail_restrict(const T* r, T* b, T* x, const Geom& gf, const Geom& gc, int tid,
                                              int nth) {
  constexpr int NC = KIND == kVisc ? D : 1;
  const int n = NC * tail_points<D, T, KIND>(gc);
  for (int t = tid; t < n; t += nth) {
    if constexpr (KIND == kNodal)
      k_restrict_nodes_at<D, T, PER>(r, b, gf, gc, t);
    else
      k_restrict_cells_at<D, T>(r, b, gf, gc, NC, t);
    x[t] = T(0);
  }
}

template <int D, typename T, int KIND, bool PER>
__device__ __forceinline__ void tail_prolong(T* xf, const T* xc, const Geom& gf, const Geom& gc, int tid, int nth) {
  constexpr int NC = KIND == kVisc ? D : 1;
  const int n = NC * tail_points<D, T, KIND>(gf);
  for (int t = tid; t < n; t += nth) {
    if constexpr (KIND == kNodal)
      k_prolong_nodes_add_at<D, T>(xf, xc, gf, gc, t);
    else
      k_prolong_cells_add_at<D, T, PER>(xf, xc, gf, gc, NC, KIND == kVisc ? T(-1) : T(1), t);
  }
}

template <typename T>
__device__ __forceinline__ void block_copy(T* dst, const T* src, int n) {
  for (int t = threadIdx.x; t < n; t += blockDim.x) dst[t] = src[t];
}

// a solo level's arrays from shared memory at p (and p past them), with the
// level's viscosities and reciprocals copied in
template <int D, typename T, int KIND>
__device__ inline void tail_carve(TailView<T>& v, char*& p, const Geom& g, const T* const* ef, const T* inv) {
  const int n = tail_points<D, T, KIND>(g) * (KIND == kVisc ? D : 1);
  T* q = (T*)p;
  v.x = q;
  v.b = q + n;
  q += 2 * n;
  if (KIND == kVisc) {
    v.inv = q;
    block_copy(q, inv, n);
    q += n;
    for (int a = 0; a < D; ++a) {
      v.ef[a] = q;
      block_copy(q, ef[a], g.nface[a]);
      q += g.nface[a];
    }
  }
  p += tail_level_bytes<D, T, KIND>(g);
}

// the coarsest level by sweeps Gauss-Seidel sweeps in FP64 (no exact inverse)
template <int D, typename T, int KIND, bool PER>
__device__ inline void tail_bottom_sweeps(const BottomArg<T>& a, const Geom& g, const T* b, T* x, char* mem,
                                          double* sh) {
  TailView<double> v;
  v.r = nullptr;
  tail_carve<D, double, KIND>(v, mem, g, a.ef, a.inv);
  double* bd = (double*)v.b;
  for (int i = threadIdx.x; i < a.n; i += blockDim.x) {
    bd[i] = (double)b[i];
    v.x[i] = 0.0;
  }
  __syncthreads();
  if (KIND != kVisc) bottom_sub_mean<D>(bd, a.n, KIND, g, sh);
  for (int s = 0; s < a.sweeps; ++s)
    tail_smooth<D, double, KIND, PER>(v, g, a.beta, threadIdx.x, blockDim.x, SyncSolo());
  if (KIND != kVisc) bottom_sub_mean<D>(v.x, a.n, KIND, g, sh);
  for (int i = threadIdx.x; i < a.n; i += blockDim.x) x[i] = (T)v.x[i];
  __syncthreads();
}

// PER = false: every level of every cavity has walls on every axis.  Grid:
// ncav clusters; ls: the first solo level (a cavity whose coarsest level is
// above it has that level solo); smem: the solo levels' arrays, a residual
// scratch of the largest, and the coarsest level's FP64 copies where it has no
// exact inverse.
template <int D, typename T, int KIND, bool PER = true>
__global__ void __launch_bounds__(tail_threads<T>()) k_vcycle_tail(TailTabs tb, int lf, int ls, int ncav,
                                                                  const int* __restrict__ mask, int nu1, int nu2) {
  extern __shared__ __align__(16) char smem[];
  __shared__ TailView<T> sv[kMaxLev];
  __shared__ Geom sg[kMaxLev];
  __shared__ double sh[33];
  __shared__ T sbeta;
  unsigned rank, nblk;
  asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
  asm("mov.u32 %0, %%cluster_nctarank;" : "=r"(nblk));
  const int c = blockIdx.x / nblk;
  if (c >= ncav || (mask && !mask[c])) return;
  const BottomArg<T>& bot = ((const BottomArg<T>*)tb.bot)[c];
  const int L = bot.level;
  if (L < lf) return;
  const int s0 = ls < L ? ls : L;  // the first solo level
  // the levels' geometry and global arrays
  for (int l = lf; l <= L; ++l) {
    const Geom* g = nullptr;
    TailView<T> v;
    if (KIND == kVisc) {
      const ViscArg<T>& a = ((const ViscArg<T>*)tb.lv[l])[c];
      g = &a.g;
      v = {a.x, a.out, a.b, a.inv, {a.ef[0], a.ef[1], a.ef[2]}};
      if (threadIdx.x == 0 && l == lf) sbeta = a.beta;
    } else {
      const PoisArg<T>& a = ((const PoisArg<T>*)tb.lv[l])[c];
      g = &a.g;
      v = {a.x, a.r, a.b, nullptr, {nullptr, nullptr, nullptr}};
    }
    for (int q = threadIdx.x; q < (int)(sizeof(Geom) / 4); q += blockDim.x) ((int*)&sg[l])[q] = ((const int*)g)[q];
    if (threadIdx.x == 0) sv[l] = v;
  }
  __syncthreads();
  const T beta = KIND == kVisc ? sbeta : T(0);
  const int nth = blockDim.x * nblk, tid = rank * blockDim.x + threadIdx.x;
  const SyncWide wide;
  const SyncSolo solo;
  if (s0 > lf) {
    if (lf > 0) {  // a coarse level starts from zero, level 0 from the given iterate
      const int n = (KIND == kVisc ? D : 1) * tail_points<D, T, KIND>(sg[lf]);
      for (int t = tid; t < n; t += nth) sv[lf].x[t] = T(0);
      wide();
    }
    for (int l = lf; l < s0; ++l) {
      const TailView<T> v = sv[l];
      for (int s = 0; s < nu1; ++s) tail_smooth<D, T, KIND, PER>(v, sg[l], beta, tid, nth, wide);
      tail_resid<D, T, KIND, PER>(v, sg[l], beta, tid, nth);
      wide();
      tail_restrict<D, T, KIND, PER>(v.r, (T*)sv[l + 1].b, sv[l + 1].x, sg[l], sg[l + 1], tid, nth);
      wide();
    }
  }
  if (rank == 0) {
    // the solo levels: shared-memory arrays, the residual scratch after them
    const int me = threadIdx.x, nb = blockDim.x;
    char* p = smem;
    TailView<T> gl = sv[s0];
    __syncthreads();  // every thread has the global view
    for (int l = s0; l <= L; ++l) {
      TailView<T> v = sv[l];
      const TailView<T> w = v;
      if (l < L) {
        tail_carve<D, T, KIND>(v, p, sg[l], w.ef, w.inv);
      } else {  // the coarsest level: x and b only
        const int n = tail_points<D, T, KIND>(sg[l]) * (KIND == kVisc ? D : 1);
        v.x = (T*)p;
        v.b = v.x + n;
        p += (2 * n * sizeof(T) + 15) / 16 * 16;
      }
      __syncthreads();
      if (me == 0) sv[l] = v;
    }
    if (me == 0)
      for (int l = s0; l <= L; ++l) sv[l].r = (T*)p;
    __syncthreads();
    if (s0 < L)
      p += ((KIND == kVisc ? D : 1) * (size_t)tail_points<D, T, KIND>(sg[s0]) * sizeof(T) + 15) / 16 * 16;
    {
      const int n = tail_points<D, T, KIND>(sg[s0]) * (KIND == kVisc ? D : 1);
      T *x = sv[s0].x, *b = (T*)sv[s0].b;
      for (int t = me; t < n; t += nb) {
        b[t] = gl.b[t];
        x[t] = s0 > 0 ? T(0) : gl.x[t];
      }
      __syncthreads();
    }
    for (int l = s0; l < L; ++l) {
      const TailView<T> v = sv[l];
      for (int s = 0; s < nu1; ++s) tail_smooth<D, T, KIND, PER>(v, sg[l], beta, me, nb, solo);
      tail_resid<D, T, KIND, PER>(v, sg[l], beta, me, nb);
      solo();
      tail_restrict<D, T, KIND, PER>(v.r, (T*)sv[l + 1].b, sv[l + 1].x, sg[l], sg[l + 1], me, nb);
      solo();
    }
    if (bot.Minv)
      bottom_block<D, T>(bot, sv[L].b, sv[L].x);
    else
      tail_bottom_sweeps<D, T, KIND, PER>(bot, sg[L], sv[L].b, sv[L].x, p, sh);
    for (int l = L - 1; l >= s0; --l) {
      const TailView<T> v = sv[l];
      tail_prolong<D, T, KIND, PER>(v.x, sv[l + 1].x, sg[l], sg[l + 1], me, nb);
      solo();
      for (int s = 0; s < nu2; ++s) tail_smooth<D, T, KIND, PER>(v, sg[l], beta, me, nb, solo);
    }
    block_copy(gl.x, (const T*)sv[s0].x, tail_points<D, T, KIND>(sg[s0]) * (KIND == kVisc ? D : 1));
    if (me == 0) sv[s0] = gl;  // the wide levels read it from global memory
    __syncthreads();
  }
  if (s0 > lf) {
    wide();
    for (int l = s0 - 1; l >= lf; --l) {
      const TailView<T> v = sv[l];
      tail_prolong<D, T, KIND, PER>(v.x, sv[l + 1].x, sg[l], sg[l + 1], tid, nth);
      wide();
      for (int s = 0; s < nu2; ++s) tail_smooth<D, T, KIND, PER>(v, sg[l], beta, tid, nth, wide);
    }
  }
}

// ---------------------------------------------------------------------------
// host side of the tail
// ---------------------------------------------------------------------------
constexpr size_t kTailSmem = 200 * 1024;  // dynamic shared memory the solo levels may take

// dynamic shared memory of the tail with solo levels s0..L of the hierarchy gs
// (sweeps: the coarsest level has no exact inverse)
template <int D, typename T, int KIND>
inline size_t tail_smem(const Geom* const* gs, int s0, int L, bool sweeps) {
  size_t b = 0;
  for (int l = s0; l < L; ++l) b += tail_level_bytes<D, T, KIND>(*gs[l]);
  const size_t nc = KIND == kVisc ? D : 1;
  b += (2 * nc * tail_points<D, T, KIND>(*gs[L]) * sizeof(T) + 15) / 16 * 16;
  if (s0 < L) b += (nc * tail_points<D, T, KIND>(*gs[s0]) * sizeof(T) + 15) / 16 * 16;
  if (sweeps) b += tail_bottom_bytes<D, KIND>(*gs[L]);
  return b;
}

// first solo level of a hierarchy gs[0..L]: the finest from lf on with at most
// kTailSolo cells whose levels fit in shared memory; -1 when not even the
// coarsest level does
template <int D, typename T>
constexpr int tail_solo_cells() {
  return sizeof(T) == 4 ? (D == 3 ? 512 : 1024) : 64;
}
template <int D, typename T, int KIND>
inline int tail_solo_level(const Geom* const* gs, int lf, int L, bool sweeps) {
  for (int l = lf; l <= L; ++l)
    if ((l == L || gs[l]->ncell <= tail_solo_cells<D, T>()) && tail_smem<D, T, KIND>(gs, l, L, sweeps) <= kTailSmem)
      return l;
  return -1;
}

// blocks per cluster for ncav cavities: as many as share the SMs without a
// second wave of clusters, 16 at most (8 where the device cannot place 16)
template <int D, typename T, int KIND, bool PER>
inline int tail_blocks(int ncav, size_t smem) {
  int nblk = 16;
  while (nblk > 1 && nblk * ncav > 152) nblk >>= 1;
  if (nblk > 8) {
    auto kern = k_vcycle_tail<D, T, KIND, PER>;
    int n = 0;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)nblk);
    cfg.blockDim = dim3((unsigned)tail_threads<T>());
    cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim = {(unsigned)nblk, 1, 1};
    cfg.attrs = at;
    cfg.numAttrs = 1;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTailSmem) != cudaSuccess ||
        cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess ||
        cudaOccupancyMaxActiveClusters(&n, kern, &cfg) != cudaSuccess || n < 1) {
      cudaGetLastError();
      nblk = 8;
    }
  }
  return nblk;
}

// the default first level of a single cavity's tail (see there): cells
template <int D, typename T>
constexpr int tail_wide_cells() {
  return sizeof(T) == 4 ? (D == 3 ? 32768 : 16384) : (D == 3 ? 4096 : 16384);
}

// launch on stream s: ncav clusters of nblk blocks
template <int D, typename T, int KIND, bool PER>
inline cudaError_t tail_launch(cudaStream_t s, const TailTabs& tb, int lf, int ls, int ncav, const int* mask, int nu1,
                               int nu2, int nblk, size_t smem) {
  auto kern = k_vcycle_tail<D, T, KIND, PER>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTailSmem);
  if (e == cudaSuccess && nblk > 8) e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(nblk * ncav));
  cfg.blockDim = dim3((unsigned)tail_threads<T>());
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim = {(unsigned)nblk, 1, 1};
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, tb, lf, ls, ncav, mask, nu1, nu2);
}

}  // namespace batch
}  // namespace hb
