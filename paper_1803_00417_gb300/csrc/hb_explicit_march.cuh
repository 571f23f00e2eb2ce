// The predictor's slopes and transverse terms (Eqs. 13-14) on large 3D grids,
// each limited difference and each face's upwind state formed once.
//
// What bounds both: FP64 instructions (two per SM and cycle).  One thread per
// cell (k_slopes, k_hats) forms the limited differences of a cell three times
// per axis (as p - 1, p and p + 1 of its neighbours) and every face's states
// twice.  Here a thread takes the neighbour's from the thread, or its own
// previous cell, that forms them.  The values, and the operations behind each,
// are those of the one-cell forms, so the bits are the same.  Slopes at 128^3:
// 472 us in one launch, 128 (x) + 163 (y and z) here.  Small boxes and boxes that
// leave the tiles half empty keep one thread per cell (slopes_march, hats_march).
#pragma once
#include "hb_explicit.cuh"

namespace hb {

// cells per thread of a marching slope: 16 against the two limited differences
// that a chunk forms again at its start
constexpr int kPredChunk = 16;
constexpr int kPredX = 64, kPredY = 4;  // block of the slopes along y and z
constexpr int kRowX = 128, kRowY = 2;   // block of the slopes along x

// the limited difference of the cell with values wm, w0, wp (slope5's s-th)
struct SlopePart {
  double dC, dlim, df;
};
__host__ __device__ __forceinline__ SlopePart slope_part(double dL, double dR, double wm, double wp) {
  SlopePart s;
  s.dC = dhalf(wp - wm);
  s.dlim = dsame_sign(dL, dR) ? dtwice(dminabs(dL, dR)) : 0.0;
  s.df = dsgn_min(s.dC, s.dlim);
  return s;
}
__host__ __device__ __forceinline__ double slope_of(const SlopePart& s, double df0, double df2) {
  const double d4 = (4.0 / 3.0) * s.dC - (1.0 / 6.0) * (df2 + df0);
  return dsgn_min(d4, s.dlim);
}

// u_c at q along axis A of the line through (i, j, k): inside the box, or the
// wall ghost / the wrapped cell
template <int A>
__host__ __device__ __forceinline__ double line_value(const double* __restrict__ uc, const Geom& g, int c, int i, int j,
                                                      int k, int q) {
  if (A == 0) i = q;
  if (A == 1) j = q;
  if (A == 2) k = q;
  if (q >= 0 && q < g.n[A]) return uc[i + g.n[0] * (j + g.n[1] * k)];
  return uget<3>(uc, g, c, i, j, k, false);
}

// slopes along A of the cells q0 <= q < q1 of a line
template <int A>
__host__ __device__ __forceinline__ void slope_line(const double* __restrict__ u, double* __restrict__ slopes,
                                                    const Geom& g, int c, int i, int j, int k, int q0, int q1) {
  const double* uc = u + (size_t)c * g.ncell;
  double* out = slopes + (size_t)(A * 3 + c) * g.ncell;
  const int s = A == 1 ? g.n[0] : g.n[0] * g.n[1];
  double wm = line_value<A>(uc, g, c, i, j, k, q0 - 1);
  double w0 = line_value<A>(uc, g, c, i, j, k, q0), wp = line_value<A>(uc, g, c, i, j, k, q0 + 1);
  double d0 = w0 - wm, d1 = wp - w0;  // differences below and above the cell at hand
  double dfm;                         // of the cell before
  {
    const double wmm = line_value<A>(uc, g, c, i, j, k, q0 - 2);
    dfm = slope_part(wm - wmm, d0, wmm, w0).df;
  }
  SlopePart cur = slope_part(d0, d1, wm, wp);
  size_t o = (size_t)((A == 1 ? i + g.n[0] * g.n[1] * k : i + g.n[0] * j) + q0 * s);
  for (int q = q0; q < q1; ++q, o += s) {
    const double w2 = line_value<A>(uc, g, c, i, j, k, q + 2);
    const double d2 = w2 - wp;
    const SlopePart nxt = slope_part(d1, d2, w0, w2);
    out[o] = slope_of(cur, dfm, nxt.df);
    dfm = cur.df;
    cur = nxt;
    w0 = wp;
    wp = w2;
    d1 = d2;
  }
}

// Slopes along y (blockIdx.z < chunks of y) and z of all components, marching:
// grid (3 components x tiles of x, tiles of the other axis, chunks of y + of z).
__global__ void __launch_bounds__(kPredX* kPredY) k_slopes_yz(const double* __restrict__ u,
                                                              double* __restrict__ slopes,
                                                              const __grid_constant__ Geom g) {
  pdl_wait();
  const int nx = (g.n[0] + kPredX - 1) / kPredX, ny = (g.n[1] + kPredChunk - 1) / kPredChunk;
  const int c = blockIdx.x / nx;
  const int i = (blockIdx.x - c * nx) * kPredX + threadIdx.x;
  const int o = blockIdx.y * kPredY + threadIdx.y;
  if (i >= g.n[0]) return;
  if ((int)blockIdx.z < ny) {
    const int q0 = blockIdx.z * kPredChunk;
    if (o < g.n[2]) slope_line<1>(u, slopes, g, c, i, 0, o, q0, min(q0 + kPredChunk, g.n[1]));
  } else {
    const int q0 = ((int)blockIdx.z - ny) * kPredChunk;
    if (o < g.n[1]) slope_line<2>(u, slopes, g, c, i, o, 0, q0, min(q0 + kPredChunk, g.n[2]));
  }
}
inline dim3 slopes_yz_grid(const Geom& g) {
  const int m = g.n[1] > g.n[2] ? g.n[1] : g.n[2];
  return dim3((unsigned)(3 * ((g.n[0] + kPredX - 1) / kPredX)), (unsigned)((m + kPredY - 1) / kPredY),
              (unsigned)((g.n[1] + kPredChunk - 1) / kPredChunk + (g.n[2] + kPredChunk - 1) / kPredChunk));
}

// Slopes along x of all components: a block takes kRowX cells of kRowY rows;
// the limited differences pass through shared memory, the two beyond the
// block's ends are formed by its first and last thread.
__global__ void __launch_bounds__(kRowX* kRowY) k_slopes_x(const double* __restrict__ u, double* __restrict__ slopes,
                                                           const __grid_constant__ Geom g) {
  pdl_wait();
  __shared__ double sdf[kRowY][3][kRowX + 2];
  const int tx = threadIdx.x, ty = threadIdx.y;
  const int i = blockIdx.y * kRowX + tx;
  const int row = blockIdx.x * kRowY + ty;  // j + n1 k
  const int k = row / g.n[1], j = row - k * g.n[1];
  const bool in = i < g.n[0] && row < g.n[1] * g.n[2];
  SlopePart s[3];
  if (in) {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const double* uc = u + (size_t)c * g.ncell;
      const double wm = line_value<0>(uc, g, c, i, j, k, i - 1), w0 = line_value<0>(uc, g, c, i, j, k, i);
      const double wp = line_value<0>(uc, g, c, i, j, k, i + 1);
      const double dL = w0 - wm, dR = wp - w0;
      s[c] = slope_part(dL, dR, wm, wp);
      sdf[ty][c][tx + 1] = s[c].df;
      if (tx == 0) {
        const double w2 = line_value<0>(uc, g, c, i, j, k, i - 2);
        sdf[ty][c][0] = slope_part(wm - w2, dL, w2, w0).df;
      }
      if (tx == kRowX - 1 || i == g.n[0] - 1) {
        const double w2 = line_value<0>(uc, g, c, i, j, k, i + 2);
        sdf[ty][c][tx + 2] = slope_part(dR, w2 - wp, w0, w2).df;
      }
    }
  }
  __syncthreads();
  if (!in) return;
#pragma unroll
  for (int c = 0; c < 3; ++c)
    slopes[(size_t)c * g.ncell + i + (size_t)g.n[0] * row] = slope_of(s[c], sdf[ty][c][tx], sdf[ty][c][tx + 2]);
}
inline dim3 slopes_x_grid(const Geom& g) {
  return dim3((unsigned)((g.n[1] * g.n[2] + kRowY - 1) / kRowY), (unsigned)((g.n[0] + kRowX - 1) / kRowX));
}

// The frame of the march: which cell a thread takes, how the three values of
// each face pass from the thread that forms them to the one above it, and how
// many planes a block marches.
constexpr int kMarchX = 64, kMarchY = 4;  // cells of a block's tile, one thread each
constexpr int kMarchMain = kMarchX * kMarchY / 32;  // warps of the tile
// and three warps for the faces before the tile (formed by the tile's own first
// warps, these are the ones that all others wait for at each plane's barrier)
constexpr int kMarchThreads = (kMarchMain + 3) * 32;

// the face values in flight, two planes deep: x faces of each warp's first
// lane, y faces of each row
struct MarchShare {
  double x[2][kMarchY][kMarchX / 32][3];
  double y[2][kMarchY][3][kMarchX];
};

struct MarchThread {
  int i, j, k0, k1;  // the cell's column and the block's planes
  int tx, ty, lane, wx;
  bool halo, in;
  __device__ __forceinline__ MarchThread(const Geom& g, int chunk) {
    const int w = threadIdx.x >> 5;
    lane = threadIdx.x & 31;
    hw = w - kMarchMain;
    halo = hw >= 0;
    wx = w % (kMarchX / 32);
    ty = w / (kMarchX / 32);
    tx = wx * 32 + lane;
    i = blockIdx.x * kMarchX + tx;
    j = blockIdx.y * kMarchY + ty;
    in = !halo && i < g.n[0] && j < g.n[1];
    n0 = g.n[0];
    n1 = g.n[1];
    k0 = blockIdx.z * chunk;
    k1 = min(k0 + chunk, g.n[2]);
  }
  // the extra warps: the faces that the tile takes from its neighbours in
  // plane k, fx(i, j, F) and fy(i, j, F) the values of the upper faces of cell
  // (i, j, k) (coordinate -1: the low wall, or the wrapped face)
  template <typename FX, typename FY>
  __device__ __forceinline__ void halo_faces(MarchShare& sh, int k, FX&& fx, FY&& fy) const {
    const int w = k & 1;
    const int i0 = blockIdx.x * kMarchX, j0 = blockIdx.y * kMarchY;
    double F[3];
    if (hw < kMarchX / 32) {
      const int r = hw * 32 + lane;
      if (i0 + r < n0) {
        fy(i0 + r, j0 - 1, F);
#pragma unroll
        for (int c = 0; c < 3; ++c) sh.y[w][0][c][r] = F[c];
      }
    } else if (lane < kMarchY && j0 + lane < n1) {
      fx(i0 - 1, j0 + lane, F);
#pragma unroll
      for (int c = 0; c < 3; ++c) sh.x[w][lane][0][c] = F[c];
    }
  }
  // the cell's upper faces, for the threads above
  __device__ __forceinline__ void put(MarchShare& sh, int k, const double* hx, const double* hy) const {
    const int w = k & 1;
    const bool px = lane == 31 && wx + 1 < kMarchX / 32;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      if (px) sh.x[w][ty][wx + 1][c] = hx[c];
      if (ty + 1 < kMarchY) sh.y[w][ty + 1][c][tx] = hy[c];
    }
  }
  // the cell's lower faces, once every warp has put plane k's.  One barrier a
  // plane: plane k + 1 goes to the other half, plane k + 2 comes after the
  // barrier of k + 1, which every warp reaches after reading k's.
  __device__ __forceinline__ void lower(const MarchShare& sh, int k, const double* hx, double* lx, double* ly) const {
    const int w = k & 1;
#pragma unroll
    for (int c = 0; c < 3; ++c) lx[c] = __shfl_up_sync(0xffffffffu, hx[c], 1);
    __syncthreads();
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      if (lane == 0) lx[c] = sh.x[w][ty][wx][c];
      ly[c] = sh.y[w][ty][c][tx];
    }
  }
  int n0, n1, hw;
};
static_assert(kMarchX == 64 && kMarchY <= 32, "two warps take the row before the tile, one the column");

inline dim3 march_grid(const Geom& g, int chunk) {
  return dim3((unsigned)((g.n[0] + kMarchX - 1) / kMarchX), (unsigned)((g.n[1] + kMarchY - 1) / kMarchY),
              (unsigned)((g.n[2] + chunk - 1) / chunk));
}
// Planes per block for a launch of that many tiles: of 6 to 24 the count that
// takes the least time when two blocks run on each of the 152 SMs, in waves of
// equal blocks whose start costs a third of a plane (128^3: 7 planes, 1216
// blocks, four full waves; 16 planes leave the second wave a third empty).
// cost: that time, in thirds of a plane.
struct MarchPlan {
  int chunk;
  long long cost;
};
inline MarchPlan march_plan(const Geom& g) {
  const dim3 t = march_grid(g, g.n[2]);
  const long long tiles = (long long)t.x * t.y;
  MarchPlan p{6, 0};
  for (int q = 6; q <= 24; ++q) {
    const long long nb = tiles * ((g.n[2] + q - 1) / q), waves = (nb + 303) / 304, cost = waves * (3 * q + 1);
    if (p.cost == 0 || cost < p.cost) p = {q, cost};
  }
  return p;
}
// a launch's y and z extents stay within 65535
inline bool march_extents(const Geom& g) { return g.n[1] <= 65535 && g.n[2] <= 65535; }

// The slopes by lines from 60^3 cells on: below, the chunks are few and their
// threads form serially what one thread per cell forms at once (40^3: 6 us
// slower; 48^3 to 56^3: within 5 us either way; 60^3: 8 us faster, 128 x 64 x
// 64: 50, 160^3: 370).  Narrower boxes than 48 leave most of a row's block idle.
inline bool slopes_march(const Geom& g) { return march_extents(g) && g.n[0] >= 48 && g.ncell >= 60 * 60 * 60; }

// The transverse terms by march where its waves take less time than one thread
// per cell: 0.33 ns a cell there, 6.1 us a third of a plane here, so at most 52
// thirds per million cells.  Boxes whose rows fill the 64-cell tiles and whose
// blocks fill a wave gain from 0.4 million cells on (64 x 96 x 64: 48 thirds per
// million cells, 22 us faster; 128 x 64 x 64: 22 us; 160^3: 253 us); 48^3 (172,
// 60 us slower), 66 x 64 x 64 (92, 62 us slower), 80^3 (72, 50 us slower) and 96
// x 64 x 64 (64, 14 us slower) do not, 48 x 128 x 128 (56) and 100^3 (52) are
// within 4 us.
inline bool hats_march(const Geom& g) {
  return march_extents(g) && march_plan(g).cost * 1000000 <= 52LL * g.ncell;
}

// k_hats marching along z: a thread forms the states of its cell's three upper
// faces and takes the lower ones' from their owners (684 -> 540 us at 128^3;
// 190 to 135 FP64 operations a cell).
__global__ void __launch_bounds__(kMarchThreads, 2) k_hats_march(const double* __restrict__ u,
                                                                 const double* __restrict__ slopes,
                                                                 const double* __restrict__ Gp,
                                                                 const double* __restrict__ Lu, Force fo, int pv,
                                                                 double* __restrict__ hats, double* __restrict__ tcom,
                                                                 const __grid_constant__ Geom g, const StepC k,
                                                                 int chunk) {
  pdl_wait();
  __shared__ MarchShare sh;
  const MarchThread th(g, chunk);
  double v;
  if (th.halo) {
    for (int kk = th.k0; kk < th.k1; ++kk) {
      auto face = [&](int b, int i, int j, double* F) {
        const int L[3] = {i, j, kk};
        prestate_face<3>(u, slopes, g, k, b, L, F, v);
      };
      th.halo_faces(sh, kk, [&](int i, int j, double* F) { face(0, i, j, F); },
                    [&](int i, int j, double* F) { face(1, i, j, F); });
      __syncthreads();
    }
    return;
  }
  // [b]: states on the lower and upper b-face; the b component is the face's normal velocity
  double lo[3][3], hi[3][3];
#pragma unroll
  for (int b = 0; b < 3; ++b)
#pragma unroll
    for (int c = 0; c < 3; ++c) lo[b][c] = hi[b][c] = 0.0;
  if (th.in) {
    const int L[3] = {th.i, th.j, th.k0 - 1};
    prestate_face<3>(u, slopes, g, k, 2, L, lo[2], v);
  }
  for (int kk = th.k0; kk < th.k1; ++kk) {
    const int p[3] = {th.i, th.j, kk};
    if (th.in) {
      prestate_face<3>(u, slopes, g, k, 0, p, hi[0], v);
      prestate_face<3>(u, slopes, g, k, 1, p, hi[1], v);
    }
    th.put(sh, kk, hi[0], hi[1]);
    if (th.in) prestate_face<3>(u, slopes, g, k, 2, p, hi[2], v);
    th.lower(sh, kk, hi[0], lo[0], lo[1]);  // behind a barrier
    if (!th.in) continue;
    double hat[3][3];
    const int t = th.i + g.n[0] * (th.j + g.n[1] * kk);
#pragma unroll
    for (int b = 0; b < 3; ++b)
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        hat[b][c] = hat_term(hi[b][b], lo[b][b], hi[b][c], lo[b][c], g);
        hats[(size_t)(b * 3 + c) * g.ncell + t] = hat[b][c];
      }
    store_tcom<3>(hat, Gp, Lu, fo, pv, tcom, g, k, t);
#pragma unroll
    for (int c = 0; c < 3; ++c) lo[2][c] = hi[2][c];
  }
}

}  // namespace hb
