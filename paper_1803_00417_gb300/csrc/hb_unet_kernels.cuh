// Kernels of the learned initial-guess network (U-Net on the nodal grid).
//
// Activations are channels-last BF16: element (point p, channel c) at
// p*C + c, points x fastest on a padded box of X*Y*Z points.  Convolutions
// are implicit GEMMs on the tensor cores (mma.sync m16n8k16, BF16 inputs,
// FP32 accumulation): rows = 16 points, columns = 8 output channels,
// k = 16 input channels of one of the 3^D taps.  Taps are the offsets in
// {-1,0,1}^D in lexicographic order (x slowest), zero padding outside.
#pragma once
#include <cuda_bf16.h>
#include <cstdint>

namespace hb {
namespace nn {

typedef __nv_bfloat16 bf16;

__device__ __forceinline__ uint32_t ld32(const bf16* p) { return *reinterpret_cast<const uint32_t*>(p); }

__device__ __forceinline__ uint32_t pack2(bf16 lo, bf16 hi) {
  return (uint32_t)__bfloat16_as_ushort(lo) | ((uint32_t)__bfloat16_as_ushort(hi) << 16);
}

__device__ __forceinline__ void mma_bf16(float* d, const uint32_t* a, uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};\n"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

template <int D>
__device__ __forceinline__ void tap_offset(int t, int* o) {
  if (D == 3) {
    o[0] = t / 9 - 1;
    o[1] = (t / 3) % 3 - 1;
    o[2] = t % 3 - 1;
  } else {
    o[0] = t / 3 - 1;
    o[1] = t % 3 - 1;
    o[2] = 0;
  }
}

struct Box {
  int X, Y, Z;
};

// point index of p shifted by o, or -1 outside the box
__device__ __forceinline__ long long shifted(const Box& b, int i, int j, int k, const int* o) {
  int a = i + o[0], c = j + o[1], e = k + o[2];
  if (a < 0 || a >= b.X || c < 0 || c >= b.Y || e < 0 || e >= b.Z) return -1;
  return (long long)a + (long long)b.X * ((long long)c + (long long)b.Y * e);
}

__device__ __forceinline__ void coords(const Box& b, long long p, int& i, int& j, int& k) {
  i = (int)(p % b.X);
  long long r = p / b.X;
  j = (int)(r % b.Y);
  k = (int)(r / b.Y);
}

// out[p, out_off + co] = act(bias[co] + sum_tap sum_ci in[p + o_tap, ci] W[tap, co, ci])
// for the NTB*8 output channels of slice blockIdx.y.  4 warps, 16 points each.
// W: [taps][Cout][Cin] BF16 (Cin multiple of 16).  bias may be null.
template <int D, int NTB>
__global__ void __launch_bounds__(128) k_conv_fwd(const bf16* __restrict__ in, int Cin, const bf16* __restrict__ W,
                                                  const float* __restrict__ bias, int Cout, bf16* __restrict__ out,
                                                  int out_stride, int out_off, int relu, Box box) {
  pdl_wait();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int g = lane >> 2, t4 = lane & 3;
  const long long P = (long long)box.X * box.Y * box.Z;
  const long long p0 = ((long long)blockIdx.x * 4 + warp) * 16;
  if (p0 >= P) return;
  const int co_base = blockIdx.y * NTB * 8;
  long long pr[2] = {p0 + g, p0 + g + 8};
  int ci[2], cj[2], ck[2];
  bool valid[2];
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    valid[r] = pr[r] < P;
    coords(box, valid[r] ? pr[r] : 0, ci[r], cj[r], ck[r]);
  }
  float acc[NTB][4];
#pragma unroll
  for (int n = 0; n < NTB; ++n) acc[n][0] = acc[n][1] = acc[n][2] = acc[n][3] = 0.f;
  const int T = D == 3 ? 27 : 9;
  const int KC = Cin / 16;
  for (int tap = 0; tap < T; ++tap) {
    int o[3];
    tap_offset<D>(tap, o);
    long long q[2];
#pragma unroll
    for (int r = 0; r < 2; ++r) q[r] = valid[r] ? shifted(box, ci[r], cj[r], ck[r], o) : -1;
    for (int kc = 0; kc < KC; ++kc) {
      uint32_t A[4];
      const int cb = kc * 16 + 2 * t4;
      A[0] = q[0] >= 0 ? ld32(in + q[0] * Cin + cb) : 0u;
      A[1] = q[1] >= 0 ? ld32(in + q[1] * Cin + cb) : 0u;
      A[2] = q[0] >= 0 ? ld32(in + q[0] * Cin + cb + 8) : 0u;
      A[3] = q[1] >= 0 ? ld32(in + q[1] * Cin + cb + 8) : 0u;
#pragma unroll
      for (int n = 0; n < NTB; ++n) {
        const bf16* wp = W + ((size_t)tap * Cout + co_base + n * 8 + g) * Cin + cb;
        mma_bf16(acc[n], A, ld32(wp), ld32(wp + 8));
      }
    }
  }
#pragma unroll
  for (int n = 0; n < NTB; ++n) {
    const int co = co_base + n * 8 + 2 * t4;
    const float b0 = bias ? bias[co] : 0.f, b1 = bias ? bias[co + 1] : 0.f;
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      if (!valid[r]) continue;
      float v0 = acc[n][2 * r] + b0, v1 = acc[n][2 * r + 1] + b1;
      if (relu) {
        v0 = fmaxf(v0, 0.f);
        v1 = fmaxf(v1, 0.f);
      }
      *reinterpret_cast<uint32_t*>(out + pr[r] * out_stride + out_off + co) =
          pack2(__float2bfloat16_rn(v0), __float2bfloat16_rn(v1));
    }
  }
}

// Weight gradient gW[tap, co, ci] += sum_p gz[p, co] x[p + o_tap, ci]: per tap
// a product of two point-major matrices over the points.  Block (bx, tap, bz)
// takes a 32 co x 32 ci tile (narrower at the edges) of one tap over one chunk
// of points: 64 points at a time of both operands are staged by cp.async (two
// buffers), each warp multiplies 16 of them (ldmatrix.trans gives the
// transposed fragments), the warps' partial sums meet in shared memory and one
// FP32 atomic per element goes to gW.  The chunks are short enough for about
// eight blocks per SM: the sum over points is the long dimension and the tiles
// alone (54 to 648 of them) leave most SMs idle; read by 2-byte gathers with a
// 64-bit division per point, 4096 points a block, a 32^3 layer took 370 us.
constexpr int kWgTile = 32, kWgPts = 64, kWgRow = kWgTile * 2 + 16;  // 80-byte rows: no ldmatrix bank conflicts

__device__ __forceinline__ void ldsm4t(uint32_t* r, uint32_t a) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(a)
               : "memory");
}

template <int D>
__global__ void __launch_bounds__(128) k_conv_wgrad(const bf16* __restrict__ x, int Cin, const bf16* __restrict__ gz,
                                                    int Cout, float* __restrict__ gW, Box box, int chunk) {
  pdl_wait();
  __shared__ __align__(16) unsigned char sm[2][2][kWgPts * kWgRow];  // [buffer][gz, x]
  __shared__ float part[4][kWgTile * kWgTile];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int nci = (Cin + kWgTile - 1) / kWgTile;
  const int co0 = (int)(blockIdx.x / nci) * kWgTile, ci0 = (int)(blockIdx.x % nci) * kWgTile;
  const int nco = min(kWgTile, Cout - co0), ncx = min(kWgTile, Cin - ci0);  // multiples of 16
  int o[3];
  tap_offset<D>(blockIdx.y, o);
  const int P = box.X * box.Y * box.Z;  // at most 2^31 / 16 (the activations' index range)
  const int pb = (int)blockIdx.z * chunk, pe = min(pb + chunk, P);
  // thread -> (point, 16-byte chunk) of a stage: 64 points x 4 chunks of each operand
  auto load = [&](int p0, int b) {
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const int pt = (tid >> 2) + 32 * r, ch = tid & 3, p = p0 + pt;
      const uint32_t dst = (uint32_t)(pt * kWgRow + ch * 16);
      const bool in = p < pe;
      const int rw = p / box.X, i = p - rw * box.X, k = rw / box.Y, j = rw - k * box.Y;
      const long long q = in ? shifted(box, i, j, k, o) : -1;
      const bool okg = in && ch * 8 < nco, okx = q >= 0 && ch * 8 < ncx;
      const uint32_t dg = (uint32_t)__cvta_generic_to_shared(&sm[b][0][0]) + dst;
      const uint32_t dx = (uint32_t)__cvta_generic_to_shared(&sm[b][1][0]) + dst;
      const bf16* sg = okg ? gz + (long long)p * Cout + co0 + ch * 8 : gz;
      const bf16* sx = okx ? x + q * Cin + ci0 + ch * 8 : x;
      const int ng = okg ? 16 : 0, nx = okx ? 16 : 0;
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(dg), "l"(sg), "r"(ng) : "memory");
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(dx), "l"(sx), "r"(nx) : "memory");
    }
    asm volatile("cp.async.commit_group;\n" ::: "memory");
  };
  float acc[2][4][4] = {};  // [16 co][8 ci]
  int b = 0;
  if (pb < pe) load(pb, 0);
  for (int p0 = pb; p0 < pe; p0 += kWgPts, b ^= 1) {
    if (p0 + kWgPts < pe) {
      load(p0 + kWgPts, b ^ 1);
      asm volatile("cp.async.wait_group 1;\n" ::: "memory");
    } else {
      asm volatile("cp.async.wait_group 0;\n" ::: "memory");
    }
    __syncthreads();
    // the warp's 16 points; lane l addresses row l % 8 of matrix l / 8
    const uint32_t row = (uint32_t)((warp * 16 + ((lane >> 4) << 3) + (lane & 7)) * kWgRow);
    const uint32_t brow = (uint32_t)((warp * 16 + (((lane >> 3) & 1) << 3) + (lane & 7)) * kWgRow);
    const uint32_t sg = (uint32_t)__cvta_generic_to_shared(&sm[b][0][0]);
    const uint32_t sx = (uint32_t)__cvta_generic_to_shared(&sm[b][1][0]);
    uint32_t A[2][4], B[2][4];
#pragma unroll
    for (int m = 0; m < 2; ++m) ldsm4t(A[m], sg + row + (uint32_t)(m * 32 + ((lane >> 3) & 1) * 16));
#pragma unroll
    for (int n = 0; n < 2; ++n) ldsm4t(B[n], sx + brow + (uint32_t)(n * 32 + (lane >> 4) * 16));
#pragma unroll
    for (int m = 0; m < 2; ++m)
#pragma unroll
      for (int n = 0; n < 4; ++n) mma_bf16(acc[m][n], A[m], B[n >> 1][2 * (n & 1)], B[n >> 1][2 * (n & 1) + 1]);
    __syncthreads();
  }
  const int g = lane >> 2, t4 = lane & 3;
#pragma unroll
  for (int m = 0; m < 2; ++m)
#pragma unroll
    for (int n = 0; n < 4; ++n)
#pragma unroll
      for (int q = 0; q < 4; ++q)
        part[warp][(m * 16 + g + (q >> 1) * 8) * kWgTile + n * 8 + 2 * t4 + (q & 1)] = acc[m][n][q];
  __syncthreads();
  for (int e = tid; e < kWgTile * kWgTile; e += 128) {
    const int r = e / kWgTile, c = e % kWgTile;
    if (r < nco && c < ncx)
      atomicAdd(gW + ((size_t)blockIdx.y * Cout + co0 + r) * Cin + ci0 + c,
                (part[0][e] + part[1][e]) + (part[2][e] + part[3][e]));
  }
}

}  // namespace nn
}  // namespace hb
