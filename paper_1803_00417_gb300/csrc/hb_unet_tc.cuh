// The U-Net convolution on the 5th-generation tensor cores (tcgen05): an
// implicit GEMM D[p, co] = sum_tap sum_ci X[p + o_tap, ci] W[tap, co, ci]
// with M = 128 points per CTA, N = a slice of Cout, K = Cin per tap.  The
// operands are staged in shared memory (K-major, no swizzle: core matrices of
// 8 rows x 16 bytes), one thread issues the tcgen05.mma (BF16 in,
// FP32 accumulate in TMEM), tcgen05.commit arrives on an mbarrier that the CTA
// waits on (bounded); the epilogue reads the accumulators with tcgen05.ld
// (warp w owns TMEM lanes 32w .. 32w+31, i.e. its 32 points), adds the bias,
// applies ReLU and stores BF16.
#pragma once
#include <cuda_bf16.h>
#include <cstdint>

#include "hb_unet_kernels.cuh"

namespace hb {
namespace nn {

constexpr int kTcM = 128;                 // points per CTA (the MMA's M)
// mbarrier polls before a wait on the tensor cores gives up.  A CTA that
// gives up sets the network's error flag (the host then reports
// HBF_ERR_TIMEOUT and discards every output of that forward pass), waits
// again on the same phase for up to kTcDrainLimit polls so that no MMA it
// issued is still writing its TMEM columns or reading its shared memory, and
// only then frees its TMEM and exits.  Completion of one CTA's MMAs takes
// microseconds, so neither limit is reached in normal operation.
constexpr long long kTcWaitLimit = 1 << 24;
constexpr long long kTcDrainLimit = 1 << 27;

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Shared-memory matrix descriptor for a K-major operand without swizzling, as
// two words: lo holds the start address / 16 and the byte stride / 16 between
// core matrices along K (leading), hi the one along M/N (stride) and the
// descriptor version 1; base offset 0, layout 0.  Moving the operand by n
// bytes adds n / 16 to lo: one thread issues every MMA of a CTA, and building
// the whole descriptor for each took it about 130 cycles an MMA.
__device__ __forceinline__ uint32_t tc_desc_lo(uint32_t saddr, uint32_t lbo) { return (saddr >> 4) | ((lbo >> 4) << 16); }
__device__ __forceinline__ uint32_t tc_desc_hi(uint32_t sbo) { return (sbo >> 4) | (1u << 14); }

// Instruction descriptor of kind::f16: FP32 accumulator, BF16 A and B, both
// K-major, shape M x N.
__host__ __device__ constexpr uint32_t tc_idesc(int M, int N) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// TMEM columns for an accumulator of n FP32 columns (a power of two >= 32)
__host__ __device__ constexpr int tc_cols(int n) {
  return n <= 32 ? 32 : (n <= 64 ? 64 : (n <= 128 ? 128 : (n <= 256 ? 256 : 512)));
}

__device__ __forceinline__ bool mbar_wait_parity(uint32_t bar, uint32_t parity,
                                                 long long limit = kTcWaitLimit) {
  for (long long it = 0; it < limit; ++it) {
    uint32_t done;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(bar), "r"(parity)
        : "memory");
    if (done) return true;
  }
  return false;
}

__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, bool ok) {
  const int n = ok ? 16 : 0;  // 0: the 16 bytes are zeros
  asm volatile("cp.async.ca.shared.global [%0], [%1], 16, %2;\n" ::"r"(dst), "l"(src), "r"(n) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

// D += A B (FIRST: D = A B)
template <bool FIRST>
__device__ __forceinline__ void tc_mma(uint32_t tmem, uint32_t alo, uint32_t ahi, uint32_t blo, uint32_t bhi,
                                       uint32_t idesc) {
  if (FIRST)
    asm volatile(
        "{\n .reg .pred p;\n .reg .b64 a, b;\n mov.b64 a, {%1, %2};\n mov.b64 b, {%3, %4};\n"
        " setp.ne.b32 p, 0, 0;\n tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %5, p;\n}\n" ::"r"(tmem),
        "r"(alo), "r"(ahi), "r"(blo), "r"(bhi), "r"(idesc)
        : "memory");
  else
    asm volatile(
        "{\n .reg .pred p;\n .reg .b64 a, b;\n mov.b64 a, {%1, %2};\n mov.b64 b, {%3, %4};\n"
        " setp.eq.b32 p, 0, 0;\n tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %5, p;\n}\n" ::"r"(tmem),
        "r"(alo), "r"(ahi), "r"(blo), "r"(bhi), "r"(idesc)
        : "memory");
}
__device__ __forceinline__ void tc_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(bar) : "memory");
}

// TMEM and barrier set-up of a CTA: warp 0 allocates tcols columns, thread 0
// initialises nbar barriers of one arrival; returns the TMEM address
__device__ __forceinline__ uint32_t tc_setup(uint32_t* slot, uint64_t* bars, int nbar, int tcols) {
  if (threadIdx.x < 32) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(slot)),
                 "r"(tcols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
  }
  if (threadIdx.x == 0) {
    for (int i = 0; i < nbar; ++i)
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(smem_u32(bars + i)) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
  return *slot;
}
__device__ __forceinline__ void tc_release(uint32_t tmem, int tcols) {
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  __syncthreads();
  if (threadIdx.x < 32)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(tcols) : "memory");
}

// bias, ReLU and BF16 of the accumulators' row tid % 128 (n columns, a multiple
// of 16, shared out over the CTA's groups of four warps), to dst when the row
// is a point; bias may be null
__device__ __forceinline__ void tc_epilogue(uint32_t tmem, int n, const float* __restrict__ bias, int relu, bf16* dst,
                                            bool valid) {
  const uint32_t lane_base = tmem + (((threadIdx.x >> 5) & 3u) << 21);  // warp w: lanes 32 (w % 4) on
  for (int c0 = (int)(threadIdx.x / kTcM) * 16; c0 < n; c0 += (int)(blockDim.x / kTcM) * 16) {
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, "
        "%14, %15}, [%16];\n"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(lane_base + (uint32_t)c0)
        : "memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
    if (valid) {
      uint32_t packed[8];
#pragma unroll
      for (int m = 0; m < 8; ++m) {
        float v0 = __uint_as_float(r[2 * m]) + (bias ? bias[c0 + 2 * m] : 0.f);
        float v1 = __uint_as_float(r[2 * m + 1]) + (bias ? bias[c0 + 2 * m + 1] : 0.f);
        if (relu) {
          v0 = fmaxf(v0, 0.f);
          v1 = fmaxf(v1, 0.f);
        }
        packed[m] = pack2(__float2bfloat16_rn(v0), __float2bfloat16_rn(v1));
      }
      uint4* d = reinterpret_cast<uint4*>(dst + c0);
      d[0] = make_uint4(packed[0], packed[1], packed[2], packed[3]);
      d[1] = make_uint4(packed[4], packed[5], packed[6], packed[7]);
    }
  }
}

constexpr int kTcSlack = 1024;           // after the operand tiles: alignment
constexpr int kTcMaxSmem = 200 * 1024;  // dynamic shared memory a convolution may use

// ---------------------------------------------------------------------------
// General variant: any box, any layer.  The CTA takes 128 points and nt output
// channels.  Per tap its 16 warps bring the 128 shifted input rows and the nt x
// Cin weights to one of two shared-memory stages, through registers: the loads
// of the next two taps are in flight while the current tap's MMAs run.  (By
// cp.async a tap took 1.15 us whatever its size and the ring's depth: the
// proxy fence that makes the stage visible to the tensor cores also waits for
// the copies still in flight.  Staged by four warps one tap at a time it took
// 2.4 us.)  nt is a slice of Cout where the points alone leave SMs without a
// CTA (the coarse levels: 1 to 46 CTAs of 128 points), and each slice then
// stages fewer weights.
// ---------------------------------------------------------------------------
constexpr int kTcThreads = 512;
__host__ __device__ constexpr int tc_stage_bytes(int cin, int nt) { return (kTcM + nt) * cin * 2; }
__host__ __device__ constexpr int tc_smem_bytes(int cin, int nt) { return 2 * tc_stage_bytes(cin, nt) + kTcSlack; }
// output channels per CTA: all of them, or the largest slice (16 at least)
// that gives every SM a CTA
__host__ __device__ constexpr int tc_slice(long long blocks, int cout) {
  int nt = cout;
  while (nt % 32 == 0 && (nt > kTcM || blocks * (cout / nt) < 152)) nt /= 2;
  return nt;
}

// out[p, out_off + co] = act(bias[co] + sum_tap sum_ci in[p + o_tap, ci] W[tap, co, ci])
// for co in slice blockIdx.y of nt channels.  Requires Cin % 16 == 0, Cin <=
// 32 KQ, nt % 16 == 0, 16 <= nt <= 128; tcols = tc_cols(nt).  *err is set when
// a wait on the tensor cores gives up (the outputs of that CTA are then not
// written).
template <int D, int KQ>
__global__ void __launch_bounds__(kTcThreads) k_conv_fwd_tc(const bf16* __restrict__ in, int Cin,
                                                            const bf16* __restrict__ W,
                                                            const float* __restrict__ bias, int Cout, int nt,
                                                            bf16* __restrict__ out, int out_stride, int out_off,
                                                            int relu, Box box, int tcols, int* __restrict__ err) {
  pdl_wait();
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ __align__(8) uint64_t bars[3];  // one per stage, and one for the last MMA
  __shared__ uint32_t tmem_slot;
  constexpr int T = D == 3 ? 27 : 9;
  const int tid = threadIdx.x;
  const int KC = Cin / 8;  // 16-byte chunks per row
  const int co0 = blockIdx.y * nt;
  const long long P = (long long)box.X * box.Y * box.Z;
  const uint32_t tmem = tc_setup(&tmem_slot, bars, 3, tcols);
  const uint32_t idesc = tc_idesc(kTcM, nt);
  const uint32_t base = smem_u32(smem), stage = (uint32_t)tc_stage_bytes(Cin, nt), boff = (uint32_t)kTcM * Cin * 2;
  const uint32_t dlo = tc_desc_lo(base, 128u), dhi = tc_desc_hi((uint32_t)KC * 128u);  // next 8-row group: KC chunks on
  // Staging: warp w copies rows 8 w .. 8 w + 7, 4 chunks at a time (lane: row
  // l % 8, chunk l / 8), so that it touches 8 lines of global memory at a time
  // and writes shared memory without conflicts.  Bit t of vm tells that tap t
  // of the lane's row of A lies in the box (taps run over (x, y(, z)) offsets,
  // x slowest: three bits per axis).
  const int lane = tid & 31, c4 = lane >> 3, row = (tid >> 5) * 8 + (lane & 7);
  const long long pr = (long long)blockIdx.x * kTcM + row;
  uint32_t vm = 0u;
  if (pr < P) {
    const int pp = (int)pr, rw = pp / box.X, pi = pp - rw * box.X, pk = rw / box.Y, pj = rw - pk * box.Y;
    auto bits = [](int q, int n) { return (q > 0 ? 1u : 0u) | 2u | (q < n - 1 ? 4u : 0u); };
    const uint32_t bx = bits(pi, box.X), by = bits(pj, box.Y), bz = bits(pk, box.Z);
    auto spread = [](uint32_t hi, uint32_t lo, int w) {
      return ((hi & 1u) ? lo : 0u) | ((hi & 2u) ? lo << w : 0u) | ((hi & 4u) ? lo << (2 * w) : 0u);
    };
    vm = D == 3 ? spread(bx, spread(by, bz, 3), 9) : spread(bx, by, 3);
  }
  const size_t place = (size_t)((row >> 3) * KC + c4) * 128u + (size_t)(row & 7) * 16u;
  const bf16* const wrow = W + ((size_t)co0 + row) * Cin + 8 * c4;
  uint4 ra[2][KQ], rb[2][KQ];
  auto fetch = [&](int tap, uint4* a, uint4* b) {
    int o[3];
    tap_offset<D>(tap, o);
    const long long sh = (long long)o[0] + (long long)box.X * ((long long)o[1] + (long long)box.Y * o[2]);
    const bool in_box = (vm >> tap) & 1u;  // zeros outside
    const bf16* src = in + (pr + sh) * Cin + 8 * c4;
    const bf16* wt = wrow + (size_t)tap * Cout * Cin;
#pragma unroll
    for (int k = 0; k < KQ; ++k) {
      a[k] = b[k] = make_uint4(0u, 0u, 0u, 0u);
      if (4 * k + c4 < KC) {
        if (in_box) a[k] = *reinterpret_cast<const uint4*>(src + 32 * k);
        if (row < nt) b[k] = *reinterpret_cast<const uint4*>(wt + 32 * k);
      }
    }
  };
  bool ok = true;  // false once a wait gave up: nothing is staged any more
  auto step = [&](int tap, uint4* a, uint4* b) {
    const int s = tap & 1;
    // the stage's previous MMAs, two taps back
    if (tap >= 2 && ok) ok = mbar_wait_parity(smem_u32(bars + s), (uint32_t)((tap >> 1) - 1) & 1u);
    if (ok) {
      unsigned char* dst = smem + (size_t)s * stage + place;
#pragma unroll
      for (int k = 0; k < KQ; ++k)
        if (4 * k + c4 < KC) {
          *reinterpret_cast<uint4*>(dst + (size_t)k * 512u) = a[k];
          if (row < nt) *reinterpret_cast<uint4*>(dst + boff + (size_t)k * 512u) = b[k];
        }
    }
    if (tap + 2 < T) fetch(tap + 2, a, b);
    // make the stage visible to the tensor cores
    asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
    __syncthreads();
    if (tid == 0) {
      asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
      const uint32_t alo = dlo + (uint32_t)s * (stage >> 4), blo = alo + (boff >> 4);
      if (tap == 0)
        tc_mma<true>(tmem, alo, dhi, blo, dhi, idesc);
      else
        tc_mma<false>(tmem, alo, dhi, blo, dhi, idesc);
#pragma unroll 4
      for (int kc = 1; kc < KC / 2; ++kc)  // K = 16: two chunks of 128 bytes per core-matrix row group
        tc_mma<false>(tmem, alo + 16u * kc, dhi, blo + 16u * kc, dhi, idesc);
      tc_commit(smem_u32(bars + s));
      if (tap == T - 1) tc_commit(smem_u32(bars + 2));
    }
  };
  fetch(0, ra[0], rb[0]);
  fetch(1, ra[1], rb[1]);
#pragma unroll 1
  for (int tap = 0; tap < T; tap += 2) {
    step(tap, ra[0], rb[0]);
    if (tap + 1 < T) step(tap + 1, ra[1], rb[1]);
  }
  if (ok) ok = mbar_wait_parity(smem_u32(bars + 2), 0u);
  ok = __syncthreads_and(ok ? 1 : 0) != 0;
  asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
  if (ok) {
    const long long p = (long long)blockIdx.x * kTcM + (tid & (kTcM - 1));
    tc_epilogue(tmem, nt, bias ? bias + co0 : nullptr, relu, out + p * out_stride + out_off + co0, p < P);
  } else {
    if (tid == 0) atomicExch(err, 1);
    mbar_wait_parity(smem_u32(bars + 2), 0u, kTcDrainLimit);  // drain before TMEM is freed
  }
  tc_release(tmem, tcols);
}

// ---------------------------------------------------------------------------
// Halo variant for the layers whose whole tap set fits in shared memory.  The
// CTA's 128 points are an 8 (x) x 16 (y) tile of one z plane.  Its input halo
// (10 x 18 x 3 points in 3D, 10 x 18 in 2D, zero outside the box) is staged as
// one plane of 16-byte channel chunks per K chunk, rows at a 16-byte stride;
// then the operand of tap (dx, dy, dz) is a descriptor into that halo: 8
// consecutive halo rows (one tile row shifted by dx) form a core matrix at any
// start row, the next tile row is 10 halo rows further (SBO = 160 bytes) and
// the next K chunk one plane further (LBO).  One thread issues all 3^d *
// Cin/16 MMAs back to back.  A CTA stages the weights of all taps once and
// walks tiles (tile += gridDim.x), the next tile's halo arriving by cp.async
// while the current one is multiplied and stored (two halo buffers where they
// fit): with one tile per CTA, staging the weights again for every 128 points
// and nothing overlapped, a 72^3 layer of 16 channels took 99 us.
// ---------------------------------------------------------------------------
constexpr int kHaloX = 10, kHaloY = 18;

__host__ __device__ constexpr int tc_halo_rows(int d) { return kHaloX * kHaloY * (d == 3 ? 3 : 1); }

__host__ __device__ constexpr int tc_halo_smem_bytes(int d, int cin, int cout, int nbuf) {
  return nbuf * tc_halo_rows(d) * cin * 2 + (d == 3 ? 27 : 9) * cout * cin * 2 + kTcSlack;
}
// halo buffers: 2 while two CTAs share an SM (about 112 KB each), else 1 (the
// CTAs then overlap each other), or none where not even one fits
__host__ __device__ constexpr int tc_halo_bufs(int d, int cin, int cout) {
  return tc_halo_smem_bytes(d, cin, cout, 2) <= 112 * 1024 ? 2
                                                           : (tc_halo_smem_bytes(d, cin, cout, 1) <= kTcMaxSmem ? 1 : 0);
}

constexpr int kTcHaloThreads = 256;
template <int D>
__global__ void __launch_bounds__(kTcHaloThreads) k_conv_fwd_tc_halo(const bf16* __restrict__ in, int Cin,
                                                           const bf16* __restrict__ W,
                                                           const float* __restrict__ bias, int Cout,
                                                           bf16* __restrict__ out, int out_stride, int out_off,
                                                           int relu, Box box, int nbuf, int tcols,
                                                           int* __restrict__ err) {
  pdl_wait();
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ __align__(8) uint64_t mbar;
  __shared__ uint32_t tmem_slot;
  constexpr int T = D == 3 ? 27 : 9;
  constexpr int HR = tc_halo_rows(D);
  const int KC = Cin / 8;
  const uint32_t plane = (uint32_t)HR * 16u;  // one 16-byte channel chunk of every halo row
  const uint32_t hbase = smem_u32(smem), hbuf = (uint32_t)KC * plane, bbase = hbase + (uint32_t)nbuf * hbuf;
  const int tid = threadIdx.x;
  const int ntx = box.X / 8, nty = (box.Y + 15) / 16, ntile = ntx * nty * box.Z;
  const uint32_t tmem = tc_setup(&tmem_slot, &mbar, 1, tcols);
  const uint32_t bar = smem_u32(&mbar), idesc = tc_idesc(kTcM, Cout);
  const uint32_t alo = tc_desc_lo(hbase, plane), ahi = tc_desc_hi((uint32_t)kHaloX * 16u);
  const uint32_t blo = tc_desc_lo(bbase, 128u), bhi = tc_desc_hi((uint32_t)KC * 128u);
  const uint32_t wtap = (uint32_t)Cout * Cin * 2 / 16;  // a tap's weights
  auto place = [&](int t, int& x0, int& y0, int& z) {
    const int r = t / ntx;
    x0 = (t - r * ntx) * 8;
    z = r / nty;
    y0 = (r - z * nty) * 16;
  };
  // input halo of tile t into buffer b, zero outside the box
  auto load_halo = [&](int t, int b) {
    int x0, y0, z;
    place(t, x0, y0, z);
    // a warp copies 32 / cl points x cl chunks at a time (neighbouring points'
    // lines are shared, and shared memory is written without conflicts)
    const int cl = KC >= 4 ? 4 : 2, np = 32 / cl, lane = tid & 31;
    const int c0 = lane / np;
    for (int h = (tid >> 5) * np + lane % np; h < HR; h += (kTcHaloThreads / 32) * np) {
      const int xx = h % kHaloX, r = h / kHaloX, yy = r % kHaloY, zz = r / kHaloY;
      const int gx = x0 - 1 + xx, gy = y0 - 1 + yy, gz = D == 3 ? z - 1 + zz : 0;
      const bool in_box = gx >= 0 && gx < box.X && gy >= 0 && gy < box.Y && gz >= 0 && gz < box.Z;
      const bf16* src =
          in_box ? in + ((long long)gx + (long long)box.X * ((long long)gy + (long long)box.Y * gz)) * Cin : in;
      const uint32_t dst = hbase + (uint32_t)b * hbuf + (uint32_t)h * 16u;
      for (int k8 = c0; k8 < KC; k8 += cl) cp_async16(dst + (uint32_t)k8 * plane, src + 8 * k8, in_box);
    }
  };
  // weights of every tap, core-matrix layout per tap
  for (int idx = tid; idx < T * Cout * KC; idx += kTcHaloThreads) {
    const int k8 = idx % KC, rr = idx / KC;  // rr = tap * Cout + row
    const int tap = rr / Cout, r = rr - tap * Cout;
    cp_async16(bbase + (uint32_t)tap * Cout * Cin * 2 + (uint32_t)((r >> 3) * KC + k8) * 128u + (uint32_t)(r & 7) * 16u,
               W + (size_t)8 * idx, true);
  }
  int t = blockIdx.x;
  if (t < ntile) load_halo(t, 0);
  cp_async_commit();
  bool ok = true;
  uint32_t parity = 0;
  for (int it = 0; t < ntile && ok; t += gridDim.x, ++it) {  // ok is the same in every thread
    const int b = nbuf == 2 ? it & 1 : 0, tn = t + (int)gridDim.x;
    cp_async_wait<0>();
    asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");  // the last tile's accumulators are read
    __syncthreads();
    if (tid == 0) {
      asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
      const uint32_t ab = alo + (uint32_t)b * (hbuf >> 4);
      uint32_t w = blo;
#pragma unroll
      for (int tap = 0; tap < T; ++tap, w += wtap) {
        int o[3];
        tap_offset<D>(tap, o);
        const int row0 = ((D == 3 ? (1 + o[2]) * kHaloY : 0) + (1 + o[1])) * kHaloX + (1 + o[0]);
        if (tap == 0)
          tc_mma<true>(tmem, ab + row0, ahi, w, bhi, idesc);
        else
          tc_mma<false>(tmem, ab + row0, ahi, w, bhi, idesc);
        for (int kc = 1; kc < KC / 2; ++kc)
          tc_mma<false>(tmem, ab + row0 + (uint32_t)(2 * kc) * HR, ahi, w + 16u * kc, bhi, idesc);
      }
      tc_commit(bar);
    }
    // the other buffer's MMAs are done: the next tile's halo
    if (nbuf == 2 && tn < ntile) load_halo(tn, b ^ 1);
    if (nbuf == 2) cp_async_commit();
    ok = __syncthreads_and(mbar_wait_parity(bar, parity) ? 1 : 0) != 0;
    if (!ok) break;  // parity keeps the phase still pending
    parity ^= 1u;
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    if (nbuf == 1) {
      if (tn < ntile) load_halo(tn, 0);
      cp_async_commit();
    }
    // row r of D is the tile point (x0 + r % 8, y0 + r / 8, z)
    int x0, y0, z;
    place(t, x0, y0, z);
    const int row = tid & (kTcM - 1), px = x0 + (row & 7), py = y0 + (row >> 3);
    const long long p = (long long)px + (long long)box.X * ((long long)py + (long long)box.Y * (D == 3 ? z : 0));
    tc_epilogue(tmem, Cout, bias, relu, out + p * out_stride + out_off, py < box.Y);
  }
  cp_async_wait<0>();
  if (!ok) {
    if (tid == 0) atomicExch(err, 1);
    mbar_wait_parity(bar, parity, kTcDrainLimit);  // drain before TMEM is freed
  }
  tc_release(tmem, tcols);
}

}  // namespace nn
}  // namespace hb
