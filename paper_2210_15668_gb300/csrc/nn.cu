// Kernels of the learned warm-start network (a small 3-D U-Net on one coarse
// multigrid level).  Activations are channels-last BF16 ([voxel][channel]);
// convolutions are implicit GEMMs on the BF16 tensor cores with FP32
// accumulation (mma.sync m16n8k16): M = voxels (16 per warp), N = output
// channels, K = 27 taps x input channels, split over three warps per voxel tile.  3x3x3 stencils are periodic in x
// and y and zero-padded in z, like the device.  Gradients with respect to the
// input use the same kernel with the taps flipped and the channel matrices
// transposed (the adjoint convolution); gradients with respect to the weights
// contract over voxels (M = input channels, N = output channels, K = voxels) into one
// FP32 partial sum per block, and the partial sums are added in a fixed order.  Grids that
// the tensor-memory convolution's tiles divide take that kernel instead of mma.sync
// (conv_tc_kernel).  Master weights, Adam moments and gradients are FP32; the kernels read
// BF16 copies.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <string>
#include <vector>

#include "ferrox_internal.cuh"

namespace fx {

namespace {

using bf16 = __nv_bfloat16;

__device__ __forceinline__ void mma_bf16(float (&d)[4], const unsigned (&a)[4], const unsigned (&b)[2]) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
      "{%8,%9}, {%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

// voxel index of the neighbour at tap (dz, dy, dx) = (tap/9, tap/3%3, tap%3) - 1,
// or -1 outside the z range
__device__ __forceinline__ int nb_index(int z, int y, int x, int tap, const NNGrid& g) {
  const int zz = z + tap / 9 - 1;
  if (zz < 0 || zz >= g.D) return -1;
  int yy = y + (tap / 3) % 3 - 1;
  yy = yy < 0 ? yy + g.H : (yy >= g.H ? yy - g.H : yy);
  int xx = x + tap % 3 - 1;
  xx = xx < 0 ? xx + g.W : (xx >= g.W ? xx - g.W : xx);
  return (zz * g.H + yy) * g.W + xx;
}

__device__ __forceinline__ void voxel_zyx(int m, const NNGrid& g, int& z, int& y, int& x) {
  const int hw = g.H * g.W;
  z = m / hw;
  const int r = m - z * hw;
  y = r / g.W;
  x = r - y * g.W;
}

// out[m][co] = act(bias[co] + sum_tap sum_ci in[nb(m, tap)][ci] w[tap][ci][co]),
// weights in the kernel layout wk[tap][co][ci] (BF16).  A block holds kConvTiles
// tiles of 16 voxels; the three warps of a tile (threadIdx.z) split the 27 taps
// by z offset (9 each), so every warp's chain of dependent gathers is one slab,
// and the partial sums meet in shared memory in a fixed order (slab 0 + slab 1
// + slab 2).
constexpr int kConvTiles = 4;

template <int COUT, bool MASK>   // MASK: the ReLU's backward on the output (an adjoint)
__global__ void __launch_bounds__(32 * kConvTiles * 3) conv_fwd_kernel(
    const bf16* in, int cin, const bf16* __restrict__ wk,
    const float* __restrict__ bias, NNGrid g, int relu, const bf16* mask, bf16* __restrict__ out_bf,
    float* __restrict__ out_f, int f_ch0) {
  pdl_enter();
  __shared__ float part[2][kConvTiles][COUT / 8][4][32];
  const int lane = threadIdx.x, tile = threadIdx.y, slab = threadIdx.z;
  const int M = g.D * g.H * g.W;
  const int m0 = (blockIdx.x * kConvTiles + tile) * 16;
  const bool active = m0 < M;
  const int gq = lane >> 2, tq = lane & 3;
  int zr[2], yr[2], xr[2];
  bool val[2];
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    const int m = m0 + gq + 8 * r;
    val[r] = m < M;
    voxel_zyx(val[r] ? m : 0, g, zr[r], yr[r], xr[r]);
  }
  float acc[COUT / 8][4];
#pragma unroll
  for (int j = 0; j < COUT / 8; ++j) acc[j][0] = acc[j][1] = acc[j][2] = acc[j][3] = 0.f;
  const unsigned* inw = reinterpret_cast<const unsigned*>(in);
  const unsigned* ww = reinterpret_cast<const unsigned*>(wk);
  const int cin2 = cin >> 1;
  if (active) {
    // the slab's nine taps unrolled: their gathers are all in flight before the
    // MMAs that consume them (the layer is latency-bound at these sizes)
#pragma unroll
    for (int t = 0; t < 9; ++t) {
      const int tap = slab * 9 + t;
      const int n0 = val[0] ? nb_index(zr[0], yr[0], xr[0], tap, g) : -1;
      const int n1 = val[1] ? nb_index(zr[1], yr[1], xr[1], tap, g) : -1;
      for (int c0 = 0; c0 < cin; c0 += 16) {
        const int off = (c0 >> 1) + tq;
        unsigned a[4];
        a[0] = n0 >= 0 ? __ldg(inw + (size_t)n0 * cin2 + off) : 0u;
        a[1] = n1 >= 0 ? __ldg(inw + (size_t)n1 * cin2 + off) : 0u;
        a[2] = n0 >= 0 ? __ldg(inw + (size_t)n0 * cin2 + off + 4) : 0u;
        a[3] = n1 >= 0 ? __ldg(inw + (size_t)n1 * cin2 + off + 4) : 0u;
#pragma unroll
        for (int j = 0; j < COUT / 8; ++j) {
          const unsigned* wp = ww + (size_t)(tap * COUT + j * 8 + gq) * cin2 + off;
          const unsigned b[2] = {__ldg(wp), __ldg(wp + 4)};
          mma_bf16(acc[j], a, b);
        }
      }
    }
  }
  if (slab > 0) {
#pragma unroll
    for (int j = 0; j < COUT / 8; ++j)
#pragma unroll
      for (int q = 0; q < 4; ++q) part[slab - 1][tile][j][q][lane] = acc[j][q];
  }
  __syncthreads();
  if (slab > 0 || !active) return;
#pragma unroll
  for (int j = 0; j < COUT / 8; ++j)
#pragma unroll
    for (int q = 0; q < 4; ++q) acc[j][q] = (acc[j][q] + part[0][tile][j][q][lane]) + part[1][tile][j][q][lane];
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    if (!val[r]) continue;
    const int m = m0 + gq + 8 * r;
#pragma unroll
    for (int j = 0; j < COUT / 8; ++j) {
      const int co = j * 8 + 2 * tq;
      float v0 = acc[j][2 * r], v1 = acc[j][2 * r + 1];
      if (bias) { v0 += bias[co]; v1 += bias[co + 1]; }
      if (relu) { v0 = fmaxf(v0, 0.f); v1 = fmaxf(v1, 0.f); }
      if (MASK) {
        const float2 am = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(mask + (size_t)m * COUT + co));
        if (!(am.x > 0.f)) v0 = 0.f;
        if (!(am.y > 0.f)) v1 = 0.f;
      }
      if (out_bf)
        *reinterpret_cast<__nv_bfloat162*>(out_bf + (size_t)m * COUT + co) = __floats2bfloat162_rn(v0, v1);
      if (out_f && f_ch0) {
        if (co == 0) out_f[m] = v0;
      } else if (out_f) {
        out_f[(size_t)m * COUT + co] = v0;
        out_f[(size_t)m * COUT + co + 1] = v1;
      }
    }
  }
}

// ---- 3x3x3 convolution on the fifth-generation tensor cores (tcgen05, TMEM) ----------
//
// A tile is 8 (x) x 16 (y) x zt (z) voxels.  Its input with a one-voxel halo
// (10 x 18 x (zt + 2) voxels, periodic in x and y, zero outside z) is staged in
// shared memory in the no-swizzle K-major layout of the tensor core's operands:
// for each 8-channel chunk a plane of 16-byte entries [z][y][x].  Eight
// consecutive x voxels are then one 8 x 16 B core matrix and the 16 y rows of a
// tile are core matrices 160 B apart, so the A operand of every tap is the same
// staged tile seen through a shifted descriptor: the 27 taps need no further
// data movement.  The weights of all taps sit beside it as [tap][ci/8][co][ci%8].
// One thread issues the 128 x COUT x 16 MMAs (27 taps x CIN/16 K-steps per
// z-plane) into FP32 accumulators in tensor memory; the four warps read their
// 32 rows back with tcgen05.ld for the bias, ReLU and BF16/FP32 store.
//
// CTAs are persistent: the weights are loaded once, and the halo buffers and
// accumulators are double-buffered, so the loads of tile i + 1 and the epilogue
// of tile i - 1 run while the tensor core works on tile i.
constexpr int kTcX = 8, kTcY = 16, kTcHX = kTcX + 2, kTcHY = kTcY + 2;
constexpr int kTcPlane = kTcHX * kTcHY;             // halo entries per z-plane
constexpr int kTcThreads = 128;
constexpr long long kTcWaitCycles = 2000000000LL;   // ~1 s at 2 GHz

__device__ __forceinline__ unsigned smem_u32(const void* p) {
  return (unsigned)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ void tc_cp16(unsigned dst, const void* src, bool valid) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(dst), "l"(src), "r"(valid ? 16 : 0)
               : "memory");
}

// shared-memory matrix descriptor: start address, leading (K-direction) and
// stride (8-row group) byte offsets, descriptor version 1, no swizzle.  The start
// address is the low field (bits 0-13, in 16-byte units), so a descriptor of an
// address 16 k bytes further is this one plus k.
__device__ __forceinline__ unsigned long long tc_desc(unsigned addr, unsigned lbo, unsigned sbo) {
  return (unsigned long long)((addr & 0x3FFFFu) >> 4) | ((unsigned long long)(lbo >> 4) << 16) |
         ((unsigned long long)(sbo >> 4) << 32) | (1ull << 46);
}

// instruction descriptor of kind::f16: FP32 accumulator, BF16 A and B, both
// K-major, M = 128, N = n
__host__ __device__ constexpr unsigned tc_idesc(int n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((unsigned)(n >> 3) << 17) | ((unsigned)(128 >> 4) << 24);
}

__device__ __forceinline__ void tc_mma(unsigned d, unsigned long long a, unsigned long long b, unsigned idesc,
                                       unsigned accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(d),
      "l"(a), "l"(b), "r"(idesc), "r"(accumulate)
      : "memory");
}

__device__ __forceinline__ bool mbar_try(unsigned mbar, unsigned parity) {
  unsigned done;
  asm volatile(
      "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}\n"
      : "=r"(done)
      : "r"(mbar), "r"(parity)
      : "memory");
  return done != 0;
}

// bounded wait on an mbarrier phase; false when the limit ran out
__device__ __forceinline__ bool mbar_wait(unsigned mbar, unsigned parity, long long limit) {
  const long long t0 = clock64();
  while (!mbar_try(mbar, parity))
    if (clock64() - t0 > limit) return false;
  return true;
}

// 16 consecutive FP32 accumulator columns of this warp's 32 rows
__device__ __forceinline__ void tc_ld16(unsigned taddr, float (&v)[16]) {
  unsigned r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, "
      "[%16];\n"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

__host__ __device__ constexpr int tc_cols(int n) {
  return n <= 32 ? 32 : n <= 64 ? 64 : n <= 128 ? 128 : n <= 256 ? 256 : 512;
}

struct TcTile {
  int x0, y0, z0;
};

__device__ __forceinline__ TcTile tc_tile(int t, const NNGrid& g, int zt) {
  const int nbx = g.W / kTcX, nby = g.H / kTcY;
  return TcTile{(t % nbx) * kTcX, ((t / nbx) % nby) * kTcY, (t / (nbx * nby)) * zt};
}

// Stage the halo of one tile: warp w takes halo rows (z, y) w, w + 4, ...; lane j
// takes entries j and j + 32 of a row, entry q = x * NCH + chunk, so a warp reads
// consecutive 16-byte chunks of consecutive voxels.  With UP the 48 input
// channels are the concatenation [up(a4) (32), s1 (16)] read in place: chunks
// 0-3 from the coarse field a4 (= in) at the parent voxel, chunks 4-5 from s1.
template <int CIN, bool UP>
__device__ __forceinline__ void tc_load_halo(const bf16* in, const bf16* s1,
                                             const NNGrid& g, TcTile t, int zt, unsigned buf, int chunk_entries) {
  constexpr int NCH = CIN / 8, PER_ROW = kTcHX * NCH;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int Hc = g.H / 2, Wc = g.W / 2;
  int goff[2], soff[2];
  bool have[2], fine[2];
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int q = lane + 32 * h;
    have[h] = q < PER_ROW;
    const int xx = have[h] ? q / NCH : 0, k = q % NCH;
    int gx = t.x0 + xx - 1;
    gx = gx < 0 ? gx + g.W : (gx >= g.W ? gx - g.W : gx);
    fine[h] = !UP || k >= 4;
    goff[h] = UP ? (k < 4 ? (gx >> 1) * 32 + 8 * k : gx * 16 + 8 * (k - 4)) : gx * CIN + 8 * k;
    soff[h] = 16 * (k * chunk_entries + xx);
  }
  const int rows = kTcHY * (zt + 2);
  for (int r = warp; r < rows; r += kTcThreads / 32) {
    const int zz = r / kTcHY, yy = r - zz * kTcHY;
    int gy = t.y0 + yy - 1;
    gy = gy < 0 ? gy + g.H : (gy >= g.H ? gy - g.H : gy);
    int gz = t.z0 + zz - 1;
    const bool okz = gz >= 0 && gz < g.D;
    gz = okz ? gz : 0;
    const bf16* row = UP ? s1 + (size_t)(gz * g.H + gy) * g.W * 16 : in + (size_t)(gz * g.H + gy) * g.W * CIN;
    const bf16* crow = UP ? in + (size_t)((gz >> 1) * Hc + (gy >> 1)) * Wc * 32 : row;
    const unsigned srow = buf + 16u * (unsigned)(r * kTcHX);
#pragma unroll
    for (int h = 0; h < 2; ++h)
      if (have[h]) tc_cp16(srow + soff[h], (fine[h] ? row : crow) + goff[h], okz);
  }
}

template <int CIN, int COUT, bool MASK>
__device__ __forceinline__ void tc_epilogue(unsigned tmem_acc, const NNGrid& g, TcTile t, int zt,
                                            const float* __restrict__ bias, int relu, const bf16* mask,
                                            bf16* __restrict__ out_bf, float* __restrict__ out_f, int f_ch0) {
  const int tid = threadIdx.x, warp = tid >> 5;
  // thread tid holds accumulator row tid = voxel (y0 + tid / 8, x0 + tid % 8)
  const int x = t.x0 + (tid & 7), y = t.y0 + (tid >> 3);
  for (int p = 0; p < zt; ++p) {
    const size_t m = ((size_t)(t.z0 + p) * g.H + y) * g.W + x;
#pragma unroll
    for (int j = 0; j < COUT / 16; ++j) {
      float v[16];
      tc_ld16(tmem_acc + ((unsigned)(32 * warp) << 16) + (unsigned)(p * COUT + 16 * j), v);
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        if (bias) v[i] += __ldg(bias + 16 * j + i);
        if (relu) v[i] = fmaxf(v[i], 0.f);
      }
      if (MASK) {   // the ReLU's backward: zero where the activation is not positive
        const uint4* mp = reinterpret_cast<const uint4*>(mask + m * COUT + 16 * j);
        const uint4 q[2] = {mp[0], mp[1]};
        const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(q);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const float2 am = __bfloat1622float2(h[i]);
          if (!(am.x > 0.f)) v[2 * i] = 0.f;
          if (!(am.y > 0.f)) v[2 * i + 1] = 0.f;
        }
      }
      if (out_bf) {
        uint4 q[2];
        __nv_bfloat162* h = reinterpret_cast<__nv_bfloat162*>(q);
#pragma unroll
        for (int i = 0; i < 8; ++i) h[i] = __floats2bfloat162_rn(v[2 * i], v[2 * i + 1]);
        uint4* o = reinterpret_cast<uint4*>(out_bf + m * COUT + 16 * j);
        o[0] = q[0];
        o[1] = q[1];
      }
      if (out_f && f_ch0) {
        if (j == 0) out_f[m] = v[0];
      } else if (out_f) {
        float4* o = reinterpret_cast<float4*>(out_f + m * COUT + 16 * j);
#pragma unroll
        for (int i = 0; i < 4; ++i) o[i] = make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
      }
    }
  }
}

template <int CIN, int COUT, bool UP, bool MASK>
__global__ void __launch_bounds__(kTcThreads) conv_tc_kernel(
    const bf16* in, const bf16* s1, const bf16* __restrict__ wt,
    const float* __restrict__ bias, NNGrid g, int zt, int relu, const bf16* mask,
    bf16* __restrict__ out_bf, float* __restrict__ out_f, int f_ch0, int* __restrict__ fault) {
  constexpr int NCH = CIN / 8;
  constexpr int WBYTES = 27 * CIN * COUT * 2;
  extern __shared__ __align__(128) unsigned char smem[];
  unsigned long long* mbar = reinterpret_cast<unsigned long long*>(smem);   // two barriers
  unsigned* tslot = reinterpret_cast<unsigned*>(smem + 16);
  const int tid = threadIdx.x, warp = tid >> 5;
  const int ncols = tc_cols(2 * zt * COUT);
  const int chunk_entries = kTcPlane * (zt + 2);
  const unsigned hbytes = 16u * NCH * chunk_entries;
  const unsigned sw = smem_u32(smem + 128);
  const unsigned hb0 = sw + WBYTES, mb0 = smem_u32(mbar);   // buffer / barrier b at + b hbytes / + 8 b
  const int ntiles = (g.W / kTcX) * (g.H / kTcY) * (g.D / zt);
  const int nmine = blockIdx.x < ntiles ? (ntiles - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;

  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(tslot)),
                 "r"(ncols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
  }
  if (tid == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(mb0) : "memory");
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(mb0 + 8) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  // weights (a straight copy of the packed array) and the first tile, one group.  The next
  // convolution's blocks may take their places now: each allocates its accumulators and
  // loads its weights while this kernel runs, and waits for it before its first input (no
  // kernel that writes weights lets its successor start early).  With the launches' own
  // work done ahead, nine dependent launches of a forward pass on 8x64x64 take 44 us
  // instead of 68; inputs of kernels that may start early are not marked __restrict__,
  // which would allow their loads before the wait.
  // The barrier puts every thread's trigger after warp 0's allocation: the successor starts
  // once all blocks here have triggered, so all hold their columns by then.  Its blocks on
  // the same SM may find none left and wait for this kernel; this kernel never waits for
  // theirs, which they keep until it is done (an allocation has no time limit).
  for (int i = tid; i < WBYTES / 16; i += kTcThreads) tc_cp16(sw + 16u * i, wt + 8 * i, true);
  __syncthreads();
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  pdl_enter();
  if (nmine > 0) tc_load_halo<CIN, UP>(in, s1, g, tc_tile(blockIdx.x, g, zt), zt, hb0, chunk_entries);
  asm volatile("cp.async.commit_group;\n" ::: "memory");

  constexpr unsigned idesc = tc_idesc(COUT);
  const unsigned a_lbo = 16u * chunk_entries, b_lbo = 16u * COUT;
  const unsigned long long bdesc0 = tc_desc(sw, b_lbo, 128u);
  unsigned tmem = 0;
  bool ok = true;
  int issued = 0;   // tiles whose MMAs were committed
  for (int i = 0; i < nmine; ++i) {
    asm volatile("cp.async.wait_group 0;\n" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    ok = !__syncthreads_or(!ok);
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    if (!ok) break;
    tmem = *tslot;
    const int cur = i & 1;
    if (tid == 0) {
      const unsigned d0 = tmem + (unsigned)(cur * zt * COUT);
      const unsigned long long adesc0 = tc_desc(hb0 + cur * hbytes, a_lbo, 16u * kTcHX);
      const unsigned long long kstep = 2ull * (unsigned long long)chunk_entries;   // 16-byte units
      for (int p = 0; p < zt; ++p) {
        const unsigned long long ap = adesc0 + (unsigned long long)(p * kTcPlane);
#pragma unroll 3
        for (int tap = 0; tap < 27; ++tap) {
          const int dz = tap / 9, dy = (tap / 3) % 3, dx = tap % 3;
          const unsigned long long at = ap + (unsigned long long)((dz * kTcHY + dy) * kTcHX + dx);
#pragma unroll
          for (int ks = 0; ks < CIN / 16; ++ks)
            tc_mma(d0 + (unsigned)(p * COUT), at + ks * kstep,
                   bdesc0 + (unsigned long long)((tap * NCH + 2 * ks) * COUT), idesc, (tap | ks) != 0);
        }
      }
      asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(mb0 + 8 * cur)
                   : "memory");
    }
    issued = i + 1;
    __syncwarp();
    if (i > 0) {   // tile i - 1: its MMAs done frees its halo buffer and accumulator
      ok = __all_sync(0xffffffffu, mbar_wait(mb0 + 8 * (cur ^ 1), ((i - 1) >> 1) & 1, kTcWaitCycles));
      asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    }
    if (ok && i + 1 < nmine)
      tc_load_halo<CIN, UP>(in, s1, g, tc_tile(blockIdx.x + (i + 1) * gridDim.x, g, zt), zt,
                            hb0 + (cur ^ 1) * hbytes, chunk_entries);
    asm volatile("cp.async.commit_group;\n" ::: "memory");
    if (ok && i > 0)
      tc_epilogue<CIN, COUT, MASK>(tmem + (unsigned)((cur ^ 1) * zt * COUT), g, tc_tile(blockIdx.x + (i - 1) * gridDim.x, g, zt),
                             zt, bias, relu, mask, out_bf, out_f, f_ch0);
  }
  if (ok && nmine > 0) {
    const int l = nmine - 1;
    ok = __all_sync(0xffffffffu, mbar_wait(mb0 + 8 * (l & 1), (l >> 1) & 1, kTcWaitCycles));
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    if (ok)
      tc_epilogue<CIN, COUT, MASK>(tmem + (unsigned)((l & 1) * zt * COUT), g, tc_tile(blockIdx.x + l * gridDim.x, g, zt), zt,
                             bias, relu, mask, out_bf, out_f, f_ch0);
  }
  asm volatile("cp.async.wait_group 0;\n" ::: "memory");
  if (!ok && tid == 0) {
    atomicExch(fault, 1);
    // let the last committed MMAs drain before the columns are freed
    if (issued > 0) mbar_wait(mb0 + 8 * ((issued - 1) & 1), ((issued - 1) >> 1) & 1, kTcWaitCycles);
  }
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  __syncthreads();
  if (warp == 0) {
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    const unsigned base = *tslot;
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(base), "r"(ncols) : "memory");
  }
}

// ---- weight gradients -------------------------------------------------------------------
// gw[tap][ci][co] += sum_m in[nb(m, tap)][ci] dout[m][co] and gb[co] += sum_m dout[m][co].
// A contraction over the voxels: a block stages tiles of 16 (x) x 8 (y) x tz voxels of
// dout and of the input with its one-voxel halo once in shared memory (16-byte entries
// [8-channel chunk][voxel], conflict-free for ldmatrix), and its nine warps take the
// (dz, dy) pairs of the 27 taps: per 16 voxels a warp loads one dout fragment and three
// shifted input fragments (ldmatrix.trans turns [voxel][channel] into the transposed
// operand) and issues the MMAs into FP32 registers, which it keeps over all tiles of the
// block.  The blocks' sums go to a workspace and are added in a fixed order, so repeated
// runs agree bit for bit.  16 -> 16 layer on 16x64x64: 85 us (one warp per tap and 1024
// voxels, gathering 2-byte elements and adding with atomics) + 9 us for the bias before,
// 8.4 us + 4.3 us for the sums now; 48 -> 16: 92 + 9 before, 16 + 6 now.
constexpr int kWgX = 16, kWgY = 8, kWgHX = kWgX + 2, kWgHY = kWgY + 2;
constexpr int kWgThreads = 288;

__device__ __forceinline__ void ldsm_x4_trans(unsigned (&r)[4], unsigned addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr)
               : "memory");
}

__host__ __device__ constexpr int wg_elems(int cin, int cout) { return 27 * cin * cout + cout; }

template <int CIN, int COUT>
__global__ void __launch_bounds__(kWgThreads) conv_wgrad_kernel(const bf16* in, const bf16* dout,
                                                                NNGrid g, int tz, float* __restrict__ part) {
  pdl_enter();
  constexpr int KC = CIN / 8, NC = COUT / 8;
  extern __shared__ __align__(128) unsigned char smem[];
  const int nv = (tz + 2) * kWgHY * kWgHX, nd = tz * kWgY * kWgX;
  const unsigned si = smem_u32(smem), sd = si + 16u * KC * nv;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int dz = warp / 3, dy = warp % 3;
  const int ntx = (g.W + kWgX - 1) / kWgX, nty = (g.H + kWgY - 1) / kWgY, ntz = (g.D + tz - 1) / tz;
  float acc[3][CIN / 16][NC][4];
#pragma unroll
  for (int t = 0; t < 3; ++t)
#pragma unroll
    for (int c = 0; c < CIN / 16; ++c)
#pragma unroll
      for (int j = 0; j < NC; ++j) acc[t][c][j][0] = acc[t][c][j][1] = acc[t][c][j][2] = acc[t][c][j][3] = 0.f;
  float bias = 0.f;
  // this lane's row of the four 8x8 matrices of a fragment: voxel and chunk
  const int lv = lane & 7, lm = lane >> 3;
  const int a_vox = lv + 8 * (lm >> 1), a_ch = lm & 1;   // input: chunk pairs first, then voxels
  const int b_vox = lv + 8 * (lm & 1), b_ch = lm >> 1;   // dout: voxel halves first, then chunks
  for (int tile = blockIdx.x; tile < ntx * nty * ntz; tile += gridDim.x) {
    const int x0 = (tile % ntx) * kWgX, y0 = ((tile / ntx) % nty) * kWgY, z0 = (tile / (ntx * nty)) * tz;
    __syncthreads();   // the previous tile's readers
    for (int q = tid; q < nv * KC; q += kWgThreads) {
      const int ch = q % KC, v = q / KC;
      const int xx = v % kWgHX, yy = (v / kWgHX) % kWgHY, zz = v / (kWgHX * kWgHY);
      const int gz = z0 + zz - 1;
      const int gx = (x0 + xx - 1 + g.W) % g.W, gy = (y0 + yy - 1 + g.H) % g.H;
      const bool ok = gz >= 0 && gz < g.D;
      tc_cp16(si + 16u * (ch * nv + v), in + ((size_t)((ok ? gz : 0) * g.H + gy) * g.W + gx) * CIN + 8 * ch, ok);
    }
    for (int q = tid; q < nd * NC; q += kWgThreads) {
      const int ch = q % NC, v = q / NC;
      const int x = x0 + v % kWgX, y = y0 + (v / kWgX) % kWgY, z = z0 + v / (kWgX * kWgY);
      const bool ok = x < g.W && y < g.H && z < g.D;   // voxels beyond the grid contribute nothing
      tc_cp16(sd + 16u * (ch * nd + v), dout + (ok ? ((size_t)(z * g.H + y) * g.W + x) * COUT + 8 * ch : 0), ok);
    }
    asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;\n" ::: "memory");
    __syncthreads();
    if (tid < 256) {   // bias: thread tid sums channel tid % COUT over every 256 / COUT-th voxel
      const bf16* d = reinterpret_cast<const bf16*>(smem + 16 * (size_t)KC * nv);
      const int c = tid % COUT;
      for (int v = tid / COUT; v < nd; v += 256 / COUT) bias += __bfloat162float(d[((c >> 3) * nd + v) * 8 + (c & 7)]);
    }
    for (int row = 0; row < tz * kWgY; ++row) {   // 16 voxels along x
      const int z = row / kWgY, y = row - z * kWgY;
      unsigned b[NC / 2][4];
#pragma unroll
      for (int j = 0; j < NC / 2; ++j) ldsm_x4_trans(b[j], sd + 16u * ((2 * j + b_ch) * nd + row * kWgX + b_vox));
      const unsigned base = (unsigned)(((z + dz) * kWgHY + y + dy) * kWgHX);
#pragma unroll
      for (int t = 0; t < 3; ++t)
#pragma unroll
        for (int c = 0; c < CIN / 16; ++c) {
          unsigned af[4];
          ldsm_x4_trans(af, si + 16u * ((2 * c + a_ch) * nv + base + t + a_vox));
#pragma unroll
          for (int j = 0; j < NC; ++j) {
            const unsigned bf[2] = {b[j >> 1][2 * (j & 1)], b[j >> 1][2 * (j & 1) + 1]};
            mma_bf16(acc[t][c][j], af, bf);
          }
        }
    }
  }
  float* out = part + (size_t)blockIdx.x * wg_elems(CIN, COUT);
  const int gq = lane >> 2, tq = lane & 3;
#pragma unroll
  for (int t = 0; t < 3; ++t)
#pragma unroll
    for (int c = 0; c < CIN / 16; ++c)
#pragma unroll
      for (int j = 0; j < NC; ++j) {
        float* o = out + (size_t)((warp * 3 + t) * CIN + c * 16 + gq) * COUT + j * 8 + 2 * tq;
        *reinterpret_cast<float2*>(o) = make_float2(acc[t][c][j][0], acc[t][c][j][1]);
        *reinterpret_cast<float2*>(o + 8 * COUT) = make_float2(acc[t][c][j][2], acc[t][c][j][3]);
      }
  __syncthreads();
  float* red = reinterpret_cast<float*>(smem);
  if (tid < 256) red[tid] = bias;
  __syncthreads();
  if (tid < COUT) {
    float s = 0.f;
    for (int q = tid; q < 256; q += COUT) s += red[q];
    out[27 * CIN * COUT + tid] = s;
  }
}

// gw, gb += the blocks' sums: 32 elements by 8 partial rows per block, a fixed order
__global__ void __launch_bounds__(256) wgrad_reduce_kernel(const float* part, int nblk, int nw, int nb,
                                                           float* __restrict__ gw, float* __restrict__ gb) {
  pdl_enter();
  __shared__ float sh[8][32];
  const int n = nw + nb, t = blockIdx.x * 32 + threadIdx.x;
  float s = 0.f;
  if (t < n)
    for (int q = threadIdx.y; q < nblk; q += 64) {
      float v[8];
#pragma unroll
      for (int w = 0; w < 8; ++w) v[w] = q + 8 * w < nblk ? __ldcg(part + (size_t)(q + 8 * w) * n + t) : 0.f;
#pragma unroll
      for (int w = 0; w < 8; ++w) s += v[w];
    }
  sh[threadIdx.y][threadIdx.x] = s;
  __syncthreads();
  if (threadIdx.y == 0 && t < n) {
#pragma unroll
    for (int q = 1; q < 8; ++q) s += sh[q][threadIdx.x];
    if (t < nw) gw[t] += s;
    else gb[t - nw] += s;
  }
}

// 2x2x2 mean of a fine channels-last field: one thread per coarse voxel and
// 8-channel chunk (16 bytes)
__global__ void pool2_kernel(const bf16* in, NNGrid f, int C, bf16* __restrict__ out) {
  pdl_enter();
  const int Dc = f.D / 2, Hc = f.H / 2, Wc = f.W / 2, nch = C / 8;
  const long long n = (long long)Dc * Hc * Wc * nch;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n; t += (long long)gridDim.x * blockDim.x) {
    const int k = (int)(t % nch);
    const long long v = t / nch;
    const int X = (int)(v % Wc), Y = (int)((v / Wc) % Hc), Z = (int)(v / ((long long)Wc * Hc));
    float s[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    for (int q = 0; q < 8; ++q) {
      const int z = 2 * Z + (q >> 2), y = 2 * Y + ((q >> 1) & 1), x = 2 * X + (q & 1);
      const uint4 u = *reinterpret_cast<const uint4*>(in + ((size_t)(z * f.H + y) * f.W + x) * C + 8 * k);
      const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&u);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float2 p = __bfloat1622float2(h[i]);
        s[2 * i] += p.x;
        s[2 * i + 1] += p.y;
      }
    }
    uint4 o;
    __nv_bfloat162* oh = reinterpret_cast<__nv_bfloat162*>(&o);
#pragma unroll
    for (int i = 0; i < 4; ++i) oh[i] = __floats2bfloat162_rn(0.125f * s[2 * i], 0.125f * s[2 * i + 1]);
    *reinterpret_cast<uint4*>(out + (size_t)v * C + 8 * k) = o;
  }
}

// cat[v] = [a4(parent of v) (32 channels), s1(v) (16 channels)]: one thread per
// voxel and 8-channel chunk (16 bytes)
__global__ void upcat_kernel(const bf16* a4, const bf16* s1, NNGrid f,
                             bf16* __restrict__ cat) {
  pdl_enter();
  const long long n = (long long)f.D * f.H * f.W * 6;
  const int Hc = f.H / 2, Wc = f.W / 2;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n; t += (long long)gridDim.x * blockDim.x) {
    const int k = (int)(t % 6);
    const long long v = t / 6;
    const int x = (int)(v % f.W), y = (int)((v / f.W) % f.H), z = (int)(v / ((long long)f.W * f.H));
    const uint4 u = k < 4 ? *reinterpret_cast<const uint4*>(a4 + ((size_t)((z / 2) * Hc + y / 2) * Wc + x / 2) * 32 + 8 * k)
                          : *reinterpret_cast<const uint4*>(s1 + (size_t)v * 16 + 8 * (k - 4));
    *reinterpret_cast<uint4*>(cat + (size_t)v * 48 + 8 * k) = u;
  }
}

// da4m[V][c] = bf16(sum over the 8 children of dcat[child][c] (c < 32), masked by a4 > 0)
__global__ void up_grad_kernel(const float* dcat, const bf16* a4, NNGrid f,
                               bf16* __restrict__ out) {
  pdl_enter();
  const int Dc = f.D / 2, Hc = f.H / 2, Wc = f.W / 2;
  const long long n = (long long)Dc * Hc * Wc * 32;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n; t += (long long)gridDim.x * blockDim.x) {
    const int c = (int)(t % 32);
    const long long v = t / 32;
    const int X = (int)(v % Wc), Y = (int)((v / Wc) % Hc), Z = (int)(v / ((long long)Wc * Hc));
    float s = 0.f;
    for (int q = 0; q < 8; ++q) {
      const int z = 2 * Z + (q >> 2), y = 2 * Y + ((q >> 1) & 1), x = 2 * X + (q & 1);
      s += dcat[((size_t)(z * f.H + y) * f.W + x) * 48 + c];
    }
    out[t] = __float2bfloat16(__bfloat162float(a4[t]) > 0.f ? s : 0.f);
  }
}

// ds1m[v][c] = bf16((dcat[v][32 + c] + dp[parent(v)][c] / 8) masked by s1 > 0)
__global__ void skip_grad_kernel(const float* dcat, const float* dp,
                                 const bf16* s1, NNGrid f, bf16* __restrict__ out) {
  pdl_enter();
  const long long n = (long long)f.D * f.H * f.W * 16;
  const int Hc = f.H / 2, Wc = f.W / 2;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n; t += (long long)gridDim.x * blockDim.x) {
    const int c = (int)(t % 16);
    const long long v = t / 16;
    const int x = (int)(v % f.W), y = (int)((v / f.W) % f.H), z = (int)(v / ((long long)f.W * f.H));
    const float g = dcat[(size_t)v * 48 + 32 + c] +
                    0.125f * dp[((size_t)((z / 2) * Hc + y / 2) * Wc + x / 2) * 16 + c];
    out[t] = __float2bfloat16(__bfloat162float(s1[t]) > 0.f ? g : 0.f);
  }
}

// loss += sum (y0 - t)^2 / M; dy[m][0] = 2 (y0 - t) / M, other channels 0
__global__ void __launch_bounds__(256) mse_kernel(const float* y, const float* tgt, int M,
                                                  bf16* __restrict__ dy, float* __restrict__ loss) {
  pdl_enter();
  __shared__ float sh[8];
  float s = 0.f;
  for (int m = blockIdx.x * blockDim.x + threadIdx.x; m < M; m += gridDim.x * blockDim.x) {
    const float d = y[m] - tgt[m];
    s += d * d;
    uint4* o = reinterpret_cast<uint4*>(dy + (size_t)m * 16);
    o[0] = make_uint4(__bfloat16_as_ushort(__float2bfloat16(2.f * d / M)), 0u, 0u, 0u);
    o[1] = make_uint4(0u, 0u, 0u, 0u);
  }
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < 8; ++w) s += sh[w];
    atomicAdd(loss, s / M);
  }
}

// the six layers' places in the parameter arrays: layer l's weights start at w0[l] (its
// packed copies too), its biases at b0[l] behind all weights
struct NNLayout {
  int w0[7], b0[7], cin[6], cout[6];
};

// kernel layouts of a weight, FP32 master [tap][ci][co]: forward wk[tap][co][ci];
// adjoint wb[tap][ci][co] = w[26 - tap][ci][co] read as a conv with Cin' = co, Cout' = ci;
// the same two in the tensor-memory kernel's operand layout [tap][cin/8][cout][cin%8]:
// wkt for the forward, wbt (Cin' = co, Cout' = ci) for the adjoint
__device__ __forceinline__ void pack_weight(int t, int cin, int cout, float w, bf16* __restrict__ wk, bf16* __restrict__ wb,
                                            bf16* __restrict__ wkt, bf16* __restrict__ wbt) {
  const int co = t % cout, ci = (t / cout) % cin, tap = t / (cin * cout);
  const bf16 val = __float2bfloat16(w);
  wk[((size_t)tap * cout + co) * cin + ci] = val;
  wb[((size_t)(26 - tap) * cin + ci) * cout + co] = val;
  wkt[(((size_t)tap * (cin / 8) + ci / 8) * cout + co) * 8 + ci % 8] = val;
  wbt[(((size_t)(26 - tap) * (cout / 8) + co / 8) * cin + ci) * 8 + co % 8] = val;
}

// Adam on every parameter (update; a step size that rounds to zero still moves the moments and
// clears the gradients) and the packed copies of the weights, all layers in one launch
__global__ void __launch_bounds__(256) adam_pack_kernel(NNLayout L, float* __restrict__ p, float* __restrict__ g,
                                                        float* __restrict__ m, float* __restrict__ v, int update, float lr,
                                                        float b1, float b2, float c1, float c2, float eps,
                                                        bf16* __restrict__ wk,
                                                        bf16* __restrict__ wb, bf16* __restrict__ wkt,
                                                        bf16* __restrict__ wbt) {
  pdl_enter();
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= L.b0[6]) return;
  float x = p[t];
  if (update) {
    const float gr = g[t];
    const float mt = b1 * m[t] + (1.f - b1) * gr;
    const float vt = b2 * v[t] + (1.f - b2) * gr * gr;
    m[t] = mt;
    v[t] = vt;
    x -= lr * (mt / c1) / (sqrtf(vt / c2) + eps);
    p[t] = x;
    g[t] = 0.f;
  }
  if (t >= L.w0[6]) return;
  int l = 0;
  while (t >= L.w0[l + 1]) ++l;
  const int o = L.w0[l];
  pack_weight(t - o, L.cin[l], L.cout[l], x, wk + o, wb + o, wkt + o, wbt + o);
}

int grid1(long long n, int threads) {
  long long b = (n + threads - 1) / threads;
  if (b > 152LL * 8) b = 152LL * 8;
  return (int)(b < 1 ? 1 : b);
}

// dynamic shared memory of a tensor-memory CTA (barriers, weights, two halo
// buffers), padded so that the CTAs of one launch that fit on one SM never ask for more
// than its 512 tensor-memory columns together.  The launches of other layers that share
// the SM are not counted: conv_tc_kernel lets the next one start only when all its own
// blocks hold their columns.
size_t tc_smem(int cin, int cout, int zt) {
  const size_t b = 128 + (size_t)27 * cin * cout * 2 + 2 * (size_t)(cin / 8) * kTcPlane * (zt + 2) * 16;
  const int per_sm = 512 / tc_cols(2 * zt * cout);
  const size_t floor_b = 233472 / (per_sm + 1) - 1024 + 16;
  return std::max(b, floor_b);
}

int tc_tiles(NNGrid g, int zt) { return (g.W / kTcX) * (g.H / kTcY) * (g.D / zt); }

int sm_count() {
  static int n = 0;
  if (!n) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    if (n < 1) n = 1;
  }
  return n;
}

// z-planes per tile: the most of {4, 2} that divides D, fits the shared memory
// and still gives every SM a tile, else 1
int tc_zt(int cin, int cout, NNGrid g) {
  for (int zt : {4, 2})
    if (g.D % zt == 0 && tc_smem(cin, cout, zt) <= 232448 && tc_tiles(g, zt) >= sm_count()) return zt;
  return 1;
}

template <int CIN, int COUT, bool UP = false>
void launch_conv_tc(const bf16* in, const bf16* s1, const bf16* wt, const float* bias, NNGrid g, int relu,
                    const bf16* mask, bf16* out_bf, float* out_f, int f_ch0, int* fault, cudaStream_t s) {
  const int zt = tc_zt(CIN, COUT, g);
  const size_t smem = tc_smem(CIN, COUT, zt);
  const int per_sm = std::max(1, std::min(16, (int)(233472 / (smem + 1024))));
  const int blocks = std::min(tc_tiles(g, zt), sm_count() * per_sm);
  auto k = mask ? conv_tc_kernel<CIN, COUT, false, true> : conv_tc_kernel<CIN, COUT, UP, false>;
  launch_k(k, dim3(blocks), dim3(kTcThreads), smem, s, in, s1, wt, bias, g, zt, relu, mask, out_bf, out_f, f_ch0, fault);
}

}  // namespace

// Shared-memory limits of the tensor-memory kernels, set once per process when
// a network is created, so that no launch (possibly inside a stream capture)
// has to configure its function first.
cudaError_t nn_tc_setup() {
  static cudaError_t done = [] {
    const int lim = 232448;
    const cudaFuncAttribute a = cudaFuncAttributeMaxDynamicSharedMemorySize;
    cudaError_t e = cudaSuccess;
    auto set = [&](const void* f) {
      const cudaError_t r = cudaFuncSetAttribute(f, a, lim);
      if (e == cudaSuccess) e = r;
    };
    set((const void*)conv_tc_kernel<16, 16, false, false>);
    set((const void*)conv_tc_kernel<16, 16, false, true>);
    set((const void*)conv_tc_kernel<16, 32, false, false>);
    set((const void*)conv_tc_kernel<16, 32, false, true>);
    set((const void*)conv_tc_kernel<16, 48, false, false>);
    set((const void*)conv_tc_kernel<16, 48, false, true>);
    set((const void*)conv_tc_kernel<32, 16, false, false>);
    set((const void*)conv_tc_kernel<32, 16, false, true>);
    set((const void*)conv_tc_kernel<32, 32, false, false>);
    set((const void*)conv_tc_kernel<32, 32, false, true>);
    set((const void*)conv_tc_kernel<48, 16, false, false>);
    set((const void*)conv_tc_kernel<48, 16, false, true>);
    set((const void*)conv_tc_kernel<48, 16, true, false>);
    set((const void*)conv_wgrad_kernel<16, 16>);
    set((const void*)conv_wgrad_kernel<16, 32>);
    set((const void*)conv_wgrad_kernel<32, 32>);
    set((const void*)conv_wgrad_kernel<48, 16>);
    return e;
  }();
  return done;
}

// The tensor-memory kernel takes grids whose x extent is a multiple of 8 and y
// extent a multiple of 16; other grids use the mma.sync kernel.
bool nn_conv_uses_tc(int cin, int cout, NNGrid g) {
  if (g.W % kTcX || g.H % kTcY || g.D < 1) return false;
  return (cin == 16 && (cout == 16 || cout == 32 || cout == 48)) || (cin == 32 && (cout == 16 || cout == 32)) ||
         (cin == 48 && cout == 16);
}

bool nn_conv_fwd(const bf16* in, int cin, const bf16* wk, const bf16* wt, const float* bias, int cout,
                 NNGrid g, int relu, const bf16* mask, bf16* out_bf, float* out_f, int f_ch0, int* fault, cudaStream_t s) {
  if (wt && fault && nn_conv_uses_tc(cin, cout, g)) {
    auto go = [&](auto launch) { launch(in, nullptr, wt, bias, g, relu, mask, out_bf, out_f, f_ch0, fault, s); };
    if (cin == 16 && cout == 16) go(launch_conv_tc<16, 16>);
    else if (cin == 16 && cout == 32) go(launch_conv_tc<16, 32>);
    else if (cin == 16 && cout == 48) go(launch_conv_tc<16, 48>);
    else if (cin == 32 && cout == 16) go(launch_conv_tc<32, 16>);
    else if (cin == 32 && cout == 32) go(launch_conv_tc<32, 32>);
    else go(launch_conv_tc<48, 16>);
    return true;
  }
  const int M = g.D * g.H * g.W;
  const int tiles = (M + 15) / 16;
  const int blocks = (tiles + kConvTiles - 1) / kConvTiles;
  const dim3 block(32, kConvTiles, 3);
  // two kernels each: the mask's branch cost the forward 9% (22x20x32: 74.8 -> 81.9 us)
  auto go = [&](auto k) { launch_k(k, dim3(blocks), block, 0, s, in, cin, wk, bias, g, relu, mask, out_bf, out_f, f_ch0); };
  if (cout == 16) go(mask ? conv_fwd_kernel<16, true> : conv_fwd_kernel<16, false>);
  else if (cout == 32) go(mask ? conv_fwd_kernel<32, true> : conv_fwd_kernel<32, false>);
  else if (cout == 48) go(mask ? conv_fwd_kernel<48, true> : conv_fwd_kernel<48, false>);
  return false;
}

// conv(48 -> 16) of [up(a4), s1] on the tensor-memory kernel without forming the
// concatenation; false (nothing launched) where the grid does not allow it
bool nn_conv_upcat_tc(const bf16* a4, const bf16* s1, const bf16* wt, const float* bias, NNGrid g, int relu,
                      bf16* out_bf, int* fault, cudaStream_t s) {
  if (!wt || !fault || !nn_conv_uses_tc(48, 16, g)) return false;
  launch_conv_tc<48, 16, true>(a4, s1, wt, bias, g, relu, nullptr, out_bf, nullptr, 0, fault, s);
  return true;
}

// Planes per tile of the weight gradient: the most of {4, 2} that leaves five of six SMs a
// tile (128 of 152).  A whole training step, us, with a tile asked for 128 or for all 152 SMs:
// 8x64x64 (two planes 128 tiles) 242 / 248, 16x48x48 (144) 256 / 260, 14x66x62 (four planes
// 144) 383 / 390, 16x72x64 (144) 424 / 432, 16x64x64 (128) 284 / 284; for 64 SMs 8x64x64
// takes 248 and 16x48x48 267: fewer, deeper tiles load less halo until SMs idle.
int wg_tz(NNGrid g) {
  const long long t = (long long)((g.W + kWgX - 1) / kWgX) * ((g.H + kWgY - 1) / kWgY);
  for (int tz : {4, 2})
    if (t * ((g.D + tz - 1) / tz) >= 128) return tz;
  return 1;
}

int wg_blocks(NNGrid g, int tz) {
  const long long t = (long long)((g.W + kWgX - 1) / kWgX) * ((g.H + kWgY - 1) / kWgY) * ((g.D + tz - 1) / tz);
  return (int)std::min<long long>(t, sm_count());
}

// floats of the weight gradients' workspace: one block's sums of the largest layer per SM
size_t nn_wgrad_workspace() { return (size_t)sm_count() * wg_elems(32, 32); }

// gw and gb of one layer; part: the workspace (one layer at a time)
void nn_conv_wgrad(const bf16* in, int cin, const bf16* dout, int cout, NNGrid g, float* gw,
                   float* gb, float* part, cudaStream_t s) {
  const int tz = wg_tz(g), blocks = wg_blocks(g, tz);
  const size_t smem = 16 * ((size_t)(cin / 8) * (tz + 2) * kWgHY * kWgHX + (size_t)(cout / 8) * tz * kWgY * kWgX);
  if (cin == 16 && cout == 16) launch_k(conv_wgrad_kernel<16, 16>, dim3(blocks), dim3(kWgThreads), smem, s, in, dout, g, tz, part);
  else if (cin == 16 && cout == 32) launch_k(conv_wgrad_kernel<16, 32>, dim3(blocks), dim3(kWgThreads), smem, s, in, dout, g, tz, part);
  else if (cin == 32 && cout == 32) launch_k(conv_wgrad_kernel<32, 32>, dim3(blocks), dim3(kWgThreads), smem, s, in, dout, g, tz, part);
  else if (cin == 48 && cout == 16) launch_k(conv_wgrad_kernel<48, 16>, dim3(blocks), dim3(kWgThreads), smem, s, in, dout, g, tz, part);
  const int nw = 27 * cin * cout;
  launch_k(wgrad_reduce_kernel, dim3((nw + cout + 31) / 32), dim3(32, 8), 0, s, part, blocks, nw, cout, gw, gb);
}

void nn_pool2(const bf16* in, NNGrid f, int C, bf16* out, cudaStream_t s) {
  launch_k(pool2_kernel, dim3(grid1((long long)f.D * f.H * f.W * C / 64, 256)), dim3(256), 0, s, in, f, C, out);
}
void nn_upcat(const bf16* a4, const bf16* s1, NNGrid f, bf16* cat, cudaStream_t s) {
  launch_k(upcat_kernel, dim3(grid1((long long)f.D * f.H * f.W * 6, 256)), dim3(256), 0, s, a4, s1, f, cat);
}
void nn_up_grad(const float* dcat, const bf16* a4, NNGrid f, bf16* out, cudaStream_t s) {
  launch_k(up_grad_kernel, dim3(grid1((long long)f.D * f.H * f.W * 4, 256)), dim3(256), 0, s, dcat, a4, f, out);
}
void nn_skip_grad(const float* dcat, const float* dp, const bf16* s1, NNGrid f, bf16* out, cudaStream_t s) {
  launch_k(skip_grad_kernel, dim3(grid1((long long)f.D * f.H * f.W * 16, 256)), dim3(256), 0, s, dcat, dp, s1, f, out);
}
void nn_mse(const float* y, const float* tgt, int M, bf16* dy, float* loss, cudaStream_t s) {
  launch_k(mse_kernel, dim3(grid1(M, 256)), dim3(256), 0, s, y, tgt, M, dy, loss);
}
void nn_adam_pack(const NNLayout& L, float* p, float* g, float* m, float* v, bool update, float lr, int step, bf16* wk,
                  bf16* wb, bf16* wkt, bf16* wbt, cudaStream_t s) {
  const float b1 = 0.9f, b2 = 0.999f;
  const float c1 = 1.f - powf(b1, (float)step), c2 = 1.f - powf(b2, (float)step);
  launch_k(adam_pack_kernel, dim3((L.b0[6] + 255) / 256), dim3(256), 0, s, L, p, g, m, v, update ? 1 : 0, lr, b1, b2, c1, c2, 1e-8f,
           wk, wb, wkt, wbt);
}

}  // namespace fx

// ======================================================================================
// Host side: the network object (weights, Adam state, activations for one grid,
// snapshot store) and its C ABI.
// ======================================================================================

namespace fx {
namespace {

constexpr int kLayers = 6;
constexpr int kCin[kLayers] = {16, 16, 16, 32, 48, 16};
constexpr int kCout[kLayers] = {16, 16, 32, 32, 16, 16};

__global__ void __launch_bounds__(256) f32_to_bf16_kernel(const float* in, long long n, int vec,
                                                          bf16* __restrict__ out) {
  pdl_enter();
  if (vec) {   // eight values by 16-byte accesses
    const long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (8 * t >= n) return;
    const float4 *p = reinterpret_cast<const float4*>(in) + 2 * t, a = p[0], b = p[1];
    uint4 q;
    __nv_bfloat162* h = reinterpret_cast<__nv_bfloat162*>(&q);
    h[0] = __floats2bfloat162_rn(a.x, a.y);
    h[1] = __floats2bfloat162_rn(a.z, a.w);
    h[2] = __floats2bfloat162_rn(b.x, b.y);
    h[3] = __floats2bfloat162_rn(b.z, b.w);
    reinterpret_cast<uint4*>(out)[t] = q;
    return;
  }
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n; t += (long long)gridDim.x * blockDim.x)
    out[t] = __float2bfloat16(in[t]);
}

void nn_to_bf16(const float* in, long long n, bf16* out, cudaStream_t s) {
  const int vec = n % 8 == 0 && reinterpret_cast<uintptr_t>(in) % 16 == 0;   // out is the network's own
  launch_k(f32_to_bf16_kernel, dim3(vec ? (unsigned)((n / 8 + 255) / 256) : (unsigned)grid1(n, 256)), dim3(256), 0, s, in, n,
           vec, out);
}

}  // namespace
}  // namespace fx

using fx::bf16;

struct ferrox_nn {
  fx::NNGrid g{}, gc{};
  int M = 0, Mc = 0;
  cudaStream_t stream = nullptr;
  // every layer's weights, then every layer's biases, in one array each for the values,
  // gradients and moments (one Adam launch, one copy per array); packed weights likewise
  fx::NNLayout lay{};
  float *par = nullptr, *grad = nullptr, *mom1 = nullptr, *mom2 = nullptr;
  bf16 *wk0 = nullptr, *wb0 = nullptr, *wkt0 = nullptr, *wbt0 = nullptr;
  // the layers' places in them
  float* w[fx::kLayers] = {};
  float* b[fx::kLayers] = {};
  float* gw[fx::kLayers] = {};
  float* gb[fx::kLayers] = {};
  bf16* wk[fx::kLayers] = {};
  bf16* wb[fx::kLayers] = {};
  bf16* wkt[fx::kLayers] = {};   // tensor-memory operand layouts of wk and wb
  bf16* wbt[fx::kLayers] = {};
  float* part = nullptr;         // weight gradients' workspace
  int* fault = nullptr;          // set by a tensor-memory convolution whose wait ran out
  bool tc = true;                // tensor-memory convolutions where the grid allows
  bf16 *x = nullptr, *a1 = nullptr, *s1 = nullptr, *p = nullptr, *a3 = nullptr, *a4 = nullptr,
       *cat = nullptr, *a5 = nullptr, *dy = nullptr, *t16a = nullptr, *t16b = nullptr,
       *t32a = nullptr, *t32b = nullptr;
  float *y = nullptr, *dcat = nullptr, *dpc = nullptr, *loss = nullptr;
  int cap = 0, count = 0, next = 0;
  bf16* snap_x = nullptr;     // [cap][M][16]
  float* snap_t = nullptr;    // [cap][M]
  int adam_step = 0;
  std::vector<void*> allocs;
  std::string err;
};

namespace {

std::string g_nn_error;

ferrox_status nfail(ferrox_nn* n, ferrox_status s, const std::string& m) {
  if (n) n->err = m; else g_nn_error = m;
  return s;
}

#define FX_NCK(call)                                                                          \
  do {                                                                                        \
    cudaError_t _e = (call);                                                                  \
    if (_e != cudaSuccess)                                                                    \
      return nfail(N, _e == cudaErrorMemoryAllocation ? FERROX_ENOMEM : FERROX_ECUDA,         \
                   std::string(#call) + ": " + cudaGetErrorString(_e));                       \
  } while (0)

template <typename P>
cudaError_t nalloc(ferrox_nn* N, P** ptr, size_t bytes) {
  void* v = nullptr;
  cudaError_t e = cudaMalloc(&v, bytes);
  if (e == cudaSuccess) {
    N->allocs.push_back(v);
    cudaMemset(v, 0, bytes);
  }
  *ptr = static_cast<P*>(v);
  return e;
}

// one Adam update with step size lr (update) and the packed copies of the weights
void adam_pack(ferrox_nn* N, bool update, float lr = 0.f) {
  fx::nn_adam_pack(N->lay, N->par, N->grad, N->mom1, N->mom2, update, lr, std::max(1, N->adam_step), N->wk0, N->wb0,
                   N->wkt0, N->wbt0, N->stream);
}

// one convolution of layer l: forward weights, or the adjoint's when adjoint is set
void conv(ferrox_nn* N, int l, bool adjoint, const bf16* in, fx::NNGrid g, int relu, bf16* out_bf, float* out_f,
          cudaStream_t s, int f_ch0 = 0, const bf16* mask = nullptr) {
  const int cin = adjoint ? fx::kCout[l] : fx::kCin[l], cout = adjoint ? fx::kCin[l] : fx::kCout[l];
  fx::nn_conv_fwd(in, cin, adjoint ? N->wb[l] : N->wk[l], !N->tc ? nullptr : adjoint ? N->wbt[l] : N->wkt[l],
                  adjoint ? nullptr : N->b[l], cout, g, relu, mask, out_bf, out_f, f_ch0, N->fault, s);
}

// forward pass from N->x; output channel 0 (FP32) in y (null: N->y).  The concatenation
// [up(a4), s1] is formed in memory only for a backward pass (keep_cat) or where
// the tensor-memory kernel cannot read it in place.
void forward(ferrox_nn* N, bool keep_cat, float* y = nullptr) {
  cudaStream_t s = N->stream;
  using namespace fx;
  conv(N, 0, false, N->x, N->g, 1, N->a1, nullptr, s);
  conv(N, 1, false, N->a1, N->g, 1, N->s1, nullptr, s);
  nn_pool2(N->s1, N->g, 16, N->p, s);
  conv(N, 2, false, N->p, N->gc, 1, N->a3, nullptr, s);
  conv(N, 3, false, N->a3, N->gc, 1, N->a4, nullptr, s);
  if (keep_cat || !N->tc ||
      !nn_conv_upcat_tc(N->a4, N->s1, N->wkt[4], N->b[4], N->g, 1, N->a5, N->fault, s)) {
    nn_upcat(N->a4, N->s1, N->g, N->cat, s);
    conv(N, 4, false, N->cat, N->g, 1, N->a5, nullptr, s);
  }
  conv(N, 5, false, N->a5, N->g, 0, nullptr, y ? y : N->y, s, 1);   // output channel 0 only
}

// backward pass from N->dy (gradient of the loss w.r.t. the output); accumulates gw, gb
void backward(ferrox_nn* N) {
  cudaStream_t s = N->stream;
  using namespace fx;
  auto wgrad = [&](int l, const bf16* in, const bf16* dout, NNGrid g) {
    nn_conv_wgrad(in, kCin[l], dout, kCout[l], g, N->gw[l], N->gb[l], N->part, s);
  };
  // the adjoints whose result passes a ReLU only are masked and rounded as they are stored
  wgrad(5, N->a5, N->dy, N->g);
  conv(N, 5, true, N->dy, N->g, 0, N->t16a, nullptr, s, 0, N->a5);            // da5
  wgrad(4, N->cat, N->t16a, N->g);
  conv(N, 4, true, N->t16a, N->g, 0, nullptr, N->dcat, s);
  nn_up_grad(N->dcat, N->a4, N->g, N->t32a, s);                               // da4
  wgrad(3, N->a3, N->t32a, N->gc);
  conv(N, 3, true, N->t32a, N->gc, 0, N->t32b, nullptr, s, 0, N->a3);         // da3
  wgrad(2, N->p, N->t32b, N->gc);
  conv(N, 2, true, N->t32b, N->gc, 0, nullptr, N->dpc, s);                    // dp
  nn_skip_grad(N->dcat, N->dpc, N->s1, N->g, N->t16b, s);                     // ds1
  wgrad(1, N->a1, N->t16b, N->g);
  conv(N, 1, true, N->t16b, N->g, 0, N->t16a, nullptr, s, 0, N->a1);          // da1
  wgrad(0, N->x, N->t16a, N->g);
}

void nn_release(ferrox_nn* N) {
  if (!N) return;
  if (N->stream) cudaStreamSynchronize(N->stream);
  for (void* p : N->allocs) cudaFree(p);
  delete N;
}

}  // namespace

namespace fx {
// used by the context when it feeds the network (engine.cu)
bf16* nn_input(ferrox_nn* N) { return N->x; }
const float* nn_output(ferrox_nn* N) { return N->y; }
void nn_run_forward(ferrox_nn* N, cudaStream_t s) {
  cudaStream_t keep = N->stream;
  N->stream = s;
  forward(N, false);
  N->stream = keep;
}
NNGrid nn_grid(const ferrox_nn* N) { return N->g; }
int nn_capacity(const ferrox_nn* N) { return N->cap; }
bf16* nn_snap_x(ferrox_nn* N) { return N->snap_x; }
float* nn_snap_t(ferrox_nn* N) { return N->snap_t; }
int nn_next_slot(const ferrox_nn* N) { return N->next; }
void nn_note_snapshots(ferrox_nn* N, int added) {
  N->count = std::min(N->cap, N->count + added);
  N->next = (N->next + added) % std::max(1, N->cap);
}
}  // namespace fx

extern "C" {

ferrox_status ferrox_nn_create(ferrox_nn** out, int D, int H, int W, int capacity,
                               const float* weights, const float* biases, void* cuda_stream) {
  if (!out) return nfail(nullptr, FERROX_EINVAL, "null output pointer");
  *out = nullptr;
  if (D < 2 || H < 2 || W < 2 || D % 2 || H % 2 || W % 2)
    return nfail(nullptr, FERROX_EINVAL, "network grid sizes must be even and >= 2");
  if (capacity < 0 || !weights || !biases) return nfail(nullptr, FERROX_EINVAL, "bad argument");
  ferrox_nn* N = new ferrox_nn();
  N->g = fx::NNGrid{D, H, W};
  N->gc = fx::NNGrid{D / 2, H / 2, W / 2};
  N->M = D * H * W;
  N->Mc = N->M / 8;
  N->cap = capacity;
  N->stream = static_cast<cudaStream_t>(cuda_stream);
  if (const cudaError_t te = fx::nn_tc_setup(); te != cudaSuccess) {
    delete N;
    return nfail(nullptr, FERROX_ECUDA, std::string("cudaFuncSetAttribute: ") + cudaGetErrorString(te));
  }
  const size_t M = N->M, Mc = N->Mc;
  auto fail_alloc = [&](cudaError_t e) {
    const std::string m = std::string("cudaMalloc: ") + cudaGetErrorString(e);
    nn_release(N);
    return nfail(nullptr, FERROX_ENOMEM, m);
  };
  cudaError_t e;
  fx::NNLayout& L = N->lay;
  for (int l = 0; l < fx::kLayers; ++l) {
    L.cin[l] = fx::kCin[l];
    L.cout[l] = fx::kCout[l];
    L.w0[l + 1] = L.w0[l] + 27 * fx::kCin[l] * fx::kCout[l];
  }
  L.b0[0] = L.w0[fx::kLayers];
  for (int l = 0; l < fx::kLayers; ++l) L.b0[l + 1] = L.b0[l] + fx::kCout[l];
  const size_t nw = L.w0[fx::kLayers], np = L.b0[fx::kLayers];
  for (float** p : {&N->par, &N->grad, &N->mom1, &N->mom2})
    if ((e = nalloc(N, p, np * sizeof(float))) != cudaSuccess) return fail_alloc(e);
  for (bf16** p : {&N->wk0, &N->wb0, &N->wkt0, &N->wbt0})
    if ((e = nalloc(N, p, nw * sizeof(bf16))) != cudaSuccess) return fail_alloc(e);
  if ((e = nalloc(N, &N->part, fx::nn_wgrad_workspace() * sizeof(float))) != cudaSuccess) return fail_alloc(e);
  for (int l = 0; l < fx::kLayers; ++l) {
    N->w[l] = N->par + L.w0[l];
    N->b[l] = N->par + L.b0[l];
    N->gw[l] = N->grad + L.w0[l];
    N->gb[l] = N->grad + L.b0[l];
    N->wk[l] = N->wk0 + L.w0[l];
    N->wb[l] = N->wb0 + L.w0[l];
    N->wkt[l] = N->wkt0 + L.w0[l];
    N->wbt[l] = N->wbt0 + L.w0[l];
  }
  cudaMemcpy(N->par, weights, nw * sizeof(float), cudaMemcpyHostToDevice);
  cudaMemcpy(N->par + nw, biases, (np - nw) * sizeof(float), cudaMemcpyHostToDevice);
  struct { bf16** p; size_t n; } bufs[] = {
      {&N->x, M * 16}, {&N->a1, M * 16}, {&N->s1, M * 16}, {&N->p, Mc * 16}, {&N->a3, Mc * 32},
      {&N->a4, Mc * 32}, {&N->cat, M * 48}, {&N->a5, M * 16}, {&N->dy, M * 16},
      {&N->t16a, M * 16}, {&N->t16b, M * 16}, {&N->t32a, Mc * 32}, {&N->t32b, Mc * 32}};
  for (auto& bq : bufs)
    if ((e = nalloc(N, bq.p, bq.n * sizeof(bf16))) != cudaSuccess) return fail_alloc(e);
  struct { float** p; size_t n; } fbufs[] = {{&N->y, M}, {&N->dcat, M * 48}, {&N->dpc, Mc * 16}, {&N->loss, 4}};
  for (auto& bq : fbufs)
    if ((e = nalloc(N, bq.p, bq.n * sizeof(float))) != cudaSuccess) return fail_alloc(e);
  if ((e = nalloc(N, &N->fault, sizeof(int))) != cudaSuccess) return fail_alloc(e);
  if (capacity > 0) {
    if ((e = nalloc(N, &N->snap_x, (size_t)capacity * M * 16 * sizeof(bf16))) != cudaSuccess) return fail_alloc(e);
    if ((e = nalloc(N, &N->snap_t, (size_t)capacity * M * sizeof(float))) != cudaSuccess) return fail_alloc(e);
  }
  adam_pack(N, false);
  if ((e = cudaDeviceSynchronize()) != cudaSuccess) {
    nn_release(N);
    return nfail(nullptr, FERROX_ECUDA, cudaGetErrorString(e));
  }
  *out = N;
  return FERROX_OK;
}

ferrox_status ferrox_nn_forward(ferrox_nn* N, const float* x_dev, float* y_dev) {
  if (!N || !x_dev || !y_dev) return nfail(N, FERROX_EINVAL, "null argument");
  fx::nn_to_bf16(x_dev, (long long)N->M * 16, N->x, N->stream);
  forward(N, false, y_dev);
  FX_NCK(cudaGetLastError());
  return FERROX_OK;
}

// forward + MSE against t_dev + backward: gradients are accumulated (not applied)
ferrox_status ferrox_nn_loss_grad(ferrox_nn* N, const float* x_dev, const float* t_dev, float* loss_host) {
  if (!N || !x_dev || !t_dev) return nfail(N, FERROX_EINVAL, "null argument");
  fx::nn_to_bf16(x_dev, (long long)N->M * 16, N->x, N->stream);
  FX_NCK(cudaMemsetAsync(N->loss, 0, sizeof(float), N->stream));
  forward(N, true);
  fx::nn_mse(N->y, t_dev, N->M, N->dy, N->loss, N->stream);
  backward(N);
  FX_NCK(cudaGetLastError());
  if (loss_host) {
    FX_NCK(cudaMemcpyAsync(loss_host, N->loss, sizeof(float), cudaMemcpyDeviceToHost, N->stream));
    FX_NCK(cudaStreamSynchronize(N->stream));
  }
  return FERROX_OK;
}

ferrox_status ferrox_nn_params(ferrox_nn* N, float* w, float* b, float* gw, float* gb) {
  if (!N) return nfail(nullptr, FERROX_EINVAL, "null network");
  FX_NCK(cudaStreamSynchronize(N->stream));
  const size_t nw = N->lay.w0[fx::kLayers], nb = N->lay.b0[fx::kLayers] - nw;
  if (w) FX_NCK(cudaMemcpy(w, N->par, nw * sizeof(float), cudaMemcpyDeviceToHost));
  if (b) FX_NCK(cudaMemcpy(b, N->par + nw, nb * sizeof(float), cudaMemcpyDeviceToHost));
  if (gw) FX_NCK(cudaMemcpy(gw, N->grad, nw * sizeof(float), cudaMemcpyDeviceToHost));
  if (gb) FX_NCK(cudaMemcpy(gb, N->grad + nw, nb * sizeof(float), cudaMemcpyDeviceToHost));
  return FERROX_OK;
}

ferrox_status ferrox_nn_set_params(ferrox_nn* N, const float* w, const float* b) {
  if (!N || !w || !b) return nfail(N, FERROX_EINVAL, "null argument");
  const size_t nw = N->lay.w0[fx::kLayers], nb = N->lay.b0[fx::kLayers] - nw;
  FX_NCK(cudaMemcpyAsync(N->par, w, nw * sizeof(float), cudaMemcpyHostToDevice, N->stream));
  FX_NCK(cudaMemcpyAsync(N->par + nw, b, nb * sizeof(float), cudaMemcpyHostToDevice, N->stream));
  adam_pack(N, false);
  FX_NCK(cudaStreamSynchronize(N->stream));
  return FERROX_OK;
}

ferrox_status ferrox_nn_adam_step(ferrox_nn* N, double lr) {
  if (!N || !(lr > 0.0)) return nfail(N, FERROX_EINVAL, "bad argument");
  N->adam_step += 1;
  adam_pack(N, true, (float)lr);
  FX_NCK(cudaGetLastError());
  return FERROX_OK;
}

ferrox_status ferrox_nn_snapshot_count(const ferrox_nn* N, int* count) {
  if (!N || !count) return FERROX_EINVAL;
  *count = N->count;
  return FERROX_OK;
}

// epochs over the stored snapshots (in storage order), Adam every `batch`
// snapshots; loss_per_epoch[e] = mean snapshot loss of epoch e
ferrox_status ferrox_nn_train(ferrox_nn* N, int epochs, double lr, int batch, float* loss_per_epoch) {
  if (!N || epochs < 0 || batch < 1 || !(lr > 0.0)) return nfail(N, FERROX_EINVAL, "bad argument");
  if (N->count < 1) return nfail(N, FERROX_ESTATE, "no snapshots collected");
  const size_t M = N->M;
  // a fresh order of the snapshots every epoch (Fisher-Yates with a splitmix64
  // stream of fixed seed, so runs repeat), and a cosine decay of the step size
  // from lr to lr / 10 over all Adam steps of the call
  std::vector<int> order(N->count);
  for (int q = 0; q < N->count; ++q) order[q] = q;
  unsigned long long state = 0x2545F4914F6CDD1Dull;
  auto next = [&state]() {
    unsigned long long z = (state += 0x9E3779B97F4A7C15ull);
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
  };
  const long long per_epoch = (N->count + batch - 1) / batch, total = std::max(1LL, per_epoch * epochs);
  long long k = 0;
  for (int ep = 0; ep < epochs; ++ep) {
    for (int q = N->count - 1; q > 0; --q) std::swap(order[q], order[(int)(next() % (unsigned long long)(q + 1))]);
    FX_NCK(cudaMemsetAsync(N->loss, 0, sizeof(float), N->stream));
    for (int j = 0; j < N->count; ++j) {
      const int q = order[j];
      FX_NCK(cudaMemcpyAsync(N->x, N->snap_x + (size_t)q * M * 16, M * 16 * sizeof(bf16),
                             cudaMemcpyDeviceToDevice, N->stream));
      forward(N, true);
      fx::nn_mse(N->y, N->snap_t + (size_t)q * M, N->M, N->dy, N->loss, N->stream);
      backward(N);
      if ((j + 1) % batch == 0 || j + 1 == N->count) {
        const double lr_k = lr * (0.1 + 0.45 * (1.0 + std::cos(3.141592653589793 * (double)k / (double)total)));
        ++k;
        N->adam_step += 1;
        adam_pack(N, true, (float)lr_k);
      }
    }
    FX_NCK(cudaGetLastError());
    float l = 0.f;
    FX_NCK(cudaMemcpyAsync(&l, N->loss, sizeof(float), cudaMemcpyDeviceToHost, N->stream));
    FX_NCK(cudaStreamSynchronize(N->stream));
    if (loss_per_epoch) loss_per_epoch[ep] = l / N->count;
  }
  return FERROX_OK;
}

ferrox_status ferrox_nn_destroy(ferrox_nn* N) {
  nn_release(N);
  return FERROX_OK;
}

const char* ferrox_nn_last_error(const ferrox_nn* N) { return N ? N->err.c_str() : g_nn_error.c_str(); }

ferrox_status ferrox_nn_use_tensor_memory(ferrox_nn* N, int on) {
  if (!N || (on != 0 && on != 1)) return nfail(N, FERROX_EINVAL, "use_tensor_memory must be 0 or 1");
  N->tc = on != 0;
  return FERROX_OK;
}

ferrox_status ferrox_nn_kernel_info(ferrox_nn* N, int* tc_forward, int* tc_backward, int* fault) {
  if (!N) return nfail(nullptr, FERROX_EINVAL, "null network");
  int f = 0, b = 0;
  if (N->tc) {
    for (int l = 0; l < fx::kLayers; ++l) {
      const fx::NNGrid g = (l == 2 || l == 3) ? N->gc : N->g;
      f += fx::nn_conv_uses_tc(fx::kCin[l], fx::kCout[l], g);
      if (l > 0) b += fx::nn_conv_uses_tc(fx::kCout[l], fx::kCin[l], g);
    }
  }
  if (tc_forward) *tc_forward = f;
  if (tc_backward) *tc_backward = b;
  if (fault) {
    FX_NCK(cudaStreamSynchronize(N->stream));
    FX_NCK(cudaMemcpy(fault, N->fault, sizeof(int), cudaMemcpyDeviceToHost));
  }
  return FERROX_OK;
}

}  // extern "C"

// ======================================================================================
// Bridge between the multigrid arenas and the network (used by the context).
// ======================================================================================
namespace fx {
namespace {

// 2x2x2 (or semi-coarsened) mean of a level field into the next level
template <typename T>
__global__ void avg_down_kernel(T* __restrict__ a, LevelDesc F, LevelDesc C) {
  pdl_enter();
  const long long n = C.ncell;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n; t += (long long)gridDim.x * blockDim.x) {
    const int I = (int)(t % C.nx), J = (int)((t / C.nx) % C.ny), K = (int)(t / ((long long)C.nx * C.ny));
    const int nxc = F.crx ? 2 : 1, nyc = F.cry ? 2 : 1, nzc = F.crz ? 2 : 1;
    double s = 0.0;
    for (int dk = 0; dk < nzc; ++dk)
      for (int dj = 0; dj < nyc; ++dj)
        for (int di = 0; di < nxc; ++di) {
          const int i = F.crx ? 2 * I + di : I, j = F.cry ? 2 * J + dj : J, k = F.crz ? 2 * K + dk : K;
          s += (double)a[F.off + ((long long)k * F.ny + j) * F.nx + i];
        }
    a[C.off + t] = (T)(s / (nxc * nyc * nzc));
  }
}

// sum of squares of a level field in fixed order: one block
template <typename T>
__global__ void rms_kernel(const T* a, long long off, long long n, double* __restrict__ out) {
  pdl_enter();
  __shared__ double sh[32];
  double s = 0.0;
  for (long long t = threadIdx.x; t < n; t += blockDim.x) {
    const double v = (double)a[off + t];
    s = fma(v, v, s);
  }
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x < 32) {
    s = threadIdx.x < (blockDim.x >> 5) ? sh[threadIdx.x] : 0.0;
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (threadIdx.x == 0) *out = sqrt(s / (double)n) + 1e-300;
  }
}

// network input: residual / rms, per-plane material features, height, bias
template <typename T>
__global__ void features_kernel(const T* r, LevelDesc L, const float* __restrict__ pf,
                                const double* scale, const DevParams* prm,
                                bf16* __restrict__ x) {
  pdl_enter();
  const long long n = L.ncell;
  const float inv = (float)(1.0 / *scale);
  const float vapp = (float)(prm->v_top - prm->v_bot);
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n; t += (long long)gridDim.x * blockDim.x) {
    const int K = (int)(t / ((long long)L.nx * L.ny));
    float f[16] = {(float)r[L.off + t] * inv, pf[4 * K], pf[4 * K + 1], pf[4 * K + 2], pf[4 * K + 3],
                   0.5f * vapp, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    __nv_bfloat162* o = reinterpret_cast<__nv_bfloat162*>(x + t * 16);
#pragma unroll
    for (int c = 0; c < 8; ++c) o[c] = __floats2bfloat162_rn(f[2 * c], f[2 * c + 1]);
  }
}

// e (level) = scale * network output channel 0
template <typename T>
__global__ void apply_kernel(const float* y, LevelDesc L, const double* scale,
                             T* __restrict__ e) {
  pdl_enter();
  const double s = *scale;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < L.ncell; t += (long long)gridDim.x * blockDim.x)
    e[L.off + t] = (T)(s * (double)y[t]);
}

// e0 = phi - phi_guess (fine level), the error the initial guess had
template <typename T>
__global__ void guess_error_kernel(const double* phi, const double* guess,
                                   long long n, T* __restrict__ e0) {
  pdl_enter();
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n; t += (long long)gridDim.x * blockDim.x)
    e0[t] = (T)(phi[t] - guess[t]);
}

// training target = restricted error / rms of the restricted initial residual
template <typename T>
__global__ void target_kernel(const T* e, LevelDesc L, const double* scale,
                              float* __restrict__ tgt) {
  pdl_enter();
  const double inv = 1.0 / *scale;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < L.ncell; t += (long long)gridDim.x * blockDim.x)
    tgt[t] = (float)((double)e[L.off + t] * inv);
}

}  // namespace

template <typename T>
void nn_bridge_restrict(T* arena, const std::vector<LevelDesc>& lv, int to, cudaStream_t s) {
  for (int l = 0; l < to; ++l)
    launch_k(avg_down_kernel<T>, dim3(grid1(lv[l + 1].ncell, 256)), dim3(256), 0, s, arena, lv[l], lv[l + 1]);
}
template <typename T>
void nn_bridge_scale(const T* arena, const LevelDesc& L, double* scale, cudaStream_t s) {
  launch_k(rms_kernel<T>, dim3(1), dim3(1024), 0, s, arena, L.off, L.ncell, scale);
}
template <typename T>
void nn_bridge_features(const T* r, const LevelDesc& L, const float* pf, const double* scale,
                        const DevParams* prm, bf16* x, cudaStream_t s) {
  launch_k(features_kernel<T>, dim3(grid1(L.ncell, 256)), dim3(256), 0, s, r, L, pf, scale, prm, x);
}
template <typename T>
void nn_bridge_apply(const float* y, const LevelDesc& L, const double* scale, T* e, cudaStream_t s) {
  launch_k(apply_kernel<T>, dim3(grid1(L.ncell, 256)), dim3(256), 0, s, y, L, scale, e);
}
template <typename T>
void nn_bridge_guess_error(const double* phi, const double* guess, long long n, T* e0, cudaStream_t s) {
  launch_k(guess_error_kernel<T>, dim3(grid1(n, 256)), dim3(256), 0, s, phi, guess, n, e0);
}
template <typename T>
void nn_bridge_target(const T* e, const LevelDesc& L, const double* scale, float* tgt, cudaStream_t s) {
  launch_k(target_kernel<T>, dim3(grid1(L.ncell, 256)), dim3(256), 0, s, e, L, scale, tgt);
}

#define FX_NNB(T)                                                                                   \
  template void nn_bridge_restrict<T>(T*, const std::vector<LevelDesc>&, int, cudaStream_t);        \
  template void nn_bridge_scale<T>(const T*, const LevelDesc&, double*, cudaStream_t);              \
  template void nn_bridge_features<T>(const T*, const LevelDesc&, const float*, const double*,      \
                                      const DevParams*, bf16*, cudaStream_t);                       \
  template void nn_bridge_apply<T>(const float*, const LevelDesc&, const double*, T*, cudaStream_t); \
  template void nn_bridge_guess_error<T>(const double*, const double*, long long, T*, cudaStream_t); \
  template void nn_bridge_target<T>(const T*, const LevelDesc&, const double*, float*, cudaStream_t);
FX_NNB(float)
FX_NNB(double)
#undef FX_NNB

}  // namespace fx
