// The middle levels of an FP64 V-cycle, and the tail below them, in one launch by one
// cluster of 16 CTAs.
//
// A colour sweep of a level of a few thousand cells is 2.6 us of launch for 0.1 to 0.6 us
// of FP64 work, and ten such launches a level are most of a V-cycle on small grids; one CTA
// alone (the tail kernel) has 1/152 of the chip's FP64 rate.  Sixteen SMs take such a level
// in about the time one launch costs, so here each CTA holds 1/16 of every level in shared
// memory (consecutive red/black pairs of the linear order), a thread one pair of each
// level, its right-hand sides, diagonals and couplings in registers during the sweeps;
// neighbours are read from wherever they lie through distributed shared memory, and a
// cluster barrier ends each colour.  The levels' residuals and shifts are restricted by
// gathering, the tail (a V-cycle of CTA 0 or the dense solve, its rows spread over the
// cluster) goes through global memory as between launches, and the corrections return the
// same way.  Each cell sees the operations of smooth_pair, cell_residual, restrict4_kernel
// and prolong_fine in the same order: a V-cycle equals the separate launches bit for bit.
#include <cuda_runtime.h>

#define FX_TAIL_LINKAGE __noinline__   // see mg_device.cuh
#include "ferrox_internal.cuh"
#include "mg_device.cuh"

namespace fx {

namespace {

using namespace dev;

// barrier of the cluster after writes to global memory
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release;\nbarrier.cluster.wait.acquire;\n" ::: "memory");
}
// ... after writes to the CTA's own shared memory only: the release restricted to those
// does not wait for the memory system (74 ns a barrier of 256-thread CTAs
// instead of 221)
__device__ __forceinline__ void cluster_sync_smem() {
  asm volatile("fence.release.sync_restrict::shared::cta.cluster;\n"
               "barrier.cluster.arrive.relaxed;\nbarrier.cluster.wait.acquire;\n" ::: "memory");
}
__device__ __forceinline__ unsigned cluster_rank() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// address of the same shared-memory place in CTA `rank` of the cluster
__device__ __forceinline__ unsigned at_rank(unsigned a, int rank) {
  unsigned r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
  return r;
}
__device__ __forceinline__ double ld_cluster(unsigned a) {
  double v;
  asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ double2 ld_cluster2(unsigned a) {
  double2 v;
  asm volatile("ld.shared::cluster.v2.f64 {%0, %1}, [%2];" : "=d"(v.x), "=d"(v.y) : "r"(a) : "memory");
  return v;
}

// x / d from ri = 1 / d rounded to nearest: one residual correction of x * ri gives the
// rounded quotient (Markstein, IBM J. Res. Dev. 34, 1990), two operations instead of a
// division's dozen in the chain of every shifted cell
__device__ __forceinline__ double over_recip(double x, double d, double ri) {
  const double t = __dmul_rn(x, ri);
  return fma(fma(-d, t, x), ri, t);
}

// a thread's pair of a level: coordinates, couplings and neighbours' addresses (of the
// pair's first cell, for x of the cell outside the pair)
struct MidPair {
  bool on;
  int ip, j, k, par;                 // par: colour of the first cell
  unsigned own, xl, xr, ym, yp, zl, zh;
  double cx, cy, cl, ch, diag, inv;  // inv: 1 / diag
  double r0, r1, d0, d1;             // right-hand sides, diagonals with shift
  double i0, i1;                     // 1 / d0, 1 / d1 (on planes with a shift)
  bool s;                            // the plane has a shift
};

struct MidView {
  int hx, ny, nz, np, sh;
  unsigned mx, my;                   // divisors by hx and ny
  unsigned e, r, s;                  // shared-memory places of the CTA's part
  __device__ __forceinline__ unsigned pair(unsigned base, int p) const {
    return at_rank(base + (unsigned)(p & ((1 << sh) - 1)) * 16u, p >> sh);
  }
  __device__ __forceinline__ unsigned cell(unsigned base, int i, int j, int k) const {
    return pair(base, (k * ny + j) * hx + (i >> 1)) + (i & 1) * 8u;
  }
};

__device__ __forceinline__ MidView mid_view(const MidLevel& L, unsigned smem) {
  return MidView{L.d.nx >> 1, L.d.ny, L.d.nz, (L.d.nx >> 1) * L.d.ny * L.d.nz, L.sh, L.mx, L.my,
                 smem + L.e_off, smem + L.r_off, smem + L.s_off};
}

// t / d for t < 2^16 (m = ceil(2^32 / d), div32; 0 for d = 1)
__device__ __forceinline__ int mid_div(int t, unsigned m) { return m ? (int)__umulhi((unsigned)t, m) : t; }

template <bool SC>
__device__ __forceinline__ void mid_setup(MidPair& m, const MidView& V, const PlaneCoef<double>* coef, unsigned zero,
                                          int rank) {
  const int p = (rank << V.sh) + (int)threadIdx.x;
  m.on = (int)threadIdx.x < (1 << V.sh) && p < V.np;
  m.ip = m.j = m.k = m.par = 0;
  m.s = false;
  if (!m.on) return;
  const int row = mid_div(p, V.mx);
  m.ip = p - row * V.hx;
  m.k = mid_div(row, V.my);
  m.j = row - m.k * V.ny;
  m.par = (m.j + m.k) & 1;
  m.own = V.e + threadIdx.x * 16u;
  const int r0 = row * V.hx, pl = V.hx * V.ny;
  m.xl = V.pair(V.e, r0 + (m.ip == 0 ? V.hx - 1 : m.ip - 1)) + 8u;
  m.xr = V.pair(V.e, r0 + (m.ip == V.hx - 1 ? 0 : m.ip + 1));
  m.ym = V.pair(V.e, m.j == 0 ? p + (V.ny - 1) * V.hx : p - V.hx);
  m.yp = V.pair(V.e, m.j == V.ny - 1 ? p - (V.ny - 1) * V.hx : p + V.hx);
  m.zl = m.k > 0 ? V.pair(V.e, p - pl) : zero;          // two zeros beyond the electrodes
  m.zh = m.k < V.nz - 1 ? V.pair(V.e, p + pl) : zero;
  const PlaneCoef<double>& c = coef[m.k];   // in shared memory
  m.cx = c.cx; m.cy = c.cy; m.cl = c.czlo; m.ch = c.czhi;
  m.diag = c.diag; m.inv = c.invdiag;
  m.s = SC && c.has_s;
}

// the pair's diagonals with its shifts
template <bool SC>
__device__ __forceinline__ void mid_diag(MidPair& m, double s0, double s1) {
  m.d0 = m.d1 = m.diag;
  if (SC && m.s) {
    m.d0 += s0;
    m.d1 += s1;
    m.i0 = 1.0 / m.d0;
    m.i1 = 1.0 / m.d1;
  }
}

// (r + couplings * neighbours) of the pair's cell w (gs_numerator); other: the pair's other cell
__device__ __forceinline__ double mid_num(const MidPair& m, int w, double other) {
  const unsigned o = w * 8u;
  const double x = ld_cluster(w ? m.xr : m.xl), ym = ld_cluster(m.ym + o), yp = ld_cluster(m.yp + o);
  const double zl = ld_cluster(m.zl + o), zh = ld_cluster(m.zh + o);
  double acc = w ? m.r1 : m.r0;
  acc = fma(m.cx, x + other, acc);
  acc = fma(m.cy, ym + yp, acc);
  acc = fma(m.cl, zl, acc);
  return fma(m.ch, zh, acc);
}

// red-black sweeps of the level; v0, v1: the pair's corrections
template <bool SC>
__device__ __forceinline__ void mid_sweeps(const MidPair& m, double* own, double& v0, double& v1, int nu, bool zero) {
#pragma unroll 1
  for (int h = 0; h < 2 * nu; ++h) {
    const int w = m.par ^ (h & 1);
    if (m.on) {
      double x;
      if (zero && h == 0) {
        x = (w ? m.r1 : m.r0) * (SC && m.s ? (w ? m.i1 : m.i0) : m.inv);
      } else {
        x = mid_num(m, w, w ? v0 : v1);
        if (SC && m.s) x = over_recip(x, w ? m.d1 : m.d0, w ? m.i1 : m.i0);
        else x *= m.inv;
      }
      if (w) v1 = x;
      else v0 = x;
      own[w] = x;
    }
    cluster_sync_smem();
  }
}

// residuals of the coarse cells (2 ip, J, K) and (2 ip + 1, J, K): the means over the red
// children on the fine level F, summed in the order of restrict4_kernel or (seq) of the
// tail's restrict_cell (q: red residuals, one per fine pair; the pairs of the two coarse
// cells lie together)
__device__ __forceinline__ double2 mid_gather(const MidView& F, unsigned q, int crz, int seq, int ip, int J, int K) {
  const int p = ((crz ? 2 * K : K) * F.ny + 2 * J) * F.hx + 2 * ip;
  const int pl = F.ny * F.hx, mask = (1 << F.sh) - 1;
  auto get = [&](int t) {
    const unsigned a = at_rank(q + (unsigned)(t & mask) * 8u, t >> F.sh);
    return F.hx > 1 ? ld_cluster2(a) : make_double2(ld_cluster(a), 0.0);   // one coarse column: one pair a row
  };
  const double2 c0 = get(p), c3 = get(p + F.hx);
  if (!crz) return make_double2((c0.x + c3.x) * 0.25, (c0.y + c3.y) * 0.25);
  const double2 c5 = get(p + pl), c6 = get(p + pl + F.hx);
  if (seq) return make_double2((((c0.x + c3.x) + c5.x) + c6.x) * 0.125, (((c0.y + c3.y) + c5.y) + c6.y) * 0.125);
  return make_double2(((c0.x + c5.x) + (c6.x + c3.x)) * 0.125, ((c0.y + c5.y) + (c6.y + c3.y)) * 0.125);
}

// mean shift of the children of one coarse cell, in the same orders
__device__ __forceinline__ double mid_gather_s(const MidView& F, int crz, int seq, int I, int J, int K) {
  const int p = ((crz ? 2 * K : K) * F.ny + 2 * J) * F.hx + I, pl = F.ny * F.hx;
  const double2 a = ld_cluster2(F.pair(F.s, p)), b = ld_cluster2(F.pair(F.s, p + F.hx));
  if (!crz) return (seq ? ((a.x + a.y) + b.x) + b.y : (a.x + a.y) + (b.x + b.y)) * 0.25;
  const double2 c = ld_cluster2(F.pair(F.s, p + pl)), d = ld_cluster2(F.pair(F.s, p + pl + F.hx));
  return (seq ? ((((((a.x + a.y) + b.x) + b.y) + c.x) + c.y) + d.x) + d.y
              : ((a.x + c.x) + (a.y + c.y)) + ((b.x + d.x) + (b.y + d.y))) * 0.125;
}

// prolongated correction of fine cell (i, j, k) (prolong_fine); e(x, y, z): coarse values
template <typename E>
__device__ __forceinline__ double mid_prolong(E e, int i, int j, int k, int crz, int nx, int ny, int nz) {
  const int I = i >> 1, J = j >> 1, K = crz ? k >> 1 : k;
  const int I2 = (i & 1) ? (I + 1 == nx ? 0 : I + 1) : (I == 0 ? nx - 1 : I - 1);
  const int J2 = (j & 1) ? (J + 1 == ny ? 0 : J + 1) : (J == 0 ? ny - 1 : J - 1);
  const int K2 = (k & 1) ? K + 1 : K - 1;
  const bool in = K2 >= 0 && K2 < nz;
  auto zcol = [&](int x, int y) -> double {
    const double c0 = e(x, y, K);
    if (!crz) return c0;
    return in ? fma(0.75, c0, quarter(e(x, y, K2))) : 0.5 * c0;
  };
  const double z11 = zcol(I, J), z12 = zcol(I, J2), z21 = zcol(I2, J), z22 = zcol(I2, J2);
  const double y1 = fma(0.75, z11, quarter(z12)), y2 = fma(0.75, z21, quarter(z22));
  return fma(0.75, y1, quarter(y2));
}

template <bool SC>
__global__ void __launch_bounds__(kMidThreadsMax) mid_kernel(MGArgs<double> g, const __grid_constant__ MidArgs a) {
  extern __shared__ __align__(16) unsigned char mid_smem[];
  PlaneCoef<double>* const coef = reinterpret_cast<PlaneCoef<double>*>(mid_smem + a.coef_off);
  {   // the levels' planes lie together in the table, which no kernel writes
    const double* src = reinterpret_cast<const double*>(g.coef + a.lv[0].d.coef_off);
    double* dst = reinterpret_cast<double*>(coef);
    for (int t = threadIdx.x; t < a.planes * (int)(sizeof(PlaneCoef<double>) / 8); t += blockDim.x) dst[t] = __ldg(src + t);
  }
  pdl_enter();
  const unsigned smem = (unsigned)__cvta_generic_to_shared(mid_smem);
  const int rank = (int)cluster_rank(), tid = threadIdx.x;
  double* const zeros = reinterpret_cast<double*>(mid_smem);
  double* const q = reinterpret_cast<double*>(mid_smem + a.q_off);
  if (tid < 2) zeros[tid] = 0.0;
  __syncthreads();
  MidPair m;
  double v0 = 0.0, v1 = 0.0;
#pragma unroll 1
  for (int l = 0; l < a.n; ++l) {
    const MidLevel& L = a.lv[l];
    const MidView V = mid_view(L, smem);
    mid_setup<SC>(m, V, coef + (L.d.coef_off - a.lv[0].d.coef_off), smem, rank);
    double s0 = 0.0, s1 = 0.0;
    if (m.on) {
      if (l == 0) {
        const long long c = L.d.off + 2 * ((long long)(rank << L.sh) + tid);
        const double2 r = *reinterpret_cast<const double2*>(g.r + c);
        m.r0 = r.x; m.r1 = r.y;
        if (SC) {
          const double2 s = *reinterpret_cast<const double2*>(g.s + c);
          s0 = s.x; s1 = s.y;
        }
      } else {
        const MidLevel& Lf = a.lv[l - 1];
        const MidView F = mid_view(Lf, smem);
        const double2 r = mid_gather(F, smem + a.q_off, Lf.d.crz, Lf.seq, m.ip, m.j, m.k);
        m.r0 = r.x; m.r1 = r.y;
        if (SC) {
          s0 = mid_gather_s(F, Lf.d.crz, Lf.seq, 2 * m.ip, m.j, m.k);
          s1 = mid_gather_s(F, Lf.d.crz, Lf.seq, 2 * m.ip + 1, m.j, m.k);
        }
      }
      double* R = reinterpret_cast<double*>(mid_smem + L.r_off) + 2 * tid;
      R[0] = m.r0; R[1] = m.r1;
      if (SC) {
        double* S = reinterpret_cast<double*>(mid_smem + L.s_off) + 2 * tid;
        S[0] = s0; S[1] = s1;
      }
      mid_diag<SC>(m, s0, s1);
    }
    double* own = reinterpret_cast<double*>(mid_smem + L.e_off) + 2 * tid;
    mid_sweeps<SC>(m, own, v0, v1, a.nu1, true);
    if (m.on) {   // the black residuals vanish
      const double num = mid_num(m, m.par, m.par ? v0 : v1);
      q[tid] = fma(-(m.par ? m.d1 : m.d0), m.par ? v1 : v0, num);
    }
    cluster_sync_smem();
  }
  // the tail's right-hand side (and shift), its correction, through global memory
  const MidLevel& Lb = a.lv[a.n - 1];
  const LevelDesc& C = a.coarse;
  {
    const MidView F = mid_view(Lb, smem);
    const int hc = (C.nx + 1) >> 1, pairs = hc * C.ny * C.nz;
    for (int t = rank * (int)blockDim.x + tid; t < pairs; t += kMidCtas * (int)blockDim.x) {
      const int row = t / hc, ip = t - row * hc, K = row / C.ny, J = row - K * C.ny;
      const long long c = C.off + (long long)row * C.nx + 2 * ip;
      const bool two = 2 * ip + 1 < C.nx;
      const double2 r = mid_gather(F, smem + a.q_off, Lb.d.crz, Lb.seq, ip, J, K);
      g.r[c] = r.x;
      if (two) g.r[c + 1] = r.y;
      if (SC) {
        g.s[c] = mid_gather_s(F, Lb.d.crz, Lb.seq, 2 * ip, J, K);
        if (two) g.s[c + 1] = mid_gather_s(F, Lb.d.crz, Lb.seq, 2 * ip + 1, J, K);
      }
    }
  }
  cluster_sync();
  if (a.dense) {
    const int n = (int)C.ncell, lane = tid & 31, warps = (int)blockDim.x >> 5;
    for (int row = rank * warps + (tid >> 5); row < n; row += kMidCtas * warps) {
      const double* A = a.dense + (size_t)row * n;
      double acc = 0.0;
#pragma unroll 4
      for (int c = lane; c < n; c += 32) acc = fma(__ldg(A + c), __ldcg(g.r + C.off + c), acc);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
      if (lane == 0) g.e[C.off + row] = acc;
    }
  } else if (rank == 0) {
    tail_vcycle<double>(g, a.tail, mid_smem + a.tail_off);
  }
  cluster_sync();
#pragma unroll 1
  for (int l = a.n - 1; l >= 0; --l) {
    const MidLevel& L = a.lv[l];
    const MidView V = mid_view(L, smem);
    double* own = reinterpret_cast<double*>(mid_smem + L.e_off) + 2 * tid;
    if (l < a.n - 1) mid_setup<SC>(m, V, coef + (L.d.coef_off - a.lv[0].d.coef_off), smem, rank);
    if (m.on) {
      if (l < a.n - 1) {
        const double* R = reinterpret_cast<const double*>(mid_smem + L.r_off) + 2 * tid;
        m.r0 = R[0]; m.r1 = R[1];
        const double* S = reinterpret_cast<const double*>(mid_smem + L.s_off) + 2 * tid;
        if (SC) mid_diag<SC>(m, S[0], S[1]);
        v0 = own[0]; v1 = own[1];
      }
      // the red cells are relaxed before they are read: only black ones are corrected
      const int w = m.par ^ 1, i = 2 * m.ip + w;
      double c;
      if (l < a.n - 1) {
        const MidLevel& Lc = a.lv[l + 1];
        const MidView B = mid_view(Lc, smem);
        c = mid_prolong([&](int x, int y, int z) { return ld_cluster(B.cell(B.e, x, y, z)); }, i, m.j, m.k, L.d.crz,
                        Lc.d.nx, Lc.d.ny, Lc.d.nz);
      } else {
        c = mid_prolong([&](int x, int y, int z) { return __ldcg(g.e + C.off + (z * C.ny + y) * C.nx + x); }, i, m.j,
                        m.k, L.d.crz, C.nx, C.ny, C.nz);
      }
      if (w) own[1] = v1 = v1 + c;
      else own[0] = v0 = v0 + c;
    }
    cluster_sync_smem();
    mid_sweeps<SC>(m, own, v0, v1, a.nu2, false);
    if (l == 0 && m.on)
      *reinterpret_cast<double2*>(g.e + L.d.off + 2 * ((long long)(rank << L.sh) + tid)) = make_double2(v0, v1);
  }
}

const void* mid_func(bool sc) { return sc ? (const void*)mid_kernel<true> : (const void*)mid_kernel<false>; }

cudaLaunchConfig_t mid_config(const MidPlan& p, cudaLaunchAttribute* at, cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(kMidCtas);
  cfg.blockDim = dim3(p.threads);
  cfg.dynamicSmemBytes = p.smem;
  cfg.stream = s;
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = kMidCtas;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = pdl_enabled() ? 2 : 1;
  return cfg;
}

}  // namespace

bool mid_prepare(const MidPlan& p, bool sc) {
  const void* f = mid_func(sc);
  cudaLaunchAttribute at[2];
  const cudaLaunchConfig_t cfg = mid_config(p, at, nullptr);
  int n = 0;
  const bool ok = cudaFuncSetAttribute(f, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
                  cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, kMidMaxSmem) == cudaSuccess &&
                  cudaOccupancyMaxActiveClusters(&n, f, &cfg) == cudaSuccess && n >= 1;
  cudaGetLastError();
  return ok;
}

void launch_mid(const MGArgs<double>& g, const MidPlan& p, cudaStream_t s) {
  cudaLaunchAttribute at[2];
  const cudaLaunchConfig_t cfg = mid_config(p, at, s);
  if (g.s) cudaLaunchKernelEx(&cfg, mid_kernel<true>, g, p.args);
  else cudaLaunchKernelEx(&cfg, mid_kernel<false>, g, p.args);
}

}  // namespace fx
