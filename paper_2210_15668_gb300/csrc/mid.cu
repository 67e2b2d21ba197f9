// The middle levels of a V-cycle, and the tail below them, in one launch by one cluster of
// 16 CTAs.
//
// A colour sweep of a level of a few thousand cells is 2.6 us of launch for 0.1 to 0.6 us
// of FP64 work, and ten such launches a level are most of a V-cycle on small grids; one CTA
// alone (the tail kernel) has 1/152 of the chip's FP64 rate, and in FP32 spends its time on
// its own latencies.  Sixteen SMs take such a level in about the time one launch costs, so
// here each CTA holds 1/16 of every level in shared memory (consecutive red/black pairs of
// the linear order), a thread one pair of each level, its right-hand sides, diagonals and
// couplings in registers during the sweeps; neighbours are read from wherever they lie
// through distributed shared memory, and a cluster barrier ends each colour.  The levels'
// residuals and shifts are restricted by gathering, the coarsest level is relaxed in the
// same way, a tail of its own (a V-cycle of CTA 0 or the dense solve, its rows spread over
// the cluster) goes through global memory as between launches.  Each cell sees the
// operations of smooth_pair, cell_residual, restrict4_kernel (restrict_cell) and
// prolong_fine in the same order: a V-cycle equals the separate launches bit for bit (FP64
// quotients by a shifted diagonal: over_recip).
//
// A colour phase is bound by its latencies, 0.35 to 0.5 us (a load from another SM, six
// dependent FP64 operations of about 27 ns, 74 ns of barrier).  Measured: 64x64x16 FP64,
// levels of 8192 and 1024 cells, 21 launches and 54 us -> 1 launch and 20 us a V-cycle;
// 64^3 with carriers 70 -> 34 us; 96x80x37 mixed with carriers (64 sweeps of a coarsest
// level of 2220 cells) 68 -> 44 us; the tail alone on 256x256x64 with carriers, FP32,
// 34 -> 26 us together with the legs of the level above it.
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
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
  return r;
}
// Loads of distributed shared memory.  Volatile keeps them between the barriers; they may
// move past other accesses, which touch other colours or arrays.
__device__ __forceinline__ void ld_cluster(unsigned a, double& v) {
  asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(a));
}
__device__ __forceinline__ void ld_cluster(unsigned a, float& v) {
  asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(a));
}
__device__ __forceinline__ void ld_cluster2(unsigned a, double& x, double& y) {
  asm volatile("ld.shared::cluster.v2.f64 {%0, %1}, [%2];" : "=d"(x), "=d"(y) : "r"(a));
}
__device__ __forceinline__ void ld_cluster2(unsigned a, float& x, float& y) {
  asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];" : "=f"(x), "=f"(y) : "r"(a));
}
template <typename T>
__device__ __forceinline__ T ld_at(unsigned a) {
  T v;
  ld_cluster(a, v);
  return v;
}
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }

// x / d from ri = 1 / d rounded to nearest: x * ri with one residual correction, two
// operations instead of a division's dozen in the chain of every shifted cell.  Markstein
// (IBM J. Res. Dev. 34, 1990) proves the rounded quotient from a start within one unit in
// the last place; x * ri may be 1.5 off, so a quotient next to a midpoint of two numbers
// could still round the other way.  Two billion pairs, half of them made to lie there, gave
// the division's bits.  Not so where the residual underflows (|x| below about 1e-290), and
// an infinite x gives NaN (a solve that ends as not finite either way).
__device__ __forceinline__ double over_recip(double x, double d, double ri) {
  const double t = __dmul_rn(x, ri);
  return fma(fma(-d, t, x), ri, t);
}
__device__ __forceinline__ float over_recip(float x, float, float ri) { return __fmul_rn(x, ri); }   // as over_shifted

// a thread's pair of a level: coordinates, couplings and neighbours' addresses (of the
// pair's first cell, for x of the cell outside the pair)
template <typename T>
struct MidPair {
  bool on;
  int ip, j, k, par;                 // par: colour of the first cell
  unsigned own, xl, xr, ym, yp, zl, zh;
  T cx, cy, cl, ch, diag, inv;       // inv: 1 / diag
  T r0, r1, d0, d1;                  // right-hand sides, diagonals with shift
  T i0, i1;                          // 1 / d0, 1 / d1 (on planes with a shift)
  bool s;                            // the plane has a shift
};

template <typename T>
struct MidView {
  int hx, ny, nz, np, sh;
  unsigned mx, my;                   // divisors by hx and ny
  unsigned e, r, s;                  // shared-memory places of the CTA's part
  __device__ __forceinline__ unsigned pair(unsigned base, int p) const {
    return at_rank(base + (unsigned)(p & ((1 << sh) - 1)) * (2u * sizeof(T)), p >> sh);
  }
  __device__ __forceinline__ unsigned cell(unsigned base, int i, int j, int k) const {
    return pair(base, (k * ny + j) * hx + (i >> 1)) + (i & 1) * (unsigned)sizeof(T);
  }
};

template <typename T>
__device__ __forceinline__ MidView<T> mid_view(const MidLevel& L, unsigned smem) {
  return MidView<T>{L.d.nx >> 1, L.d.ny, L.d.nz, (L.d.nx >> 1) * L.d.ny * L.d.nz, L.sh, L.mx, L.my,
                    smem + L.e_off, smem + L.r_off, smem + L.s_off};
}

// t / d for t < 2^16 (m = ceil(2^32 / d), div32; 0 for d = 1)
__device__ __forceinline__ int mid_div(int t, unsigned m) { return m ? (int)__umulhi((unsigned)t, m) : t; }

template <typename T, bool SC>
__device__ __forceinline__ void mid_setup(MidPair<T>& m, const MidView<T>& V, const PlaneCoef<T>* coef, unsigned zero,
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
  m.own = V.e + threadIdx.x * (2u * sizeof(T));
  const int r0 = row * V.hx, pl = V.hx * V.ny;
  m.xl = V.pair(V.e, r0 + (m.ip == 0 ? V.hx - 1 : m.ip - 1)) + (unsigned)sizeof(T);
  m.xr = V.pair(V.e, r0 + (m.ip == V.hx - 1 ? 0 : m.ip + 1));
  m.ym = V.pair(V.e, m.j == 0 ? p + (V.ny - 1) * V.hx : p - V.hx);
  m.yp = V.pair(V.e, m.j == V.ny - 1 ? p - (V.ny - 1) * V.hx : p + V.hx);
  m.zl = m.k > 0 ? V.pair(V.e, p - pl) : zero;          // two zeros beyond the electrodes
  m.zh = m.k < V.nz - 1 ? V.pair(V.e, p + pl) : zero;
  const PlaneCoef<T>& c = coef[m.k];   // in shared memory
  m.cx = c.cx; m.cy = c.cy; m.cl = c.czlo; m.ch = c.czhi;
  m.diag = c.diag; m.inv = c.invdiag;
  m.s = SC && c.has_s;
}

// the pair's diagonals with its shifts
template <typename T, bool SC>
__device__ __forceinline__ void mid_diag(MidPair<T>& m, T s0, T s1) {
  m.d0 = m.d1 = m.diag;
  if (SC && m.s) {
    m.d0 += s0;
    m.d1 += s1;
    m.i0 = T(1) / m.d0;
    m.i1 = T(1) / m.d1;
  }
}

// (r + couplings * neighbours) of the pair's cell w (gs_numerator); other: the pair's other cell
template <typename T>
__device__ __forceinline__ T mid_num(const MidPair<T>& m, int w, T other) {
  const unsigned o = w * (unsigned)sizeof(T);
  const T x = ld_at<T>(w ? m.xr : m.xl), ym = ld_at<T>(m.ym + o), yp = ld_at<T>(m.yp + o);
  const T zl = ld_at<T>(m.zl + o), zh = ld_at<T>(m.zh + o);
  T acc = w ? m.r1 : m.r0;
  acc = fma(m.cx, x + other, acc);
  acc = fma(m.cy, ym + yp, acc);
  acc = fma(m.cl, zl, acc);
  return fma(m.ch, zh, acc);
}

// red-black sweeps of the level; v0, v1: the pair's corrections.  zero: from zero (1: the
// first red cells as smooth_pair, 2: as tail_smooth_held relaxes them)
template <typename T, bool SC>
__device__ __forceinline__ void mid_sweeps(const MidPair<T>& m, T* own, T& v0, T& v1, int nu, int zero) {
#pragma unroll 1
  for (int h = 0; h < 2 * nu; ++h) {
    const int w = m.par ^ (h & 1);
    if (m.on) {
      T x;
      if (zero == 1 && h == 0) {
        x = mul_rn(w ? m.r1 : m.r0, SC && m.s ? (w ? m.i1 : m.i0) : m.inv);
      } else {
        x = zero && h == 0 ? (w ? m.r1 : m.r0) : mid_num(m, w, w ? v0 : v1);
        if (SC && m.s) x = over_recip(x, w ? m.d1 : m.d0, w ? m.i1 : m.i0);
        else x = mul_rn(x, m.inv);
      }
      if (w) v1 = x;
      else v0 = x;
      own[w] = x;
    }
    cluster_sync_smem();
  }
}

// Means over the children of the coarse cells (2 ip, J, K) and (2 ip + 1, J, K) on the
// fine level F: of the red residuals (q: one per fine pair; black ones vanish) and of the
// shifts.  Summed in the order of restrict4_kernel, four partial sums of the children
// c and c + 4, or (seq) one after another as restrict_cell in the tail.
template <typename T>
struct Sum4 {
  T s[4] = {T(0), T(0), T(0), T(0)};
  T all = T(0);
  __device__ __forceinline__ void add(int c, T v) {
#pragma unroll
    for (int q = 0; q < 4; ++q) s[q] += (c & 3) == q ? v : T(0);
    all += v;
  }
  __device__ __forceinline__ T get(int seq) const { return seq ? all : (s[0] + s[1]) + (s[2] + s[3]); }
};

// one coarse cell of a level that is not halved in both x and y
template <typename T, bool SHIFT>
__device__ __noinline__ T mid_gather_part(MidView<T> F, unsigned q, int crx, int cry, int crz, int seq, int I, int J, int K) {
  const int nxc = crx ? 2 : 1, nyc = cry ? 2 : 1, nzc = crz ? 2 : 1;
  const int j0 = cry ? 2 * J : J, k0 = crz ? 2 * K : K, mask = (1 << F.sh) - 1;
  Sum4<T> sum;
  for (int dk = 0; dk < nzc; ++dk)
    for (int dj = 0; dj < nyc; ++dj)
      for (int di = 0; di < nxc; ++di) {
        const int i = crx ? 2 * I + di : I, j = j0 + dj, k = k0 + dk, c = di + nxc * (dj + nyc * dk);
        const int p = (k * F.ny + j) * F.hx + (i >> 1);
        if (SHIFT) sum.add(c, ld_at<T>(F.pair(F.s, p) + (i & 1) * (unsigned)sizeof(T)));
        else if (!((i + j + k) & 1)) sum.add(c, ld_at<T>(at_rank(q + (unsigned)(p & mask) * (unsigned)sizeof(T), p >> F.sh)));
      }
  return sum.get(seq) * (T(1) / T(nxc * nyc * nzc));
}

template <typename T, bool SC>
__device__ __forceinline__ void mid_gather(const MidView<T>& F, unsigned q, const LevelDesc& d, int seq, int ip, int J,
                                           int K, T& r0, T& r1, T& s0, T& s1) {
  if (!d.crx || !d.cry) {
    const int w = d.crx ? F.hx : 2 * F.hx;   // coarse cells in a row
    const bool two = 2 * ip + 1 < w;
    r0 = mid_gather_part<T, false>(F, q, d.crx, d.cry, d.crz, seq, 2 * ip, J, K);
    r1 = two ? mid_gather_part<T, false>(F, q, d.crx, d.cry, d.crz, seq, 2 * ip + 1, J, K) : T(0);
    if (SC) {
      s0 = mid_gather_part<T, true>(F, q, d.crx, d.cry, d.crz, seq, 2 * ip, J, K);
      s1 = two ? mid_gather_part<T, true>(F, q, d.crx, d.cry, d.crz, seq, 2 * ip + 1, J, K) : T(0);
    }
    return;
  }
  // rows (dj, dk) of the fine pairs 2 ip and 2 ip + 1, which lie together (one coarse
  // column: one pair a row); all loads first
  const int rows = d.crz ? 4 : 2, mask = (1 << F.sh) - 1;
  const int p = ((d.crz ? 2 * K : K) * F.ny + 2 * J) * F.hx + 2 * ip, pl = F.ny * F.hx;
  T a[4], b[4], u[4][2], v[4][2];
#pragma unroll
  for (int w = 0; w < 4; ++w) {
    a[w] = b[w] = u[w][0] = u[w][1] = v[w][0] = v[w][1] = T(0);
    if (w >= rows) continue;
    const int t = p + (w & 1) * F.hx + (w >> 1) * pl;
    const unsigned at = at_rank(q + (unsigned)(t & mask) * (unsigned)sizeof(T), t >> F.sh);
    if (F.hx > 1) ld_cluster2(at, a[w], b[w]);
    else ld_cluster(at, a[w]);
    if (SC) {
      ld_cluster2(F.pair(F.s, t), u[w][0], u[w][1]);
      if (F.hx > 1) ld_cluster2(F.pair(F.s, t + 1), v[w][0], v[w][1]);
    }
  }
  const T mean = d.crz ? T(0.125) : T(0.25);
  // red children of rows 0 .. 3: c = 0, 3, 5, 6 (an odd plane alone: 1, 2, the same sum)
  auto red = [&](const T (&x)[4]) { return (seq ? ((x[0] + x[1]) + x[2]) + x[3] : (x[0] + x[2]) + (x[3] + x[1])) * mean; };
  auto all = [&](const T (&x)[4][2]) {
    return (seq ? ((((((x[0][0] + x[0][1]) + x[1][0]) + x[1][1]) + x[2][0]) + x[2][1]) + x[3][0]) + x[3][1]
                : ((x[0][0] + x[2][0]) + (x[0][1] + x[2][1])) + ((x[1][0] + x[3][0]) + (x[1][1] + x[3][1]))) * mean;
  };
  r0 = red(a);
  r1 = red(b);
  if (SC) {
    s0 = all(u);
    s1 = all(v);
  }
}

// prolongated correction of fine cell (i, j, k) (prolong_fine) of level l; e(x, y, z): coarse
// values of a level of nx x ny x nz cells, all loaded first
template <typename T, typename E>
__device__ __forceinline__ T mid_prolong(E e, const LevelDesc& l, int i, int j, int k, int nx, int ny, int nz) {
  const int I = l.crx ? i >> 1 : i, J = l.cry ? j >> 1 : j, K = l.crz ? k >> 1 : k;
  const int I2 = !l.crx ? I : (i & 1) ? (I + 1 == nx ? 0 : I + 1) : (I == 0 ? nx - 1 : I - 1);
  const int J2 = !l.cry ? J : (j & 1) ? (J + 1 == ny ? 0 : J + 1) : (J == 0 ? ny - 1 : J - 1);
  const int K2 = (k & 1) ? K + 1 : K - 1;
  const bool in = K2 >= 0 && K2 < nz;
  T c[4], o[4] = {T(0), T(0), T(0), T(0)};   // columns (I, J), (I, J2), (I2, J), (I2, J2)
#pragma unroll
  for (int q = 0; q < 4; ++q) c[q] = e(q & 2 ? I2 : I, q & 1 ? J2 : J, K);
  if (l.crz && in) {
#pragma unroll
    for (int q = 0; q < 4; ++q) o[q] = e(q & 2 ? I2 : I, q & 1 ? J2 : J, K2);
  }
  if (l.crz) {
#pragma unroll
    for (int q = 0; q < 4; ++q) c[q] = in ? fma(T(0.75), c[q], quarter(o[q])) : T(0.5) * c[q];
  }
  const T y1 = l.cry ? fma(T(0.75), c[0], quarter(c[1])) : c[0], y2 = l.cry ? fma(T(0.75), c[2], quarter(c[3])) : c[2];
  return l.crx ? fma(T(0.75), y1, quarter(y2)) : y1;
}

template <typename T, bool SC>
__global__ void __launch_bounds__(mid_threads_max<T>()) mid_kernel(MGArgs<T> g, const __grid_constant__ MidArgs a) {
  extern __shared__ __align__(16) unsigned char mid_smem[];
  PlaneCoef<T>* const coef = reinterpret_cast<PlaneCoef<T>*>(mid_smem + a.coef_off);
  {   // the levels' planes lie together in the table, which no kernel writes
    const double* src = reinterpret_cast<const double*>(g.coef + a.lv[0].d.coef_off);
    double* dst = reinterpret_cast<double*>(coef);
    for (int t = threadIdx.x; t < a.planes * (int)(sizeof(PlaneCoef<T>) / 8); t += blockDim.x) dst[t] = __ldg(src + t);
  }
  pdl_enter();
  const unsigned smem = (unsigned)__cvta_generic_to_shared(mid_smem);
  const int rank = (int)cluster_rank(), tid = threadIdx.x;
  T* const zeros = reinterpret_cast<T*>(mid_smem);
  T* const q = reinterpret_cast<T*>(mid_smem + a.q_off);
  if (tid < 2) zeros[tid] = T(0);
  __syncthreads();
  MidPair<T> m;
  T v0 = T(0), v1 = T(0);
#pragma unroll 1
  for (int l = 0; l < a.n; ++l) {
    const MidLevel& L = a.lv[l];
    const MidView<T> V = mid_view<T>(L, smem);
    mid_setup<T, SC>(m, V, coef + (L.d.coef_off - a.lv[0].d.coef_off), smem, rank);
    T s0 = T(0), s1 = T(0);
    if (m.on) {
      if (l == 0) {
        const long long c = L.d.off + 2 * ((long long)(rank << L.sh) + tid);
        m.r0 = g.r[c]; m.r1 = g.r[c + 1];
        if (SC) {
          s0 = g.s[c]; s1 = g.s[c + 1];
        }
      } else {
        const MidLevel& Lf = a.lv[l - 1];
        const MidView<T> F = mid_view<T>(Lf, smem);
        mid_gather<T, SC>(F, smem + a.q_off, Lf.d, Lf.seq, m.ip, m.j, m.k, m.r0, m.r1, s0, s1);
      }
      T* R = reinterpret_cast<T*>(mid_smem + L.r_off) + 2 * tid;
      R[0] = m.r0; R[1] = m.r1;
      if (SC) {
        T* S = reinterpret_cast<T*>(mid_smem + L.s_off) + 2 * tid;
        S[0] = s0; S[1] = s1;
      }
      mid_diag<T, SC>(m, s0, s1);
    }
    T* own = reinterpret_cast<T*>(mid_smem + L.e_off) + 2 * tid;
    const bool bottom = a.bottom && l == a.n - 1;
    mid_sweeps<T, SC>(m, own, v0, v1, bottom ? a.bottom : a.nu1, bottom && a.bottom >= kTailHeldSweeps ? 2 : 1);
    if (bottom) break;
    if (m.on) {   // the black residuals vanish
      const T num = mid_num(m, m.par, m.par ? v0 : v1);
      q[tid] = fma(-(m.par ? m.d1 : m.d0), m.par ? v1 : v0, num);
    }
    cluster_sync_smem();
  }
  const LevelDesc& C = a.coarse;
  if (!a.bottom) {
    // the tail's right-hand side (and shift), its correction, through global memory
    const MidLevel& Lb = a.lv[a.n - 1];
    const MidView<T> F = mid_view<T>(Lb, smem);
    const int hc = (C.nx + 1) >> 1, pairs = hc * C.ny * C.nz;
    for (int t = rank * (int)blockDim.x + tid; t < pairs; t += kMidCtas * (int)blockDim.x) {
      const int row = t / hc, ip = t - row * hc, K = row / C.ny, J = row - K * C.ny;
      const long long c = C.off + (long long)row * C.nx + 2 * ip;
      const bool two = 2 * ip + 1 < C.nx;
      T r0, r1, s0 = T(0), s1 = T(0);
      mid_gather<T, SC>(F, smem + a.q_off, Lb.d, Lb.seq, ip, J, K, r0, r1, s0, s1);
      if (a.single) {   // one cell, relaxed once from zero
        const PlaneCoef<T> k = ldg_struct(g.coef + C.coef_off);
        g.e[C.off] = mul_rn(r0, SC && k.has_s ? T(1) / (k.diag + s0) : k.invdiag);
        continue;
      }
      g.r[c] = r0;
      if (SC) g.s[c] = s0;
      if (two) {
        g.r[c + 1] = r1;
        if (SC) g.s[c + 1] = s1;
      }
    }
    cluster_sync();
    if (a.dense) {
      const int n = (int)C.ncell, lane = tid & 31, warps = (int)blockDim.x >> 5;
      for (int row = rank * warps + (tid >> 5); row < n; row += kMidCtas * warps) {
        const T* A = static_cast<const T*>(a.dense) + (size_t)row * n;
        T acc = T(0);
#pragma unroll 4
        for (int c = lane; c < n; c += 32) acc = fma(__ldg(A + c), __ldcg(g.r + C.off + c), acc);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        if (lane == 0) g.e[C.off + row] = acc;
      }
      cluster_sync();
    } else if (!a.single) {
      if (rank == 0) tail_vcycle<T>(g, a.tail, mid_smem + a.tail_off);
      cluster_sync();
    }
  }
#pragma unroll 1
  for (int l = a.n - (a.bottom ? 2 : 1); l >= 0; --l) {
    const MidLevel& L = a.lv[l];
    const MidView<T> V = mid_view<T>(L, smem);
    T* own = reinterpret_cast<T*>(mid_smem + L.e_off) + 2 * tid;
    if (l < a.n - 1) mid_setup<T, SC>(m, V, coef + (L.d.coef_off - a.lv[0].d.coef_off), smem, rank);
    if (m.on) {
      if (l < a.n - 1) {
        const T* R = reinterpret_cast<const T*>(mid_smem + L.r_off) + 2 * tid;
        m.r0 = R[0]; m.r1 = R[1];
        const T* S = reinterpret_cast<const T*>(mid_smem + L.s_off) + 2 * tid;
        if (SC) mid_diag<T, SC>(m, S[0], S[1]);
        v0 = own[0]; v1 = own[1];
      }
      // the red cells are relaxed before they are read: only black ones are corrected
      const int w = m.par ^ 1, i = 2 * m.ip + w;
      T c;
      if (l < a.n - 1) {
        const MidLevel& Lc = a.lv[l + 1];
        const MidView<T> B = mid_view<T>(Lc, smem);
        c = mid_prolong<T>([&](int x, int y, int z) { return ld_at<T>(B.cell(B.e, x, y, z)); }, L.d, i, m.j, m.k, Lc.d.nx,
                           Lc.d.ny, Lc.d.nz);
      } else {
        c = mid_prolong<T>([&](int x, int y, int z) { return __ldcg(g.e + C.off + (z * C.ny + y) * C.nx + x); }, L.d, i,
                           m.j, m.k, C.nx, C.ny, C.nz);
      }
      if (w) own[1] = v1 = v1 + c;
      else own[0] = v0 = v0 + c;
    }
    cluster_sync_smem();
    mid_sweeps<T, SC>(m, own, v0, v1, a.nu2, 0);
    if (l == 0 && m.on) {
      T* e = g.e + L.d.off + 2 * ((long long)(rank << L.sh) + tid);
      e[0] = v0;
      e[1] = v1;
    }
  }
}

template <typename T>
const void* mid_func(bool sc) { return sc ? (const void*)mid_kernel<T, true> : (const void*)mid_kernel<T, false>; }

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

template <typename T>
bool mid_prepare(const MidPlan& p, bool sc) {
  const void* f = mid_func<T>(sc);
  cudaLaunchAttribute at[2];
  const cudaLaunchConfig_t cfg = mid_config(p, at, nullptr);
  int n = 0;
  const bool ok = cudaFuncSetAttribute(f, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
                  cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, kMidMaxSmem) == cudaSuccess &&
                  cudaOccupancyMaxActiveClusters(&n, f, &cfg) == cudaSuccess && n >= 1;
  cudaGetLastError();
  return ok;
}

template <typename T>
void launch_mid(const MGArgs<T>& g, const MidPlan& p, cudaStream_t s) {
  cudaLaunchAttribute at[2];
  const cudaLaunchConfig_t cfg = mid_config(p, at, s);
  if (g.s) cudaLaunchKernelEx(&cfg, mid_kernel<T, true>, g, p.args);
  else cudaLaunchKernelEx(&cfg, mid_kernel<T, false>, g, p.args);
}

template bool mid_prepare<double>(const MidPlan&, bool);
template bool mid_prepare<float>(const MidPlan&, bool);
template void launch_mid<double>(const MGArgs<double>&, const MidPlan&, cudaStream_t);
template void launch_mid<float>(const MGArgs<float>&, const MidPlan&, cudaStream_t);

}  // namespace fx
