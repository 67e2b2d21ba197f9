// Per-cell and per-column device functions of the multigrid and of the FP64
// outer residual, shared by the multi-kernel path (multigrid.cu) and the
// persistent batched engine (persistent.cu).  See multigrid.cu for the method.
#pragma once
#include <cuda_runtime.h>
#include <math.h>

#include "carrier_exp.cuh"
#include "df_arith.cuh"
#include "ferrox_internal.cuh"

namespace fx {
namespace dev {

// arenas hold fewer than 2^31 elements (checked at init), so 32-bit indices suffice
__device__ __forceinline__ int lidx(const LevelDesc& L, int i, int j, int k) {
  return (int)L.off + (k * L.ny + j) * L.nx + i;
}

// (r + sum of couplings * neighbours) of one cell; the Gauss-Seidel numerator.
template <typename T>
__device__ __forceinline__ T gs_numerator(const T* e, const T* r, const PlaneCoef<T>& c,
                                          const LevelDesc& L, int i, int j, int k, int id) {
  const int im = (i == 0) ? L.nx - 1 : i - 1;
  const int ip = (i == L.nx - 1) ? 0 : i + 1;
  const int jm = (j == 0) ? L.ny - 1 : j - 1;
  const int jp = (j == L.ny - 1) ? 0 : j + 1;
  const int row = id - i;
  const int plane = L.nx * L.ny;
  T sx = e[row + im] + e[row + ip];
  T sy = e[id + (jm - j) * L.nx] + e[id + (jp - j) * L.nx];
  T ed = (k > 0) ? e[id - plane] : T(0);
  T eu = (k < L.nz - 1) ? e[id + plane] : T(0);
  T acc = r[id];
  acc = fma(c.cx, sx, acc);
  acc = fma(c.cy, sy, acc);
  acc = fma(c.czlo, ed, acc);
  acc = fma(c.czhi, eu, acc);
  return acc;
}

// a numerator over the shifted diagonal d = diag + s; in FP32 by the reciprocal, as
// level 0 does with its stored 1 / (diag + s) and the V-cycle legs at every level
template <typename T>
__device__ __forceinline__ T over_shifted(T num, T d) {
  if constexpr (sizeof(T) == sizeof(float)) return num * (T(1) / d);
  else return num / d;
}

struct Upd {
  double* phi;      // fine-level potential (null: no fused update)
  double clamp;     // |e| limit of one update (infinite without carriers)
  int zero;         // set phi = 0 (degenerate zero right-hand side)
  float clampf;     // the limit rounded to FP32 (FP32 corrections)
};

// phi += e, e clamped to [-clamp, clamp].  An FP32 correction is clamped in FP32
// against the limit rounded to float and widened with integer operations: one FP64 add
// per cell instead of two FP64 min/max, a conversion and the add (GB300 runs FP64, and
// conversions to it, at 1/58 of the FP32 rate; both fine legs on 256x256x32, timed one by
// one, 56 -> 52 us, the update alone 14.3 -> 12.2).  With an infinite limit (no carriers)
// the result is the same bit for bit (corrections below 2^-126 count as zero).
template <typename T>
__device__ __forceinline__ void apply_update(const Upd& u, int idx, T e) {
  if (u.zero) {
    u.phi[idx] = 0.0;
  } else if constexpr (sizeof(T) == sizeof(float)) {
    u.phi[idx] += f64_of_float(fminf(fmaxf(e, -u.clampf), u.clampf));
  } else {
    u.phi[idx] += fmin(fmax(e, -u.clamp), u.clamp);
  }
}

// One red/black pair position (ip) of a row: update the cell of `color`; on a
// zero-start sweep also zero the other cell; optionally fold both cells' final
// corrections into phi (last black sweep of the fine level).
template <typename T>
__device__ __forceinline__ void smooth_pair(const MGArgs<T>& a, const LevelDesc& L, int ip, int j,
                                            int k, int color, int zero_init, const Upd& u) {
  const int par = (j + k + color) & 1;
  const int i = 2 * ip + par;
  const int i2 = 2 * ip + (par ^ 1);
  const PlaneCoef<T> c = ldg_struct(a.coef + L.coef_off + k);
  T ev = T(0);
  int id = -1;
  if (i < L.nx) {
    id = lidx(L, i, j, k);
    if (zero_init) {
      const T d = c.has_s ? (a.sinv ? a.sinv[id - L.off] : T(1) / (c.diag + a.s[id])) : c.invdiag;
      ev = a.r[id] * d;
    } else {
      const T num = gs_numerator(a.e, a.r, c, L, i, j, k, id);
      ev = c.has_s ? (a.sinv ? num * a.sinv[id - L.off] : over_shifted<T>(num, c.diag + a.s[id])) : num * c.invdiag;
    }
    a.e[id] = ev;
  }
  if (i2 < L.nx) {
    const int id2 = lidx(L, i2, j, k);
    if (zero_init) a.e[id2] = T(0);
    if (u.phi) apply_update(u, id2 - L.off, a.e[id2]);
  }
  if (u.phi && id >= 0) apply_update(u, id - L.off, ev);
}

// residual of one fine cell: r - (A + s) e
template <typename T>
__device__ __forceinline__ T cell_residual(const MGArgs<T>& a, const LevelDesc& L, int i, int j,
                                           int k) {
  const PlaneCoef<T> c = ldg_struct(a.coef + L.coef_off + k);
  const int id = lidx(L, i, j, k);
  T num = gs_numerator(a.e, a.r, c, L, i, j, k, id);   // r + couplings * neighbours
  T d = c.has_s ? c.diag + a.s[id] : c.diag;
  return fma(-d, a.e[id], num);
}

// A red/black pre-smoothing ends with the black colour ((i + j + k) odd), whose
// cells were just relaxed against red neighbours that have not changed since:
// their residual is zero up to rounding.  With skip_black set, restriction
// sums the residuals of the red children only (half the arithmetic).  The
// colouring is a proper 2-colouring only if every periodic lateral size is
// even (or 1); black_residual_zero() tells the callers when that holds.
__host__ __device__ __forceinline__ int black_residual_zero(const LevelDesc& F, int nu1) {
  return nu1 > 0 && (F.nx == 1 || !(F.nx & 1)) && (F.ny == 1 || !(F.ny & 1));
}

// Residual of the children of coarse cell (I, J, K) on level F, their mean written to the
// coarse right-hand side (and the mean Newton shift).
template <typename T>
__device__ __forceinline__ void restrict_cell(const MGArgs<T>& a, const LevelDesc& F,
                                              const LevelDesc& C, int I, int J, int K,
                                              int skip_black = 0) {
  const int nxc = F.crx ? 2 : 1, nyc = F.cry ? 2 : 1, nzc = F.crz ? 2 : 1;
  const int i0 = F.crx ? 2 * I : I, j0 = F.cry ? 2 * J : J, k0 = F.crz ? 2 * K : K;
  T sum = T(0), ssum = T(0);
  for (int dk = 0; dk < nzc; ++dk)
    for (int dj = 0; dj < nyc; ++dj)
      for (int di = 0; di < nxc; ++di) {
        const int i = i0 + di, j = j0 + dj, k = k0 + dk;
        if (!(skip_black && ((i + j + k) & 1))) sum += cell_residual(a, F, i, j, k);
        if (a.s) ssum += a.s[lidx(F, i, j, k)];
      }
  const T inv = T(1) / T(nxc * nyc * nzc);
  const int idc = lidx(C, I, J, K);
  a.r[idc] = sum * inv;
  if (a.s) a.s[idc] = ssum * inv;
}

// x / 4.  In FP64 by the exponent where x and the result are normal numbers: the same value
// as the multiplication, which would take 19 clocks of an SM's FP64 pipe per warp (7 of
// prolong_fine's 15 FP64 operations and 10 of prolong_tiled_kernel's 24 are these).
template <typename T>
__device__ __forceinline__ T quarter(T x) {
  if constexpr (sizeof(T) == sizeof(double)) {
    const int hi = __double2hiint(x);
    if (((unsigned)(hi >> 20) & 0x7ffu) - 3u < 0x7fcu) return __hiloint2double(hi - (2 << 20), __double2loint(x));
  }
  return T(0.25) * x;   // zero, subnormal numbers, infinities, NaN
}

// Prolongation + correction for the children of coarse cell (I, J, K).
// Cell-centred trilinear interpolation, separable: along every coarsened
// direction a child takes 3/4 of its own coarse value and 1/4 of the coarse
// neighbour on its side; an electrode beyond the coarse grid acts as a ghost
// cell holding -e (zero correction on the electrode face).
template <typename T>
__device__ __forceinline__ void prolong_cell(const MGArgs<T>& a, const LevelDesc& F,
                                             const LevelDesc& C, int I, int J, int K, int constant) {
  const int nxc = F.crx ? 2 : 1, nyc = F.cry ? 2 : 1, nzc = F.crz ? 2 : 1;
  T* e = a.e;
  if (constant) {
    const T E0 = e[lidx(C, I, J, K)];
    for (int c = 0; c < nzc; ++c)
      for (int b = 0; b < nyc; ++b)
        for (int q = 0; q < nxc; ++q)
          e[lidx(F, F.crx ? 2 * I + q : I, F.cry ? 2 * J + b : J, F.crz ? 2 * K + c : K)] += E0;
    return;
  }
  const int Im = I == 0 ? C.nx - 1 : I - 1, Ip = I + 1 == C.nx ? 0 : I + 1;
  const int Jm = J == 0 ? C.ny - 1 : J - 1, Jp = J + 1 == C.ny ? 0 : J + 1;
  const int xs[3] = {Im, I, Ip}, ys[3] = {Jm, J, Jp};
  T Z[2][3][3];
#pragma unroll
  for (int yy = 0; yy < 3; ++yy)
#pragma unroll
    for (int xx = 0; xx < 3; ++xx) {
      if ((!F.cry && yy != 1) || (!F.crx && xx != 1)) continue;
      const T Ec = e[lidx(C, xs[xx], ys[yy], K)];
      if (F.crz) {
        Z[0][yy][xx] = (K > 0) ? fma(T(0.75), Ec, T(0.25) * e[lidx(C, xs[xx], ys[yy], K - 1)])
                               : T(0.5) * Ec;
        Z[1][yy][xx] = (K + 1 < C.nz) ? fma(T(0.75), Ec, T(0.25) * e[lidx(C, xs[xx], ys[yy], K + 1)])
                                      : T(0.5) * Ec;
      } else {
        Z[0][yy][xx] = Ec;
      }
    }
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    if (c >= nzc) break;
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      if (b >= nyc) break;
      T Y[3];
#pragma unroll
      for (int xx = 0; xx < 3; ++xx) {
        if (!F.crx && xx != 1) continue;
        Y[xx] = F.cry ? fma(T(0.75), Z[c][1][xx], T(0.25) * Z[c][b ? 2 : 0][xx]) : Z[c][1][xx];
      }
      const int fj = F.cry ? 2 * J + b : J, fk = F.crz ? 2 * K + c : K;
      if (F.crx) {
        const int f0 = lidx(F, 2 * I, fj, fk);
        e[f0] += fma(T(0.75), Y[1], T(0.25) * Y[0]);
        e[f0 + 1] += fma(T(0.75), Y[1], T(0.25) * Y[2]);
      } else {
        e[lidx(F, I, fj, fk)] += Y[1];
      }
    }
  }
}

// Prolongation + correction of one fine cell (i, j, k) of F: the separable
// trilinear interpolation of prolong_cell (z, then y, then x, the same
// operations in the same order), evaluated per fine cell, so that a tiny level
// spreads its arithmetic over one thread per fine cell.
template <typename T>
__device__ __forceinline__ void prolong_fine(const MGArgs<T>& a, const LevelDesc& F,
                                             const LevelDesc& C, int i, int j, int k,
                                             int constant) {
  T* e = a.e;
  const int I = F.crx ? i >> 1 : i, J = F.cry ? j >> 1 : j, K = F.crz ? k >> 1 : k;
  if (constant) {
    e[lidx(F, i, j, k)] += e[lidx(C, I, J, K)];
    return;
  }
  // the coarse neighbour on the child's side in each coarsened direction
  const int I2 = !F.crx ? I : (i & 1) ? (I + 1 == C.nx ? 0 : I + 1) : (I == 0 ? C.nx - 1 : I - 1);
  const int J2 = !F.cry ? J : (j & 1) ? (J + 1 == C.ny ? 0 : J + 1) : (J == 0 ? C.ny - 1 : J - 1);
  const int K2 = (k & 1) ? K + 1 : K - 1;   // outside [0, C.nz): electrode ghost (-e)
  auto zcol = [&](int x, int y) -> T {
    const T c0 = e[lidx(C, x, y, K)];
    if (!F.crz) return c0;
    return (K2 >= 0 && K2 < C.nz) ? fma(T(0.75), c0, quarter(e[lidx(C, x, y, K2)]))
                                  : T(0.5) * c0;
  };
  const T z11 = zcol(I, J);
  T y1 = z11, y2 = T(0);
  if (F.cry) y1 = fma(T(0.75), z11, quarter(zcol(I, J2)));
  if (F.crx) {
    const T z21 = zcol(I2, J);
    y2 = F.cry ? fma(T(0.75), z21, quarter(zcol(I2, J2))) : z21;
    e[lidx(F, i, j, k)] += fma(T(0.75), y1, quarter(y2));
  } else {
    e[lidx(F, i, j, k)] += y1;
  }
}

// ---- single-CTA tail: the smallest levels in shared memory ---------------------------

// Division by a level constant d without the integer divide sequence: with
// m = ceil(2^32 / d) = floor((2^32 - 1) / d) + 1 (one 32-bit divide per call),
// floor(t m / 2^32) = floor(t / d) for all t < 2^16 and d <= 2^16 (Granlund and
// Montgomery, PLDI 1994: the error t (m d - 2^32) / d stays below 2^32 / d).
// The tail's shared-memory budget keeps every tail level below 2^16 cells, so
// all indices of a tail sweep are in range.
static_assert(kTailMaxSmem / (2 * sizeof(float)) < 65536, "tail indices must stay below 2^16");

__device__ __forceinline__ unsigned long long magic32(unsigned d) {
  return (unsigned long long)(0xFFFFFFFFu / d) + 1ull;
}
__device__ __forceinline__ int div32(int t, unsigned long long m) {
  return (int)(((unsigned long long)(unsigned)t * m) >> 32);
}

// FX_TAIL_LINKAGE: how tail_smooth and tail_vcycle are compiled in this
// translation unit.  The batched engines (persistent.cu) set __noinline__:
// inlined there, the FP64 instantiation lost the tail's smoothing (the first
// tail level kept its old shared-memory contents; 35 V-cycles per solve instead
// of 8 on a 32x32x16 stack), depending only on the surrounding code.  The
// single-instance tail kernel inlines them (same V-cycle counts either way,
// checked by the solver tests' cycle bounds).
#ifndef FX_TAIL_LINKAGE
#define FX_TAIL_LINKAGE
#endif
template <typename T>
__device__ FX_TAIL_LINKAGE void tail_smooth(const MGArgs<T>& a, const LevelDesc& L, int sweeps, int zero_first) {
  const int hx = (L.nx + 1) >> 1;
  const int items = hx * L.ny * L.nz;
  const unsigned long long mx = magic32(hx), my = magic32(L.ny);
  const Upd none{nullptr, 0.0, 0, 0.0f};
  for (int sw = 0; sw < sweeps; ++sw)
    for (int color = 0; color < 2; ++color) {
      const int zi = (zero_first && sw == 0 && color == 0);
      for (int t = threadIdx.x; t < items; t += blockDim.x) {
        const int rest = div32(t, mx), k = div32(rest, my);
        smooth_pair(a, L, t - rest * hx, rest - k * L.ny, k, color, zi, none);
      }
      __syncthreads();
    }
}

// Many sweeps of one level (a coarsest level that cannot be halved further, relaxed
// bottom_sweeps times) with two red/black pairs per thread held in registers: their
// right-hand sides, reciprocal diagonals, couplings, neighbour indices and own
// corrections are set up once, so a colour phase is five shared-memory loads, six
// operations and one store per cell, and a barrier.  tail_smooth decodes every pair and
// loads its level, plane coefficients and shift anew in every phase; it stays the better
// one for the two sweeps of the other levels, where a tail's time is the first pass over
// its code (both measured, 256x256x64 MFISM: 28 us a V-cycle either way).  96x80x37
// MFISM, coarsest level 6x10x37 cells, 64 sweeps: the tail 118 -> 43 us a V-cycle.
constexpr int kTailHeldSweeps = 8;   // sweeps from which the set-up pays
template <typename T>
__device__ __forceinline__ void tail_smooth_held(const MGArgs<T>& a, const LevelDesc& L, int sweeps) {
  constexpr int ITEMS = 2;
  const int hx = (L.nx + 1) >> 1, items = hx * L.ny * L.nz;
  const unsigned long long mx = magic32(hx), my = magic32(L.ny);
  const int plane = L.nx * L.ny;
  T* e = a.e + L.off;
  T v[ITEMS][2], r[ITEMS][2], inv[ITEMS][2], cx[ITEMS], cy[ITEMS], cl[ITEMS], ch[ITEMS];
  int id[ITEMS], xo[ITEMS][2], ym[ITEMS], yp[ITEMS], zl[ITEMS], zh[ITEMS], par[ITEMS];
  bool two[ITEMS], div[ITEMS];
#pragma unroll
  for (int q = 0; q < ITEMS; ++q) {
    const int t = (int)threadIdx.x + q * (int)blockDim.x;
    par[q] = -1;
    if (t >= items) continue;
    const int rest = div32(t, mx), k = div32(rest, my);
    const int ip = t - rest * hx, j = rest - k * L.ny, i = 2 * ip;
    id[q] = (k * L.ny + j) * L.nx + i;
    two[q] = i + 1 < L.nx;
    par[q] = (j + k) & 1;                       // colour of the pair's first cell
    // the x neighbour outside the pair (of a single cell: itself)
    xo[q][0] = two[q] ? (i == 0 ? L.nx - 1 : -1) : 0;
    xo[q][1] = i + 2 >= L.nx ? 1 - L.nx : 1;
    ym[q] = ((j == 0) ? L.ny - 1 : -1) * L.nx;
    yp[q] = ((j == L.ny - 1) ? 1 - L.ny : 1) * L.nx;
    const PlaneCoef<T> c = ldg_struct(a.coef + L.coef_off + k);
    cx[q] = c.cx; cy[q] = c.cy;
    cl[q] = k > 0 ? c.czlo : T(0);
    ch[q] = k < L.nz - 1 ? c.czhi : T(0);
    zl[q] = k > 0 ? -plane : 0;                 // times a zero coupling at the electrodes
    zh[q] = k < L.nz - 1 ? plane : 0;
    // FP64 divides by the shifted diagonal, FP32 multiplies by its reciprocal (over_shifted)
    div[q] = sizeof(T) == sizeof(double) && c.has_s;
#pragma unroll
    for (int w = 0; w < 2; ++w) {
      const int t2 = id[q] + (w && two[q] ? 1 : 0);
      r[q][w] = a.r[L.off + t2];
      if (!c.has_s) inv[q][w] = c.invdiag;
      else if constexpr (sizeof(T) == sizeof(float)) inv[q][w] = T(1) / (c.diag + a.s[L.off + t2]);
      else inv[q][w] = c.diag + a.s[L.off + t2];
      v[q][w] = T(0);
      e[t2] = T(0);
    }
  }
  __syncthreads();
  for (int sw = 0; sw < sweeps; ++sw)
#pragma unroll
    for (int color = 0; color < 2; ++color) {
#pragma unroll
      for (int q = 0; q < ITEMS; ++q) {
        if (par[q] < 0) continue;
        const int w = par[q] ^ color;            // which cell of the pair has this colour
        if (w && !two[q]) continue;
        const int t = id[q] + w;
        const T own = two[q] ? (w ? v[q][0] : v[q][1]) : v[q][0];
        T acc = w ? r[q][1] : r[q][0];
        acc = fma(cx[q], e[t + (w ? xo[q][1] : xo[q][0])] + own, acc);
        acc = fma(cy[q], e[t + ym[q]] + e[t + yp[q]], acc);
        acc = fma(cl[q], e[t + zl[q]], acc);
        acc = fma(ch[q], e[t + zh[q]], acc);
        const T d = w ? inv[q][1] : inv[q][0];
        const T x = div[q] ? acc / d : acc * d;
        if (w) v[q][1] = x;
        else v[q][0] = x;
        e[t] = x;
      }
      __syncthreads();
    }
}

// e = A^-1 r on a level of n <= kDenseMax cells: the inverse (row-major, computed
// on the host in FP64) times r, four lanes per row and a fixed-order reduction.
template <typename T>
__device__ void tail_dense(const T* __restrict__ inv, int n, const T* r, T* e) {
  const int tid = threadIdx.x;
  if ((tid >> 5) < ((4 * n + 31) >> 5)) {   // whole warps, for the shuffles
    const int row = tid >> 2, p = tid & 3;
    T acc = T(0);
    if (row < n)
      for (int c = p; c < n; c += 4) acc = fma(__ldg(inv + row * n + c), r[c], acc);
    acc += __shfl_xor_sync(0xffffffffu, acc, 1);
    acc += __shfl_xor_sync(0xffffffffu, acc, 2);
    if (row < n && p == 0) e[row] = acc;
  }
  __syncthreads();
}

// A complete V-cycle over the tail levels of one instance, by one CTA, with the
// level arrays in shared memory (smem holds 2 or 3 arrays of t.elems values).
// With t.dense the level t.dense_lev is solved exactly by its inverse and the
// levels below it are not visited; otherwise the coarsest level is relaxed
// t.bottom_sweeps times.
template <typename T>
__device__ FX_TAIL_LINKAGE void tail_vcycle(const MGArgs<T>& g, const TailArgs& t, unsigned char* tail_smem) {
  T* se = reinterpret_cast<T*>(tail_smem);
  T* sr = se + t.elems;
  T* ss = g.s ? sr + t.elems : nullptr;
  const LevelDesc* lv = t.lv;
  const int n0 = (int)lv[0].ncell;
  for (int q = threadIdx.x; q < n0; q += blockDim.x) {
    sr[q] = g.r[t.base + q];
    if (ss) ss[q] = g.s[t.base + q];
  }
  __syncthreads();
  MGArgs<T> a;
  a.e = se; a.r = sr; a.s = ss; a.coef = g.coef; a.lv = lv;
  const int bottom = t.dense ? t.dense_lev : t.nlev - 1;
  for (int l = 0; l < bottom; ++l) {
    const LevelDesc F = ldg_struct(lv + l), C = ldg_struct(lv + l + 1);
    tail_smooth(a, F, t.nu1, 1);
    const int nc = (int)C.ncell;
    const unsigned long long mx = magic32(C.nx), my = magic32(C.ny);
    const int skip = black_residual_zero(F, t.nu1);
    for (int q = threadIdx.x; q < nc; q += blockDim.x) {
      const int rest = div32(q, mx), K = div32(rest, my);
      restrict_cell(a, F, C, q - rest * C.nx, rest - K * C.ny, K, skip);
    }
    __syncthreads();
  }
  if (t.dense) {
    const LevelDesc B = ldg_struct(lv + bottom);
    tail_dense(static_cast<const T*>(t.dense), (int)B.ncell, sr + B.off, se + B.off);
  } else {
    const LevelDesc B = ldg_struct(lv + bottom);
    if (t.bottom_sweeps >= kTailHeldSweeps && ((B.nx + 1) >> 1) * B.ny * B.nz <= 2 * (int)blockDim.x)
      tail_smooth_held(a, B, t.bottom_sweeps);
    else
      tail_smooth(a, B, t.bottom_sweeps, 1);
  }
  for (int l = bottom - 1; l >= 0; --l) {
    const LevelDesc F = ldg_struct(lv + l), C = ldg_struct(lv + l + 1);
    const int nf = (int)F.ncell;
    const unsigned long long mx = magic32(F.nx), my = magic32(F.ny);
    for (int q = threadIdx.x; q < nf; q += blockDim.x) {
      const int rest = div32(q, mx), k = div32(rest, my);
      prolong_fine(a, F, C, q - rest * F.nx, rest - k * F.ny, k, t.constant);
    }
    __syncthreads();
    tail_smooth(a, F, t.nu2, 0);
  }
  for (int q = threadIdx.x; q < n0; q += blockDim.x) g.e[t.base + q] = se[q];
}

__device__ __forceinline__ double warp_sum(double v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Block sum of one value; result valid in thread 0.
__device__ __forceinline__ void block_sum1(double& x) {
  __shared__ double sh1[32];
  const int tid = threadIdx.x + threadIdx.y * blockDim.x;
  const int nthr = blockDim.x * blockDim.y;
  x = warp_sum(x);
  const int w = tid >> 5, l = tid & 31;
  if (l == 0) sh1[w] = x;
  __syncthreads();
  if (w == 0) x = warp_sum(l < ((nthr + 31) >> 5) ? sh1[l] : 0.0);
  __syncthreads();
}

// Block sum of three values; result valid in thread 0.
__device__ __forceinline__ float warp_sum_f(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// FP32 block sums of two per-thread values (the double-float residual's norms, which
// decide a tolerance: FP32 sums within a block are ample); valid in thread 0
__device__ __forceinline__ void block_sum2f(float& x, float& y) {
  __shared__ float shf[2][32];
  const int tid = threadIdx.x + threadIdx.y * blockDim.x;
  const int nthr = blockDim.x * blockDim.y;
  x = warp_sum_f(x); y = warp_sum_f(y);
  const int w = tid >> 5, l = tid & 31;
  if (l == 0) { shf[0][w] = x; shf[1][w] = y; }
  __syncthreads();
  const int nw = (nthr + 31) >> 5;
  if (w == 0) {
    x = l < nw ? shf[0][l] : 0.0f;
    y = l < nw ? shf[1][l] : 0.0f;
    x = warp_sum_f(x); y = warp_sum_f(y);
  }
  __syncthreads();
}

__device__ __forceinline__ void block_sum3(double& x, double& y, double& z) {
  __shared__ double sh[3][32];
  const int tid = threadIdx.x + threadIdx.y * blockDim.x;
  const int nthr = blockDim.x * blockDim.y;
  x = warp_sum(x); y = warp_sum(y); z = warp_sum(z);
  const int w = tid >> 5, l = tid & 31;
  if (l == 0) { sh[0][w] = x; sh[1][w] = y; sh[2][w] = z; }
  __syncthreads();
  const int nw = (nthr + 31) >> 5;
  if (w == 0) {
    x = l < nw ? sh[0][l] : 0.0;
    y = l < nw ? sh[1][l] : 0.0;
    z = l < nw ? sh[2][l] : 0.0;
    x = warp_sum(x); y = warp_sum(y); z = warp_sum(z);
  }
  __syncthreads();
}

// FP64 -> FP32 store of the outer residual (mixed form) by integer truncation:
// sign, rebiased exponent and the top 23 mantissa bits, rounding toward zero
// (within 1 FP32 ulp; the FP64 defect correction absorbs it).  Magnitudes below
// the FP32 normal range store a signed zero, above it (and NaN) infinity; the
// norms and the convergence decision use the FP64 value.  The conversion
// instruction would run on the FP64 pipe that bounds this kernel.
template <typename T>
__device__ __forceinline__ T narrow_resid(double x) {
  if (sizeof(T) == sizeof(float)) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    const unsigned sign = (unsigned)(b >> 32) & 0x80000000u;
    const int e = (int)((b >> 52) & 0x7ff) - 1023 + 127;
    if (e <= 0) return (T)__uint_as_float(sign);
    if (e >= 255) return (T)__uint_as_float(sign | 0x7f800000u);
    return (T)__uint_as_float(sign | ((unsigned)e << 23) | (unsigned)((b >> 29) & 0x7fffffu));
  }
  return (T)x;
}

// The same to the nearest float (ties away from zero), half the error and no bias: a run
// that takes several V-cycles per residual accepts corrections of about 1e-2 whose last
// bits come from here.
__device__ __forceinline__ float round_resid(double x) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(x), b = u + (1ull << 28);
  const unsigned sign = (unsigned)(u >> 32) & 0x80000000u;
  const int e = (int)((b >> 52) & 0x7ff) - 1023 + 127;
  if (e >= 255 || ((u >> 52) & 0x7ff) == 0x7ff) return __uint_as_float(sign | 0x7f800000u);
  if (e <= 0) return __uint_as_float(sign);
  return __uint_as_float(sign | ((unsigned)e << 23) | (unsigned)((b >> 29) & 0x7fffffu));
}

// Fermi-Dirac integral of order 1/2 (normalised to e^eta for eta -> -inf) and its
// derivative, by the approximation of Bednarczyk & Bednarczyk (1978) that the paper
// uses for the carrier integrals: F = 1/(e^-eta + xi), xi = (3 sqrt(pi)/4) v^(-3/8),
// v = eta^4 + 50 + 33.6 eta (1 - 0.68 e^(-0.17 (eta + 1)^2)).  Far below the band
// edge (eta < -700, where e^-eta overflows) F = e^eta to double precision.
__device__ __forceinline__ double fd_half(double eta, double& dF) {
  if (eta < -700.0) {
    dF = exp(eta);
    return dF;
  }
  const double g = exp(-0.17 * (eta + 1.0) * (eta + 1.0));
  const double w = fma(-0.68, g, 1.0);
  const double e2 = eta * eta;
  const double v = fma(e2, e2, fma(33.6 * eta, w, 50.0));
  const double dv = fma(4.0 * e2, eta, 33.6 * fma(eta * 0.2312 * g, eta + 1.0, w));
  const double xi = 1.3293403881791355 * exp(-0.375 * log(v));   // (3 sqrt(pi)/4) v^(-3/8)
  const double dxi = -0.375 * xi * dv / v;
  const double em = exp(-eta);
  const double F = 1.0 / (em + xi);
  dF = (em - dxi) * F * F;
  return F;
}

// The same for |eta| < 700 with em = e^-eta given, in a quarter of the FP64 operations:
//   * xi = c v^(-3/8) without log and exp: y = v^(-1/8) from FP32 to about 1e-6, one step of
//     Householder's third-order iteration, y (1 + h/8 + 9 h^2/128) with h = 1 - v y^8 (the
//     binomial series of (1 - h)^(-1/8), the next term is below 1e-17), and 1/v = y^8;
//   * the Gaussian in v is left out where 0.68 of it is below 2^-60 (it is next to 1).
constexpr double kFdGaussMax = 42.0;
__device__ __forceinline__ double fd_half_em(double eta, double em, double& dF) {
  const double e1 = __dadd_rn(eta, 1.0), q = __dmul_rn(__dmul_rn(0.17, e1), e1);
  double w = 1.0, d = 1.0;   // 1 - 0.68 g and the derivative of eta (1 - 0.68 g)
  if (q < kFdGaussMax) {
    const double g = exp_minus(q);
    w = fma(-0.68, g, 1.0);
    d = fma(__dmul_rn(__dmul_rn(eta, 0.2312), g), e1, w);
  }
  const double e2 = __dmul_rn(eta, eta);
  const double v = fma(e2, e2, fma(__dmul_rn(33.6, eta), w, 50.0));
  const double dv = fma(__dmul_rn(4.0, e2), eta, __dmul_rn(33.6, d));
  const double y0 = f64_of_float(exp2f(-0.125f * __log2f(df_from_double(v).h)));
  double y2 = __dmul_rn(y0, y0), y4 = __dmul_rn(y2, y2), y8 = __dmul_rn(y4, y4);
  const double h = fma(-v, y8, 1.0);
  const double y = fma(__dmul_rn(y0, h), fma(h, 9.0 / 128.0, 0.125), y0);
  y2 = __dmul_rn(y, y);
  y4 = __dmul_rn(y2, y2);
  y8 = __dmul_rn(y4, y4);
  const double xi = __dmul_rn(__dmul_rn(1.3293403881791355, y2), y);   // (3 sqrt(pi)/4) v^(-3/8)
  const double dxi = __dmul_rn(__dmul_rn(__dmul_rn(-0.375, xi), dv), y8);
  const double F = __drcp_rn(__dadd_rn(em, xi));
  dF = __dmul_rn(__dmul_rn(__dadd_rn(em, -dxi), F), F);
  return F;
}

// Carrier charge rho = kq (p - n + Nnet) of a semiconductor cell and the Newton shift
// -d rho/d phi, FP64.  Every rounding is spelled out, so that the residual's variants
// (and the two batched engines) agree bit for bit whatever they are inlined into.
template <int SC>
__device__ __forceinline__ void carrier_charge(const PlaneTDGL& pt, double phi, double& rho, double& shift) {
  const double u = __dmul_rn(phi, pt.inv_vt);
  double diff, sum;   // p - n; dp + dn in units of 1 / V_T
  if (SC == 2 && pt.fd) {
    // n = Nc F(eta_e0 + u), p = Nv F(eta_p0 - u); -d rho/d phi = kq (dn + dp)/VT
    // both exponentials from one reduction of u and e^-eta_e0, e^-eta_p0 of the host; the
    // general form where one of them could leave the range
    double dn, dp, Fe, Fp;
    const double ee = __dadd_rn(pt.eta_e0, u), ep = __dadd_rn(pt.eta_p0, -u);
    if (fabs(u) < 300.0 && fabs(pt.eta_e0) < 300.0 && fabs(pt.eta_p0) < 300.0) {
      double up, um;
      exp_pm(u, up, um);
      Fe = fd_half_em(ee, __dmul_rn(pt.em_e0, um), dn);
      Fp = fd_half_em(ep, __dmul_rn(pt.em_p0, up), dp);
    } else {
      Fe = fd_half(ee, dn);
      Fp = fd_half(ep, dp);
    }
    const double n = __dmul_rn(pt.Nc, Fe);
    diff = fma(pt.Nv, Fp, -n);
    sum = fma(pt.Nc, dn, __dmul_rn(pt.Nv, dp));
  } else {
    double ep, em;
    exp_pm(u, ep, em);
    const double n = __dmul_rn(pt.n0, ep);
    diff = fma(pt.p0, em, -n);
    sum = fma(pt.p0, em, n);
  }
  rho = __dmul_rn(pt.kq, __dadd_rn(diff, pt.Nnet));
  shift = __dmul_rn(__dmul_rn(pt.kq, sum), pt.inv_vt);
}

// FP64 residual of planes [k0, k1) of one (x, y) column, marching up with a
// register window; accumulates r^2, b^2 (first residual of a solve only) and
// rho^2.  SC = 0 compiles out the carrier term (stacks without a semiconductor
// layer), SC = 1 keeps Boltzmann statistics only, SC = 2 also Fermi-Dirac.
// The Newton shift of a level-0 cell, and with sinv_out the reciprocal of the
// shifted diagonal (in T, from the diagonal as the sweeps' T coefficients hold
// it), which the level-0 sweeps multiply by instead of dividing in every sweep.
template <typename T>
__device__ __forceinline__ void put_shift(const ResidArgs& a, long long t, double sv, T diag_t) {
  const T s = (T)sv;
  static_cast<T*>(a.s_out)[t] = s;
  if (a.sinv_out) static_cast<T*>(a.sinv_out)[t] = T(1) / (diag_t + s);
}

// the level-0 diagonal in T from its double-float pair (float: the high part is
// the nearest float)
template <typename T>
__device__ __forceinline__ T diag_of_df(const PlaneCoefDF& c) {
  if constexpr (sizeof(T) == sizeof(float)) return c.diag_h;
  else return (double)c.diag_h + (double)c.diag_l;
}

template <typename T, int SC = 2>
__device__ __forceinline__ void resid_column(const ResidArgs& a, int i, int j, int k0, int k1,
                                             double& acc_r, double& acc_b, double& acc_rho) {
  const int nx = a.nx, ny = a.ny, nz = a.nz;
  const long long plane = (long long)nx * ny;
  T* r_out = static_cast<T*>(a.r_out);
  T* s_out = static_cast<T*>(a.s_out);
  const double v_bot = a.params->v_bot, v_top = a.params->v_top;
  const int im = (i == 0) ? nx - 1 : i - 1, ip = (i == nx - 1) ? 0 : i + 1;
  const long long dxm = im - i, dxp = ip - i;
  const long long dym = (long long)((j == 0) ? ny - 1 : j - 1) * nx - (long long)j * nx;
  const long long dyp = (long long)((j == ny - 1) ? 0 : j + 1) * nx - (long long)j * nx;
  const double* phi = a.phi;
  const long long col = (long long)j * nx + i;
  double pd = k0 > 0 ? phi[(long long)(k0 - 1) * plane + col] : 0.0;
  double pc = phi[(long long)k0 * plane + col];
  for (int k = k0; k < k1; ++k) {
    const long long t = k * plane + col;
    const double pu = (k < nz - 1) ? phi[t + plane] : 0.0;
    const PlaneCoef<double> c = ldg_struct(a.coef0 + k);
    const PlaneTDGL pt = ldg_struct(a.planes + k);
    const double sx = phi[t + dxm] + phi[t + dxp];
    const double sy = phi[t + dym] + phi[t + dyp];
    double bb;
    if (pt.b_dyn) {
      bb = a.b[t];
    } else {
      bb = 0.0;
      if (k == 0) bb += pt.lift * v_bot;
      if (k == nz - 1) bb += pt.lift * v_top;
    }
    double rho = 0.0;
    if (SC && pt.sc) {
      double s;
      carrier_charge<SC>(pt, pc, rho, s);
      if (s_out) put_shift<T>(a, t, s, (T)c.diag);
      acc_rho = fma(rho, rho, acc_rho);
    }
    // r = b + rho - A phi = (b + rho) - diag phi + couplings * neighbours
    double r = fma(-c.diag, pc, SC ? __dadd_rn(bb, rho) : bb);
    r = fma(c.czhi, pu, r);
    r = fma(c.czlo, pd, r);
    r = fma(c.cy, sy, r);
    r = fma(c.cx, sx, r);
    r_out[t] = narrow_resid<T>(r);
    acc_r = fma(r, r, acc_r);
    if (a.first) acc_b = fma(bb, bb, acc_b);
    pd = pc;
    pc = pu;
  }
}

// The same residual of planes [k0, k1) of R rows (j0 .. j0 + R - 1) and the 32 cells of a
// warp: the operations of resid_column in the same order, with each potential loaded
// once per warp column (z neighbours from the march, x neighbours from the adjacent
// lanes, inner y neighbours from the thread's other rows) instead of five times.  The
// FP64 pipe bounds it: seven operations per cell and one for the FP64 norm.  Every lane of
// the warp has to call it; `in` marks those that hold a cell.
//   DFC: Boltzmann carriers in double-float on the FP32 pipe, beside the FP64 stencil (the
//     mixed form), added to the FP64 sum as pairs: FP32 and FP64 pipes overlap, and the
//     exponentials cost no FP64 instruction.
//   ROUND: the FP32 residual rounded to nearest (the single stack's mixed form).
//   N: the type of the squared norms (float where they decide a tolerance from an FP32
//     residual, as in resid_column_df).
template <typename T, int SC, bool DFC, int R, typename N, bool ROUND = false>
__device__ __forceinline__ void resid_rows(const ResidArgs& a, int i, int j0, int k0, int k1, bool in, N& acc_r,
                                           N& acc_b, double& acc_rho) {
  const int nx = a.nx, ny = a.ny, nz = a.nz;
  const long long plane = (long long)nx * ny;
  T* r_out = static_cast<T*>(a.r_out);
  T* s_out = static_cast<T*>(a.s_out);
  // electrode lift of static boundary planes (nz >= 2: two planes)
  double lift_bot = 0.0, lift_top = 0.0;
  if (k0 == 0) lift_bot = __ldg(&a.planes[0].lift) * a.params->v_bot;
  if (k1 == nz) lift_top = __ldg(&a.planes[nz - 1].lift) * a.params->v_top;
  const int lane = threadIdx.x & 31;
  const int x = in ? i : 0, y = in ? j0 : 0;         // idle lanes read cell 0 of the plane
  const bool edge_m = lane == 0, edge_p = lane == 31 || i == nx - 1;
  const long long col = (long long)y * nx + x;
  const long long dxm = (x == 0) ? nx - 1 : -1, dxp = (x == nx - 1) ? 1 - nx : 1;
  const long long lo = (long long)((y == 0) ? ny - 1 : y - 1) * nx + x;
  const long long hi = (long long)((y + R >= ny) ? 0 : y + R) * nx + x;
  const double* phi = a.phi;
  float rho2f = 0.0f;   // rho^2 of the double-float carriers (enters only the scale of the test)
  double pd[R], pc[R];
#pragma unroll
  for (int q = 0; q < R; ++q) {
    pd[q] = k0 > 0 ? phi[(long long)(k0 - 1) * plane + col + (long long)q * nx] : 0.0;
    pc[q] = phi[(long long)k0 * plane + col + (long long)q * nx];
  }
  for (int k = k0; k < k1; ++k) {
    const long long o = k * plane;
    const PlaneCoef<double> c = ldg_struct(a.coef0 + k);
    const PlaneTDGL* pk = a.planes + k;
    const int b_dyn = __ldg(&pk->b_dyn);
    const double ylo = phi[o + lo], yhi = phi[o + hi];
    const bool sc = SC && __ldg(&pk->sc);
    PlaneTDGL pt;
    PlaneCarrierDF cd;
    float diag_f = 0.0f;
    if (sc) {
      pt = ldg_struct(pk);
      if (DFC) {
        cd = ldg_struct(a.carriers_df + k);
        diag_f = (float)c.diag;
      }
    }
    double pu[R], bb[R];
#pragma unroll
    for (int q = 0; q < R; ++q) {
      const long long t = o + col + (long long)q * nx;
      pu[q] = (k < nz - 1) ? phi[t + plane] : 0.0;
      bb[q] = b_dyn ? a.b[t] : k == 0 ? lift_bot : k == nz - 1 ? lift_top : 0.0;
    }
#pragma unroll
    for (int q = 0; q < R; ++q) {
      const long long t = o + col + (long long)q * nx;
      double xm = __shfl_up_sync(0xffffffffu, pc[q], 1), xp = __shfl_down_sync(0xffffffffu, pc[q], 1);
      if (edge_m) xm = phi[t + dxm];
      if (edge_p) xp = phi[t + dxp];
      const double sx = xm + xp;
      const double sy = (q ? pc[q - 1] : ylo) + (q < R - 1 ? pc[q + 1] : yhi);
      double b_rho = bb[q];
      df rho_df{0.0f, 0.0f};
      bool add_df = false;
      if (sc) {
        df u{0.0f, 0.0f};
        if (DFC) u = df_mul(df_from_double(pc[q]), df{cd.inv_vt_h, cd.inv_vt_l});
        if (DFC && !(SC == 2 && pt.fd) && fabsf(u.h) <= kExpDFMax) {
          // rho = kq p0 e^{-u} - kq n0 e^{u} + kq Nnet, u = phi / V_T
          df ep, em;
          exp_pm_df(u, ep, em);
          const df kn = df_mul(df{cd.kqn0_h, cd.kqn0_l}, ep);
          const df kp = df_mul(df{cd.kqp0_h, cd.kqp0_l}, em);
          rho_df = df_add(df_add(kp, df_neg(kn)), df{cd.kqN_h, cd.kqN_l});
          add_df = true;
          if (in) rho2f = fmaf(rho_df.h, rho_df.h, rho2f);
          if (s_out && in) {
            const float sv = (kn.h + kp.h) * cd.inv_vt_h;
            s_out[t] = (T)sv;
            if (a.sinv_out) static_cast<T*>(a.sinv_out)[t] = (T)(1.0f / (diag_f + sv));
          }
        } else {
          double s, rho;
          carrier_charge<SC>(pt, pc[q], rho, s);
          b_rho = __dadd_rn(b_rho, rho);
          if (in) {
            acc_rho = fma(rho, rho, acc_rho);
            if (s_out) put_shift<T>(a, t, s, (T)c.diag);
          }
        }
      }
      // r = b + rho - A phi = (b + rho) - diag phi + couplings * neighbours
      double r = fma(-c.diag, pc[q], b_rho);
      r = fma(c.czhi, pu[q], r);
      r = fma(c.czlo, pd[q], r);
      r = fma(c.cy, sy, r);
      r = fma(c.cx, sx, r);
      float rf = 0.0f;
      if (DFC && add_df) {
        rf = df_add(df_from_double(r), rho_df).h;
        if (in) r_out[t] = (T)rf;
      } else {
        T rt;
        if constexpr (ROUND) rt = round_resid(r);
        else rt = narrow_resid<T>(r);
        if (in) r_out[t] = rt;
        rf = (float)rt;
      }
      if (in) {
        if constexpr (sizeof(N) == sizeof(float)) {
          acc_r = fmaf(rf, rf, acc_r);
          if (a.first) {
            const float bf = df_from_double(bb[q]).h;
            acc_b = fmaf(bf, bf, acc_b);
          }
        } else {
          acc_r = fma(r, r, acc_r);
          if (a.first) acc_b = fma(bb[q], bb[q], acc_b);
        }
      }
    }
#pragma unroll
    for (int q = 0; q < R; ++q) {
      pd[q] = pc[q];
      pc[q] = pu[q];
    }
  }
  if (DFC) acc_rho += (double)rho2f;
}

// The same residual with the stencil in double-float arithmetic too (df_arith.cuh), for
// the diagnostic entry: the potentials, the right-hand side b + rho and the coefficients
// enter as h + l pairs, the products and sums keep about 48 bits, so r agrees with the
// FP64 residual to a few 2^-48 of the largest term.
template <typename T, int SC>
__device__ __forceinline__ void resid_column_df(const ResidArgs& a, int i, int j, int k0, int k1,
                                                float& acc_r, float& acc_b, double& acc_rho) {
  const int nx = a.nx, ny = a.ny, nz = a.nz;
  const long long plane = (long long)nx * ny;
  T* r_out = static_cast<T*>(a.r_out);
  T* s_out = static_cast<T*>(a.s_out);
  const double v_bot = a.params->v_bot, v_top = a.params->v_top;
  const int im = (i == 0) ? nx - 1 : i - 1, ip = (i == nx - 1) ? 0 : i + 1;
  const long long dxm = im - i, dxp = ip - i;
  const long long dym = (long long)((j == 0) ? ny - 1 : j - 1) * nx - (long long)j * nx;
  const long long dyp = (long long)((j == ny - 1) ? 0 : j + 1) * nx - (long long)j * nx;
  const double* phi = a.phi;
  const long long col = (long long)j * nx + i;
  double pc_d = phi[(long long)k0 * plane + col];
  df pd = k0 > 0 ? df_from_double(phi[(long long)(k0 - 1) * plane + col]) : df{0.0f, 0.0f};
  df pc = df_from_double(pc_d);
  float rho2f = 0.0f;   // rho^2 of the double-float carrier path (enters only the scale of the test)
  for (int k = k0; k < k1; ++k) {
    const long long t = k * plane + col;
    const double pu_d = (k < nz - 1) ? phi[t + plane] : 0.0;
    const df pu = df_from_double(pu_d);
    const PlaneCoefDF c = ldg_struct(a.coef_df + k);
    // only the plane fields this cell needs (the whole record is 28 words)
    const PlaneTDGL* pk = a.planes + k;
    const int b_dyn = __ldg(&pk->b_dyn);
    // x neighbours: the centre pairs of the neighbouring lanes when a warp holds 32
    // cells of one row (the row's ends convert their own)
    df xm, xp;
    if (a.warp_rows) {
      const int lane = threadIdx.x & 31;
      xm.h = __shfl_up_sync(0xffffffffu, pc.h, 1);
      xm.l = __shfl_up_sync(0xffffffffu, pc.l, 1);
      xp.h = __shfl_down_sync(0xffffffffu, pc.h, 1);
      xp.l = __shfl_down_sync(0xffffffffu, pc.l, 1);
      if (lane == 0) xm = df_from_double(phi[t + dxm]);
      if (lane == 31) xp = df_from_double(phi[t + dxp]);
    } else {
      xm = df_from_double(phi[t + dxm]);
      xp = df_from_double(phi[t + dxp]);
    }
    const df sx = df_add_fast(xm, xp);
    const df sy = df_add_fast(df_from_double(phi[t + dym]), df_from_double(phi[t + dyp]));
    double bb;
    if (b_dyn) {
      bb = a.b[t];
    } else {
      bb = 0.0;
      if (k == 0) bb += __ldg(&pk->lift) * v_bot;
      if (k == nz - 1) bb += __ldg(&pk->lift) * v_top;
    }
    df b_df = df_from_double(bb);
    if (SC && __ldg(&pk->sc)) {
      const PlaneTDGL pt = ldg_struct(pk);
      // Boltzmann densities in double-float on the FP32 pipe while |u| <= kExpDFMax:
      // rho = kq p0 e^{-u} - kq n0 e^{u} + kq Nnet, u = phi / V_T
      const df inv_vt = df_from_double(pt.inv_vt);
      const df u = df_mul(pc, inv_vt);
      if (!(SC == 2 && pt.fd) && fabsf(u.h) <= kExpDFMax) {
        df ep, em;
        exp_pm_df(u, ep, em);
        const df kn = df_mul(df_from_double(pt.kqn0), ep);
        const df kp = df_mul(df_from_double(pt.kqp0), em);
        const df rho = df_add(df_add(kp, df_neg(kn)), df_from_double(pt.kqN));
        b_df = df_add(b_df, rho);
        rho2f = fmaf(rho.h, rho.h, rho2f);
        if (s_out) {
          const float sv = (kn.h + kp.h) * inv_vt.h;
          s_out[t] = (T)sv;
          if (a.sinv_out) static_cast<T*>(a.sinv_out)[t] = (T)(1.0f / (c.diag_h + sv));
        }
      } else {
        double rho;
        double s;
        carrier_charge<SC>(pt, pc_d, rho, s);
        if (s_out) put_shift<T>(a, t, s, diag_of_df<T>(c));
        b_df = df_from_double(bb + rho);
        acc_rho = fma(rho, rho, acc_rho);
      }
    }
    // r = ((b + rho) - diag phi) + (z couplings) + (lateral couplings), as a tree
    const df r0 = df_add_fast(b_df, df_neg(df_mul(df{c.diag_h, c.diag_l}, pc)));
    const df rz = df_add_fast(df_mul(df{c.czhi_h, c.czhi_l}, pu), df_mul(df{c.czlo_h, c.czlo_l}, pd));
    const df rl = df_add_fast(df_mul(df{c.cy_h, c.cy_l}, sy), df_mul(df{c.cx_h, c.cx_l}, sx));
    const df r = df_add_fast(df_add_fast(r0, rz), rl);
    if (sizeof(T) == sizeof(float))
      r_out[t] = (T)r.h;
    else
      r_out[t] = (T)((double)r.h + (double)r.l);
    acc_r = fmaf(r.h, r.h, acc_r);
    if (a.first) {
      const float bh = df_from_double(bb).h;
      acc_b = fmaf(bh, bh, acc_b);
    }
    pd = pc;
    pc = pu;
    pc_d = pu_d;
  }
  if (SC) acc_rho += (double)rho2f;
}

// Convergence decision of one solve from its summed norms (one thread).
__device__ __forceinline__ int decide(DevStats* st, double sr, double sb, double sq, int first,
                                      double tol, int max_cycles, int launches_per_cycle,
                                      int adapt_max = 0, int launches_per_vcycle = 0,
                                      int inner_fixed = 1) {
  if (first) {
    st->solves += 1;
    st->cycles_this_solve = 0;
    st->zero_phi = 0;
    st->launches += 1;
    st->bnorm2 = sb;          // b is fixed during a solve
  }
  const double rn = sqrt(sr);
  const double scale = fmax(sqrt(st->bnorm2), sqrt(sq));
  int cond;
  if (!isfinite(rn) || !isfinite(scale)) {
    if (st->status == 0) st->status = FERROX_ENONFINITE;
    cond = 0;
  } else if (rn <= tol * scale) {
    cond = 0;
  } else if (st->cycles_this_solve >= max_cycles) {
    if (st->status == 0) st->status = FERROX_ENOCONV;
    cond = 0;
  } else {
    // scale == 0 with r != 0: b = 0 and rho(phi) = 0, whose solution is phi = 0
    if (scale == 0.0) st->zero_phi = 1;
    cond = 1;
  }
  if (cond) {
    st->cycles_this_solve += 1;
    st->cycles += 1;
    st->launches += launches_per_cycle;
    if (adapt_max <= 0) st->vcycles += inner_fixed;
  }
  if (adapt_max > 0 && !first && st->inner_k > 0 && st->prev_rnorm > 0.0 && rn > 0.0) {
    // contraction per V-cycle over the outer iteration just finished, measured
    // whether or not it reached the tolerance (kept for the next solves)
    st->rho_v = fmin(fmax(pow(rn / st->prev_rnorm, 1.0 / st->inner_k), 0.02), 0.9);
  }
  if (cond && adapt_max > 0) {
    // V-cycles for the next outer iteration: enough, at the estimated contraction
    // (0.2 before any measurement), to bring ||r|| to the tolerance
    const double rho = st->rho_v > 0.0 ? st->rho_v : 0.2;
    const double need = (rn > 0.0 && scale > 0.0) ? log(tol * scale / rn) / log(rho) : 1.0;
    const int k = (int)fmin(fmax(ceil(need), 1.0), (double)adapt_max);
    st->inner_k = k;
    st->inner_left = k;
    st->prev_rnorm = rn;
    st->launches += k * launches_per_vcycle;
    st->vcycles += k;
  }
  st->last_cond = cond;
  st->last_cycles = st->cycles_this_solve;
  st->last_rnorm = rn;
  st->last_scale = scale;
  st->last_rel = scale > 0.0 ? rn / scale : (rn > 0.0 ? INFINITY : 0.0);
  return cond;
}

}  // namespace dev
}  // namespace fx
