// Per-column device functions of the fused TDGL update (Eq. TDGL2) and the
// Poisson right-hand side, shared by tdgl.cu and the persistent batched engine.
// See tdgl.cu for the method.
#pragma once
#include <cuda_runtime.h>

#include "ferrox_internal.cuh"

namespace fx {
namespace dev {

__device__ __forceinline__ double landau(double a, double b, double g, double P) {
  const double P2 = P * P;
  return P * fma(P2, fma(g, P2, b), a);
}

// The FP64 update of P_z along a column, plane by plane upwards.  The face potential,
// polarization step and potential that a plane shares with the next one are kept, so each
// is computed and loaded once: 18 FP64 operations for the force and update of a cell and 4
// for its right-hand side (38 executed per cell before, with both faces of every cell
// evaluated on their own).  The gradient terms are formed from differences of P, so their
// roundings are relative to the terms and not to g/h^2 P, which is the larger by far in
// smooth domains (one operation more than with P's coefficients collected in `lin`).
// Every rounding is spelled out: all kernels that march, from whatever plane they start,
// agree bit for bit.
struct PzMarch {
  double P, dP, ph, face;    // of the plane updated next: P, its step from the plane below, potential, lower face potential
  bool ready = false;        // they are its own (the plane below was ferroelectric)
};

// potential of the face between planes k - 1 and k (f: plane k's table entry; dP: the step of P)
__device__ __forceinline__ double face_potential(const PlaneForce& f, double ph_lo, double ph_hi, double dP) {
  return fma(-f.fpc, dP, fma(f.fw_L, ph_lo, __dmul_rn(f.fw_R, ph_hi)));
}

// new P of ferroelectric plane k (cell t) of column (i, j)
__device__ __forceinline__ double advance_z(const TDGLArgs& a, PzMarch& m, const double* Pz, long long t, long long ti,
                                            int k, int i, int j, int im, int ip, int jm, int jp, double v_bot,
                                            double v_top) {
  const long long plane = (long long)a.nx * a.ny;
  const PlaneForce f = ldg_struct(a.force + k);
  if (!m.ready) {
    m.P = Pz[t];
    m.ph = a.phi[t];
    m.dP = __dadd_rn(m.P, -(k > 0 && __ldg(&a.force[k - 1].fe) ? Pz[t - plane] : 0.0));
    m.face = k == 0 ? v_bot : face_potential(f, a.phi[t - plane], m.ph, m.dP);
  }
  const double lat = __dadd_rn(__dadd_rn(Pz[t - i + im], Pz[t - i + ip]),
                               __dadd_rn(Pz[t + (long long)(jm - j) * a.nx], Pz[t + (long long)(jp - j) * a.nx]));
  double Pup = 0.0, dP_up = 0.0, ph_up = 0.0, face_up = v_top;
  bool fe_up = false;
  if (k < a.nz - 1) {
    const PlaneForce* u = a.force + k + 1;
    fe_up = __ldg(&u->fe);
    if (fe_up) Pup = Pz[t + plane];
    ph_up = a.phi[t + plane];
    PlaneForce fu;
    fu.fw_L = __ldg(&u->fw_L); fu.fw_R = __ldg(&u->fw_R); fu.fpc = __ldg(&u->fpc);
    dP_up = __dadd_rn(Pup, -m.P);
    face_up = face_potential(fu, m.ph, ph_up, dP_up);
  }
  const double P2 = __dmul_rn(m.P, m.P);
  double dF = __dmul_rn(m.P, fma(P2, fma(f.gamma, P2, f.beta), f.lin));
  dF = fma(f.w_dn, m.dP, dF);
  dF = fma(f.w_up, dP_up, dF);
  dF = fma(f.glat, fma(-4.0, m.P, lat), dF);
  dF = fma(__dadd_rn(face_up, -m.face), a.inv_h, dF);
  double pn;
  if (a.mode == 0) {
    pn = fma(f.gdt, dF, m.P);
  } else {
    const double fz = __dmul_rn(f.gam, dF);
    if (a.mode == 1) {
      a.F_store[ti] = fz;
      pn = fma(a.dt, fz, m.P);
    } else {
      pn = fma(0.5 * a.dt, __dadd_rn(a.F_store[ti], fz), a.P_base[ti]);
    }
  }
  m.dP = dP_up;
  m.P = Pup;
  m.ph = ph_up;
  m.face = face_up;
  m.ready = fe_up;
  return pn;
}

// polarization of the face below plane k from the new P of planes k - 1 and k (the cell's
// own on electrode faces)
__device__ __forceinline__ double face_polarization(const TDGLArgs& a, int k, double lo, double hi) {
  if (k == 0) return hi;
  if (k == a.nz) return lo;
  return fma(__ldg(&a.force[k].fw_R), lo, __dmul_rn(__ldg(&a.force[k].fw_L), hi));
}

// right-hand side of plane k from its two face polarizations
__device__ __forceinline__ double rhs_faces(const TDGLArgs& a, int k, double pf_dn, double pf_up, double v_bot,
                                            double v_top) {
  double b = __dmul_rn(__dadd_rn(pf_dn, -pf_up), a.b_scale);
  if (k == 0) b = fma(__ldg(&a.planes[0].lift), v_bot, b);
  if (k == a.nz - 1) b = fma(__ldg(&a.planes[a.nz - 1].lift), v_top, b);
  return b;
}

// One of CZ chunks of a column's dynamic planes (one component): the new P of its planes,
// and their right-hand sides; those of the chunk's first and last planes take the
// neighbouring chunks' edge values from shared memory (first_s, last_s: [CZ] of this
// column, STRIDE apart).  Every thread of the block has to call it.
template <int CZ>
__device__ __forceinline__ void tdgl_chunk(const TDGLArgs& a, int mode, int i, int j, bool col, int c, double* first_s,
                                           double* last_s, int stride) {
  const int per = (a.kd_hi - a.kd_lo + 1 + CZ - 1) / CZ;
  const int k0 = a.kd_lo + c * per, k1 = min(a.kd_hi, k0 + per - 1);   // empty when k0 > k1
  const long long plane = (long long)a.nx * a.ny, cix = (long long)j * a.nx + i;
  const double v_bot = a.params->v_bot, v_top = a.params->v_top;
  double p_first = 0.0, pm1 = 0.0, pf_second = 0.0, pf = 0.0;
  if (col && k0 <= k1) {
    const int im = (i == 0) ? a.nx - 1 : i - 1, ip = (i == a.nx - 1) ? 0 : i + 1;
    const int jm = (j == 0) ? a.ny - 1 : j - 1, jp = (j == a.ny - 1) ? 0 : j + 1;
    PzMarch m;
    for (int k = k0; k <= k1; ++k) {
      const long long t = k * plane + cix;
      double pn = 0.0;
      if (__ldg(&a.force[k].fe)) {
        if (mode == 3) {
          pn = a.P_in[t];
        } else {
          pn = advance_z(a, m, a.P_in, t, t, k, i, j, im, ip, jm, jp, v_bot, v_top);
          a.P_out[t] = pn;
        }
      } else {
        m.ready = false;
      }
      if (k == k0) {
        p_first = pn;
      } else {
        const double up = face_polarization(a, k, pm1, pn);
        if (k == k0 + 1) pf_second = up;
        else a.b[(k - 1) * plane + cix] = rhs_faces(a, k - 1, pf, up, v_bot, v_top);
        pf = up;
      }
      pm1 = pn;
    }
    first_s[c * stride] = p_first;
    last_s[c * stride] = pm1;
  }
  __syncthreads();
  if (!col || k0 > k1) return;
  const double below = k0 - 1 >= a.kd_lo ? last_s[(c - 1) * stride] : 0.0;
  const double above = k1 + 1 <= a.kd_hi ? first_s[(c + 1) * stride] : 0.0;
  const double pf_lo = face_polarization(a, k0, below, p_first), pf_hi = face_polarization(a, k1 + 1, pm1, above);
  a.b[k0 * plane + cix] = rhs_faces(a, k0, pf_lo, k1 == k0 ? pf_hi : pf_second, v_bot, v_top);
  if (k1 > k0) a.b[k1 * plane + cix] = rhs_faces(a, k1, pf, pf_hi, v_bot, v_top);
}

// in-plane component (3-component model): own Landau polynomial and dPhi/dx
// from in-plane face potentials (equal permittivity on both sides of the face)
__device__ __forceinline__ double force_xy(const TDGLArgs& a, const PlaneTDGL& pt,
                                           const PlaneTDGL* planes, const double* Pc,
                                           const double* phi, long long t, int k, int i, int j,
                                           int im, int ip, int jm, int jp, int comp,
                                           double inv_eps_abs) {
  const long long plane = (long long)a.nx * a.ny;
  const double P = Pc[t];
  const long long tm = comp == 0 ? t - i + im : t + (long long)(jm - j) * a.nx;
  const long long tp = comp == 0 ? t - i + ip : t + (long long)(jp - j) * a.nx;
  const double lat = (Pc[t - i + im] + Pc[t - i + ip]) +
                     (Pc[t + (long long)(jm - j) * a.nx] + Pc[t + (long long)(jp - j) * a.nx]);
  const bool fe_dn = k > 0 && __ldg(&planes[k - 1].fe);
  const bool fe_up = k < a.nz - 1 && __ldg(&planes[k + 1].fe);
  const double Pdn = fe_dn ? Pc[t - plane] : 0.0;
  const double Pup = fe_up ? Pc[t + plane] : 0.0;
  const double lap = fma(-4.0, P, lat) * a.inv_h2;
  const double d2z = fma(pt.wz_dn, Pdn, fma(pt.wz_c, P, pt.wz_up * Pup));
  // (Phi_f(+) - Phi_f(-))/h = (phi_p - phi_m)/(2h) - (P_p - 2P + P_m)/(4 eps)
  const double dphi = 0.5 * (phi[tp] - phi[tm]) * a.inv_h -
                      0.25 * (Pc[tp] - 2.0 * P + Pc[tm]) * inv_eps_abs;
  double dF = landau(pt.alpha_xy, pt.beta_xy, pt.gamma_xy, P);
  dF = fma(-pt.g44, lap, dF);
  dF = fma(-pt.g11, d2z, dF);
  dF += dphi;
  return -pt.Gamma * dF;
}

__device__ __forceinline__ double advance(const TDGLArgs& a, long long idx, double f) {
  if (a.mode == 0) return a.P_in[idx] + a.dt * f;
  if (a.mode == 1) {
    a.F_store[idx] = f;
    return a.P_in[idx] + a.dt * f;
  }
  return a.P_base[idx] + 0.5 * a.dt * (a.F_store[idx] + f);
}

__device__ __forceinline__ double rhs_value(const TDGLArgs& a, const PlaneTDGL* planes, int k,
                                            double pn_dn, double pn, double pn_up, double v_bot,
                                            double v_top) {
  const double Pf_dn =
      (k == 0) ? pn : fma(__ldg(&planes[k].fw_R), pn_dn, __ldg(&planes[k].fw_L) * pn);
  const double Pf_up = (k == a.nz - 1)
                           ? pn
                           : fma(__ldg(&planes[k + 1].fw_R), pn, __ldg(&planes[k + 1].fw_L) * pn_up);
  double b = -(Pf_up - Pf_dn) * a.b_scale;
  if (k == 0) b = fma(__ldg(&planes[0].lift), v_bot, b);
  if (k == a.nz - 1) b = fma(__ldg(&planes[a.nz - 1].lift), v_top, b);
  return b;
}

// One (x, y) column of the TDGL update: march up the dynamic planes, write the
// new P of the FE planes and (uniaxial) the right-hand side b of every dynamic plane.
__device__ __forceinline__ void tdgl_column(const TDGLArgs& a, int i, int j) {
  const int im = (i == 0) ? a.nx - 1 : i - 1, ip = (i == a.nx - 1) ? 0 : i + 1;
  const int jm = (j == 0) ? a.ny - 1 : j - 1, jp = (j == a.ny - 1) ? 0 : j + 1;
  const long long plane = (long long)a.nx * a.ny;
  const long long N = plane * a.nz;
  const long long col = (long long)j * a.nx + i;
  const double v_bot = a.params->v_bot, v_top = a.params->v_top;
  const PlaneTDGL* planes = a.planes;
  const double* Pz_in = a.P_in + (long long)(a.ncomp - 1) * N;
  PzMarch m;
  double pm1 = 0.0, pf = 0.0;   // new P of the plane below, polarization of its lower face
  for (int k = a.kd_lo; k <= a.kd_hi + 1; ++k) {
    double pn = 0.0;
    if (k <= a.kd_hi && __ldg(&a.force[k].fe)) {
      const long long t = k * plane + col;
      if (a.mode == 3) {
        pn = Pz_in[t];                        // right-hand side of the current P only
      } else {
        if (a.ncomp == 3) {
          const PlaneTDGL pt = ldg_struct(planes + k);
          const double inv_eps_abs = 1.0 / (8.8541878128e-12 * pt.eps_r);
          for (int c = 0; c < 2; ++c) {
            const double* Pc = a.P_in + (long long)c * N;
            const double f =
                force_xy(a, pt, planes, Pc, a.phi, t, k, i, j, im, ip, jm, jp, c, inv_eps_abs);
            a.P_out[c * N + t] = advance(a, c * N + t, f);
          }
        }
        const long long zi = (long long)(a.ncomp - 1) * N + t;
        pn = advance_z(a, m, Pz_in, t, zi, k, i, j, im, ip, jm, jp, v_bot, v_top);
        a.P_out[zi] = pn;
      }
    } else {
      m.ready = false;
    }
    if (a.ncomp == 1) {   // b of plane k - 1 once P(k) is known
      const double up = face_polarization(a, k, pm1, pn);
      if (k > a.kd_lo) a.b[(k - 1) * plane + col] = rhs_faces(a, k - 1, pf, up, v_bot, v_top);
      pf = up;
    }
    pm1 = pn;
  }
}

}  // namespace dev
}  // namespace fx
