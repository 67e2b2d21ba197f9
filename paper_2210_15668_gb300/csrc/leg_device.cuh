// One leg of a V-cycle on one level, FP32, in one pass over memory: the down leg
// (two red-black sweeps, residual, restriction) and the up leg (prolongation +
// correction, two red-black sweeps, on the fine level also phi += e), shared by the
// multi-kernel path (legs.cu) and the batched phases (persistent.cu).
//
// A colour sweep per launch reads and writes the level's arrays once per colour:
// ten launches and about 60 bytes per cell and V-cycle, each launch with a ramp of a
// few microseconds.  Here a block owns a lateral tile and marches up the planes; the
// sweeps follow one another one plane apart (a wavefront in z), so each array
// element is read and written once per leg.
//   * A thread owns a 2 x 2 column of cells (two rows, one red/black pair each), the
//     children of one coarse column: own-pair partners, own-row neighbours and all z
//     neighbours are registers; the other lateral neighbours come from shared
//     memory, where each stage publishes its colour of its newest plane.
//   * Step i relaxes red on plane i, black on i - 1, red on i - 2, black on i - 3 and
//     (down) takes the residual on i - 4.  A stage needs the previous stage's plane
//     above its own (computed earlier in the same step, in the same thread) and its
//     lateral neighbours on its own plane (published one step ago), so one barrier
//     per step suffices and two slots per stage alternate.  Four steps are unrolled:
//     plane parities and the rings of per-plane values are then fixed registers.
//   * Rows a and b of a thread are the two halves of packed FP32 operations (f32x2),
//     half the instructions of scalar ones.
//   * Latency bounds the loop: 8 to 16 warps an SM (92 to 140 registers a thread) issue in
//     20 to 46% of the cycles, and wait for the chain of stages, for shared memory and for
//     the barrier of a plane; 512x512x128 with a shift waits for memory (down 314 us for
//     530 MB from DRAM, up 225 us for 510 MB, timed one by one).
//   * The tile is surrounded by a halo of 2 HP cells whose values are recomputed
//     from the same inputs by the same operations as in the block that owns them;
//     each stage leaves one more ring of the halo stale, and the outputs are exact.
//     The same holds in z at chunk ends (kHaloZ planes).
//   * Gauss-Seidel overwrites a colour without reading it, so after the down leg
//     only the black values are needed again: they are stored alone (eb, half an
//     array), and the up leg prolongates onto black cells only.
// Every cell sees the operations of smooth_pair / cell_residual / prolong_cell in
// the same order: a leg equals the separate launches bit for bit (the relaxed values
// are rounded products, __fmul_rn, which the compiler may not fuse into the sums that
// read them from registers).
// Red cells are (i + j + k) even; lateral sizes must be even (periodic).
#pragma once
#include "mg_device.cuh"

namespace fx {
namespace dev {

// per-plane coefficients (zero outside the level, so that planes beyond the electrodes
// relax to zero)
struct LegCoef {
  float cx, cy, czlo, czhi;
  float diag, invdiag;
  int has_s, pad;
};

template <int TX, int TY, int HP_>
struct LegShape {
  static constexpr int HP = HP_;                       // halo in pairs / row pairs
  static constexpr int BX = TX / 2 + 2 * HP, BY = TY / 2 + 2 * HP;
  static constexpr int THREADS = BX * BY;
  // row pitch: the two-row stride of consecutive thread rows continues the bank
  // sequence of a row (2 pitch = BX mod 32), so a warp's accesses spread over the banks
  static constexpr int pitch_() {
    int p = BX + 2;
    while ((2 * p - BX) % 32) ++p;
    return p;
  }
  static constexpr int PITCH = (BX % 2) ? BX + 2 : pitch_();
  static constexpr int PLANE = (2 * BY + 2) * PITCH;   // one published colour of one plane
};

// Blocks per SM the register allocation has to allow: with a Newton shift or the phi update
// 16 warps (128 registers instead of 130 to 150, one 240-thread block per SM otherwise);
// the others keep the 72 to 124 registers they ask for (80 forced: 256x256x32
// mixed step 5.65 -> 6.14 ms for five solves)
__host__ __device__ constexpr int leg_min_blocks(int threads, bool cap) {
  const int w = (threads + 31) / 32;
  return cap && w < 16 ? 16 / w : 1;
}

constexpr int kLegHaloZ = 6;      // planes recomputed below a z chunk at most (even)
constexpr int kLegLag = 4;        // deepest stage's lag behind the newest relaxed plane
// coefficient planes a chunk touches: from kLegLag below its first recomputed plane to
// the planes the last unrolled steps look ahead to
__host__ __device__ constexpr int leg_coef_planes(int kz) { return kz + kLegHaloZ + 2 * kLegLag + 8; }

template <int TX, int TY, int HP>
__host__ __device__ constexpr size_t leg_smem_bytes(int stages, int kz) {
  return (size_t)leg_coef_planes(kz) * sizeof(LegCoef) + (size_t)stages * 2 * LegShape<TX, TY, HP>::PLANE * sizeof(float);
}

__device__ __forceinline__ float2 both(float x) { return make_float2(x, x); }

// numerators r + sum of couplings * neighbours of the RED (or black) cells of a
// thread's two rows on a plane of parity P: S the published plane of the other
// colour, lo / cu / hi the thread's own values of it one plane below / here / above
template <bool RED, int P>
__device__ __forceinline__ float2 leg_num(const float* S, int my, int pitch, float2 lo, float2 cu, float2 hi, float2 r,
                                          const LegCoef& c) {
  // x neighbour outside the own pair: of the left pair where the cell is the pair's first
  constexpr int o = (RED == (P == 1)) ? 1 : -1;
  const float2 x = make_float2(S[my + o], S[my + pitch - o]);
  const float2 sy = make_float2(S[my - pitch] + cu.y, cu.x + S[my + 2 * pitch]);
  float2 n = __ffma2_rn(both(c.cx), __fadd2_rn(cu, x), r);
  n = __ffma2_rn(both(c.cy), sy, n);
  n = __ffma2_rn(both(c.czlo), lo, n);
  return __ffma2_rn(both(c.czhi), hi, n);
}

// position of a thread in the level (periodic images of the tile and its halo)
struct LegPos {
  int my;            // shared-memory index of the upper row (row a)
  int base;          // cell index of row a's pair in a plane
  int hbase;         // index of row a's pair in a plane of pairs
  int cbase;         // index of the thread's coarse column in a coarse plane
  bool own;          // inside the tile and the level
};

template <typename G>
__device__ __forceinline__ LegPos leg_pos(int tid, int bx, int by, int nx, int ny) {
  const int tx = tid % G::BX, ty = tid / G::BX;
  const int hx = nx >> 1, hy = ny >> 1;
  constexpr int tpx = G::BX - 2 * G::HP, tpy = G::BY - 2 * G::HP;
  const int ux = bx * tpx - G::HP + tx, uy = by * tpy - G::HP + ty;
  int px = ux % hx, py = uy % hy;
  if (px < 0) px += hx;
  if (py < 0) py += hy;
  LegPos q;
  q.my = (1 + 2 * ty) * G::PITCH + 1 + tx;
  q.base = (2 * py) * nx + 2 * px;
  q.hbase = (2 * py) * hx + px;
  q.cbase = py * hx + px;
  q.own = tx >= G::HP && tx < G::BX - G::HP && ty >= G::HP && ty < G::BY - G::HP && ux < hx && uy < hy;
  return q;
}

// coefficients of planes p0 .. p0 + n - 1 into shared memory
__device__ __forceinline__ void leg_load_coef(LegCoef* C, const PlaneCoef<float>* coef, int p0, int n, int nz, int tid,
                                              int threads) {
  for (int q = tid; q < n; q += threads) {
    const int p = p0 + q;
    LegCoef c{0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0, 0};
    if (p >= 0 && p < nz) {
      const PlaneCoef<float> g = ldg_struct(coef + p);
      c = LegCoef{g.cx, g.cy, g.czlo, g.czhi, g.diag, g.invdiag, g.has_s, 0};
    }
    C[q] = c;
  }
}

// the red (black) elements of rows a and b on a plane of parity P: the pair's first
// element is red in row a on even planes
template <bool RED, int P>
__device__ __forceinline__ float2 leg_sel(float2 a, float2 b) {
  return (P == 0) == RED ? make_float2(a.x, b.y) : make_float2(a.y, b.x);
}

// a pair row of plane n (zero beyond the level)
__device__ __forceinline__ void leg_fetch2(const float* p, int nx, bool in, float2& a, float2& b) {
  a = b = make_float2(0.f, 0.f);
  if (in) {
    a = *reinterpret_cast<const float2*>(p);
    b = *reinterpret_cast<const float2*>(p + nx);
  }
}

// Values of the two latest planes of a stage: cu on its consumer's plane, lo one below
struct LegWin {
  float2 lo, cu;
  __device__ __forceinline__ void push(float2 v) {
    lo = cu;
    cu = v;
  }
};

// What both legs keep per plane: right-hand sides and, with a Newton shift, the
// reciprocals 1 / (diag + s), as rings indexed by plane mod 4 (mod 2)
template <bool SC>
struct LegRing {
  float2 rr[4], rk[4];                    // right-hand sides: red, black
  float2 ir[SC ? 2 : 1], ik[SC ? 4 : 1];  // reciprocals: red (lags 0 and 2), black (lags 1 and 3)
  float2 ra[2], rb[2];                    // the next two planes in flight, rows a and b
  float2 ia[SC ? 2 : 1], ib[SC ? 2 : 1];

  template <int P>
  __device__ __forceinline__ void fetch(const LegArgs& a, const LegPos& q, int n, int plane, bool has_s) {
    const size_t o = (size_t)n * plane + q.base;
    leg_fetch2(a.r + o, a.nx, n < a.nz, ra[P], rb[P]);
    if (SC) leg_fetch2(a.sinv + o, a.nx, has_s, ia[P], ib[P]);
  }
  // plane i = Q mod 4 from its landed pairs; the red reciprocals of plane i - 2 leave
  template <int Q>
  __device__ __forceinline__ float2 take(float2 ra_, float2 rb_, float2 ia_, float2 ib_, const LegCoef& c) {
    constexpr int P = Q & 1;
    rr[Q] = leg_sel<true, P>(ra_, rb_);
    rk[Q] = leg_sel<false, P>(ra_, rb_);
    const float2 old = ir[SC ? P : 0];
    if (SC) {
      ir[SC ? P : 0] = c.has_s ? leg_sel<true, P>(ia_, ib_) : both(c.invdiag);
      ik[SC ? Q : 0] = c.has_s ? leg_sel<false, P>(ia_, ib_) : both(c.invdiag);
    }
    return old;
  }
};

// ---- down leg ------------------------------------------------------------------------
// CONT: the sweeps start from the corrections a.e_in (full array) instead of zero; their
// black values are published one plane ahead.
template <int TX, int TY, bool SC, bool CONT>
struct LegDown {
  using G = LegShape<TX, TY, CONT ? 3 : 2>;
  static constexpr int STAGES = CONT ? 5 : 4;   // published: red, black, red, black (, start)
  static constexpr int HALO_Z = CONT ? 6 : 4;

  static __host__ __device__ constexpr size_t smem_bytes(int kz) { return leg_smem_bytes<TX, TY, G::HP>(STAGES, kz); }

  struct State {
    LegRing<SC> g;
    LegWin w[4], we;                     // red, black, red, black sweeps; start
    float2 sa[SC ? 2 : 1], sb[SC ? 2 : 1];   // shifts in flight for the residual's next two planes
    float2 acc;                          // restriction: the even plane's red residuals
    float2 ua, ub;                       // ... and its shifts
    float2 ea[CONT ? 2 : 1], eb[CONT ? 2 : 1];   // starting corrections in flight
  };

  // step i, Q = i mod 4
  template <int Q>
  static __device__ __forceinline__ void step(const LegArgs& a, State& st, const LegPos& q, const LegCoef* C, float* S,
                                              int i, int z0, int z1, int plane) {
    constexpr int P = Q & 1;
    auto buf = [&](int stage, int par) { return S + (stage * 2 + par) * G::PLANE; };
    auto publish = [&](int stage, int par, float2 v) {
      float* W = buf(stage, par);
      W[q.my] = v.x;
      W[q.my + G::PITCH] = v.y;
    };
    LegRing<SC>& g = st.g;
    const LegCoef c0 = C[i], c4 = C[i - 4];
    const float2 ra = g.ra[P], rb = g.rb[P], ia = g.ia[SC ? P : 0], ib = g.ib[SC ? P : 0];
    g.template fetch<P>(a, q, i + 2, plane, SC && C[i + 2].has_s);   // in flight during two steps
    const float2 rr4 = g.rr[Q];                                      // plane i - 4
    const float2 ir2 = g.template take<Q>(ra, rb, ia, ib, c0);       // plane i - 2
    float2 d4 = both(c4.diag);
    if (SC) {
      const float2 sa = st.sa[SC ? P : 0], sb = st.sb[SC ? P : 0];
      leg_fetch2(a.s + (size_t)(i - 2) * plane + q.base, a.nx, C[i - 2].has_s, st.sa[SC ? P : 0], st.sb[SC ? P : 0]);
      d4 = __fadd2_rn(d4, leg_sel<true, P>(sa, sb));
      if (a.sc && q.own && i - 4 >= z0 && i - 4 < z1) {     // mean shift of the coarse cell
        if (!a.crz || P) {
          const float2 ua = st.ua, ub = st.ub;      // the even plane's
          float t;
          if (a.seq)
            t = a.crz ? ((((((ua.x + ua.y) + ub.x) + ub.y) + sa.x) + sa.y) + sb.x) + sb.y
                      : ((sa.x + sa.y) + sb.x) + sb.y;
          else
            t = a.crz ? ((ua.x + sa.x) + (ua.y + sa.y)) + ((ub.x + sb.x) + (ub.y + sb.y))
                      : (sa.x + sa.y) + (sb.x + sb.y);
          const int K = a.crz ? (i - 4) >> 1 : i - 4;
          const size_t o = (size_t)K * (plane >> 2) + q.cbase;
          t *= a.crz ? 0.125f : 0.25f;
          a.sc[o] = t;
          if (a.sinvc) a.sinvc[o] = 1.0f / (__ldg(&a.coefc[K].diag) + t);
        }
        st.ua = sa;
        st.ub = sb;
      }
    }
    // first red sweep, plane i
    float2 v;
    if (CONT) {
      const float2 hi = leg_sel<false, P ^ 1>(st.ea[P ^ 1], st.eb[P ^ 1]);   // start, plane i + 1
      const int n = i + 3;
      leg_fetch2(a.e_in + (size_t)n * plane + q.base, a.nx, n < a.nz, st.ea[P ^ 1], st.eb[P ^ 1]);
      publish(4, P ^ 1, hi);
      v = leg_num<true, P>(buf(4, P), q.my, G::PITCH, st.we.lo, st.we.cu, hi, g.rr[Q], c0);
      st.we.push(hi);
    } else {
      v = g.rr[Q];
    }
    v = __fmul2_rn(v, SC ? g.ir[SC ? P : 0] : both(c0.invdiag));
    publish(0, P, v);
    // first black sweep, plane i - 1
    const LegCoef c1 = C[i - 1];
    float2 b = leg_num<false, P ^ 1>(buf(0, P ^ 1), q.my, G::PITCH, st.w[0].lo, st.w[0].cu, v, g.rk[(Q + 3) & 3], c1);
    b = __fmul2_rn(b, SC ? g.ik[SC ? (Q + 3) & 3 : 0] : both(c1.invdiag));
    publish(1, P ^ 1, b);
    st.w[0].push(v);
    // second red sweep, plane i - 2
    const LegCoef c2 = C[i - 2];
    v = leg_num<true, P>(buf(1, P), q.my, G::PITCH, st.w[1].lo, st.w[1].cu, b, g.rr[(Q + 2) & 3], c2);
    v = __fmul2_rn(v, SC ? ir2 : both(c2.invdiag));
    publish(2, P, v);
    st.w[1].push(b);
    // second black sweep, plane i - 3: the level's black corrections
    const LegCoef c3 = C[i - 3];
    b = leg_num<false, P ^ 1>(buf(2, P ^ 1), q.my, G::PITCH, st.w[2].lo, st.w[2].cu, v, g.rk[(Q + 1) & 3], c3);
    b = __fmul2_rn(b, SC ? g.ik[SC ? (Q + 1) & 3 : 0] : both(c3.invdiag));
    publish(3, P ^ 1, b);
    if (q.own && i - 3 >= z0 && i - 3 < z1) {
      float* o = a.eb + (size_t)(i - 3) * (plane >> 1) + q.hbase;
      o[0] = b.x;
      o[a.nx >> 1] = b.y;
    }
    // residual of the red cells of plane i - 4, restricted
    const float2 n = leg_num<true, P>(buf(3, P), q.my, G::PITCH, st.w[3].lo, st.w[3].cu, b, rr4, c4);
    const float2 f = __ffma2_rn(make_float2(-d4.x, -d4.y), st.w[2].lo, n);   // w[2].lo: second red sweep there
    if (q.own && i - 4 >= z0 && i - 4 < z1 && (!a.crz || P)) {
      const float t = !a.crz ? f.x + f.y
                      : a.seq ? ((st.acc.x + st.acc.y) + f.x) + f.y
                              : (st.acc.x + f.x) + (st.acc.y + f.y);
      a.rc[(size_t)(a.crz ? (i - 4) >> 1 : i - 4) * (plane >> 2) + q.cbase] = t * (a.crz ? 0.125f : 0.25f);
    }
    st.acc = f;
    st.w[2].push(v);
    st.w[3].push(b);
    __syncthreads();
  }

  static __device__ __forceinline__ void run(const LegArgs& a, int bx, int by, int bz, unsigned char* smem) {
    const int tid = threadIdx.x;
    const int z0 = bz * a.kz, z1 = min(a.nz, z0 + a.kz);
    const int ps = max(0, z0 - HALO_Z), pe = z1 - 1 + kLegLag;
    const int ncoef = leg_coef_planes(a.kz);
    LegCoef* C0 = reinterpret_cast<LegCoef*>(smem);
    float* S = reinterpret_cast<float*>(smem + (size_t)ncoef * sizeof(LegCoef));
    const LegPos q = leg_pos<G>(tid, bx, by, a.nx, a.ny);
    const int plane = a.nx * a.ny;
    State st = {};
    if (!SC) {   // in flight while the coefficients arrive
      st.g.template fetch<0>(a, q, ps, plane, false);
      st.g.template fetch<1>(a, q, ps + 1, plane, false);
    }
    leg_load_coef(C0, a.coef, ps - kLegLag, ncoef, a.nz, tid, G::THREADS);
    for (int t = tid; t < STAGES * 2 * G::PLANE; t += G::THREADS) S[t] = 0.f;
    const LegCoef* C = C0 - (ps - kLegLag);
    __syncthreads();
    if (SC) {
      st.g.template fetch<0>(a, q, ps, plane, C[ps].has_s);
      st.g.template fetch<1>(a, q, ps + 1, plane, C[ps + 1].has_s);
    }
    if (CONT) {
      float2 ea, eb;
      const float* e = a.e_in + (size_t)ps * plane + q.base;
      leg_fetch2(e, a.nx, true, ea, eb);
      leg_fetch2(e + plane, a.nx, ps + 1 < a.nz, st.ea[1], st.eb[1]);
      leg_fetch2(e + 2 * plane, a.nx, ps + 2 < a.nz, st.ea[0], st.eb[0]);
      const float2 v = leg_sel<false, 0>(ea, eb);
      st.we.cu = v;
      float* W = S + 4 * 2 * G::PLANE;
      W[q.my] = v.x;
      W[q.my + G::PITCH] = v.y;
      __syncthreads();
    }
    // ps is even: z0 and the halo are
    if (ps & 2) {
      step<2>(a, st, q, C, S, ps, z0, z1, plane);
      step<3>(a, st, q, C, S, ps + 1, z0, z1, plane);
    }
    for (int i = ps + (ps & 2); i <= pe; i += 4) {
      step<0>(a, st, q, C, S, i, z0, z1, plane);
      step<1>(a, st, q, C, S, i + 1, z0, z1, plane);
      if (i + 2 > pe) break;
      step<2>(a, st, q, C, S, i + 2, z0, z1, plane);
      step<3>(a, st, q, C, S, i + 3, z0, z1, plane);
    }
  }
};

// ---- up leg --------------------------------------------------------------------------
// The prolongated black values of plane i + 1 are published at step i; the sweeps follow
// as in the down leg, and plane i - 3 leaves.  PHI: the fine level's last V-cycle of an
// outer iteration: phi += e (clamped) instead of storing e.
template <int TX, int TY, bool SC, bool PHI>
struct LegUp {
  using G = LegShape<TX, TY, 2>;
  static constexpr int STAGES = 4;              // published: red, black, red, prolongated black
  // coarse values interpolated in z for one fine plane: the block's columns and a ring around them
  static constexpr int ZP = G::BX + 2, ZPLANE = (G::BY + 2) * ZP;
  static constexpr int RING = 2 * (G::BX + 2) + 2 * G::BY;
  static_assert(RING <= G::THREADS, "one ring column per thread");

  static __host__ __device__ constexpr size_t smem_bytes(int kz) {
    return leg_smem_bytes<TX, TY, G::HP>(STAGES, kz) + 2 * (size_t)ZPLANE * sizeof(float);
  }

  struct State {
    LegRing<SC> g;
    LegWin w[4];           // prolongated black, red, black, red
    float2 e[2];           // black corrections in flight (by parity of their plane)
    float zc;              // own coarse column interpolated at the plane prolongated next
    float km, kc, kp;      // own coarse column: planes K - 1, K, K + 1
    float gm, gc, gp;      // the same of the thread's ring column
    double2 fa, fb;        // PHI: the potential of the next output plane
  };

  struct Cols {
    int own, ring;         // cell index of the own / ring coarse column in a coarse plane
    int zown, zring;       // their shared-memory places (ring: -1 when the thread has none)
  };

  // two neighbouring potentials, in one access where the caller's array is 16-byte aligned
  static __device__ __forceinline__ double2 load2(const double* p, int vec) {
    if (vec) return *reinterpret_cast<const double2*>(p);
    return make_double2(p[0], p[1]);
  }
  static __device__ __forceinline__ void store2(double* p, double2 v, int vec) {
    if (vec) {
      *reinterpret_cast<double2*>(p) = v;
    } else {
      p[0] = v.x;
      p[1] = v.y;
    }
  }

  // the coarse column's value on a fine plane of parity P (prolong_cell's z part)
  template <int P>
  static __device__ __forceinline__ float zint(const LegArgs& a, float m, float c, float p, int K) {
    if (!a.crz) return c;
    const float o = P ? p : m;
    const bool in = P ? K + 1 < a.ncz : K > 0;
    return in ? fmaf(0.75f, c, 0.25f * o) : 0.5f * c;
  }

  // interpolate plane n (parity P) of the own and ring columns into the slot of its parity;
  // moves the coarse windows when the coarse plane changes
  template <int P>
  static __device__ __forceinline__ void zplane(const LegArgs& a, State& st, const Cols& k, float* Z, int n, int cplane) {
    const int K = a.crz ? n >> 1 : n;
    if (!a.crz || P == 0) {   // a new coarse plane: its upper neighbour is requested
      st.km = st.kc;
      st.kc = st.kp;
      st.gm = st.gc;
      st.gc = st.gp;
      st.kp = st.gp = 0.f;
      if (K + 1 < a.ncz) {
        const float* e = a.ec + (size_t)(K + 1) * cplane;
        st.kp = e[k.own];
        if (k.zring >= 0) st.gp = e[k.ring];
      }
    }
    if (K >= a.ncz) {
      st.zc = 0.f;
      return;
    }
    st.zc = zint<P>(a, st.km, st.kc, st.kp, K);
    float* W = Z + P * ZPLANE;
    W[k.zown] = st.zc;
    if (k.zring >= 0) W[k.zring] = zint<P>(a, st.gm, st.gc, st.gp, K);
  }

  // black values of plane n (parity P) after the correction: y, then x (z was done a step ago)
  template <int P>
  static __device__ __forceinline__ float2 prolonged(const LegArgs& a, const State& st, const Cols& k, const float* Z,
                                                     float2 e, int n) {
    const float* R = Z + P * ZPLANE + k.zown;
    // the black cell of row a is the pair's second on even planes, its first on odd ones
    constexpr int o = P == 0 ? 1 : -1;
    const float zc = st.zc;
    const float2 y = __ffma2_rn(both(0.75f), both(zc), __fmul2_rn(both(0.25f), make_float2(R[-ZP], R[ZP])));
    const float2 yn = __ffma2_rn(both(0.75f), make_float2(R[o], R[-o]),
                                 __fmul2_rn(both(0.25f), make_float2(R[o - ZP], R[ZP - o])));
    const float2 v = __fadd2_rn(e, __ffma2_rn(both(0.75f), y, __fmul2_rn(both(0.25f), yn)));
    return n < a.nz ? v : make_float2(0.f, 0.f);
  }

  // black corrections of plane n in flight
  static __device__ __forceinline__ float2 fetch_e(const LegArgs& a, const LegPos& q, int n, int plane) {
    float2 e = make_float2(0.f, 0.f);
    if (n < a.nz) {
      const float* p = a.eb + (size_t)n * (plane >> 1) + q.hbase;
      e = make_float2(p[0], p[a.nx >> 1]);
    }
    return e;
  }

  template <int Q>
  static __device__ __forceinline__ void step(const LegArgs& a, State& st, const LegPos& q, const Cols& k, const LegCoef* C,
                                              float* S, float* Z, const Upd& u, int i, int z0, int z1, int plane) {
    constexpr int P = Q & 1;
    auto buf = [&](int stage, int par) { return S + (stage * 2 + par) * G::PLANE; };
    auto publish = [&](int stage, int par, float2 v) {
      float* W = buf(stage, par);
      W[q.my] = v.x;
      W[q.my + G::PITCH] = v.y;
    };
    LegRing<SC>& g = st.g;
    const int po = i - 3;
    const bool out = q.own && po >= z0 && po < z1;
    const double2 fa = st.fa, fb = st.fb;
    if (PHI && q.own && po + 1 >= z0 && po + 1 < z1) {
      const double* f = u.phi + (size_t)(po + 1) * plane + q.base;
      st.fa = load2(f, a.phi_vec);
      st.fb = load2(f + a.nx, a.phi_vec);
    }
    const LegCoef c0 = C[i];
    const float2 ra = g.ra[P], rb = g.rb[P], ia = g.ia[SC ? P : 0], ib = g.ib[SC ? P : 0];
    g.template fetch<P>(a, q, i + 2, plane, SC && C[i + 2].has_s);   // in flight during two steps
    const float2 ir2 = g.template take<Q>(ra, rb, ia, ib, c0);       // plane i - 2
    // prolongated black, plane i + 1
    const float2 e = st.e[P ^ 1];
    st.e[P ^ 1] = fetch_e(a, q, i + 3, plane);
    const float2 hi = prolonged<P ^ 1>(a, st, k, Z, e, i + 1);
    publish(3, P ^ 1, hi);
    zplane<P>(a, st, k, Z, i + 2, plane >> 2);      // for the next step
    // red, plane i
    float2 v = leg_num<true, P>(buf(3, P), q.my, G::PITCH, st.w[0].lo, st.w[0].cu, hi, g.rr[Q], c0);
    v = __fmul2_rn(v, SC ? g.ir[SC ? P : 0] : both(c0.invdiag));
    publish(0, P, v);
    st.w[0].push(hi);
    // black, plane i - 1
    const LegCoef c1 = C[i - 1];
    float2 b = leg_num<false, P ^ 1>(buf(0, P ^ 1), q.my, G::PITCH, st.w[1].lo, st.w[1].cu, v, g.rk[(Q + 3) & 3], c1);
    b = __fmul2_rn(b, SC ? g.ik[SC ? (Q + 3) & 3 : 0] : both(c1.invdiag));
    publish(1, P ^ 1, b);
    st.w[1].push(v);
    // red, plane i - 2
    const LegCoef c2 = C[i - 2];
    v = leg_num<true, P>(buf(1, P), q.my, G::PITCH, st.w[2].lo, st.w[2].cu, b, g.rr[(Q + 2) & 3], c2);
    v = __fmul2_rn(v, SC ? ir2 : both(c2.invdiag));
    publish(2, P, v);
    st.w[2].push(b);
    // black, plane i - 3: both colours leave
    const LegCoef c3 = C[i - 3];
    b = leg_num<false, P ^ 1>(buf(2, P ^ 1), q.my, G::PITCH, st.w[3].lo, st.w[3].cu, v, g.rk[(Q + 1) & 3], c3);
    b = __fmul2_rn(b, SC ? g.ik[SC ? (Q + 1) & 3 : 0] : both(c3.invdiag));
    if (out) {
      const float2 r = st.w[3].cu;                  // red values of the plane (parity P ^ 1)
      const float2 va = P ? make_float2(r.x, b.x) : make_float2(b.x, r.x);
      const float2 vb = P ? make_float2(b.y, r.y) : make_float2(r.y, b.y);
      if (PHI) {
        auto upd = [&](double p, float e) { return u.zero ? 0.0 : p + f64_of_float(fminf(fmaxf(e, -u.clampf), u.clampf)); };
        double* f = u.phi + (size_t)po * plane + q.base;
        store2(f, make_double2(upd(fa.x, va.x), upd(fa.y, va.y)), a.phi_vec);
        store2(f + a.nx, make_double2(upd(fb.x, vb.x), upd(fb.y, vb.y)), a.phi_vec);
      } else {
        float* o = a.e_out + (size_t)po * plane + q.base;
        *reinterpret_cast<float2*>(o) = va;
        *reinterpret_cast<float2*>(o + a.nx) = vb;
      }
    }
    st.w[3].push(v);
    __syncthreads();
  }

  static __device__ __forceinline__ void run(const LegArgs& a, const Upd& u, int bx, int by, int bz, unsigned char* smem) {
    const int tid = threadIdx.x;
    const int z0 = bz * a.kz, z1 = min(a.nz, z0 + a.kz);
    const int ps = max(0, z0 - 4), pe = z1 - 1 + 3;
    const int ncoef = leg_coef_planes(a.kz);
    LegCoef* C0 = reinterpret_cast<LegCoef*>(smem);
    float* S = reinterpret_cast<float*>(smem + (size_t)ncoef * sizeof(LegCoef));
    float* Z = S + STAGES * 2 * G::PLANE;
    const LegPos q = leg_pos<G>(tid, bx, by, a.nx, a.ny);
    const int plane = a.nx * a.ny, cplane = plane >> 2;
    const int hx = a.nx >> 1, hy = a.ny >> 1;
    State st = {};
    if (!SC) {   // in flight while the coefficients arrive
      st.g.template fetch<0>(a, q, ps, plane, false);
      st.g.template fetch<1>(a, q, ps + 1, plane, false);
    }
    const float2 e0 = fetch_e(a, q, ps, plane);
    st.e[1] = fetch_e(a, q, ps + 1, plane);
    st.e[0] = fetch_e(a, q, ps + 2, plane);
    Cols k;
    k.own = q.cbase;
    k.zown = (1 + tid / G::BX) * ZP + 1 + tid % G::BX;
    k.ring = 0;
    k.zring = -1;
    if (tid < RING) {
      // ring place tid: the row above, the row below, then the columns left and right
      int rx, ry;
      if (tid < 2 * (G::BX + 2)) {
        ry = tid < G::BX + 2 ? 0 : G::BY + 1;
        rx = tid < G::BX + 2 ? tid : tid - (G::BX + 2);
      } else {
        const int t = tid - 2 * (G::BX + 2);
        ry = 1 + (t >> 1);
        rx = (t & 1) ? G::BX + 1 : 0;
      }
      k.zring = ry * ZP + rx;
      constexpr int tpx = G::BX - 2 * G::HP, tpy = G::BY - 2 * G::HP;
      int cx = (bx * tpx - G::HP + rx - 1) % hx, cy = (by * tpy - G::HP + ry - 1) % hy;
      if (cx < 0) cx += hx;
      if (cy < 0) cy += hy;
      k.ring = cy * hx + cx;
    }
    // coarse window so that the first plane's shift makes K current: kp holds plane K
    const int K0 = a.crz ? ps >> 1 : ps;
    if (K0 > 0) {
      st.kc = a.ec[(size_t)(K0 - 1) * cplane + k.own];
      if (k.zring >= 0) st.gc = a.ec[(size_t)(K0 - 1) * cplane + k.ring];
    }
    st.kp = a.ec[(size_t)K0 * cplane + k.own];
    if (k.zring >= 0) st.gp = a.ec[(size_t)K0 * cplane + k.ring];
    leg_load_coef(C0, a.coef, ps - kLegLag, ncoef, a.nz, tid, G::THREADS);
    for (int t = tid; t < STAGES * 2 * G::PLANE + 2 * ZPLANE; t += G::THREADS) S[t] = 0.f;
    const LegCoef* C = C0 - (ps - kLegLag);
    __syncthreads();
    if (SC) {
      st.g.template fetch<0>(a, q, ps, plane, C[ps].has_s);
      st.g.template fetch<1>(a, q, ps + 1, plane, C[ps + 1].has_s);
    }
    zplane<0>(a, st, k, Z, ps, cplane);
    __syncthreads();
    {
      const float2 v = prolonged<0>(a, st, k, Z, e0, ps);
      st.w[0].cu = v;
      float* W = S + 3 * 2 * G::PLANE;
      W[q.my] = v.x;
      W[q.my + G::PITCH] = v.y;
      zplane<1>(a, st, k, Z, ps + 1, cplane);
      __syncthreads();
    }
    if (ps & 2) {
      step<2>(a, st, q, k, C, S, Z, u, ps, z0, z1, plane);
      step<3>(a, st, q, k, C, S, Z, u, ps + 1, z0, z1, plane);
    }
    for (int i = ps + (ps & 2); i <= pe; i += 4) {
      step<0>(a, st, q, k, C, S, Z, u, i, z0, z1, plane);
      step<1>(a, st, q, k, C, S, Z, u, i + 1, z0, z1, plane);
      if (i + 2 > pe) break;
      step<2>(a, st, q, k, C, S, Z, u, i + 2, z0, z1, plane);
      step<3>(a, st, q, k, C, S, Z, u, i + 3, z0, z1, plane);
    }
  }
};

}  // namespace dev
}  // namespace fx
