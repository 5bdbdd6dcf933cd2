// stage_tile.cuh — the fused right-hand-side + stage-combination tile of one
// MPRK2 stage in FP64 (device code; included by the kernel translation units).
//
// One CTA owns a TX x TZR tile of cells (TZR = TZ rows, or TZ/2 or TZ/4 for
// launches of few tiles). It
//   1. stages the stage state of the tile plus a two-cell halo in shared
//      memory (x periodic; stage values q + h R_a rebuilt on the fly in
//      double), as doubles and as 64-bit fixed point, and computes u, w and
//      e = T / (gamma (gamma - 1)) on the tile plus a one-cell ring,
//   2. computes every x and z face flux of the tile once (Lax–Friedrichs
//      inviscid flux of Sec. 2.1 on the linear reconstruction of the
//      conserved variables, minus the common-value viscous flux of App. B),
//      in one direction-generic routine written in the face frame, with
//      mirror or wall-state ghosts beyond walls and the interface and the
//      interface's bulk fluxes and wall states (App. B),
//   3. forms R = -div F* + s per cell and applies the partition's stage
//      combination (Eq. MRK2 in low-storage form) in double precision.
// Only two barriers separate them (with phases of their own for the ring, the
// tangential differences and the interface state, and faces dealt to threads
// in three uneven rounds, the step below took 2.39 ms).
//
// The fluxes of mass, normal momentum and energy run in 64-bit fixed point
// (fixed_point.cuh): as double arithmetic the faces were 300 of the tile's 309
// operations per cell on a pipe that completes two per clock and SM, which
// bound every FP64 launch: the pipe was 86 % busy. The flux of the tangential
// momentum has no term as large as density or pressure (in fixed point a shear
// of 1e-6 in a flow uniform along x had 3e4 times the double form's error), so
// its integers carry an exponent (fixed_flux.cuh). Measured: a slow step of
// 2048 x 1024 cells with m = 8 11.7 -> 2.37 ms (2.06 with that flux in fixed
// point too), 64 x 64 with m = 4 185 -> 63.5 us (58.4). Faces with
// a state outside the fixed-point range take the same formulas in double
// (slow_faces), a row of 32 at a time (row_in_range); which form a face takes
// depends on its row's cells alone, so results do not depend on the tile shape
// or the launch.
#pragma once

#include "fixed_flux.cuh"
#include "fp64_recip.cuh"
#include "mprk_internal.h"

namespace mprk {

template <int TZR = TZ>
struct TileSmem {
  double q[4][TZR + 4][TX + 4];  // stage state, rows k0-2.., cols i0-2..
  i64 qi[4][TZR + 4][TX + 4];    // the same: rho, rho E .58, momenta .60
  i64 v[3][TZR + 2][TX + 2];     // u, w, e (.59), rows k0-1.., cols i0-1..
  i64 qw[2][TZR + 4][TX + 4];     // rho u, rho w packed (fixed_point.cuh)
  i64 vp[2][TZR + 2][TX + 2];     // u, w under the exponents of qw
  // face fluxes over half the divergence factor (.57; the tangential momentum's
  // and every component of a slow face as the bits of a double)
  i64 fx[4][TZR][TX + 1];  // face f between cols f-1, f
  i64 fz[4][TZR + 1][TX];  // seen from above at the interface
  i64 fg[4][TX];           // the interface seen from fluid 1 (below)
  unsigned char slow[(2 * TZR + 3) * TX];  // per face: its job and lane (face_id)
};

// Lax–Friedrichs flux in the face frame, in double (faces outside the
// fixed-point range). A state is (rho, m_n, m_t, rho E): m_n is the momentum
// along the face normal, m_t along the face. Output is f(q_L) + f(q_R) +
// lambda (q_L - q_R) - V: V the viscous or interface part of (m_n, m_t, rho E).
// lambda is the largest |u_n| + a over the left, right and Roe-averaged
// states (Sec. 2.1).
__device__ __forceinline__ void lf_face(const Geom& g, const double L[4], const double R[4], const double V[3],
                                        double out[4]) {
  const double lr = L[0], lmn = L[1], lmt = L[2], lE = L[3], rr = R[0], rmn = R[1], rmt = R[2], rE = R[3];
  const double invL = recip_f64(lr), invR = recip_f64(rr);
  const double unL = __dmul_rn(lmn, invL), utL = __dmul_rn(lmt, invL);
  const double unR = __dmul_rn(rmn, invR), utR = __dmul_rn(rmt, invR);
  const double kL = __fma_rn(lmt, utL, __dmul_rn(lmn, unL)), kR = __fma_rn(rmt, utR, __dmul_rn(rmn, unR));
  const double pL = __dmul_rn(g.gm1, __fma_rn(-0.5, kL, lE)), pR = __dmul_rn(g.gm1, __fma_rn(-0.5, kR, rE));
  const double eL = __dadd_rn(lE, pL), eR = __dadd_rn(rE, pR);
  const double lam = face_speed(g, lr, rr, unL, unR, __dsub_rn(utR, utL), 0.0, __dmul_rn(__dmul_rn(g.gamma, pL), invL),
                                __dmul_rn(__dmul_rn(g.gamma, pR), invR));
  out[0] = __fma_rn(lam, __dsub_rn(lr, rr), __dadd_rn(lmn, rmn));
  const double f1 = __dsub_rn(__dadd_rn(__fma_rn(lmn, unL, pL), __fma_rn(rmn, unR, pR)), V[0]);
  out[1] = __fma_rn(lam, __dsub_rn(lmn, rmn), f1);
  out[2] = __fma_rn(lam, __dsub_rn(lmt, rmt), __fma_rn(rmt, unR, __fma_rn(lmt, unL, -V[1])));
  out[3] = __fma_rn(lam, __dsub_rn(lE, rE), __fma_rn(unR, eR, __fma_rn(unL, eL, -V[2])));
}

// Viscous flux in the face frame from the common values of App. B: face
// velocity = mean of the two cells, normal derivatives = two-point
// differences, tangential derivatives = mean of the two cells' central
// differences. Output (0, sigma_nn, sigma_nt, u.sigma_n + kappa dT/dn).
template <typename Real>
__device__ __forceinline__ void visc_face(Real unL, Real utL, Real TL, Real gnL, Real gtL,
                                          Real unR, Real utR, Real TR, Real gnR, Real gtR,
                                          Real inv_dn, Real mu, Real kap, Real out[4]) {
  const Real half = Real(0.5);
  const Real un = half * (unL + unR), ut = half * (utL + utR);
  const Real dn_un = (unR - unL) * inv_dn;
  const Real dn_ut = (utR - utL) * inv_dn;
  const Real dn_T = (TR - TL) * inv_dn;
  const Real dt_un = half * (gnL + gnR);  // tangential derivative of u_n
  const Real dt_ut = half * (gtL + gtR);  // tangential derivative of u_t
  const Real snn = mu * (Real(2) * dn_un - Real(2.0 / 3.0) * (dn_un + dt_ut));
  const Real snt = mu * (dn_ut + dt_un);
  out[0] = Real(0);
  out[1] = snn;
  out[2] = snt;
  out[3] = un * snn + ut * snt + kap * dn_T;
}

__device__ __forceinline__ int wrap_col(int i, int nx) {
  if (i < 0) i += nx;
  if (i >= nx) i %= nx;
  return i;
}

// The cell that halo column i stands for: its periodic image, or with x
// walls its mirror image across the nearer wall. In that case *ghost is set
// and the caller builds the wall ghosts: rho u flips (mirror state), u flips
// and, at a no-slip wall, w flips ((u, w, T) ghost = 2 wall state - cell).
// Far ghosts of a tile wider than the grid feed no cell of the grid and are
// clamped into it.
__device__ __forceinline__ int halo_col(int i, int nx, int xwall, bool* ghost) {
  *ghost = false;
  if (!xwall) return wrap_col(i, nx);
  if (i < 0) {
    *ghost = true;
    i = -1 - i;
  } else if (i >= nx) {
    *ghost = true;
    i = 2 * nx - 1 - i;
  }
  return i < 0 ? 0 : (i >= nx ? nx - 1 : i);
}
// Is halo column i an x-wall ghost?
__device__ __forceinline__ bool x_ghost(int i, int nx, int xwall) { return xwall && (i < 0 || i >= nx); }

// The stage values of the four components of a general s-stage base (GEN):
// base + h sum_{q<p} A_pq R_q over the R_a slots of the current substep (slot
// q at Ra + q * slot, the components `plane` apart); p = 0 gives the base
// value. Every product-sum is an explicit fused multiply-add, so no launch
// shape or kernel that compiles this code can round it differently. Zero
// coefficients are skipped by their bits: compared as doubles, per component,
// they held the double pipe as long as the sums. The loops here and below take
// the components together and are not unrolled (unrolled, the tile spilled 116
// bytes): 1024 x 512 cells, RK4, m = 4, 1.030 -> 0.813 ms per step.
__device__ __forceinline__ void gen_stage_values(const Geom& g, const double* base, const double* Ra, size_t slot,
                                                 size_t plane, int p, double h, double val[4]) {
  double sum[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll 1
  for (int q = 0; q < p; q++) {
    const double A = g.bA[p][q];
    if (__double_as_longlong(A) == 0) continue;
    const double* R = Ra + (size_t)q * slot;
#pragma unroll
    for (int c = 0; c < 4; c++) sum[c] = __fma_rn(A, R[c * plane], sum[c]);
  }
#pragma unroll
  for (int c = 0; c < 4; c++) val[c] = p == 0 ? base[c * plane] : __fma_rn(h, sum[c], base[c * plane]);
}

// sum_q b_q R_q of the four components over the first s - 1 R_a slots and the
// current R (slot s - 1), as explicit fused multiply-adds in ascending q.
__device__ __forceinline__ void gen_weighted_sums(const Geom& g, const double* Ra, size_t slot, size_t plane,
                                                  const double R[4], double out[4]) {
  double sum[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll 1
  for (int q = 0; q < g.s - 1; q++) {
#pragma unroll
    for (int c = 0; c < 4; c++) sum[c] = __fma_rn(g.bb[q], Ra[(size_t)q * slot + c * plane], sum[c]);
  }
#pragma unroll
  for (int c = 0; c < 4; c++) out[c] = __fma_rn(g.bb[g.s - 1], R[c], sum[c]);
}

// The stage state lies inside the fixed-point range?
__device__ __forceinline__ bool cell_in_range(double r, double mu, double mw, double E) {
  return in_range(r, max(abs_word(mu), abs_word(mw)), E);
}

// Cell values of the two arithmetics: i64 (fixed point) or double.
template <typename T>
struct Arith;
template <>
struct Arith<i64> {
  template <int TZR>
  static __device__ __forceinline__ const i64* q(const TileSmem<TZR>& S) { return &S.qi[0][0][0]; }
  // q + (upper - lower neighbour) / 4
  static __device__ __forceinline__ i64 rec(i64 a, i64 up, i64 dn) { return (a << 2) + (up - dn); }
  // u, w, e of a cell; 1/rho .61
  static __device__ __forceinline__ i64 prims(i64 r, i64 mu, i64 mw, i64 E, i64 out[3]) {
    const i64 inv_ = fx::recip(r << 2);
    const FxW inv = fx::split(inv_);
    const FxW m1 = fx::split(mu << 2), m2 = fx::split(mw << 2);
    out[0] = fx::mul(m1, inv);
    out[1] = fx::mul(m2, inv);
    const i64 k = fx::mul(m1, fx::split(out[0])) + fx::mul(m2, fx::split(out[1]));  // .57; k/2 is .58
    out[2] = fx::mul(fx::split((E - k) << 2), inv) << 2;
    return inv_;
  }
};
template <>
struct Arith<double> {
  template <int TZR>
  static __device__ __forceinline__ const double* q(const TileSmem<TZR>& S) { return &S.q[0][0][0]; }
  static __device__ __forceinline__ double rec(double a, double up, double dn) { return __fma_rn(0.25, __dsub_rn(up, dn), a);
  }
  static __device__ __forceinline__ double prims(double r, double mu, double mw, double E, double out[3]) {
    const double inv = recip_f64(r);
    out[0] = __dmul_rn(mu, inv);
    out[1] = __dmul_rn(mw, inv);
    out[2] = __dmul_rn(__fma_rn(-0.5, __fma_rn(mw, out[1], __dmul_rn(mu, out[0])), E), inv);
    return inv;
  }
};

// u, w, e of the cell of halo row rr, column cc into the ring (phase 1); in
// fixed point also u and w from the packed momenta.
template <typename T, int TZR>
__device__ __forceinline__ void ring_cell(const Geom& g, TileSmem<TZR>& S, int rr, int cc, int i0, T r, T mu, T mw, T E) {
  constexpr int VP = (TZR + 2) * (TX + 2);
  if (rr < 1 || rr > TZR + 2 || cc < 1 || cc > TX + 2) return;
  T* v = reinterpret_cast<T*>(&S.v[0][0][0]) + (rr - 1) * (TX + 2) + cc - 1;
  T o[3];
  const T inv = Arith<T>::prims(r, mu, mw, E, o);
  // the mirror state's u is already flipped; a no-slip x wall flips w too
  const bool flip = x_ghost(i0 - 2 + cc, g.nx, g.xwall) && g.wall == 0;
  v[0] = o[0];
  v[VP] = flip ? -o[1] : o[1];
  v[2 * VP] = o[2];
  if constexpr (sizeof(inv) == 8 && (T)0.5 == (T)0) {
    const FxW iw = fx::split(inv);
    const i64 w = fx::packed_velocity(S.qw[1][rr][cc], iw);
    S.vp[0][rr - 1][cc - 1] = fx::packed_velocity(S.qw[0][rr][cc], iw);
    S.vp[1][rr - 1][cc - 1] = flip ? -w : w;
  }
}

// Interface (App. B, Eq. bulk-flux and the wall states after it), from the
// velocities and e of the two cells touching it: the ghost velocity 2 u_w - u
// of the cell `own` in fluid f + 1, and twice u_w sigma and -Pi, which with
// twice sigma make the flux both fluids share. In double from the state, by 34 threads of the tile
// before its faces, these took the launch of 64 x 64 cells a quarter of its
// time: a warp's double operation occupies its scheduler for 64 clocks.
__device__ __forceinline__ i64 lid_ghost(const Geom&, const FxConst& k, int f, i64 own, i64 other) {
  return own + (fx::mul(fx::split((other - own) << 2), k.lid[LID_1 + f]) << 1);
}
__device__ __forceinline__ double lid_ghost(const Geom&, const FxConst& k, int f, double own, double other) {
  return __fma_rn(k.tlid[LID_1 + f], __dsub_rn(other, own), own);
}
// The energy's part of one wall velocity component (sig: its sigma .59); the
// heat flux.
__host__ __device__ __forceinline__ i64 lid_work(const FxConst& k, i64 u1, i64 u2, i64 sig) {
  const i64 uw = u1 + fx::mul(fx::split((u2 - u1) << 2), k.lid[LID_1]);
  return fx::mul(fx::split(uw << 3), fx::split(sig));
}
__host__ __device__ __forceinline__ i64 lid_heat(const FxConst& k, i64 e1, i64 e2) {
  return fx::mul(fx::split(e2 - e1), k.lid[LID_T]);
}
__device__ __forceinline__ double lid_work(const FxConst& k, double u1, double u2, double sig) {
  return __dmul_rn(__fma_rn(__dmul_rn(0.5, k.tlid[LID_1]), __dsub_rn(u2, u1), u1), sig);
}
__device__ __forceinline__ double lid_heat(const FxConst& k, double e1, double e2) {
  return __dmul_rn(k.tlid[LID_T], __dsub_rn(e2, e1));
}

// ---- aligned velocity differences of the tangential stresses ----------------
// u: a cell's velocity under its momentum's exponent, w: the packed momentum
// or that exponent; vs, qs (vt, qt): the strides of either along the face normal (across it).
// The two cells at the face are at 0 and vs.
__device__ __forceinline__ FxA vel_diff(const i64* u, const i64* w, int vs, int qs) {
  const int a = fx::pack_exp(w[0]), b = fx::pack_exp(w[qs]), e = max(a, b);
  return FxA{vel_at(u[vs], b, e) - vel_at(u[0], a, e), e};
}
// The sum of both cells' central differences across the normal.
template <typename W>
__device__ __forceinline__ FxA vel_cross(const i64* u, const W* w, int vs, int qs, int vt, int qt) {
  const int a = fx::pack_exp(w[-qt]), b = fx::pack_exp(w[qt]), c = fx::pack_exp(w[qs - qt]), d = fx::pack_exp(w[qs + qt]);
  const int e = max(max(a, b), max(c, d));
  return FxA{(vel_at(u[vt], b, e) - vel_at(u[-vt], a, e)) + (vel_at(u[vs + vt], d, e) - vel_at(u[vs - vt], c, e)), e};
}
// The same along z for a component tangential to walls and interface, of the
// cells ua and ub of row k, with the ghosts 2 (wall state) - cell beyond them.
template <typename W>
__device__ __forceinline__ FxA dz_pair(const Geom& g, const FxConst& c, int k, const i64* ua, const i64* ub, int vr,
                                       const W* wa, const W* wb, int qr) {
  const bool top = k + 1 == g.nz || k + 1 == g.n1, bot = k == 0 || k == g.n1;
  int e = max(max(fx::pack_exp(wa[-qr]), fx::pack_exp(wa[qr])), max(fx::pack_exp(wb[-qr]), fx::pack_exp(wb[qr])));
  if (top || bot) e = max(e, max(fx::pack_exp(wa[0]), fx::pack_exp(wb[0])));
  i64 sum = 0;
#pragma unroll
  for (int s = 0; s < 2; s++) {
    const i64* u = s ? ub : ua;
    const W* w = s ? wb : wa;
    i64 up = vel_at(u[vr], fx::pack_exp(w[qr]), e), dn = vel_at(u[-vr], fx::pack_exp(w[-qr]), e);
    if (top || bot) {
      const i64 own = vel_at(u[0], fx::pack_exp(w[0]), e);
      if (top) up = k + 1 == g.nz ? (g.wall ? own : -own) : lid_ghost(g, c, 0, own, up);
      if (bot) dn = k == 0 ? (g.wall ? own : -own) : lid_ghost(g, c, 1, own, dn);
    }
    sum += up - dn;
  }
  return FxA{sum, e};
}

// ---- phase 2: face fluxes ---------------------------------------------------
// The faces of the tile as jobs of one warp each: TZR rows of z faces, TZR
// rows of x faces (columns 0 to TX - 1), the z faces above the last row, the
// x faces right of the last column (one lane per row), and in a tile at the
// interface its faces seen from below. With TZR + 1 warps these are two jobs
// per warp, with 2 TZR + 3 one: no round leaves warps waiting for a few last
// faces.
struct FaceId {
  int isx, f, c;  // z: face row f, column c; x: tile row f, face column c
  int ku;         // row above a z face, or the row of an x face
  int below;      // the interface from fluid 1
};
// Face of a job and lane; false if no cell of the tile needs it.
template <int TZR>
__device__ __forceinline__ bool face_id(const Geom& g, int job, int lane, int k0, int row_hi, FaceId* id) {
  id->below = 0;
  id->c = lane;
  if (job < TZR || job == 2 * TZR) {
    id->isx = 0;
    id->f = job < TZR ? job : TZR;
    id->ku = k0 + id->f;
    // needed by the cell below (f >= 1) or above (f < TZR); at the interface
    // this is the side of fluid 2
    return id->ku - 1 < row_hi && !(id->f == TZR && id->ku == g.n1);
  }
  if (job <= 2 * TZR + 1) {
    const bool edge = job > 2 * TZR;
    id->isx = 1;
    id->f = edge ? lane : job - TZR;
    id->c = edge ? TX : lane;
    id->ku = k0 + id->f;
    return id->ku < row_hi && id->f < TZR;
  }
  id->isx = 0;
  id->f = g.n1 - k0;
  id->ku = g.n1;
  id->below = 1;
  return id->f >= 1 && id->f <= TZR && g.n1 - 1 < row_hi;
}

// States of the face in the face frame (rho, m_n, m_t, rho E) on both sides,
// reconstructed from the four cells across it, and the two cells' velocities,
// e and tangential differences (un, ut, e, gn, gt). A boundary face (outer
// wall or interface) has the inner cell's state on one side and its mirror
// on the other; an outer wall's viscous ghost is 2 wall state - cell, and at
// the interface only (ut, e) are set. Returns the fluid of the face's
// coefficients, 2 at the interface.
template <typename T, int TZR>
__device__ __forceinline__ int face_sides(const Geom& g, const FxConst& fk, const TileSmem<TZR>& S, const FaceId& id,
                                          T L[4], T R[4], T vL[5], T vR[5]) {
  constexpr int QP = (TZR + 4) * (TX + 4), VP = (TZR + 2) * (TX + 2);
  const int n1 = g.n1, nz = g.nz, ku = id.ku, kd = ku - 1;
  // first of the four cells, their stride, and the planes of m_n, m_t
  const int qs = id.isx ? 1 : TX + 4;
  const int q0 = id.isx ? (id.f + 2) * (TX + 4) + id.c : id.f * (TX + 4) + id.c + 2;
  const int pn = id.isx ? QP : 2 * QP, pt = 3 * QP - pn;
  const bool wall = !id.isx && (ku == 0 || ku == nz), lid = !id.isx && ku == n1;
  const bool from_above = ku == 0 || (lid && !id.below);  // of a boundary face: the inner cell is the upper one
  const bool mir0 = !id.isx && (kd == 0 || kd == n1), mir3 = !id.isx && (ku == nz - 1 || ku == n1 - 1);
  const T* q = Arith<T>::q(S) + q0;
  const int planes[4] = {0, pn, pt, 3 * QP};
  if (wall || lid || mir0 || mir3) {
#pragma unroll
    for (int c = 0; c < 4; c++) {
      const bool odd = c == 1;  // mirror ghosts beyond a wall or the interface: rho w odd
      const T* p = q + planes[c];
      T a0 = p[0], a1 = p[qs], a2 = p[2 * qs], a3 = p[3 * qs];
      if (wall || lid) {
        if (from_above) a1 = odd ? -a2 : a2;
        else a2 = odd ? -a1 : a1;
      }
      if (mir0) a0 = odd ? -a1 : a1;
      if (mir3) a3 = odd ? -a2 : a2;
      L[c] = Arith<T>::rec(a1, a2, a0);
      R[c] = Arith<T>::rec(a2, a1, a3);
      if (wall || lid) {
        if (from_above) L[c] = odd ? -R[c] : R[c];
        else R[c] = odd ? -L[c] : L[c];
      }
    }
  } else {
#pragma unroll
    for (int c = 0; c < 4; c++) {
      const T* p = q + planes[c];
      const T a0 = p[0], a1 = p[qs], a2 = p[2 * qs], a3 = p[3 * qs];
      L[c] = Arith<T>::rec(a1, a2, a0);
      R[c] = Arith<T>::rec(a2, a1, a3);
    }
  }
  // velocities, e and tangential central differences of the cells at the face
  const T* v = reinterpret_cast<const T*>(&S.v[0][0][0]);
  if (lid) {
    const T* p = v + id.f * (TX + 2) + id.c + 1;
    vL[1] = p[0];
    vR[1] = p[TX + 2];
    vL[2] = p[2 * VP];
    vR[2] = p[2 * VP + TX + 2];
    return 2;
  }
  if (id.isx) {
    const T* p = v + (id.f + 1) * (TX + 2) + id.c;
    const bool top = ku + 1 == nz || ku + 1 == n1, bot = ku == 0 || ku == n1;
#pragma unroll
    for (int s = 0; s < 2; s++, p++) {
      T* o = s ? vR : vL;
      const T u = p[0], w = p[VP];
      o[0] = u;
      o[1] = w;
      o[2] = p[2 * VP];
      // z differences of u, w, with the ghost 2 (wall state) - cell beyond a
      // wall or the interface
      T uu, wu, ud, wd;
      if (top) {
        uu = ku + 1 == nz ? (g.wall ? u : -u) : lid_ghost(g, fk, 0, u, p[TX + 2]);
        wu = -w;
      } else {
        uu = p[TX + 2];
        wu = p[VP + TX + 2];
      }
      if (bot) {
        ud = ku == 0 ? (g.wall ? u : -u) : lid_ghost(g, fk, 1, u, p[-(TX + 2)]);
        wd = -w;
      } else {
        ud = p[-(TX + 2)];
        wd = p[VP - (TX + 2)];
      }
      o[3] = uu - ud;
      o[4] = wu - wd;
    }
    return ku >= n1;
  }
  const T* p = v + id.f * (TX + 2) + id.c + 1;
#pragma unroll
  for (int s = 0; s < 2; s++, p += TX + 2) {
    T* o = s ? vR : vL;
    o[0] = p[VP];
    o[1] = p[0];
    o[2] = p[2 * VP];
    o[3] = p[VP + 1] - p[VP - 1];
    o[4] = p[1] - p[-1];
  }
  if (wall) {
    const T* c = from_above ? vR : vL;
    T* o = from_above ? vL : vR;
    o[0] = -c[0];
    o[1] = g.wall ? c[1] : -c[1];
    o[2] = c[2];
    o[3] = -c[3];
    o[4] = g.wall ? c[4] : -c[4];
  }
  return (ku == 0 ? 0 : kd) >= n1;
}

// A tile none of whose faces lies at, or next to, a wall or the interface, and
// none beyond the launch's rows: its faces need no ghosts and no row tests.
template <int TZR>
__device__ __forceinline__ bool tile_plain(const Geom& g, int k0, int row_hi) {
  return k0 >= 2 && k0 + TZR <= g.nz - 2 && k0 + TZR <= row_hi && (g.n1 < k0 - 1 || g.n1 > k0 + TZR + 1);
}
// face_id and face_sides of such a tile, per direction: every cell at a fixed
// offset from the face's first one. Without the row tests and the addresses
// by direction 2048 x 1024 cells, m = 8, went from 2.118 to 2.058 ms per step,
// 1024 x 512 with the RK4 base from 1.049 to 1.030 ms.
// The general form stays for the tiles at the walls and the interface and
// those with a cell outside the fixed-point range.
template <int TZR>
__device__ __forceinline__ bool face_id_plain(int job, int lane, int k0, FaceId* id) {
  const bool edge = job == 2 * TZR + 1;
  id->below = 0;
  id->isx = job >= TZR && job != 2 * TZR;
  id->f = edge ? lane : job < TZR ? job : job - TZR;
  id->c = edge ? TX : lane;
  id->ku = k0 + id->f;
  return !edge || lane < TZR;
}
template <bool X, int TZR>
__device__ __forceinline__ void face_sides_plain(const TileSmem<TZR>& S, const FaceId& id, i64 L[4], i64 R[4], i64 vL[5],
                                                 i64 vR[5]) {
  constexpr int QP = (TZR + 4) * (TX + 4), VP = (TZR + 2) * (TX + 2), VW = TX + 2;
  constexpr int qs = X ? 1 : TX + 4, vs = X ? 1 : VW, vt = X ? VW : 1;  // along the normal; across it
  constexpr int pn = X ? 1 : 2, pt = 3 - pn;
  const i64* q = &S.qi[0][X ? id.f + 2 : id.f][X ? id.c : id.c + 2];
  constexpr int planes[4] = {0, pn * QP, pt * QP, 3 * QP};
#pragma unroll
  for (int c = 0; c < 4; c++) {
    const i64* p = q + planes[c];
    const i64 a0 = p[0], a1 = p[qs], a2 = p[2 * qs], a3 = p[3 * qs];
    L[c] = Arith<i64>::rec(a1, a2, a0);
    R[c] = Arith<i64>::rec(a2, a1, a3);
  }
  const i64* v = &S.v[0][X ? id.f + 1 : id.f][X ? id.c : id.c + 1];
  constexpr int vn = (pn - 1) * VP, vu = (pt - 1) * VP;
#pragma unroll
  for (int s = 0; s < 2; s++) {
    const i64* p = v + s * vs;
    i64* o = s ? vR : vL;
    o[0] = p[vn];
    o[1] = p[vu];
    o[2] = p[2 * VP];
    o[4] = p[vu + vt] - p[vu - vt];
  }
}

// The viscous flux of the normal momentum and the energy over half the
// divergence factor from the common values of App. B: sigma_nn and u .
// sigma_n + kappa dT/dn, .57; snt: sigma_nt .59.
__host__ __device__ __forceinline__ void fx_visc(const FxW* fc, const i64 vL[5], const i64 vR[5], i64 snt, i64* Vn, i64* VE) {
  *Vn = fx::mul2(fc[FXC_A], fx::split(vR[0] - vL[0]), fc[FXC_B], fx::split(vL[4] + vR[4]));
  // (u_L + u_R) . sigma: .61 x .59 -> .56, half of it at .57
  *VE = fx::mul2(fx::split((vL[0] + vR[0]) << 2), fx::split(*Vn << 2), fx::split((vL[1] + vR[1]) << 2), fx::split(snt)) +
        fx::mul(fc[FXC_K], fx::split(vR[2] - vL[2]));
}

// The same flux in double.
__device__ __forceinline__ void double_visc(const double* fc, const double vL[5], const double vR[5], double V[3]) {
  V[0] = __fma_rn(fc[FXC_A], __dsub_rn(vR[0], vL[0]), __dmul_rn(fc[FXC_B], __dadd_rn(vL[4], vR[4])));
  V[1] = __fma_rn(fc[FXC_C], __dsub_rn(vR[1], vL[1]), __dmul_rn(fc[FXC_D], __dadd_rn(vL[3], vR[3])));
  const double us = __fma_rn(__dadd_rn(vL[1], vR[1]), V[1], __dmul_rn(__dadd_rn(vL[0], vR[0]), V[0]));
  V[2] = __fma_rn(0.5, us, __dmul_rn(fc[FXC_K], __dsub_rn(vR[2], vL[2])));
}

// The tangential stress of face id in fluid fl (2: the interface), with the
// ghosts of face_sides; and the flux of the tangential momentum from it.
template <int TZR>
__device__ __forceinline__ FxStress visc_tan(const Geom& g, const FxConst& fk, const TileSmem<TZR>& S, const FaceId& id,
                                             int fl) {
  constexpr int VS = TX + 2, QS = TX + 4;
  const int ku = id.ku, r = id.isx ? id.f + 1 : id.f, c = id.isx ? id.c : id.c + 1;
  const i64* u = &S.vp[0][r][c];  // of the first cell at the face
  const i64* w = &S.vp[1][r][c];
  const i64* mu = &S.qw[0][r + 1][c + 1];
  const i64* mw = &S.qw[1][r + 1][c + 1];
  if (id.isx)
    return tan_stress(fk.tc[0][fl][0], vel_diff(w, mw, 1, 1), fk.tc[0][fl][1],
                      dz_pair(g, fk, ku, u, u + 1, VS, mu, mu + 1, QS));
  if (ku == 0 || ku == g.nz) {  // the ghost's u is +-u and its difference of w the opposite
    if (g.wall) return FxStress{0, 0};
    const int e = fx::pack_exp(ku == 0 ? mu[QS] : mu[0]);
    const i64 x = vel_at(ku == 0 ? u[VS] : u[0], e, e) << 1;
    return tan_stress(fk.tc[1][fl][0], FxA{ku == 0 ? x : -x, e});
  }
  const FxA du = vel_diff(u, mu, VS, QS);
  if (fl == 2) return tan_stress(fk.ts, du);
  return tan_stress(fk.tc[1][fl][0], du, fk.tc[1][fl][1], vel_cross(w, mw, VS, QS, 1, 1));
}
template <int TZR>
__device__ __forceinline__ i64 face_tan(const Geom& g, const TileSmem<TZR>& S, const FaceId& id, const FxTan& t,
                                        FxStress V) {
  constexpr int QS = TX + 4;
  const int n1 = g.n1, nz = g.nz, ku = id.ku;
  if (id.isx) {
    const i64* q = &S.qw[1][id.f + 2][id.c];
    return tan_flux(t, q[0], q[1], q[2], q[3], V);
  }
  const i64* q = &S.qw[0][id.f][id.c + 2];
  const i64 a1 = q[QS], a2 = q[2 * QS];
  if (ku == 0 || ku == nz || ku == n1) return tan_flux(t, 0, 0, 0, 0, V);  // nothing flows through
  return tan_flux(t, ku == 1 || ku == n1 + 1 ? a1 : q[0], a1, a2, ku == nz - 1 || ku == n1 - 1 ? a2 : q[3 * QS], V);
}
template <bool X, int TZR>
__device__ __forceinline__ FxStress visc_tan_plain(const FxConst& fk, const TileSmem<TZR>& S, const FaceId& id, int fl) {
  constexpr int VS = TX + 2, QS = TX + 4;
  const int r = X ? id.f + 1 : id.f, c = X ? id.c : id.c + 1;
  constexpr int n = X ? 0 : 1, t = 1 - n;  // planes of the normal and the tangential component
  return tan_stress(fk.tc[t ? 0 : 1][fl][0], vel_diff(&S.vp[t][r][c], &S.qw[t][r + 1][c + 1], X ? 1 : VS, X ? 1 : QS),
                    fk.tc[t ? 0 : 1][fl][1],
                    vel_cross(&S.vp[n][r][c], &S.qw[n][r + 1][c + 1], X ? 1 : VS, X ? 1 : QS, X ? VS : 1, X ? QS : 1));
}
template <bool X, int TZR>
__device__ __forceinline__ i64 face_tan_plain(const TileSmem<TZR>& S, const FaceId& id, const FxTan& t, FxStress V) {
  constexpr int qs = X ? 1 : TX + 4;
  const i64* q = &S.qw[X ? 1 : 0][X ? id.f + 2 : id.f][X ? id.c : id.c + 2];
  return tan_flux(t, q[0], q[qs], q[2 * qs], q[3 * qs], V);
}

// Fluxes (mass, normal and tangential momentum, energy) to shared memory, back
// in (rho, rho u, rho w, rho E) order.
template <int TZR>
__device__ __forceinline__ void store_flux(TileSmem<TZR>& S, const FaceId& id, const i64 F[4]) {
  i64* p;
  int plane, n;
  if (id.isx) {
    p = &S.fx[0][id.f][id.c], plane = TZR * (TX + 1), n = 1;
  } else if (id.below) {
    p = &S.fg[0][id.c], plane = TX, n = 2;
  } else {
    p = &S.fz[0][id.f][id.c], plane = (TZR + 1) * TX, n = 2;
  }
  p[0] = F[0];
  p[n * plane] = F[1];
  p[(3 - n) * plane] = F[2];
  p[3 * plane] = F[3];
}

// Do the cells that face id reads (four across it, and the tangential
// neighbours of the two at it) lie in the fixed-point range? Asked only in tiles where some cell does not.
template <int TZR>
__device__ __noinline__ bool face_in_range(const Geom& g, const TileSmem<TZR>& S, const FaceId id, int k0) {
  auto cell = [&](int r, int c) {  // halo row and column
    const int k = k0 - 2 + r;
    return k < 0 || k >= g.nz || cell_in_range(S.q[0][r][c], S.q[1][r][c], S.q[2][r][c], S.q[3][r][c]);
  };
  bool ok = true;
  if (id.isx) {
    for (int j = 0; j < 4; j++) ok = ok && cell(id.f + 2, id.c + j);
    for (int j = 0; j < 4; j++) ok = ok && cell(id.f + 1 + 2 * (j >> 1), id.c + 1 + (j & 1));
  } else {
    for (int j = 0; j < 4; j++) ok = ok && cell(id.f + j, id.c + 2);
    for (int j = 0; j < 4; j++) ok = ok && cell(id.f + 1 + (j >> 1), id.c + 1 + 2 * (j & 1));
  }
  return ok;
}

// Is the face of this lane evaluated in fixed point (out: its own cells are
// not in range)? The double pass runs a job's 32 faces together, so one of them
// outside takes the whole row of faces there, and the fixed-point pass is spared
// (30 % of the cells outside: 512 x 256, m = 4, 618 -> 579 us). An x face that two tiles
// evaluate, on a tile's edge or the wrap, asks its own cells alone.
__device__ __forceinline__ bool row_in_range(const FaceId& id, int i0, int nx, bool out) {
  const bool alone = id.isx && (id.c == 0 || id.c == TX || i0 + id.c == nx);
  const bool any = __any_sync(0xffffffffu, out && !alone);
  return !(out || (any && !alone));
}

// The faces marked slow (all: every face), in double: the ring again as
// doubles (in the same storage), then their fluxes. Ends with the tile's
// barrier. Against the tile that did everything in double, us per step: 2048 x
// 1024, m = 8, wholly outside 9378 (11683), 30 % of the cells outside 9957
// (11690); 512 x 256, m = 4, 442 (519) and 490 (519); with the Roe speed of
// every face and coefficients computed per tile 11556, 11979, 552 and 579.
template <int NT, int TZR>
__device__ __noinline__ void slow_faces(const Geom& g, const FxConst& fk, TileSmem<TZR>& S, int k0, int i0, int row_hi, bool all) {
  for (int e = threadIdx.x; e < (TZR + 2) * (TX + 2); e += NT) {
    const int rr = e / (TX + 2) + 1, cc = e % (TX + 2) + 1, k = k0 - 2 + rr;
    if (k >= 0 && k < g.nz)
      ring_cell<double, TZR>(g, S, rr, cc, i0, S.q[0][rr][cc], S.q[1][rr][cc], S.q[2][rr][cc], S.q[3][rr][cc]);
  }
  __syncthreads();
  for (int job = threadIdx.x / 32; job < 2 * TZR + 3; job += NT / 32) {
    const int lane = threadIdx.x % 32, e = job * TX + lane;
    FaceId id;
    if (!face_id<TZR>(g, job, lane, k0, row_hi, &id) || !(all || S.slow[e])) continue;
    if (all) S.slow[e] = 1;
    double L[4], R[4], vL[5], vR[5], V[3], F[4];
    const int fl = face_sides<double, TZR>(g, fk, S, id, L, R, vL, vR);
    if (fl < 2) {
      double_visc(fk.fd[id.isx ? 0 : 1][fl], vL, vR, V);
    } else {
      V[0] = 0.0;
      V[1] = __dmul_rn(fk.tlid[LID_S], __dsub_rn(vR[1], vL[1]));
      V[2] = __dadd_rn(lid_work(fk, vL[1], vR[1], V[1]), lid_heat(fk, vL[2], vR[2]));
    }
    lf_face(g, L, R, V, F);
    i64 o[4];
#pragma unroll
    for (int c = 0; c < 4; c++) o[c] = __double_as_longlong(F[c]);
    store_flux(S, id, o);
  }
  __syncthreads();
}

// The tile body. tile = linear tile index within the launch's row range.
// Inlined into each kernel, so that the single-instance kernel takes its
// arguments from the constant bank and the batch kernel from shared memory;
// every double operation names its rounding (no contraction is left to the
// compiler) and the rest is integer, so an instance's results are bitwise
// the same alone and in a batch.
//
// GEN selects the general s-stage base method (Sec. 3 remark) in place of
// Heun's low-storage path: s R_a slots, the stage values of the region
// tableaus built from the base, and its weights b in the combinations.
// NT: threads of the CTA. TZR + 1 warps make two rounds of face jobs;
// launches with fewer tiles than the GPU has SMs take 2 TZR + 3, one round,
// so that each SM holds more warps of the few tiles there are. Every phase
// but the last spreads its work over all threads, and the last (one cell per
// thread) uses the first TX x TZR. TZR: tile rows.
template <bool GEN = false, int NT = FP64_THREADS, int TZR = TZ>
__device__ __forceinline__ void stage_tile(const StageArgs& a, int tile, TileSmem<TZR>& S) {
  const Geom& g = a.g;
  const int tid = threadIdx.x;
  const int tzi = tile / a.tiles_x;
  const int txi = tile - tzi * a.tiles_x;
  const int k0 = a.row0 + tzi * TZR;
  const int i0 = txi * TX;
  const int nz = g.nz, nx = g.nx, n1 = g.n1;
  const int row_hi = a.rhs_only ? a.rhs_hi : nz;
  const size_t plane = (size_t)nz * g.pitch;
  const bool odd_stage = !a.rhs_only && (a.stage & 1);  // stages 2, 4, ... (1-based)
  const double* Ra = reinterpret_cast<const double*>(a.b.Ra);
  const double hF = g.hF;

  // stage value of component c at row k, column i of the grid
  auto stage_value = [&](int c, int k, int i) -> double {
    const size_t off = (size_t)c * plane + (size_t)k * g.pitch + i;
    if (a.rhs_only) return a.rhs_in[off];
    const bool slow_rows = k < g.n1_r;
    const double* base = slow_rows ? a.b.qA : a.qF;
    const double h = slow_rows ? g.dt : hF;
    return odd_stage ? __fma_rn(h, Ra[off], base[off]) : base[off];
  };

  // ---- 1. stage state of the tile and its halo; u, w, e on the ring ------
  bool bad = false, good = false;  // some cell outside, inside the fixed-point range
  for (int e = tid; e < (TZR + 4) * (TX + 4); e += NT) {
    const int rr = e / (TX + 4), cc = e - rr * (TX + 4);
    const int k = k0 - 2 + rr;
    if (k < 0 || k >= nz) {
      // read by faces next to a wall, which replace it by the mirror cell
#pragma unroll
      for (int c = 0; c < 4; c++) {
        S.q[c][rr][cc] = 0.0;
        S.qi[c][rr][cc] = 0;
      }
      S.qw[0][rr][cc] = S.qw[1][rr][cc] = 0;
      continue;
    }
    bool gh;
    const int i = halo_col(i0 - 2 + cc, nx, g.xwall, &gh);
    double val[4];
    if (GEN && !a.rhs_only) {
      const size_t off = (size_t)k * g.pitch + i;
      const bool slow_rows = k < g.n1_r;
      gen_stage_values(g, (slow_rows ? a.b.qA : a.qF) + off, Ra + off, 4 * plane, plane, a.stage % g.s,
                       slow_rows ? g.dt : hF, val);
    } else {
#pragma unroll
      for (int c = 0; c < 4; c++) val[c] = stage_value(c, k, i);
    }
    if (gh) val[1] = -val[1];  // mirror state beyond an x wall
#pragma unroll
    for (int c = 0; c < 4; c++) S.q[c][rr][cc] = val[c];
    const bool in = a.fx.on && cell_in_range(val[0], val[1], val[2], val[3]);
    bad |= !in;
    good |= in;
    if (!in) continue;  // no face in fixed point reads the cell
    i64 t[4];
#pragma unroll
    for (int c = 0; c < 4; c++) {
      t[c] = c == 1 || c == 2 ? fx::from_double(__double_as_longlong(val[c]), fx::S_MOM - 2)
                              : fx::from_positive(__double_as_longlong(val[c]), fx::S_RHO - 2);
      S.qi[c][rr][cc] = t[c];
      if (c == 1 || c == 2) S.qw[c - 1][rr][cc] = fx::pack(__double_as_longlong(val[c]));
    }
    ring_cell<i64, TZR>(g, S, rr, cc, i0, t[0], t[1], t[2], t[3]);
  }
  const bool has_gamma = (n1 >= k0 && n1 <= k0 + TZR);
  bad = __syncthreads_or(bad);
  bool none = false;  // no cell inside: every face in double
  if (bad) none = !__syncthreads_or(good);

  // ---- 2. face fluxes ----------------------------------------------------
  static_assert(TX == 32 && NT % 32 == 0, "a job is one warp wide");
  bool slow = false;
  const int jobs = none ? 0 : 2 * TZR + 2 + has_gamma;
  const int warp = __shfl_sync(0xffffffffu, tid / 32, 0), lane = tid % 32;
  const bool plain = !bad && tile_plain<TZR>(g, k0, row_hi);
  for (int job = warp; job < jobs; job += NT / 32) {
    FaceId id;
    i64 L[4], R[4], vL[5], vR[5], Vn = 0, VE, F[4];
    int fl;
    bool ok = true;
    FxStress Vt;
    if (plain) {
      if (!face_id_plain<TZR>(job, lane, k0, &id)) continue;
      fl = k0 >= n1;
      if (id.isx) {
        face_sides_plain<true, TZR>(S, id, L, R, vL, vR);
        Vt = visc_tan_plain<true, TZR>(a.fx, S, id, fl);
      } else {
        face_sides_plain<false, TZR>(S, id, L, R, vL, vR);
        Vt = visc_tan_plain<false, TZR>(a.fx, S, id, fl);
      }
    } else {
      const bool valid = face_id<TZR>(g, job, lane, k0, row_hi, &id);
      if (bad) ok = row_in_range(id, i0, nx, valid && !face_in_range<TZR>(g, S, id, k0));
      if (!valid) continue;
      if (ok) {
        fl = face_sides<i64, TZR>(g, a.fx, S, id, L, R, vL, vR);
        Vt = visc_tan<TZR>(g, a.fx, S, id, fl);
      }
    }
    if (ok) {
      const i64 snt = stress59(Vt);
      if (fl < 2) fx_visc(a.fx.fc[id.isx ? 0 : 1][fl], vL, vR, snt, &Vn, &VE);
      else VE = lid_work(a.fx, vL[1], vR[1], snt) + lid_heat(a.fx, vL[2], vR[2]);
      FxTan t;
      ok = fx_flux<2>(g, a.fx, L, R, Vn, VE, F, &t);
      if (ok) {
        F[3] = F[2];
        F[2] = !plain   ? face_tan<TZR>(g, S, id, t, Vt)
               : id.isx ? face_tan_plain<true, TZR>(S, id, t, Vt)
                        : face_tan_plain<false, TZR>(S, id, t, Vt);
        store_flux(S, id, F);
      }
    }
    S.slow[job * TX + lane] = !ok;
    slow |= !ok;
  }
  slow = none || __syncthreads_or(slow);
  if (slow) slow_faces<NT, TZR>(g, a.fx, S, k0, i0, row_hi, none);

  chain_next();

  // ---- 3. R = -div F* + s and the stage combination ----------------------
  {
    const int rr = tid / TX, cc = tid - rr * TX;
    const int k = k0 + rr, i = i0 + cc;
    if (rr >= TZR || k >= row_hi || i >= nx) return;
    const bool under_gamma = (k == n1 - 1);
    const double hx = 0.5 * g.inv_dx, hz = 0.5 * (k < n1 ? g.inv_dz1 : g.inv_dz2);
    const double s57 = 1.0 / (double)(1ll << fx::S_FLUX);
    double R[4];
    bool s0 = false, s1 = false, s2 = false, s3 = false;  // slow faces of the cell: left, right, lower, upper
    if (slow) {
      s0 = S.slow[(TZR + rr) * TX + cc];
      s1 = S.slow[cc < TX - 1 ? (TZR + rr) * TX + cc + 1 : (2 * TZR + 1) * TX + rr];
      s2 = S.slow[rr * TX + cc];
      s3 = S.slow[(under_gamma ? 2 * TZR + 2 : rr + 1 < TZR ? rr + 1 : 2 * TZR) * TX + cc];
    }
    if (s0 && s1 && s2 && s3) {
#pragma unroll
      for (int c = 0; c < 4; c++) {
        auto val = [&](i64 f) { return __longlong_as_double(f); };
        const double dx = __dsub_rn(val(S.fx[c][rr][cc]), val(S.fx[c][rr][cc + 1]));
        const double dz = __dsub_rn(val(S.fz[c][rr][cc]), val(under_gamma ? S.fg[c][cc] : S.fz[c][rr + 1][cc]));
        R[c] = __fma_rn(hx, dx, __dmul_rn(hz, dz));
      }
    } else if (s0 || s1 || s2 || s3) {
#pragma unroll
      for (int c = 0; c < 4; c++) {
        auto val = [&](i64 f, bool sl) { return sl ? __longlong_as_double(f) : __dmul_rn((double)f, s57); };
        const bool tx = c == 2, tz = c == 1;  // the tangential momentum of x and z faces
        const double dx = __dsub_rn(val(S.fx[c][rr][cc], s0 || tx), val(S.fx[c][rr][cc + 1], s1 || tx));
        const double dz = __dsub_rn(val(S.fz[c][rr][cc], s2 || tz),
                                    val(under_gamma ? S.fg[c][cc] : S.fz[c][rr + 1][cc], s3 || tz));
        R[c] = __fma_rn(hx, dx, __dmul_rn(hz, dz));
      }
    } else {
      const double sz = a.fx.scale_z[k >= n1];
#pragma unroll
      for (int c = 0; c < 4; c++) {
        const i64 x0 = S.fx[c][rr][cc], x1 = S.fx[c][rr][cc + 1];
        const i64 z0 = S.fz[c][rr][cc], z1 = under_gamma ? S.fg[c][cc] : S.fz[c][rr + 1][cc];
        auto diff = [&](i64 f, i64 h) { return __dsub_rn(__longlong_as_double(f), __longlong_as_double(h)); };
        if (c == 1) R[c] = __fma_rn(a.fx.scale, (double)(x0 - x1), __dmul_rn(hz, diff(z0, z1)));
        else if (c == 2) R[c] = __fma_rn(sz, (double)(z0 - z1), __dmul_rn(hx, diff(x0, x1)));
        else if (a.fx.square) R[c] = __dmul_rn(a.fx.scale, (double)((x0 - x1) + (z0 - z1)));
        else R[c] = __fma_rn(a.fx.scale, (double)(x0 - x1), __dmul_rn(sz, (double)(z0 - z1)));
      }
    }
    R[2] = __fma_rn(-g.G, S.q[0][rr + 2][cc + 2], R[2]);
    R[3] = __fma_rn(-g.G, S.q[2][rr + 2][cc + 2], R[3]);

    const size_t row_off = (size_t)k * g.pitch + i;
    if (a.rhs_only) {
#pragma unroll
      for (int c = 0; c < 4; c++) a.rhs_out[(size_t)c * plane + row_off] = R[c];
      return;
    }
    double* Ra_w = reinterpret_cast<double*>(a.b.Ra);
    const int st = a.stage;
    const double h2 = g.h2;
    if (GEN) {
      // general s-stage base: R to slot p; F rows finish a substep with the
      // weights b/m, B rows accumulate b_p R over the slow step, S rows finish
      // after the first substep
      double* Rs = reinterpret_cast<double*>(a.b.Ra);
      const size_t slot = 4 * plane;
      const int s = g.s, p = st % s;
      const bool sub_end = (p == s - 1);
      const bool b_row = k >= g.nS_r && k < g.n1_r;
      double w[4];
      if (sub_end && !b_row) gen_weighted_sums(g, Rs + row_off, slot, plane, R, w);
#pragma unroll
      for (int c = 0; c < 4; c++) {
        const size_t o = (size_t)c * plane + row_off;
        const double r = R[c];
        if (!sub_end) Rs[(size_t)p * slot + o] = r;
        if (b_row) {
          const size_t pb = (size_t)(g.n1_r - g.nS_r) * g.pitch;
          double* acc = a.b.accB + (size_t)c * pb + (size_t)(k - g.nS_r) * g.pitch + i;
          const double v = (st == 0) ? __dmul_rn(g.bb[p], r) : __fma_rn(g.bb[p], r, *acc);
          *acc = (st == s * g.m - 1) ? __fma_rn(g.hF, v, a.b.qA[o]) : v;
        } else if (sub_end) {
          if (k >= g.n1_r) a.qF_next[o] = __fma_rn(g.hF, w[c], a.qF[o]);
          else a.b.accS[(size_t)c * ((size_t)g.nS_r * g.pitch) + row_off] = __fma_rn(g.dt, w[c], a.b.qA[o]);
        }
      }
      return;
    }
    if (k >= g.n1_r) {
      // fast region: m Heun substeps of dt/m
      if (!(st & 1)) {
#pragma unroll
        for (int c = 0; c < 4; c++) Ra_w[(size_t)c * plane + row_off] = R[c];
      } else {
#pragma unroll
        for (int c = 0; c < 4; c++) {
          const size_t o = (size_t)c * plane + row_off;
          a.qF_next[o] = __fma_rn(h2, __dadd_rn(Ra[o], R[c]), a.qF[o]);
        }
      }
    } else if (k >= g.nS_r) {
      // buffer: RK2 restarted from q_n each substep, weights 1/(2m)
      const size_t pb = (size_t)(g.n1_r - g.nS_r) * g.pitch;
      const size_t ob = (size_t)(k - g.nS_r) * g.pitch + i;
      const bool last = (st == 2 * g.m - 1);
#pragma unroll
      for (int c = 0; c < 4; c++) {
        const size_t o = (size_t)c * plane + row_off;
        double* acc = a.b.accB + (size_t)c * pb + ob;
        if (!(st & 1)) Ra_w[o] = R[c];
        if (st == 0) {
          *acc = R[c];
        } else if (last) {
          *acc = __fma_rn(h2, __dadd_rn(*acc, R[c]), a.b.qA[o]);
        } else {
          *acc = __dadd_rn(*acc, R[c]);
        }
      }
    } else {
      // slow region: evaluated at stages 1 and 2 only (Algorithm 1)
      const size_t ps = (size_t)g.nS_r * g.pitch;
#pragma unroll
      for (int c = 0; c < 4; c++) {
        const size_t o = (size_t)c * plane + row_off;
        if (st == 0) {
          Ra_w[o] = R[c];
        } else {
          a.b.accS[(size_t)c * ps + row_off] = __fma_rn(g.hdt, __dadd_rn(Ra[o], R[c]), a.b.qA[o]);
        }
      }
    }
  }
}

}  // namespace mprk
