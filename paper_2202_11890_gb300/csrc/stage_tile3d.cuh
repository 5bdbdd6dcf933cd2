// stage_tile3d.cuh — the 3-D stage (App. B, Eq. ns-fv-cartesian-3d in full),
// FP64: five conserved variables (rho, rho u, rho v, rho w, rho E), x and y
// periodic, the S/B/F row bands and Gamma in z as in 2-D. Layout of every
// state-sized array: [5][nz][ny][pitch].
//
// A stage is two launches over the active rows:
//  * yface3: one CTA per TX x TZ tile of an x–z plane j computes the y-face
//    fluxes G* between planes j and j+1 of its cells and stores them (face
//    j+1/2 at index j) in a state-sized buffer;
//  * stage3: one CTA per TX x TZ3 tile of plane j computes its x and z faces
//    as the 2-D tile does, takes the y divergence from the stored y faces,
//    adds the source and applies the stage combination.
// Every face is computed once. Viscous fluxes use the common face values
// of App. B: mean velocity, two-point normal derivatives, tangential
// derivatives averaged from the two cells' central differences, sigma =
// mu (grad u + grad u^T - 2/3 div u I), heat flux -kappa grad T.
//
// As in the 2-D tile, the fluxes of mass, normal momentum and energy run in
// 64-bit fixed point (fixed_point.cuh), because the double pipe bound both
// kernels (80 to 86 % busy with 125 + 238 operations per cell), and those of
// the tangential momenta in integers with an exponent. Measured: a slow step
// of 512 x 64 x 200 cells with m = 4 44.1 -> 11.3 ms. Faces whose cells leave
// the range are evaluated in double by a second pass over the tile, a row of 32
// at a time (row_in_range in stage_tile.cuh), so neighbouring tiles agree on the
// faces they share. Fluxes come over half the divergence factor of their
// direction, as .57 integers or as doubles (flux_tag).
#pragma once

#include "fixed_flux.cuh"
#include "fp64_recip.cuh"
#include "mprk_internal.h"
#include "stage_tile.cuh"

namespace mprk {

constexpr int NC3 = 5;

// Lax–Friedrichs flux (Sec. 2.1) in a face frame, in double: a state is (rho,
// m_n, m_t1, m_t2, rho E); lambda is the largest |u_n| + a over the left,
// right and Roe-averaged states. V: the viscous part.
__device__ __forceinline__ void lf_face5(const Geom& g, const double l[5], const double r[5], const double V[4],
                                         double out[5]) {
  const double invL = recip_f64(l[0]), invR = recip_f64(r[0]);
  const double unL = __dmul_rn(l[1], invL), t1L = __dmul_rn(l[2], invL), t2L = __dmul_rn(l[3], invL);
  const double unR = __dmul_rn(r[1], invR), t1R = __dmul_rn(r[2], invR), t2R = __dmul_rn(r[3], invR);
  const double kL = __fma_rn(l[3], t2L, __fma_rn(l[2], t1L, __dmul_rn(l[1], unL)));
  const double kR = __fma_rn(r[3], t2R, __fma_rn(r[2], t1R, __dmul_rn(r[1], unR)));
  const double pL = __dmul_rn(g.gm1, __fma_rn(-0.5, kL, l[4])), pR = __dmul_rn(g.gm1, __fma_rn(-0.5, kR, r[4]));
  const double eL = __dadd_rn(l[4], pL), eR = __dadd_rn(r[4], pR);
  const double lam = face_speed(g, l[0], r[0], unL, unR, __dsub_rn(t1R, t1L), __dsub_rn(t2R, t2L),
                                __dmul_rn(__dmul_rn(g.gamma, pL), invL), __dmul_rn(__dmul_rn(g.gamma, pR), invR));
  out[0] = __fma_rn(lam, __dsub_rn(l[0], r[0]), __dadd_rn(l[1], r[1]));
  const double f1 = __dsub_rn(__dadd_rn(__fma_rn(l[1], unL, pL), __fma_rn(r[1], unR, pR)), V[0]);
  out[1] = __fma_rn(lam, __dsub_rn(l[1], r[1]), f1);
  out[2] = __fma_rn(lam, __dsub_rn(l[2], r[2]), __fma_rn(r[2], unR, __fma_rn(l[2], unL, -V[1])));
  out[3] = __fma_rn(lam, __dsub_rn(l[3], r[3]), __fma_rn(r[3], unR, __fma_rn(l[3], unL, -V[2])));
  out[4] = __fma_rn(lam, __dsub_rn(l[4], r[4]), __fma_rn(unR, eR, __fma_rn(unL, eL, -V[3])));
}

// One side of a face in its frame: velocity (u_n, u_t1, u_t2), e = T / (gamma
// (gamma - 1)), and the cell's central differences (unscaled) of u_n and u_t1
// along t1 (g1) and of u_n and u_t2 along t2 (g2). The fixed-point form uses
// neither difference of u_n.
template <typename T>
struct VSide {
  T u[3], e, g1[2], g2[2];
};

// ---- shared helpers --------------------------------------------------------

struct Geo3 {
  int nx, ny, nz, n1, pitch;
  size_t plane;  // elements of one component
  __device__ __forceinline__ size_t at(int c, int k, int j, int i) const {
    return ((size_t)c * nz + k) * ny * (size_t)pitch + (size_t)j * pitch + i;
  }
};
__device__ __forceinline__ Geo3 geo3(const Geom& g) {
  Geo3 s;
  s.nx = g.nx;
  s.ny = g.ny;
  s.nz = g.nz;
  s.n1 = g.n1;
  s.pitch = g.pitch;
  s.plane = (size_t)g.nz * g.ny * g.pitch;
  return s;
}
__device__ __forceinline__ int wrap3(int i, int n) {
  if (i < 0) i += n;
  if (i >= n) i -= n;
  if (i < 0 || i >= n) i = ((i % n) + n) % n;  // only for grids narrower than the tile halo
  return i;
}

// The stage value (q_n, or q_n + h R_a on the second stage of a substep) of
// every component at (k, j, i); the full state given by rhs_in for the test
// hook.
__device__ __forceinline__ void stage_val3(const StageArgs& a, const Geo3& G, int k, int j, int i, double q[5]) {
  const Geom& g = a.g;
  const bool slow = k < g.n1_r;
  const double* base = a.rhs_only ? a.rhs_in : (slow ? a.b.qA : a.qF);
  const size_t o = G.at(0, k, j, i);
#pragma unroll
  for (int c = 0; c < 5; c++) q[c] = base[o + c * G.plane];
  if (!a.rhs_only && (a.stage & 1)) {
    const double h = slow ? g.dt : g.hF;
    const double* Ra = reinterpret_cast<const double*>(a.b.Ra);
#pragma unroll
    for (int c = 0; c < 5; c++) q[c] = __fma_rn(h, Ra[o + c * G.plane], q[c]);
  }
}
__device__ __forceinline__ bool cell_in_range3(const double q[5]) {
  return in_range(q[0], max(abs_word(q[1]), max(abs_word(q[2]), abs_word(q[3]))), q[4]);
}

// The two arithmetics of the tiles: i64 (fixed point) and double.
template <typename T>
struct Arith3;
template <>
struct Arith3<i64> {
  static __device__ __forceinline__ i64 cell(double q, int c) {  // rho, rho E .58, momenta .60
    return fx::from_double(__double_as_longlong(q), c == 0 || c == 4 ? fx::S_RHO - 2 : fx::S_MOM - 2);
  }
  static __device__ __forceinline__ i64 rec(i64 a, i64 up, i64 dn) { return (a << 2) + (up - dn); }
  // u, v, w, e of a cell; 1/rho .61
  static __device__ __forceinline__ i64 prims(const i64 q[5], i64 v[4]) {
    const i64 inv_ = fx::recip(q[0] << 2);
    const FxW inv = fx::split(inv_);
    i64 k = 0;
#pragma unroll
    for (int c = 0; c < 3; c++) {
      const FxW m = fx::split(q[c + 1] << 2);
      v[c] = fx::mul(m, inv);
      k += fx::mul(m, fx::split(v[c]));
    }
    v[3] = fx::mul(fx::split((q[4] - k) << 2), inv) << 2;  // k .57: k/2 .58
    return inv_;
  }
};
template <>
struct Arith3<double> {
  static __device__ __forceinline__ double cell(double q, int) { return q; }
  static __device__ __forceinline__ double rec(double a, double up, double dn) {
    return __fma_rn(0.25, __dsub_rn(up, dn), a);
  }
  static __device__ __forceinline__ double prims(const double q[5], double v[4]) {
    const double inv = recip_f64(q[0]);
    double k = 0.0;
#pragma unroll
    for (int c = 0; c < 3; c++) {
      v[c] = __dmul_rn(q[c + 1], inv);
      k = __fma_rn(q[c + 1], v[c], k);
    }
    v[3] = __dmul_rn(__fma_rn(-0.5, k, q[4]), inv);
    return inv;
  }
};

// A stored flux of mass, normal momentum or energy: the .57 integer itself
// (|F| < 8, so its top four bits agree) or the bits of a double, whose top
// four bits differ for 2^-511 <= |F| < 2^513. Smaller doubles store as zero,
// larger ones and NaN as the positive NaN. Tangential momenta are doubles.
__device__ __forceinline__ bool flux_is_double(i64 f) {
  return (unsigned)((int)(f >> 32) + 0x10000000) >= 0x20000000u;
}
__device__ __forceinline__ i64 flux_tag(double f) {
  const unsigned h = (unsigned)__double2hiint(f) & 0x7fffffffu;
  if (h < 0x20000000u) return 0;
  return h < 0x60000000u ? __double_as_longlong(f) : 0x7ff8000000000000ll;
}
__device__ __forceinline__ double flux_value(i64 f) {
  if (flux_is_double(f)) return __longlong_as_double(f);
  return __dmul_rn((double)f, 1.0 / (double)(1ll << fx::S_FLUX));
}

// Central z difference (unscaled) of velocity component comp at row k from
// the cell and its neighbours above and below (v, rows of stride vr), with
// the ghost 2 (wall state) - cell beyond a wall or Gamma; component 2 (w) is
// normal there.
template <typename T>
__device__ __forceinline__ T dz_vel(const Geom& g, const FxConst& c, int k, int comp, const T* v, int vr) {
  const T u = v[0];
  T up, dn;
  if (k + 1 == g.nz) up = (comp == 2 || !g.wall) ? -u : u;
  else if (k + 1 == g.n1) up = comp == 2 ? -u : lid_ghost(g, c, 0, u, v[vr]);  // fluid 1's top row
  else up = v[vr];
  if (k == 0) dn = (comp == 2 || !g.wall) ? -u : u;
  else if (k == g.n1) dn = comp == 2 ? -u : lid_ghost(g, c, 1, u, v[-vr]);  // fluid 2's bottom row
  else dn = v[-vr];
  return up - dn;
}

// Viscous flux in the face frame over half the divergence factor: (sigma_nn,
// sigma_nt1, sigma_nt2, u^.sigma_n + kappa dT/dn). With G[a][b] = d u_a /
// d x_b (b = normal, t1, t2): sigma_nn = mu (4/3 G00 - 2/3 (G11 + G22)),
// sigma_nt = mu (G_t0 + G_0t); the derivative factors sit in the coefficients.
// In fixed point only sigma_nn and the energy, with the other two (snt) .59.
__host__ __device__ __forceinline__ void visc3(const FxW* f, const VSide<i64>& L, const VSide<i64>& R, const i64 snt[2],
                                               i64* Vn, i64* VE) {
  *Vn = fx::mul2(f[F3_A], fx::split(R.u[0] - L.u[0]), f[F3_B1], fx::split(L.g1[1] + R.g1[1])) +
        fx::mul(fx::split(L.g2[1] + R.g2[1]), f[F3_B2]);
  // (u_L + u_R) . sigma: .61 x .59 -> .56, half of it at .57
  i64 us = fx::mul(fx::split((L.u[0] + R.u[0]) << 2), fx::split(*Vn << 2));
#pragma unroll
  for (int t = 0; t < 2; t++) us += fx::mul(fx::split((L.u[1 + t] + R.u[1 + t]) << 2), fx::split(snt[t]));
  *VE = us + fx::mul(fx::split(R.e - L.e), f[F3_K]);
}
__device__ __forceinline__ void visc3(const Fx3Const& c, int dir, int fl, const VSide<double>& L,
                                      const VSide<double>& R, double V[4]) {
  const double* f = c.fd[dir][fl];
  V[0] = __fma_rn(f[F3_A], __dsub_rn(R.u[0], L.u[0]),
                  __fma_rn(f[F3_B1], __dadd_rn(L.g1[1], R.g1[1]), __dmul_rn(f[F3_B2], __dadd_rn(L.g2[1], R.g2[1]))));
  V[1] = __fma_rn(f[F3_C], __dsub_rn(R.u[1], L.u[1]), __dmul_rn(f[F3_D1], __dadd_rn(L.g1[0], R.g1[0])));
  V[2] = __fma_rn(f[F3_C], __dsub_rn(R.u[2], L.u[2]), __dmul_rn(f[F3_D2], __dadd_rn(L.g2[0], R.g2[0])));
  double us = 0.0;
#pragma unroll
  for (int q = 0; q < 3; q++) us = __fma_rn(__dadd_rn(L.u[q], R.u[q]), V[q], us);
  V[3] = __fma_rn(0.5, us, __dmul_rn(f[F3_K], __dsub_rn(R.e, L.e)));
}

// The face flux in double: the tangential momenta as they are, the others
// tagged.
__device__ __forceinline__ void flux3(const Geom& g, const double L[5], const double R[5], const double V[4], i64 F[5]) {
  double o[5];
  lf_face5(g, L, R, V, o);
#pragma unroll
  for (int q = 0; q < 5; q++) F[q] = q == 2 || q == 3 ? __double_as_longlong(o[q]) : flux_tag(o[q]);
}

// ---- y faces ------------------------------------------------------------------

constexpr int RING3 = (TZ + 2) * (TX + 2);  // tile plus a one-cell ring
struct YfaceSmem {
  i64 q[2][5][TZ + 2][TX + 2];    // planes j and j+1, rows k0-1.., cols i0-1..
  i64 v[2][4][TZ + 2][TX + 2];    // u, v, w, e on the ring
  // packed momenta (fixed_point.cuh) and velocities under their exponents: u
  // and w in the tile's cells, v on the ring with its exponents alone
  i64 vn[2][TZ + 2][TX + 2];
  short wn[2][TZ + 2][TX + 2];
  i64 wt[2][2][TZ][TX], vt[2][2][TZ][TX];
  unsigned char ok[2][TZ + 2][TX + 2];
};

// The y face between planes j and j+1 of the thread's cell (k, i), in T, from
// the tile's cells restaged as T. First pass (T = i64): returns whether the
// face was stored in fixed point; its barrier-separated second pass (T =
// double) stores the others (want).
template <typename T>
__device__ __forceinline__ bool yface_pass(const StageArgs& a, const Fx3Const& C, int k0, int i0, int j, YfaceSmem& S,
                                           bool want) {
  constexpr bool FX = sizeof(T) == 8 && (T)0.5 == (T)0;
  const Geom& g = a.g;
  const Geo3 G = geo3(g);
  const int tid = threadIdx.x;
  const int nz = g.nz, n1 = g.n1;
  const int row_hi = a.rhs_only ? a.rhs_hi : nz;
  const int j1 = wrap3(j + 1, g.ny);
  T* Sq = reinterpret_cast<T*>(&S.q[0][0][0][0]);
  T* Sv = reinterpret_cast<T*>(&S.v[0][0][0][0]);
  bool bad = false;
  for (int e = tid; e < 2 * RING3; e += NTHREADS) {
    const int side = e >= RING3, rem = e - side * RING3;
    const int rr = rem / (TX + 2), cc = rem - rr * (TX + 2);
    const int k = k0 - 1 + rr;
    if (k < 0 || k >= nz) {
      if (FX) S.wn[side][rr][cc] = 0;
      continue;
    }
    double q[5];
    stage_val3(a, G, k, side ? j1 : j, wrap3(i0 - 1 + cc, g.nx), q);
    bool in = true;
    if (FX) {
      in = cell_in_range3(q);
      S.ok[side][rr][cc] = in;
      bad |= !in;
    }
    if (FX && !in) continue;  // no face in fixed point reads the cell
    T t[5], v[4];
#pragma unroll
    for (int c = 0; c < 5; c++) {
      t[c] = Arith3<T>::cell(q[c], c);
      Sq[(side * 5 + c) * RING3 + rem] = t[c];
    }
    const T inv = Arith3<T>::prims(t, v);
#pragma unroll
    for (int c = 0; c < 4; c++) Sv[(side * 4 + c) * RING3 + rem] = v[c];
    if constexpr (FX) {
      const FxW iw = fx::split(inv);
      const i64 w = fx::pack(__double_as_longlong(q[2]));
      S.wn[side][rr][cc] = (short)fx::pack_exp(w);
      S.vn[side][rr][cc] = fx::packed_velocity(w, iw);
      if (rr >= 1 && rr <= TZ && cc >= 1 && cc <= TX) {
#pragma unroll
        for (int c = 0; c < 2; c++) {
          const i64 m = fx::pack(__double_as_longlong(q[2 * c + 1]));
          S.wt[side][c][rr - 1][cc - 1] = m;
          S.vt[side][c][rr - 1][cc - 1] = fx::packed_velocity(m, iw);
        }
      }
    }
  }
  const int rr = tid / TX, cc = tid - rr * TX;
  const int k = k0 + rr, i = i0 + cc;
  const bool mine = k < row_hi && i < g.nx;
  // the outer two of the four cells across the face
  T am[5], ap[5];
  i64 wm[2], wp[2];  // their rho u, rho w packed
  bool out_ok = true;
  if (mine && want) {
    double q[5];
    stage_val3(a, G, k, wrap3(j - 1, g.ny), i, q);
    out_ok = cell_in_range3(q);
    if (FX) wm[0] = fx::pack(__double_as_longlong(q[1])), wm[1] = fx::pack(__double_as_longlong(q[3]));
#pragma unroll
    for (int c = 0; c < 5; c++) am[c] = Arith3<T>::cell(q[c], c);
    stage_val3(a, G, k, wrap3(j + 2, g.ny), i, q);
    out_ok = out_ok && cell_in_range3(q);
    if (FX) wp[0] = fx::pack(__double_as_longlong(q[1])), wp[1] = fx::pack(__double_as_longlong(q[3]));
#pragma unroll
    for (int c = 0; c < 5; c++) ap[c] = Arith3<T>::cell(q[c], c);
  }
  if (FX) bad = __syncthreads_or(bad);
  else __syncthreads();
  if (FX) {
    if (bad && mine) {
      // the face's own cells: the four across it and the x and z neighbours
      // of the two at it (inside the grid)
      for (int s = 0; s < 2; s++) {
        out_ok = out_ok && S.ok[s][rr + 1][cc + 1] && S.ok[s][rr + 1][cc] && S.ok[s][rr + 1][cc + 2];
        if (k > 0) out_ok = out_ok && S.ok[s][rr][cc + 1];
        if (k + 1 < nz) out_ok = out_ok && S.ok[s][rr + 2][cc + 1];
      }
    }
    // one face outside takes its row to the double pass (row_in_range)
    if (__any_sync(0xffffffffu, !out_ok)) return !mine;
  }
  if (!mine || !want) return true;
  // face frame: normal rho v, t1 rho u, t2 rho w
  const int at = (rr + 1) * (TX + 2) + cc + 1;
  T L[5], R[5];
#pragma unroll
  for (int c = 0; c < 5; c++) {
    const int f = c == 1 ? 2 : (c == 2 ? 1 : c);
    const T a0 = Sq[f * RING3 + at], a1 = Sq[(5 + f) * RING3 + at];
    L[c] = Arith3<T>::rec(a0, a1, am[f]);
    R[c] = Arith3<T>::rec(a1, a0, ap[f]);
  }
  VSide<T> s[2];
#pragma unroll
  for (int side = 0; side < 2; side++) {
    const T* V = Sv + side * 4 * RING3 + at;
    s[side].u[0] = V[RING3];
    s[side].u[1] = V[0];
    s[side].u[2] = V[2 * RING3];
    s[side].e = V[3 * RING3];
    if (!FX) {
      s[side].g1[0] = V[RING3 + 1] - V[RING3 - 1];             // x and z differences of v
      s[side].g2[0] = dz_vel(g, C.k, k, 1, V + RING3, TX + 2);
    }
    s[side].g1[1] = V[1] - V[-1];                              // x difference of u
    s[side].g2[1] = dz_vel(g, C.k, k, 2, V + 2 * RING3, TX + 2);  // z difference of w
  }
  i64 F[5];
  if constexpr (FX) {
    const FxN* tc = C.tc[1][k >= n1];
    const i64* vn = &S.vn[0][rr + 1][cc + 1];
    const short* wn = &S.wn[0][rr + 1][cc + 1];
    const i64* vt = &S.vt[0][0][rr][cc];
    const i64* wt = &S.wt[0][0][rr][cc];
    constexpr int CELLS = TZ * TX;
    const FxStress sig[2] = {
        tan_stress(tc[0], vel_diff(vt, wt, 2 * CELLS, 2 * CELLS), tc[1], vel_cross(vn, wn, RING3, RING3, 1, 1)),
        tan_stress(tc[0], vel_diff(vt + CELLS, wt + CELLS, 2 * CELLS, 2 * CELLS), tc[2],
                   dz_pair(g, C.k, k, vn, vn + RING3, TX + 2, wn, wn + RING3, TX + 2))};
    i64 Vn, VE, o[3];
    FxTan t;
    const i64 snt[2] = {stress59(sig[0]), stress59(sig[1])};
    visc3(C.fc[1][k >= n1], s[0], s[1], snt, &Vn, &VE);
    if (!fx_flux<3>(g, C.k, L, R, Vn, VE, o, &t)) return false;
    F[0] = o[0], F[1] = o[1], F[4] = o[2];
#pragma unroll
    for (int c = 0; c < 2; c++)
      F[2 + c] = tan_flux(t, wm[c], wt[c * CELLS], wt[(2 + c) * CELLS], wp[c], sig[c]);
  } else {
    T V[4];
    visc3(C, 1, k >= n1, s[0], s[1], V);
    flux3(g, L, R, V, F);
  }
#pragma unroll
  for (int c = 0; c < 5; c++) {
    const int f = c == 1 ? 2 : (c == 2 ? 1 : c);
    reinterpret_cast<i64*>(a.gy)[G.at(f, k, j, i)] = F[c];
  }
  return true;
}
__device__ __noinline__ void yface_slow(const StageArgs& a, const Fx3Const& C, int k0, int i0, int j, YfaceSmem& S,
                                        bool want) {
  yface_pass<double>(a, C, k0, i0, j, S, want);
}
__device__ __forceinline__ void yface_tile(const StageArgs& a, const Fx3Const& C, int k0, int i0, int j,
                                           YfaceSmem& S) {
  const bool done = C.k.on && yface_pass<i64>(a, C, k0, i0, j, S, true);
  if (__syncthreads_or(!done)) yface_slow(a, C, k0, i0, j, S, !done);
}

// ---- x and z faces, divergence and stage combination ----------------------

// TX x TZ3 cells: 13 warps, two face jobs each (face_id in stage_tile.cuh). 110
// KB of shared memory, two CTAs (26 warps) per SM; as TX x 8 tiles the packed
// momenta and their velocities would not leave room for three.
constexpr int TZ3 = 12;
constexpr int TILE3_THREADS = TX * (TZ3 + 1);
constexpr int RINGS = (TZ3 + 2) * (TX + 2);
struct Tile3Smem {
  i64 q[5][TZ3 + 4][TX + 4];       // plane j, rows k0-2.., cols i0-2..
  i64 qw[3][TZ3 + 4][TX + 4];      // rho u, rho v, rho w packed (fixed_point.cuh)
  i64 v[4][TZ3 + 2][TX + 2];       // u, v, w, e on the ring
  i64 vp[3][TZ3 + 2][TX + 2];      // u, v, w under the exponents of qw
  // central y differences of u, v, w on the ring: in fixed point v .59, u and w
  // .57 under the exponents ye
  i64 vy[3][TZ3 + 2][TX + 2];
  short ye[2][TZ3 + 2][TX + 2];
  // fluxes: the tangential momenta as doubles, the others tagged
  i64 fx[5][TZ3][TX + 1];          // x face f between cols f-1, f
  i64 fz[5][TZ3 + 1][TX];          // z faces seen from above
  i64 fg[5][TX];                   // interface flux seen from fluid 1
  unsigned char ok[TZ3 + 4][TX + 4];
  unsigned char oky[TZ3 + 2][TX + 2];  // the cells in planes j-1 and j+1
  unsigned char slow[(2 * TZ3 + 3) * TX];  // per face: its job and lane
};

// Phase 1 in T: stage state, velocities and their y differences. Returns
// (T = i64) 0, or 1 where some cell leaves the fixed-point range, or 2 where every
// cell does. Ends with a barrier.
template <typename T>
__device__ __forceinline__ int tile3_cells(const StageArgs& a, const Geo3& G, int k0, int i0, int j, Tile3Smem& S) {
  constexpr bool FX = (T)0.5 == (T)0;
  const Geom& g = a.g;
  const int tid = threadIdx.x, nz = g.nz, n1 = g.n1;
  const int jm = wrap3(j - 1, g.ny), jp = wrap3(j + 1, g.ny);
  constexpr int QP = (TZ3 + 4) * (TX + 4);
  T* q = reinterpret_cast<T*>(&S.q[0][0][0]);
  T* v = reinterpret_cast<T*>(&S.v[0][0][0]);
  bool bad = false, good = false;
  for (int e = tid; e < QP; e += TILE3_THREADS) {
    const int rr = e / (TX + 4), cc = e - rr * (TX + 4);
    const int k = k0 - 2 + rr;
    if (k < 0 || k >= nz) {
      // read by the faces next to a wall, which replace it by the mirror cell
#pragma unroll
      for (int c = 0; c < 5; c++) q[c * QP + e] = (T)0;
      if (FX)
#pragma unroll
        for (int c = 0; c < 3; c++) (&S.qw[0][0][0])[c * QP + e] = 0;
      continue;
    }
    double x[5];
    stage_val3(a, G, k, j, wrap3(i0 - 2 + cc, g.nx), x);
    if (FX) {
      const bool in = cell_in_range3(x);
      S.ok[rr][cc] = in;
      bad |= !in;
      good |= in;
      if (!in) continue;  // no face in fixed point reads the cell
    }
    T t[5];
#pragma unroll
    for (int c = 0; c < 5; c++) {
      t[c] = Arith3<T>::cell(x[c], c);
      q[c * QP + e] = t[c];
    }
    if (FX)
#pragma unroll
      for (int c = 0; c < 3; c++) (&S.qw[0][0][0])[c * QP + e] = fx::pack(__double_as_longlong(x[c + 1]));
    // velocities on the one-cell ring
    if (rr >= 1 && rr <= TZ3 + 2 && cc >= 1 && cc <= TX + 2) {
      T o[4];
      const T inv = Arith3<T>::prims(t, o);
      const int at = (rr - 1) * (TX + 2) + cc - 1;
#pragma unroll
      for (int c = 0; c < 4; c++) v[c * RINGS + at] = o[c];
      if constexpr (FX) {
        const FxW iw = fx::split(inv);
#pragma unroll
        for (int c = 0; c < 3; c++)
          (&S.vp[0][0][0])[c * RINGS + at] = fx::packed_velocity((&S.qw[0][0][0])[c * QP + e], iw);
      }
    }
  }
  for (int e = tid; e < RINGS; e += TILE3_THREADS) {
    const int rr = e / (TX + 2), cc = e - rr * (TX + 2);
    const int k = k0 - 1 + rr;
    if (k < 0 || k >= nz) continue;
    const int i = wrap3(i0 - 1 + cc, g.nx);
    double x[5];
    T d[3], u[2];
    int ex[2];
    bool in = true;
#pragma unroll
    for (int s = 0; s < 2; s++) {
      stage_val3(a, G, k, s ? jm : jp, i, x);
      if (FX) in = in && cell_in_range3(x);
      if (!in) break;
      if constexpr (FX) {
        const FxW inv = fx::split(fx::recip(Arith3<i64>::cell(x[0], 0) << 2));
        const i64 v_ = fx::mul(fx::split(Arith3<i64>::cell(x[2], 2) << 2), inv);
        d[1] = s ? d[1] - v_ : v_;
#pragma unroll
        for (int c = 0; c < 2; c++) {
          const i64 w = fx::pack(__double_as_longlong(x[2 * c + 1])), p = fx::packed_velocity(w, inv);
          const int ew = fx::pack_exp(w);
          if (s) {
            const int em = max(ew, ex[c]);
            d[2 * c] = vel_at(u[c], ex[c], em) - vel_at(p, ew, em);
            S.ye[c][rr][cc] = (short)em;
          } else {
            u[c] = p;
            ex[c] = ew;
          }
        }
      } else {
        const double inv = recip_f64(x[0]);
#pragma unroll
        for (int c = 0; c < 3; c++) d[c] = s ? __dsub_rn(d[c], __dmul_rn(x[c + 1], inv)) : __dmul_rn(x[c + 1], inv);
      }
    }
    if (FX) {
      S.oky[rr][cc] = in;
      bad |= !in;
    }
    if (!in) continue;
#pragma unroll
    for (int c = 0; c < 3; c++) reinterpret_cast<T*>(&S.vy[0][0][0])[c * RINGS + e] = d[c];
  }
  if (!FX) {
    __syncthreads();
    return 0;
  }
  bad = __syncthreads_or(bad);
  if (bad && !__syncthreads_or(good)) return 2;
  return bad;
}

// The flux of face id in T, stored; false where it leaves the range. A
// boundary face (outer wall or interface) has the inner cell's reconstructed
// state on one side and its mirror on the other; an outer wall's viscous
// ghost is 2 wall state - cell.
template <typename T>
__device__ __forceinline__ bool face3(const Geom& g, const Fx3Const& C, Tile3Smem& S, const FaceId& id) {
  constexpr bool FX = (T)0.5 == (T)0;
  constexpr int QP = (TZ3 + 4) * (TX + 4), VW = TX + 2;
  const int n1 = g.n1, nz = g.nz, ku = id.ku, kd = ku - 1;
  const int qs = id.isx ? 1 : TX + 4;
  const int q0 = id.isx ? (id.f + 2) * (TX + 4) + id.c : id.f * (TX + 4) + id.c + 2;
  // component planes of the normal and the tangents: x (u; v, w), z (w; u, v)
  const int pn = id.isx ? 1 : 3, p1 = id.isx ? 2 : 1, p2 = id.isx ? 3 : 2;
  const bool wall = !id.isx && (ku == 0 || ku == nz), lidf = !id.isx && ku == n1;
  const bool from_above = ku == 0 || (lidf && !id.below);
  const bool mir0 = !id.isx && (kd == 0 || kd == n1), mir3 = !id.isx && (ku == nz - 1 || ku == n1 - 1);
  const int dir = id.isx ? 0 : 2, fl = (id.isx ? ku : (ku == 0 ? 0 : kd)) >= n1;
  // the first cell at the face on the ring; in double its velocity planes
  const int vo = id.isx ? (id.f + 1) * VW + id.c : id.f * VW + id.c + 1, vs = id.isx ? 1 : VW;
  const T* q = reinterpret_cast<const T*>(&S.q[0][0][0]) + q0;
  const T* v = reinterpret_cast<const T*>(&S.v[0][0][0]) + vo;
  const T* vy1 = reinterpret_cast<const T*>(&S.vy[1][0][0]) + vo;
  T L[5], R[5], V[4];  // FX: V[0] and V[3] only
  FxStress sig[2];     // FX: the tangential stresses
  i64 snt[2];          // the same .59
  if (FX) {
    const i64* p = &S.vp[0][0][0] + vo;
    const i64* m = &S.qw[0][0][0] + q0 + qs;  // the same cell
    const int o1 = (p1 - 1) * RINGS, o2 = (p2 - 1) * RINGS, m1 = (p1 - 1) * QP, m2 = (p2 - 1) * QP;
    if (wall) {  // the ghosts' velocities are +-those of the cell, their differences of w the opposite
      sig[0] = sig[1] = FxStress{0, 0};
      if (!g.wall) {
        const int ov = ku == 0 ? vs : 0, om = ku == 0 ? qs : 0;
#pragma unroll
        for (int c = 0; c < 2; c++) {
          const int e = fx::pack_exp(m[(c ? m2 : m1) + om]);
          const i64 x = vel_at(p[(c ? o2 : o1) + ov], e, e) << 1;
          sig[c] = tan_stress(C.tc[2][fl][0], FxA{ku == 0 ? x : -x, e});
        }
      }
    } else {
      const FxA t1 = vel_diff(p + o1, m + m1, vs, qs), t2 = vel_diff(p + o2, m + m2, vs, qs);
      if (lidf) {
        sig[0] = tan_stress(C.k.ts, t1);
        sig[1] = tan_stress(C.k.ts, t2);
      } else {
        const FxN* tc = C.tc[dir][fl];
        const i64* n = p + (pn - 1) * RINGS;
        const i64* mn = m + (pn - 1) * QP;
        // differences of u_n along y and along the third direction, of both cells
        const i64* y = &S.vy[pn - 1][0][0] + vo;
        const short* ye = &S.ye[id.isx ? 0 : 1][0][0] + vo;
        const int ey = max(ye[0], ye[vs]);
        const FxA gy = {fx::shr(y[0], ey - ye[0]) + fx::shr(y[vs], ey - ye[vs]), ey};
        const FxA gt = id.isx ? dz_pair(g, C.k, ku, n, n + 1, VW, mn, mn + 1, TX + 4) : vel_cross(n, mn, vs, qs, 1, 1);
        sig[0] = tan_stress(tc[0], t1, tc[1], id.isx ? gy : gt);
        sig[1] = tan_stress(tc[0], t2, tc[2], id.isx ? gt : gy);
      }
    }
#pragma unroll
    for (int c = 0; c < 2; c++) snt[c] = stress59(sig[c]);
  }
  if (lidf) {
    // the bulk fluxes, with the wall velocities (one value for both fluids)
    V[0] = 0;
    V[3] = lid_heat(C.k, v[3 * RINGS], v[3 * RINGS + VW]);
#pragma unroll
    for (int c = 0; c < 2; c++) {
      const T u1 = v[c * RINGS], u2 = v[c * RINGS + VW];
      if constexpr (FX) {
        V[3] += lid_work(C.k, u1, u2, snt[c]);
      } else {
        V[1 + c] = __dmul_rn(C.k.tlid[LID_S], __dsub_rn(u2, u1));
        V[3] = __dadd_rn(V[3], lid_work(C.k, u1, u2, V[1 + c]));
      }
    }
  } else {
    VSide<T> s[2];
#pragma unroll
    for (int side = 0; side < 2; side++) {
      const T* p = v + side * vs;
      const T* y = vy1 + side * vs;
      s[side].u[0] = p[(pn - 1) * RINGS];
      s[side].u[1] = p[(p1 - 1) * RINGS];
      s[side].u[2] = p[(p2 - 1) * RINGS];
      s[side].e = p[3 * RINGS];
      if (id.isx) {  // t1 = y: du, dv; t2 = z: du, dw
        s[side].g1[0] = y[-RINGS];
        s[side].g1[1] = y[0];
        if (!FX) s[side].g2[0] = dz_vel(g, C.k, ku, 0, p, VW);
        s[side].g2[1] = dz_vel(g, C.k, ku, 2, p + 2 * RINGS, VW);
      } else {  // t1 = x: dw, du; t2 = y: dw, dv
        s[side].g1[0] = p[2 * RINGS + 1] - p[2 * RINGS - 1];
        s[side].g1[1] = p[1] - p[-1];
        s[side].g2[0] = y[RINGS];
        s[side].g2[1] = y[0];
      }
    }
    if (wall) {
      VSide<T> o = from_above ? s[1] : s[0];
      o.u[0] = -o.u[0];
      o.g1[0] = -o.g1[0];
      o.g2[0] = -o.g2[0];
      if (!g.wall) {
        o.u[1] = -o.u[1];
        o.u[2] = -o.u[2];
        o.g1[1] = -o.g1[1];
        o.g2[1] = -o.g2[1];
      }
      if (from_above) s[0] = o;
      else s[1] = o;
    }
    if constexpr (FX) visc3(C.fc[dir][fl], s[0], s[1], snt, V, V + 3);
    else visc3(C, dir, fl, s[0], s[1], V);
  }
  const int planes[5] = {0, pn * QP, p1 * QP, p2 * QP, 4 * QP};
  const bool edge = wall || lidf;
  if (edge || mir0 || mir3) {
#pragma unroll
    for (int c = 0; c < 5; c++) {
      const bool odd = c == 1;  // mirror ghosts beyond a wall or the interface: rho w odd
      const T* p = q + planes[c];
      T a0 = p[0], a1 = p[qs], a2 = p[2 * qs], a3 = p[3 * qs];
      if (edge) {
        if (from_above) a1 = odd ? -a2 : a2;
        else a2 = odd ? -a1 : a1;
      }
      if (mir0) a0 = odd ? -a1 : a1;
      if (mir3) a3 = odd ? -a2 : a2;
      L[c] = Arith3<T>::rec(a1, a2, a0);
      R[c] = Arith3<T>::rec(a2, a1, a3);
      if (edge) {
        if (from_above) L[c] = odd ? -R[c] : R[c];
        else R[c] = odd ? -L[c] : L[c];
      }
    }
  } else {
#pragma unroll
    for (int c = 0; c < 5; c++) {
      const T* p = q + planes[c];
      const T a0 = p[0], a1 = p[qs], a2 = p[2 * qs], a3 = p[3 * qs];
      L[c] = Arith3<T>::rec(a1, a2, a0);
      R[c] = Arith3<T>::rec(a2, a1, a3);
    }
  }
  i64 F[5];
  if constexpr (FX) {
    i64 m[3];
    FxTan t;
    if (!fx_flux<3>(g, C.k, L, R, V[0], V[3], m, &t)) return false;
    F[0] = m[0], F[1] = m[1], F[4] = m[2];
#pragma unroll
    for (int c = 0; c < 2; c++) {
      const i64* p = &S.qw[0][0][0] + q0 + ((c ? p2 : p1) - 1) * QP;
      const i64 a1 = p[qs], a2 = p[2 * qs];
      F[2 + c] = edge ? tan_flux(t, 0, 0, 0, 0, sig[c])  // nothing flows through
                      : tan_flux(t, mir0 ? a1 : p[0], a1, a2, mir3 ? a2 : p[3 * qs], sig[c]);
    }
  } else {
    flux3(g, L, R, V, F);
  }
  i64* o;
  int plane;
  if (id.isx) {
    o = &S.fx[0][id.f][id.c], plane = TZ3 * (TX + 1);
  } else if (id.below) {
    o = &S.fg[0][id.c], plane = TX;
  } else {
    o = &S.fz[0][id.f][id.c], plane = (TZ3 + 1) * TX;
  }
  o[0] = F[0];
  o[pn * plane] = F[1];
  o[p1 * plane] = F[2];
  o[p2 * plane] = F[3];
  o[4 * plane] = F[4];
  return true;
}

// Do the cells that face id reads lie in the range? The four across it, the
// y neighbours and the third-direction neighbours of the two at it. Asked only in tiles where some cell does not.
__device__ __noinline__ bool face3_in_range(const Geom& g, const Tile3Smem& S, const FaceId id, int k0) {
  auto cell = [&](int r, int c) {  // halo row and column
    const int k = k0 - 2 + r;
    return k < 0 || k >= g.nz || S.ok[r][c];
  };
  auto celly = [&](int r, int c) {  // ring row and column
    const int k = k0 - 1 + r;
    return k < 0 || k >= g.nz || S.oky[r][c];
  };
  bool ok = true;
  if (id.isx) {
    for (int s = 0; s < 4; s++) ok = ok && cell(id.f + 2, id.c + s);
    for (int s = 0; s < 2; s++)
      ok = ok && cell(id.f + 1, id.c + 1 + s) && cell(id.f + 3, id.c + 1 + s) && celly(id.f + 1, id.c + s);
  } else {
    for (int s = 0; s < 4; s++) ok = ok && cell(id.f + s, id.c + 2);
    for (int s = 0; s < 2; s++)
      ok = ok && cell(id.f + 1 + s, id.c + 1) && cell(id.f + 1 + s, id.c + 3) && celly(id.f + s, id.c + 1);
  }
  return ok;
}

// The faces marked slow (all: every face), in double, from the tile's cells
// restaged as doubles.
__device__ __noinline__ void slow_faces3(const StageArgs& a, const Fx3Const& C, int k0, int i0, int j, int row_hi,
                                         Tile3Smem& S, bool all) {
  tile3_cells<double>(a, geo3(a.g), k0, i0, j, S);
  for (int job = threadIdx.x / 32; job < 2 * TZ3 + 3; job += TILE3_THREADS / 32) {
    const int lane = threadIdx.x % 32;
    FaceId id;
    if (face_id<TZ3>(a.g, job, lane, k0, row_hi, &id) && (all || S.slow[job * TX + lane])) face3<double>(a.g, C, S, id);
  }
  __syncthreads();
}

__device__ __forceinline__ void stage_tile3(const StageArgs& a, const Fx3Const& C, int k0, int i0, int j,
                                            Tile3Smem& S) {
  const Geom& g = a.g;
  const Geo3 G = geo3(g);
  const int tid = threadIdx.x;
  const int nz = g.nz, nx = g.nx, ny = g.ny, n1 = g.n1;
  const int row_hi = a.rhs_only ? a.rhs_hi : nz;

  // ---- 1. stage state, velocities -------------------------
  const int out = C.k.on ? tile3_cells<i64>(a, G, k0, i0, j, S) : 2;

  // ---- 2. face fluxes -----------------------------------------------------
  const bool has_gamma = (n1 >= k0 && n1 <= k0 + TZ3);
  const int jobs = out == 2 ? 0 : 2 * TZ3 + 2 + has_gamma;
  const int warp = __shfl_sync(0xffffffffu, tid / 32, 0), lane = tid % 32;
  bool slow = false;
  for (int job = warp; job < jobs; job += TILE3_THREADS / 32) {
    FaceId id;
    const bool valid = face_id<TZ3>(g, job, lane, k0, row_hi, &id);
    bool ok = true;
    if (out) ok = row_in_range(id, i0, nx, valid && !face3_in_range(g, S, id, k0));
    if (!valid) continue;
    ok = ok && face3<i64>(g, C, S, id);
    S.slow[job * TX + lane] = !ok;
    slow |= !ok;
  }
  slow = out == 2 || __syncthreads_or(slow);
  if (slow) slow_faces3(a, C, k0, i0, j, row_hi, S, out == 2);

  // ---- 3. R = -div F* + s and the stage combination -------------------------
  const int rr = tid / TX, cc = tid - rr * TX;
  const int k = k0 + rr, i = i0 + cc;
  if (rr >= TZ3 || k >= row_hi || i >= nx) return;
  const bool under_gamma = (k == n1 - 1);
  const size_t row = (size_t)(k * ny + j) * g.pitch + i;  // offset within a component
  const size_t plane = G.plane;
  const int jm = wrap3(j - 1, ny);
  const i64* gy = reinterpret_cast<const i64*>(a.gy);
  const double hx = 0.5 * g.inv_dx, hy = 0.5 * g.inv_dy, hz = 0.5 * (k < n1 ? g.inv_dz1 : g.inv_dz2);
  const double sz = C.k.scale_z[k >= n1];
  double R[5];
  i64 y0[5], y1[5];
  int any = 0;
#pragma unroll
  for (int c = 0; c < 5; c++) {
    y0[c] = gy[G.at(c, k, jm, i)];
    y1[c] = gy[G.at(c, k, j, i)];
    if (c == 1 || c == 3) continue;  // the tangential momenta
    const int h0 = (int)(y0[c] >> 32), h1 = (int)(y1[c] >> 32);
    any |= (h0 ^ (h0 >> 31)) | (h1 ^ (h1 >> 31));
  }
  bool dbl = any >= 0x10000000;  // some y flux is a double
  if (out == 2) dbl = true;
  else if (slow)
    dbl = dbl || S.slow[(TZ3 + rr) * TX + cc] ||
          S.slow[cc < TX - 1 ? (TZ3 + rr) * TX + cc + 1 : (2 * TZ3 + 1) * TX + rr] || S.slow[rr * TX + cc] ||
          S.slow[(under_gamma ? 2 * TZ3 + 2 : rr + 1 < TZ3 ? rr + 1 : 2 * TZ3) * TX + cc];
  if (dbl) {
#pragma unroll
    for (int c = 0; c < 5; c++) {
      auto diff = [&](i64 f, i64 h, bool tangential) {
        return tangential ? __dsub_rn(__longlong_as_double(f), __longlong_as_double(h))
                          : __dsub_rn(flux_value(f), flux_value(h));
      };
      const double dx = diff(S.fx[c][rr][cc], S.fx[c][rr][cc + 1], c == 2 || c == 3);
      const double dz = diff(S.fz[c][rr][cc], under_gamma ? S.fg[c][cc] : S.fz[c][rr + 1][cc], c == 1 || c == 2);
      const double dy = diff(y0[c], y1[c], c == 1 || c == 3);
      R[c] = __fma_rn(hx, dx, __fma_rn(hy, dy, __dmul_rn(hz, dz)));
    }
  } else {
#pragma unroll
    for (int c = 0; c < 5; c++) {
      const i64 x0 = S.fx[c][rr][cc], x1 = S.fx[c][rr][cc + 1];
      const i64 z0 = S.fz[c][rr][cc], z1 = under_gamma ? S.fg[c][cc] : S.fz[c][rr + 1][cc];
      auto sum = [&](double sn, i64 n, double ha, i64 a0, i64 a1, double hb, i64 b0, i64 b1) {
        const double da = __dsub_rn(__longlong_as_double(a0), __longlong_as_double(a1));
        const double db = __dsub_rn(__longlong_as_double(b0), __longlong_as_double(b1));
        return __fma_rn(sn, (double)n, __fma_rn(ha, da, __dmul_rn(hb, db)));
      };
      if (c == 1) R[c] = sum(C.k.scale, x0 - x1, hy, y0[c], y1[c], hz, z0, z1);
      else if (c == 2) R[c] = sum(C.scale_y, y0[c] - y1[c], hx, x0, x1, hz, z0, z1);
      else if (c == 3) R[c] = sum(sz, z0 - z1, hx, x0, x1, hy, y0[c], y1[c]);
      else if (C.k.square) R[c] = __dmul_rn(C.k.scale, (double)((x0 - x1) + (y0[c] - y1[c]) + (z0 - z1)));
      else
        R[c] = __fma_rn(C.k.scale, (double)(x0 - x1),
                        __fma_rn(C.scale_y, (double)(y0[c] - y1[c]), __dmul_rn(sz, (double)(z0 - z1))));
    }
  }
  {
    // the source, from the stage state itself
    double q[5];
    stage_val3(a, G, k, j, i, q);
    R[3] = __fma_rn(-g.G, q[0], R[3]);
    R[4] = __fma_rn(-g.G, q[3], R[4]);
  }

  if (a.rhs_only) {
#pragma unroll
    for (int c = 0; c < 5; c++) a.rhs_out[(size_t)c * plane + row] = R[c];
    return;
  }
  double* Ra = reinterpret_cast<double*>(a.b.Ra);
  const int sg = a.stage;
  if (k >= g.n1_r) {
    // fast region: m Heun substeps of dt/m
#pragma unroll
    for (int c = 0; c < 5; c++) {
      const size_t o = (size_t)c * plane + row;
      if (!(sg & 1)) Ra[o] = R[c];
      else a.qF_next[o] = __fma_rn(g.h2, __dadd_rn(Ra[o], R[c]), a.qF[o]);
    }
  } else if (k >= g.nS_r) {
    // buffer: RK2 restarted from q_n each substep, weights 1/(2m)
    const size_t pb = (size_t)(g.n1_r - g.nS_r) * ny * g.pitch;
    const size_t ob = (size_t)((k - g.nS_r) * ny + j) * g.pitch + i;
    const bool last = (sg == 2 * g.m - 1);
#pragma unroll
    for (int c = 0; c < 5; c++) {
      const size_t o = (size_t)c * plane + row;
      double* acc = a.b.accB + (size_t)c * pb + ob;
      if (!(sg & 1)) Ra[o] = R[c];
      if (sg == 0) *acc = R[c];
      else if (last) *acc = __fma_rn(g.h2, __dadd_rn(*acc, R[c]), a.b.qA[o]);
      else *acc = __dadd_rn(*acc, R[c]);
    }
  } else {
    // slow region: stages 1 and 2 only (Algorithm 1)
    const size_t ps = (size_t)g.nS_r * ny * g.pitch;
#pragma unroll
    for (int c = 0; c < 5; c++) {
      const size_t o = (size_t)c * plane + row;
      if (sg == 0) Ra[o] = R[c];
      else a.b.accS[(size_t)c * ps + row] = __fma_rn(g.hdt, __dadd_rn(Ra[o], R[c]), a.b.qA[o]);
    }
  }
}

}  // namespace mprk
