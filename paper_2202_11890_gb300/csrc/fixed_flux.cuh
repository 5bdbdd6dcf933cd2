// fixed_flux.cuh — the Lax–Friedrichs face flux of Sec. 2.1 in 64-bit fixed
// point (fixed_point.cuh), for ND = 2 or 3 velocity components.
//
// A state is (rho, m_n, m_t.., rho E) in the face frame: rho and rho E .60,
// momenta .62. Per face: two reciprocals, two square roots and some thirty
// 64 x 64-bit products, some 1000 integer instructions against 87 double
// ones that held the double pipe for 1400 clocks per warp.
#pragma once

#include "fixed_point.cuh"
#include "fp64_recip.cuh"

namespace mprk {

using fx::i64;

// The stage state lies inside the fixed-point range (fixed_point.cuh)? m: the
// largest upper word of the momenta without their signs (abs_word). NaN, zero
// and negative densities and energies do not.
__device__ __forceinline__ bool in_range(double r, unsigned m, double E) {
  const unsigned hr = (unsigned)__double2hiint(r), he = (unsigned)__double2hiint(E);
  return hr - fx::RHO_LO < fx::RHO_HI - fx::RHO_LO && he - fx::E_LO < fx::E_HI - fx::E_LO && m < fx::MOM_HI;
}
__device__ __forceinline__ unsigned abs_word(double m) { return (unsigned)__double2hiint(m) & 0x7fffffffu; }

// One side of a face.
template <int ND>
struct FxSide {
  FxW un, mn, mt[ND - 1];
  i64 un_, ut[ND - 1];  // velocities .59
  i64 mu, p, c2;        // m_n u_n .57, p .57, c^2 .55
  i64 k;                // |m|^2 / rho .57
  i64 eh;               // rho E + p .59
};
template <int ND>
__device__ __forceinline__ void fx_side(const FxConst& c, const i64 q[ND + 2], FxSide<ND>* s) {
  const FxW inv = fx::split(fx::recip(q[0]));
  s->mn = fx::split(q[1]);
  s->un_ = fx::mul(s->mn, inv);
  s->un = fx::split(s->un_);
  s->mu = fx::mul(s->mn, s->un);
  s->k = s->mu;
#pragma unroll
  for (int t = 0; t < ND - 1; t++) {
    s->mt[t] = fx::split(q[2 + t]);
    s->ut[t] = fx::mul(s->mt[t], inv);
    s->k += fx::mul(s->mt[t], fx::split(s->ut[t]));
  }
  const FxW pe = fx::split(q[ND + 1] - (s->k << 2));  // p / (gamma - 1) .60
  s->p = fx::mul(pe, c.gm1);
  s->c2 = fx::mul(fx::split(fx::mul(pe, inv)), c.gg);
  s->eh = (q[ND + 1] >> 1) + (s->p << 2);
}

// The Roe-averaged speed |u_n| + a from the two states' densities, velocities
// and sound speeds squared (rarely needed): w the weight sqrt(rho_R) /
// (sqrt(rho_L) + sqrt(rho_R)), a^2 = (1 - w) a_L^2 + w a_R^2 + (gamma - 1)/2
// w (1 - w) |du|^2, which equals the Roe-averaged enthalpy's (gamma - 1)(H -
// |u|^2 / 2). un, c2: u_n and a^2 of the left state; du, d1, d2, dc2: the
// differences to the right one of u_n, the tangential velocities and a^2.
__device__ __forceinline__ double roe_speed(double rL, double rR, double un, double du, double d1, double d2, double c2,
                                            double dc2, double gm1) {
  const double w = recip_f64(__dadd_rn(1.0, sqrt_f64(__dmul_rn(rL, recip_f64(rR)))));
  const double q = __dmul_rn(__dmul_rn(__dmul_rn(0.5, gm1), w), __dsub_rn(1.0, w));
  const double a2 = __fma_rn(q, __fma_rn(du, du, __fma_rn(d1, d1, __dmul_rn(d2, d2))), __fma_rn(w, dc2, c2));
  return __dadd_rn(fabs(__fma_rn(w, du, un)), sqrt_f64(a2));
}
__device__ __noinline__ i64 fx_roe_speed(i64 rL, i64 rR, i64 unL, i64 unR, i64 dt1, i64 dt2, i64 c2L, i64 c2R,
                                         double gm1) {
  const double sv = 1.0 / (double)(1ll << fx::S_VEL), sc = 1.0 / (double)(1ll << 55);
  const double s = roe_speed((double)rL, (double)rR, __dmul_rn((double)unL, sv), __dmul_rn((double)(unR - unL), sv),
                             __dmul_rn((double)dt1, sv), __dmul_rn((double)dt2, sv), __dmul_rn((double)c2L, sc),
                             __dmul_rn((double)(c2R - c2L), sc), gm1);
  return __double2ll_rn(__dmul_rn(s, (double)(1ll << fx::S_VEL)));
}

// A double as a float, cut to 23 bits, on the integer pipes (0 and infinity
// beyond the float range, NaN as infinity).
__device__ __forceinline__ float cut_float(double x) {
  const unsigned h = (unsigned)__double2hiint(x);
  const int e = (int)(h >> 20 & 0x7ff) - 896;
  const unsigned m = (h & 0xfffffu) << 3 | (unsigned)__double2loint(x) >> 29;
  return __uint_as_float((h & 0x80000000u) | (e <= 0 ? 0u : e >= 255 ? 0x7f800000u : (unsigned)e << 23 | m));
}
// The largest speed of a face from the double states: that of the left, the
// right and the Roe-averaged state. The latter lies below (1 - w) s_L + w s_R
// + w (1 - w) D / (2 min a), D = (a_L - a_R)^2 + (gamma - 1)/2 |du|^2, so it
// cannot be the largest where 2 min(a) |s_L - s_R| > D: its 31 double
// operations of a face's 113 are spared but for a few faces. The comparison
// is false for NaN and beyond the float range.
__device__ __forceinline__ double face_speed(const Geom& g, double rL, double rR, double unL, double unR, double d1,
                                             double d2, double c2L, double c2R) {
  const double cL = sqrt_f64(c2L), cR = sqrt_f64(c2R);
  const double sL = __dadd_rn(fabs(unL), cL), sR = __dadd_rn(fabs(unR), cR);
  const double lam = max_speed(sL, sR);
  const double du = __dsub_rn(unR, unL);
  const float dn = cut_float(du), t1 = cut_float(d1), t2 = cut_float(d2);
  const float dc = cut_float(__dsub_rn(cL, cR)), ds = fabsf(cut_float(__dsub_rn(sL, sR)));
  const float D = fmaf(dc, dc, 0.5f * g.gm1f * fmaf(dn, dn, fmaf(t1, t1, t2 * t2)));
  const float amin = fminf(cut_float(cL), cut_float(cR));
  if (fmaf(D, 1.0001f, 1e-36f) < 2.0f * amin * ds) return lam;
  return max_speed(lam, roe_speed(rL, rR, unL, du, d1, d2, c2L, __dsub_rn(c2R, c2L), g.gm1));
}

// ---- tangential momenta -------------------------------------------------
// Unlike the other components their fluxes have no term of the size of density
// or pressure, so the rounding has to follow the momenta themselves, however
// small: they and their velocities are integers under an exponent of their
// own, aligned to the largest exponent among the cells of a face, with 57 and
// 58 bits below it where a double has 53, and the flux comes out as a double.
// In double arithmetic (thirteen operations per face) they held the double
// pipe longer: a step of 2048 x 1024 cells, m = 8, took 2.85 ms, with only the
// stress in double 2.65, this way 2.37; 512 x 64 x 200 cells, m = 4, 15.0, 13.3
// and 11.3 ms.

// x 2^-57 2^(e - 1023): a sum of velocity differences.
struct FxA {
  i64 x;
  int e;
};
// The tangential stress V over half the divergence factor, v 2^-55 2^(e - 1023).
struct FxStress {
  i64 v;
  int e;
};
// A velocity of exponent field ex (packed_velocity) for the exponent field e.
__host__ __device__ __forceinline__ i64 vel_at(i64 u, int ex, int e) { return fx::shr(u, 1 + e - ex); }
// From the difference across the face and the two cells' tangential differences.
__host__ __device__ __forceinline__ FxStress tan_stress(const FxN& C, FxA du, const FxN& D, FxA gn) {
  const int ec = du.e - C.s, ed = gn.e - D.s, e = ec > ed ? ec : ed;
  return FxStress{fx::shr(fx::mul(fx::split(du.x), C.f), e - ec) + fx::shr(fx::mul(fx::split(gn.x), D.f), e - ed), e};
}
__host__ __device__ __forceinline__ FxStress tan_stress(const FxN& C, FxA du) {
  return FxStress{fx::mul(fx::split(du.x), C.f), du.e - C.s};
}
// The stress .59.
__host__ __device__ __forceinline__ i64 stress59(FxStress s) {
  const int r = 1019 - s.e;
  return r >= 0 ? fx::shr(s.v, r) : s.v << -r;
}

// The flux, the bits of a double, from the four cells across the face as packed
// doubles (L1, R1 those at it): f(q_L) + f(q_R) + lambda (q_L - q_R) - V
// regrouped as L (u_L + u_R) + (L - R) (lambda - u_R) - V.
struct FxTan {
  i64 us, lr;  // u_nL + u_nR, lambda - u_nR (.59)
};
__host__ __device__ __forceinline__ i64 tan_flux(const FxTan& t, i64 L2, i64 L1, i64 R1, i64 R2, FxStress V) {
  const int x0 = fx::pack_exp(L2), x1 = fx::pack_exp(L1), x2 = fx::pack_exp(R1), x3 = fx::pack_exp(R2);
  const int x01 = x0 > x1 ? x0 : x1, x23 = x2 > x3 ? x2 : x3, em = x01 > x23 ? x01 : x23;
  const i64 a0 = fx::unpack(L2, em), a1 = fx::unpack(L1, em), a2 = fx::unpack(R1, em), a3 = fx::unpack(R2, em);
  const i64 L = (a1 << 2) + (a2 - a0), R = (a2 << 2) + (a1 - a3);  // .60 of 2^(em - 1023)
  const i64 F = fx::mul2(fx::split(L), fx::split(t.us), fx::split(L - R), fx::split(t.lr));  // .55
  const int e = em > V.e ? em : V.e;
  return fx::to_double(fx::shr(F, e - em) - fx::shr(V.v, e - V.e), 55 + 1023 - e);
}

// The fluxes of mass, normal momentum and energy over half the divergence
// factor (.57), or false where a state leaves the range: F = f(q_L) + f(q_R) +
// lambda (q_L - q_R) - V, lambda the largest |u_n| + a over the left, right
// and Roe-averaged states. Vn, VE: the viscous (or interface) part of the
// normal momentum and the energy. t: the factors of the tangential momenta.
template <int ND>
__device__ __forceinline__ bool fx_flux(const Geom& g, const FxConst& k, const i64 L[ND + 2], const i64 R[ND + 2],
                                        i64 Vn, i64 VE, i64 F[3], FxTan* t) {
  constexpr int E = ND + 1;
  FxSide<ND> l, r;
  fx_side<ND>(k, L, &l);
  fx_side<ND>(k, R, &r);
  const int c2l = (int)(l.c2 >> 32), c2r = (int)(r.c2 >> 32);
  if (min((int)(L[0] >> 32), (int)(R[0] >> 32)) < fx::RHO_MIN ||
      max((int)(l.k >> 32), (int)(r.k >> 32)) >= fx::KIN_MAX || min(c2l, c2r) < fx::C2_MIN ||
      max(c2l, c2r) >= fx::C2_MAX)
    return false;
  const i64 cl = fx::sqroot(l.c2 << 6), cr = fx::sqroot(r.c2 << 6);
  const i64 sl = (l.un_ < 0 ? -l.un_ : l.un_) + cl, sr = (r.un_ < 0 ? -r.un_ : r.un_) + cr;
  i64 lam = sl > sr ? sl : sr;  // .59
  {
    // The Roe speed lies below (1 - w) sl + w sr + w (1 - w) / (2 min a) D
    // with D = (a_L - a_R)^2 + (gamma - 1)/2 |du|^2, so it cannot be the
    // largest where |sl - sr| >= D (min a > 0.5 and w in [0.2, 0.8] within
    // the range): all but a few faces of a smooth flow skip it.
    const float df = fx::to_float(sl - sr), dc = fx::to_float(cl - cr), dn = fx::to_float(l.un_ - r.un_);
    float u2 = dn * dn;
#pragma unroll
    for (int t = 0; t < ND - 1; t++) {
      const float d = fx::to_float(l.ut[t] - r.ut[t]);
      u2 = fmaf(d, d, u2);
    }
    if (fabsf(df) * 5.7646075e17f /* 2^59 */ < fmaf(dc, dc, 0.5f * g.gm1f * u2)) {
      const i64 roe = fx_roe_speed(L[0], R[0], l.un_, r.un_, r.ut[0] - l.ut[0], ND > 2 ? r.ut[ND - 2] - l.ut[ND - 2] : 0,
                                   l.c2, r.c2, g.gm1);
      lam = roe > lam ? roe : lam;
    }
  }
  const FxW lam59 = fx::split(lam), lam61 = fx::split(lam << 2);
  // one rounding of the sum: exactly zero at a wall, where m_nR = -m_nL
  F[0] = ((L[1] + R[1] + 16) >> 5) + fx::mul(fx::split(L[0] - R[0]), lam61);
  F[1] = (l.mu + l.p) + (r.mu + r.p) + fx::mul(fx::split(L[1] - R[1]), lam59) - Vn;
  F[2] = fx::mul(fx::split(l.eh), fx::split(l.un_ << 3)) + fx::mul(fx::split(r.eh), fx::split(r.un_ << 3)) +
         fx::mul(fx::split(L[E] - R[E]), lam61) - VE;
  t->us = l.un_ + r.un_;
  t->lr = lam - r.un_;
  // room for the sums of the divergence: |F| < 8
  int top = 0;
#pragma unroll
  for (int c = 0; c < 3; c++) {
    const int h = (int)(F[c] >> 32);
    top |= h ^ (h >> 31);
  }
  return top < (8 << (fx::S_FLUX - 32));
}

}  // namespace mprk
