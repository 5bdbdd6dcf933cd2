// fixed_point.cuh — 64-bit fixed-point arithmetic of the FP64 face fluxes.
//
// This GPU completes two double-precision operations per clock and SM
// (measured: 2.0 DFMA, 1.7 DADD lanes per clock), but 64 lanes of 32-bit
// integer adds and shifts and about 25-32 of 32 x 32 -> 64-bit multiply-adds.
// A double operation therefore costs a warp 16 clocks, a 64-bit integer add
// one, and a 64 x 64-bit product taken to its upper half about four. The
// face fluxes of the FP64 tile run here: states, speeds and fluxes of a
// nondimensional flow (density, sound speed and pressure near one) as 64-bit
// integers in units of 2^-57 to 2^-62, except the flux of the tangential
// momentum (fixed_flux.cuh). A face whose states leave the representable
// range is evaluated in double instead (stage_tile.cuh).
//
// Errors are absolute. A product errs by at most 3/4 of its unit (mul), a pair
// of products by one (mul2). A flux in units of 2^-57 sums its products: 1.25
// units for mass, 3.75 for the normal momentum (and 1 to 1.75 for sigma_nn),
// 2.25 for the energy, whose viscous part adds up to 3.5 units in 2-D and 6 in 3-D
// (fx_visc, visc3; 2.5 and 4 at the interface; tests/test_fixed_flux.py), plus
// the errors of its factors, of units up to 2^-57. Over the states tested the
// right-hand side errs by 3 to 14 % of the double form's in mass, normal
// momentum and energy (root mean square, tests/test_gpu_flux_precision.py).
//
// Notation: x.s means the integer x * 2^s. Products drop 64 bits, so
// a.s * b.t gives (a b).(s + t - 64).
#pragma once

#include <cuda_runtime.h>

#include "mprk_internal.h"

namespace mprk {
namespace fx {

typedef long long i64;
typedef unsigned long long u64;
typedef unsigned int u32;

// Scales (binary digits after the point).
constexpr int S_RHO = 60;   // reconstructed density and energy; cells are kept 2 bits coarser
constexpr int S_MOM = 62;   // reconstructed momentum; cells 2 bits coarser
constexpr int S_VEL = 59;   // velocities, sound speed, e = T / (gamma (gamma - 1))
constexpr int S_FLUX = 57;  // face fluxes over half the divergence factor

// Cell states within these bounds keep every reconstructed state and every
// intermediate inside its 64 bits (upper words of the doubles).
constexpr u32 RHO_LO = 0x3FE00000u, RHO_HI = 0x40100000u;  // [0.5, 4)
constexpr u32 MOM_HI = 0x3FE50000u;                        // |m| < 0.65625
constexpr u32 E_LO = 0x3FB00000u, E_HI = 0x40100000u;      // [2^-4, 4)
// Bounds on a reconstructed state, as upper words of the integers.
constexpr int RHO_MIN = (int)(0.30 * (1 << (S_RHO - 32)));      // density
constexpr int KIN_MAX = 1 << (S_FLUX - 32);                     // |m|^2 / rho below 1
constexpr int C2_MIN = (int)(0.26 * (1 << 23));                 // sound speed squared (.55)
constexpr int C2_MAX = (int)(3.90 * (1 << 23));

// a b + c with a 64-bit result: one instruction (written out because the
// compiler widens the operands first and multiplies 64 x 64 bits).
__host__ __device__ __forceinline__ i64 mad(int a, int b, i64 c) {
#ifdef __CUDA_ARCH__
  i64 r;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
  return r;
#else
  return (i64)a * b + c;
#endif
}
__host__ __device__ __forceinline__ u32 mulhi_u(u32 a, u32 b) {
#ifdef __CUDA_ARCH__
  return __umulhi(a, b);
#else
  return (u32)((u64)a * b >> 32);
#endif
}

// A multiplicand: x = hi 2^32 + lo with lo signed, so that every partial
// product is one signed 32 x 32 -> 64-bit multiply-add. x < 2^63 - 2^31.
__host__ __device__ __forceinline__ FxW split(i64 x) {
  FxW w;
  w.lo = (int)x;
  w.hi = (int)(x >> 32) + (int)((u32)w.lo >> 31);
  return w;
}

// a b / 2^64, rounded: the low product (at most 2^62) is dropped.
__host__ __device__ __forceinline__ i64 mul(FxW a, FxW b) {
  const i64 t = mad(a.hi, b.lo, mad(a.lo, b.hi, 0x80000000ll));
  return mad(a.hi, b.hi, (i64)(int)(t >> 32));
}
__host__ __device__ __forceinline__ i64 mul(i64 a, FxW b) { return mul(split(a), b); }

// (a b + c d) / 2^64: the cross products share one rounding.
__host__ __device__ __forceinline__ i64 mul2(FxW a, FxW b, FxW c, FxW d) {
  i64 t = mad(a.hi, b.lo, mad(a.lo, b.hi, 0x80000000ll));
  t = mad(c.hi, d.lo, mad(c.lo, d.hi, t));
  return mad(c.hi, d.hi, mad(a.hi, b.hi, (i64)(int)(t >> 32)));
}

// a b / 2^32, b a factor in [0, 2^31).
__host__ __device__ __forceinline__ i64 mul31(i64 a, int b) {
  return mad((int)(a >> 32), b, (i64)mulhi_u((u32)a, (u32)b));
}

__host__ __device__ __forceinline__ float to_float(i64 x) {
  return fmaf((float)(int)(x >> 32), 4294967296.0f, (float)(u32)x);
}

__host__ __device__ __forceinline__ int float_bits(float x) {
#ifdef __CUDA_ARCH__
  return __float_as_int(x);
#else
  int b;
  memcpy(&b, &x, 4);
  return b;
#endif
}
__host__ __device__ __forceinline__ float rcp_seed(float x) {
#ifdef __CUDA_ARCH__
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
#else
  return 1.0f / x;
#endif
}
__host__ __device__ __forceinline__ float rsqrt_seed(float x) {
#ifdef __CUDA_ARCH__
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
#else
  return 1.0f / sqrtf(x);
#endif
}
__host__ __device__ __forceinline__ int mulhi32(int a, int b) { return (int)(mad(a, b, 0) >> 32); }

// 1/rho: rho.60 in [0.3, 4.9] -> .61. Seed y from the float reciprocal,
// rounded to a 21-bit fraction by adding 2^23, then y (1 + e + e^2) with
// e = 1 - rho y (|e| < 2^-19; the next term is below 2^-57).
__host__ __device__ __forceinline__ i64 recip(i64 rho) {
  const float s = rcp_seed((float)(int)(rho >> 32));
  const int y = float_bits(fmaf(s, 562949953421312.0f /* 2^49 */, 8388608.0f)) << 8;  // .29
  const i64 e = (1ll << 57) - mul31(rho, y);                                          // .57
  const int e50 = (int)(e >> 7);
  const i64 g = (e + (mulhi32(e50, e50) >> 11)) << 7;  // (e + e^2).64
  return ((i64)y << 32) + mul31(g, y);
}

// sqrt(x): x.61 in [0.26, 3.9] -> .59. Seed y of 1/sqrt(x) rounded to 22
// fraction bits; t = x y, e = 1 - t y, sqrt = t (1 + e/2 + 3 e^2 / 8)
// (|e| < 2^-19; the next term is below 2^-58).
__host__ __device__ __forceinline__ i64 sqroot(i64 x) {
  const float s = rsqrt_seed((float)(int)(x >> 32));
  const int y = float_bits(fmaf(s, 97184015999.0f /* 2^36.5 */, 8388608.0f)) << 8;  // .30
  const i64 t = mul31(x, y);                                                         // .59
  const i64 e = (1ll << 57) - mul31(t, y);                                           // .57
  const int e50 = (int)(e >> 7);
  const i64 g = (e << 6) + ((3 * mulhi32(e50, e50)) >> 7);  // (e/2 + 3 e^2 / 8).64
  return t + mul(split(t), split(g));
}

// x.s as a double, rounded to nearest (halves away from zero): the mantissa
// shifted to bit 62, whose leading one raises the exponent field by one, as
// does a carry of the rounding. On the integer pipes: a conversion
// instruction runs at the double pipe's rate.
__host__ __device__ __forceinline__ i64 to_double(i64 x, int s) {
  const u64 a = x < 0 ? 0ull - (u64)x : (u64)x;
  if (a == 0) return 0;
#ifdef __CUDA_ARCH__
  const int z = __clzll((i64)a);
#else
  const int z = __builtin_clzll(a);
#endif
  const u64 m = ((a << z >> 10) + 1) >> 1;
  const int e = 1085 - s - z;
  if (e <= 0) return 0;  // below the normal doubles
  return (i64)(((u64)e << 52) + m) | (x & (i64)(1ull << 63));
}

// A double below one in magnitude as a signed 53-bit mantissa, its leading one
// at bit 62, over its 10-bit exponent field (subnormals as zero); and such a
// mantissa with its leading one at bit 58 for the exponent field e, its own or
// a larger one.
__host__ __device__ __forceinline__ i64 pack(i64 bits) {
  const int e = (int)((u64)bits >> 52 & 0x7ff);
  const i64 m = (i64)(((u64)bits << 10 & 0x3fffffffffffffffull) | 1ull << 62), n = bits >> 63;
  return e == 0 ? 0 : ((m ^ n) - n) | e;
}
__host__ __device__ __forceinline__ int pack_exp(i64 w) { return (int)w & 1023; }
__host__ __device__ __forceinline__ i64 shr(i64 x, int s) { return x >> (s < 63 ? s : 63); }
__host__ __device__ __forceinline__ i64 unpack(i64 w, int e) { return shr(w & ~1023ll, 4 + e - pack_exp(w)); }
// The velocity of a cell, .58 of 2^(its momentum's exponent - 1023), from the
// packed momentum and 1/rho .61. Halved, because split's carry needs |x| below
// 2^63 - 2^31, which a mantissa of 31 leading ones exceeds.
__host__ __device__ __forceinline__ i64 packed_velocity(i64 w, FxW inv) { return mul(split((w & ~1023ll) >> 1), inv); }

// A double of a cell state within the bounds above, as an integer of scale
// s (truncated toward zero; exact when its last bit is at least 2^-s).
__host__ __device__ __forceinline__ i64 from_double(i64 bits, int s) {
  const u64 m = ((u64)bits << 10 | 1ull << 62) & 0x7fffffffffffffffull;
  int sh = 1085 - s - (int)((u64)bits >> 52 & 0x7ff);
  sh = sh > 63 ? 63 : sh;
  const i64 v = (i64)(m >> sh), n = bits >> 63;
  return (v ^ n) - n;
}

// The same of a positive double.
__host__ __device__ __forceinline__ i64 from_positive(i64 bits, int s) {
  const u64 m = (u64)bits << 10 | 1ull << 62;
  const int sh = 1085 - s - (int)((u64)bits >> 52);
  return (i64)((m & 0x7fffffffffffffffull) >> (sh & 63));
}

}  // namespace fx
}  // namespace mprk
