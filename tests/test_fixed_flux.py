"""The 64-bit fixed-point arithmetic of the FP64 faces, compiled for the host,
against exact rational numbers: the products, reciprocal, square root and
conversions, and the viscous part of the normal momentum and the energy in 2-D,
in 3-D and at the interface.

Bounds, in units of the result's last digit. A product drops the low 32 x 32
bits (at most 1/4) and rounds the cross products (1/2): 3/4 alone, 1 for two
that share a rounding. With velocities |u| <= 1.32 and stresses taken .57
(sigma_nn) or truncated to .59 (sigma_nt), the viscous energy errs by its own
products, by 1.32 times the error of sigma_nn and by 1.32 / 4 per sigma_nt:
2-D 1 + 3/4 + 1.32 (1 + 1/4), 3-D 4 (3/4) + 1.32 (7/4 + 2/4), the interface per
component 3/4 + 1.32 / 4 + |sigma| (3/4)(1/4) and 3/4 for the heat."""
import ctypes as C
import random
import subprocess
from fractions import Fraction as Fr

import numpy as np
import pytest

from paper_2202_11890_gb300 import build

SHIM = r"""
#include <cuda_runtime.h>
#include <cstring>
#include "mprk_internal.h"
#include "stage_tile.cuh"
#include "stage_tile3d.cuh"
using namespace mprk;
extern "C" {
void prim(const i64* in, i64* o) {  // in: a, b, c, d; rho .60; x .61; the bits of a double
  const FxW a = fx::split(in[0]), b = fx::split(in[1]), c = fx::split(in[2]), d = fx::split(in[3]);
  o[0] = fx::mul(a, b);
  o[1] = fx::mul2(a, b, c, d);
  o[2] = fx::recip(in[4]);
  o[3] = fx::sqroot(in[5]);
  o[4] = fx::from_double(in[6], 60);
  o[5] = fx::to_double(in[0], 59);
}
void velocity(const i64* in, i64* o) {  // the bits of a momentum, rho .60; for the exponent field in[2]
  const i64 w = fx::pack(in[0]);
  o[0] = vel_at(fx::packed_velocity(w, fx::split(fx::recip(in[1]))), fx::pack_exp(w), (int)in[2]);
}
void tangent(const i64* in, i64* o) {  // in: bits of L2, L1, R1, R2; us, lr; V, its e; C, its shift; x, its e
  i64 w[4];
  for (int j = 0; j < 4; j++) w[j] = fx::pack(in[j]);
  o[0] = tan_flux(FxTan{in[4], in[5]}, w[0], w[1], w[2], w[3], FxStress{in[6], (int)in[7]});
  const FxN c = {fx::split(in[8]), (int)in[9]};
  const FxStress s = tan_stress(c, FxA{in[10], (int)in[11]}, c, FxA{in[10] / 3, (int)in[11] - 9});
  o[1] = s.v;
  o[2] = s.e;
  o[3] = stress59(s);
}
void visc2(const i64* f, const i64* v, i64* o) {  // f: coefficients; v: L, R of five, snt
  FxW fc[FXC_N];
  for (int j = 0; j < FXC_N; j++) fc[j] = fx::split(f[j]);
  fx_visc(fc, v, v + 5, v[10], o, o + 1);
}
void visc3d(const i64* f, const i64* v, i64* o) {  // v: L, R of (u[3], e, g1, g2), snt[2]
  FxW fc[F3_N];
  for (int j = 0; j < F3_N; j++) fc[j] = fx::split(f[j]);
  VSide<i64> s[2];
  for (int k = 0; k < 2; k++) {
    for (int j = 0; j < 3; j++) s[k].u[j] = v[6 * k + j];
    s[k].e = v[6 * k + 3];
    s[k].g1[1] = v[6 * k + 4];
    s[k].g2[1] = v[6 * k + 5];
  }
  visc3(fc, s[0], s[1], v + 12, o, o + 1);
}
void lid(const i64* f, const i64* v, i64* o) {  // u1, u2, e1, e2, snt
  FxConst k;
  for (int j = 0; j < LID_N; j++) k.lid[j] = fx::split(f[j]);
  o[0] = lid_work(k, v[0], v[1], v[4]) + lid_heat(k, v[2], v[3]);
}
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("fx")
    (d / "fx.cu").write_text(SHIM)
    out = str(d / "fx.so")
    r = subprocess.run([build.nvcc(), *build.ARCH, *build.FLAGS, "-shared", "-o", out, str(d / "fx.cu")],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return C.CDLL(out)


def call(fn, *args, n):
    out = (C.c_longlong * n)()
    fn(*[(C.c_longlong * len(a))(*a) for a in args], out)
    return list(out)


def bits(x):
    return int(np.float64(x).view(np.int64))


def value(b):
    return Fr(float(np.int64(b).view(np.float64)))


def test_primitives_within_their_bounds(lib):
    rng = random.Random(3)
    one = Fr(2) ** 64
    for _ in range(4000):
        a, b, c, d = (int(rng.uniform(-1, 1) * 2 ** rng.uniform(30, 61.5)) for _ in range(4))
        rho, x = int(rng.uniform(0.3, 4.9) * 2 ** 60), int(rng.uniform(0.26, 3.9) * 2 ** 61)
        y = rng.uniform(-1, 1) * 2.0 ** rng.uniform(-70, 1)
        o = call(lib.prim, [a, b, c, d, rho, x, bits(y)], n=6)
        assert abs(o[0] - Fr(a) * b / one) <= Fr(3, 4)
        assert abs(o[1] - (Fr(a) * b + Fr(c) * d) / one) <= 1
        # one third-order step from a seed of 2^-19: a rest of 2^-57, and roundings
        # of the last two products relative to results of at least 2^58
        assert abs(Fr(o[2]) * rho / Fr(2) ** 121 - 1) <= Fr(2) ** -56
        assert abs(Fr(o[3]) ** 2 / (Fr(x) / Fr(2) ** 61 * Fr(2) ** 118) - 1) <= Fr(2) ** -55
        exact = Fr(y) * 2 ** 60
        assert abs(o[4]) <= abs(exact) < abs(o[4]) + 1 and (o[4] == 0 or (o[4] > 0) == (y > 0))
        assert value(o[5]) == Fr(a / 2 ** 59) or abs(value(o[5]) - Fr(a) / 2 ** 59) <= abs(Fr(a)) / 2 ** 112
    for a in (0, 1, -1, 2 ** 53 + 1, 2 ** 62 - 1, -(2 ** 62) + 1, 2 ** 63 - 1, -(2 ** 63)):
        o = call(lib.prim, [a, 1, 1, 1, 2 ** 60, 2 ** 60, 0], n=6)
        assert abs(value(o[5]) * 2 ** 59 - a) <= abs(Fr(a)) / 2 ** 53


# mantissas at the ends of their words: the carries of split, pack and unpack
ENDS = [0, 1, 2 ** 52 - 1, 2 ** 52 - 2, 2 ** 51, 2 ** 21, 2 ** 21 - 1, 2 ** 20, 2 ** 22 - 1, 2 ** 52 - 2 ** 21,
        2 ** 52 - 2 ** 20, 2 ** 52 - 2 ** 22, 2 ** 53 - 2 ** 31 & (2 ** 52 - 1)]


def from_parts(mantissa, exponent, negative):
    x = float(np.int64(exponent << 52 | mantissa).view(np.float64))
    return -x if negative else x


@pytest.mark.parametrize("ends", [True, False])
def test_velocity_of_any_mantissa(lib, ends):
    """m / rho under m's exponent, .57: the product's 3/4 of a unit at twice that
    resolution, the cut to .57, and 1/rho within 2^-56."""
    rng = random.Random(13)
    for n in range(4000):
        man = rng.choice(ENDS) if ends else rng.getrandbits(52)
        e = rng.choice([1, 2, 500, 1000, 1020, 1021, rng.randint(1, 1021)])
        m, rho = from_parts(man, e, rng.random() < 0.5), int(rng.uniform(0.5, 4.0) * 2 ** 60)
        o, = call(lib.velocity, [bits(m), rho, e], n=1)
        exact = Fr(m) / (Fr(rho) / 2 ** 60) * Fr(2) ** (57 - e + 1023)
        assert abs(o - exact) <= Fr(3, 2) + abs(exact) / 2 ** 56, (m, rho)


@pytest.mark.parametrize("ends", [True, False])
def test_tangential_flux_follows_the_momenta(lib, ends):
    """Momenta of every size down to 1e-300, zeros and neighbours of other sizes
    among them. Units of 2^-55 of the largest one's power of two: the pair of
    products 1; each momentum cut at 2^-58 with weights up to 3/2 of u_L + u_R
    (3.66) and 2 of lambda - u_R (5.64), (5.49 + 11.28) / 8; the two parts
    aligned, 1 each at the larger exponent; and the double's rounding."""
    rng = random.Random(11)
    for _ in range(6000):
        scale = 2.0 ** -rng.choice([0, 1, 7, 20, 33, 60, 200, 900])
        m = [rng.choice([rng.uniform(-0.65, 0.65), rng.uniform(-0.65, 0.65) * 2.0 ** -rng.randint(0, 70), 0.0]) * scale
             for _ in range(4)]
        if ends:
            top = max(bits(scale) >> 52, 4) - 2
            m = [from_parts(rng.choice(ENDS), max(top - rng.choice([0, 0, 1, 5, 31, 60]), 1), rng.random() < 0.5)
                 for _ in range(4)]
        us, lr = int(rng.uniform(-3.66, 3.66) * 2 ** 59), int(rng.uniform(0.5, 5.64) * 2 ** 59)
        big = max(map(abs, m))
        em = max((bits(abs(x)) >> 52) for x in m)
        v, ev = int(rng.uniform(-1, 1) * 2 ** 58), max(em + rng.randint(-70, 3), -40)
        fac, sh, x = int(rng.uniform(0.5, 1) * 2 ** 62), rng.randint(0, 30), int(rng.uniform(-1, 1) * 2 ** 60)
        ex = rng.randint(1, 1022)
        o = call(lib.tangent, [bits(t) for t in m] + [us, lr, v, ev, fac, sh, x, ex], n=4)
        a0, a1, a2, a3 = map(Fr, m)
        L, R = a1 + (a2 - a0) / 4, a2 + (a1 - a3) / 4
        exact = (L * us + (L - R) * lr) / Fr(2) ** 59 - Fr(v) * Fr(2) ** (ev - 1023 - 55)
        unit = lambda e: Fr(2) ** (e - 1023 - 55)  # noqa: E731
        bound = (1 + Fr(17, 8)) * unit(em) + 2 * unit(max(em, ev)) + abs(exact) / 2 ** 53 + Fr(2) ** -1022
        assert abs(value(o[0]) - exact) <= bound, (m, big)
        # the stress from two differences: 3/4 each, 1 for the alignment
        e = ex - sh
        s = Fr(x) * fac / Fr(2) ** 64 * unit(e) + int(Fr(x, 3)) * fac / Fr(2) ** 64 * unit(e - 9)
        assert o[2] == e and abs(o[1] * unit(e) - s) <= Fr(11, 4) * unit(e)
        assert abs(Fr(o[3]) - o[1] * unit(e) * Fr(2) ** 59) < 1


U, E, N = 1.32, 4.8, 59  # cell velocities and e as the range bounds them, .59


def coefficients(rng, n):
    """(8/3) mu / d and the rest below one, as the launch constants allow."""
    f = [rng.uniform(0, 1), -rng.uniform(0, 0.125), -rng.uniform(0, 0.125), rng.uniform(0, 1), 0, 0, rng.uniform(0, 1)]
    f = f if n == 7 else [f[0], f[1], 0, 0, f[6]]
    return [int(x * 2 ** 62) for x in f]


def scaled(rng):
    """Factors for velocities and their differences, from the range's ends to weak flows."""
    return rng.choice([1.0, 1.0, 2.0 ** -rng.uniform(0, 40)])


@pytest.mark.parametrize("dim", [2, 3])
def test_viscous_energy_within_its_bound(lib, dim):
    rng = random.Random(dim)
    for _ in range(6000):
        s = scaled(rng)
        r = lambda m: int(rng.choice([rng.uniform(-m, m), m, -m]) * s * 2 ** N)  # noqa: E731
        f = coefficients(rng, 5 if dim == 2 else 7)
        exact = rng.uniform(-2, 2) * s, rng.uniform(-2, 2) * s  # the double stresses
        snt = [int(x * 2 ** N) for x in exact]  # truncated toward zero
        if dim == 2:
            v = [[r(U), r(U), r(E), 0, r(5.25)] for _ in range(2)]
            Vn, VE = call(lib.visc2, f, v[0] + v[1] + snt[:1], n=2)
            L, R = v
            sn = Fr(f[0]) * (R[0] - L[0]) + Fr(f[1]) * (L[4] + R[4])
            sums, heat, kap, bn, be = [L[0] + R[0], L[1] + R[1]], R[2] - L[2], f[4], 1, 1.75 + U * 1.25
        else:
            v = [[r(U), r(U), r(U), r(E), r(2.64), r(5.25)] for _ in range(2)]
            Vn, VE = call(lib.visc3d, f, v[0] + v[1] + snt, n=2)
            L, R = v
            sn = Fr(f[0]) * (R[0] - L[0]) + Fr(f[1]) * (L[4] + R[4]) + Fr(f[2]) * (L[5] + R[5])
            sums = [L[j] + R[j] for j in range(3)]
            heat, kap, bn, be = R[3] - L[3], f[6], 1.75, 3.0 + U * 2.25
        sn = sn / Fr(2) ** 64  # .57
        assert abs(Vn - sn) <= bn
        work = Fr(sums[0], 2) * sn / Fr(2) ** N
        for t, x in zip(sums[1:], exact):
            work += Fr(t, 2) * Fr(x) * Fr(2) ** 57 / Fr(2) ** N
        assert abs(VE - (work + Fr(kap) * heat / Fr(2) ** 64)) <= be, (s, float(VE - work))


def test_interface_energy_within_its_bound(lib):
    rng = random.Random(5)
    for _ in range(6000):
        s = scaled(rng)
        r = lambda m: int(rng.choice([rng.uniform(-m, m), m, -m]) * s * 2 ** N)  # noqa: E731
        f = [0] + [int(rng.uniform(0, 1) * 2 ** 62) for _ in range(3)]
        u1, u2, e1, e2 = r(U), r(U), r(E), r(E)
        sig = rng.uniform(-2.6, 2.6) * s
        out, = call(lib.lid, f, [u1, u2, e1, e2, int(sig * 2 ** N)], n=1)
        uw = u1 + Fr(f[1]) * (u2 - u1) / Fr(2) ** 62
        exact = uw * Fr(sig) / Fr(4) + Fr(f[3]) * (e2 - e1) / Fr(2) ** 64
        assert abs(out - exact) <= 1.5 + U / 4 + 2.6 * 0.75 / 4
