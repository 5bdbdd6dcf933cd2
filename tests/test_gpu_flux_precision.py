"""The FP64 right-hand side is as accurate as plain double arithmetic, also
where the momenta are far below one: errors against extended precision
(long double: 64 or 113 bits) beside those of the FP64 oracle on the same
state, for noise of every size, weak shears of a flow that is uniform along
one direction, and Gaussian bumps with their tails.

Tolerance: both evaluate the same formulas and round each flux a few dozen
times; the root mean square over all cells may differ by the order of the
operations, which is bounded by a factor of 1.5. A shear's errors are the same
in every column, some twenty independent ones: 16 draws make one mean (a
single draw's ratio scatters by 0.3)."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2202_11890_gb300 import workloads as W
from pairs import oracle_threads, pair, rel_err
from test_gpu_3d import gpu_rhs3, pair3, rel3
from test_gpu_parity import gpu_rhs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

LD = np.longdouble


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    if np.finfo(LD).nmant < 63:
        pytest.skip("long double is no wider than double")
    from paper_2202_11890_gb300 import build
    build.build()
    oracle_threads()


# ---- -div(F^I - F^V) + s in long double -------------------------------------

def pressure(q):
    return (LD(W.GAMMA) - 1) * (q[-1] - (q[1:-1] ** 2).sum(0) / q[0] / 2)


def lax_friedrichs(L, R, n):
    g = LD(W.GAMMA)
    F, roe, weight, lam = 0, 0, 0, 0
    for s in (L, R):
        p, r = pressure(s), np.sqrt(s[0])
        f = s * (s[n] / s[0])
        f[n] += p
        f[-1] += p * s[n] / s[0]
        F = F + f / 2
        lam = np.maximum(lam, np.abs(s[n] / s[0]) + np.sqrt(g * p / s[0]))
        roe = roe + np.concatenate([s[1:-1], (s[-1] + p)[None]]) / r
        weight = weight + r
    roe = roe / weight
    sound = np.sqrt((g - 1) * (roe[-1] - (roe[:-1] ** 2).sum(0) / 2))
    return F + np.maximum(lam, np.abs(roe[n - 1]) + sound) * (L - R) / 2


def ghosts(a, ax, lo, hi):
    """One ghost layer on both ends of axis ax; lo and hi map the end layers
    to their ghosts, None is periodic."""
    first, last = np.take(a, [0], ax), np.take(a, [-1], ax)
    return np.concatenate([last if lo is None else lo(first), a, first if hi is None else hi(last)], ax)


def cut(a, ax, lo, n):
    return a[(slice(None),) * ax + (slice(lo, lo + n),)]


def rhs(grid, q, wall):
    """[nc][nz][ny][nx] of both fluids, x and y periodic."""
    q = q.astype(LD)
    n1, dx = grid.nS + grid.nB, LD(grid.dx)
    mus, out = (LD(W.MU1), LD(W.MU2)), []
    fl = [q[:, :n1], q[:, n1:]]
    kap = [m / (LD(W.GAMMA) - 1) / LD(W.PR) for m in mus]
    vel = [f[1:-1] / f[0] for f in fl]
    T = [LD(W.GAMMA) * pressure(f) / f[0] for f in fl]
    dv, dT = (vel[1][:, :1] - vel[0][:, -1:])[:-1], T[1][:1] - T[0][-1:]
    shear = 2 * mus[0] * mus[1] / (dx * (mus[0] + mus[1])) * dv
    heat = -2 * kap[0] * kap[1] / (dx * (kap[0] + kap[1])) * dT
    uw = vel[0][:-1, -1:] + shear * dx / (2 * mus[0])
    for up in (0, 1):
        out.append(fluid_rhs(fl[up], up, dx, mus[up], kap[up], vel[up], T[up], shear, heat, uw, 1 if wall else -1))
    return np.concatenate(out, 1)


def fluid_rhs(q, up, d, mu, kap, vel, T, shear, heat, uw, slip):
    nd = len(vel)
    axes = {0: 3, nd - 1: 1}
    if nd == 3:
        axes[1] = 2
    sign = lambda s: (lambda t: t * np.array(s, LD).reshape(-1, 1, 1, 1))  # noqa: E731
    lid = lambda v: np.concatenate([2 * uw - v[:-1], -v[-1:]])  # noqa: E731
    mirror = sign([1] * nd + [-1, 1])          # conserved variables at a wall or the interface
    wall = sign([slip] * (nd - 1) + [-1])      # velocities at an outer wall
    ends = lambda c, w, li: ((w, li) if up == 0 else (li, w)) if c == nd - 1 else (None, None)  # noqa: E731

    def central(a, c, lo, hi):
        e, n = ghosts(a, axes[c], lo, hi), a.shape[axes[c]]
        return cut(e, axes[c], 2, n) - cut(e, axes[c], 0, n)

    grad = {c: central(vel, c, *ends(c, wall, lid)) / (2 * d) for c in axes}
    R = np.zeros_like(q)
    for c, ax in axes.items():
        n = q.shape[ax]
        mir = ends(c, mirror, mirror)
        slope = central(q, c, *mir) / 4
        upper, lower = q + slope, q - slope
        left = np.take(upper, [-1], ax) if mir[0] is None else mir[0](np.take(lower, [0], ax))
        right = np.take(lower, [0], ax) if mir[1] is None else mir[1](np.take(upper, [-1], ax))
        F = lax_friedrichs(np.concatenate([left, upper], ax), np.concatenate([lower, right], ax), c + 1)
        face = lambda a: (cut(a, ax, 0, n + 1), cut(a, ax, 1, n + 1))  # noqa: E731
        vL, vR = face(ghosts(vel, ax, *ends(c, wall, lid)))
        same = lambda t: t  # noqa: E731
        TL, TR = face(ghosts(T[None], ax, *ends(c, same, same)))
        mean, dn = (vL + vR) / 2, (vR - vL) / d
        tan = {t: sum(face(ghosts(grad[t], ax, *ends(c, wall, wall)))) / 2 for t in axes if t != c}
        V = np.zeros_like(F)
        for j in range(nd):
            div = dn[c] + sum(tan[t][t] for t in tan)
            V[j + 1] = mu * (2 * dn[c] - div * 2 / 3) if j == c else mu * (tan[j][c] + dn[j])
        V[-1] = (mean * V[1:-1]).sum(0) + kap * ((TR - TL) / d)[0]
        if c == nd - 1:  # the interface's bulk fluxes in place of the recipe
            at = V[:, n:n + 1] if up == 0 else V[:, :1]
            at[:] = 0
            at[1:nd] = shear
            at[-1] = (uw * shear).sum(0) - heat
        F = F - V
        R -= (cut(F, ax, 1, n) - cut(F, ax, 0, n)) / d
    R[nd] -= LD(-W.G_SIGNED) * q[0]
    R[-1] -= LD(-W.G_SIGNED) * q[nd]
    return R


# ---- states -------------------------------------------------------------------

GRID = W.Grid(70, 13, 6, 22)
GRID3 = W.Grid3(40, 6, 7, 4, 10)
KINDS = [("noise", a) for a in (2e-2, 1e-4, 1e-7)] + \
        [("shear", a) for a in (1e-1, 1e-4, 1e-6, 1e-10, 1e-14)] + [("bumps", 1e-2)]


def fields(kind, amp, rho, p, nd, rng):
    """rho, p and nd velocities over [nz][..][nx] rest fields."""
    shape = rho.shape
    rand = lambda s: rng.uniform(-1, 1, s)  # noqa: E731
    if kind == "noise":
        return [rho * (1 + amp * rand(shape)), p * (1 + amp * rand(shape))] + [amp * rand(shape) for _ in range(nd)]
    if kind == "shear":  # horizontal velocities that vary along z only, in the stratified fluid
        prof = (shape[0],) + (1,) * (len(shape) - 1)
        return [rho, p] + [amp * rand(prof) * np.ones(shape) for _ in range(nd - 1)] + [np.zeros(shape)]
    centre = [0.6 * shape[0]] + [2.0] * (len(shape) - 2) + [0.4 * shape[-1]]
    at = np.meshgrid(*[np.arange(n) - c for n, c in zip(shape, centre)], indexing="ij")
    env = amp * np.exp(-sum(x * x for x in at) / 18.0)
    return [rho * (1 + env), p] + [w * env for w in (0.6, -0.5, 0.3)[:nd]]


def draws(kind):
    return 16 if kind == "shear" else 1


def compare(err_gpu, err_double):
    """Lists of errors [component][..] of one right-hand side each."""
    rms = lambda es: np.sqrt(np.mean([(e.astype(np.float64) ** 2).reshape(len(e), -1).mean(1)  # noqa: E731
                                      for e in es], 0))
    a, b = rms(err_gpu), rms(err_double)
    assert np.all(a <= 1.5 * b), (a / np.where(b > 0, b, 1), b)


@pytest.mark.parametrize("wall", [0, 1])
@pytest.mark.parametrize("kind,amp", KINDS)
def test_rhs_as_accurate_as_double(kind, amp, wall):
    errors = [], []
    for seed in range(53, 53 + draws(kind)):
        rho, p, u, w = fields(kind, amp, *W.rest_primitives(GRID), 2, np.random.default_rng(seed))
        q = W.conserved(rho, u, w, p)
        cfg, P, _ = pair(GRID, 2, dt=0.001, wall=wall)
        true = rhs(GRID, q[:, :, None, :], wall)[:, :, 0]
        errors[0].append(gpu_rhs(cfg, q) - true)
        errors[1].append(O.rhs(P, q) - true)
    compare(*errors)


@pytest.mark.parametrize("wall", [0, 1])
@pytest.mark.parametrize("kind,amp", KINDS)
def test_rhs3_as_accurate_as_double(kind, amp, wall):
    shape = (GRID3.nz, GRID3.ny, GRID3.nx)
    errors = [], []
    for seed in range(59, 59 + draws(kind)):
        rho, p = (np.broadcast_to(f[:, None, :], shape) for f in W.rest_primitives(GRID3.column_grid()))
        rho, p, u, v, w = fields(kind, amp, rho, p, 3, np.random.default_rng(seed))
        q = W.conserved3(rho, u, v, w, p)
        cfg, P, _ = pair3(GRID3, 2, dt=0.001, wall=wall)
        true = rhs(GRID3, q, wall)
        errors[0].append(gpu_rhs3(cfg, q) - true)
        errors[1].append(O.rhs3(P, q) - true)
    compare(*errors)


def end_mantissas(shape, rng):
    """Momenta of one to 2^-12 of 0.3 whose mantissas are at the ends of their
    words: all ones, 31 or 32 leading ones, one bit at the words' border."""
    man = np.array([0, 1, 2 ** 52 - 1, 2 ** 52 - 2, 2 ** 52 - 2 ** 21, 2 ** 52 - 2 ** 20, 2 ** 52 - 2 ** 22, 2 ** 31,
                    2 ** 21 - 1, 2 ** 32 - 1], np.uint64)
    e = rng.integers(1009, 1022, shape).astype(np.uint64)
    x = (rng.choice(man, shape) | e << np.uint64(52)).view(np.float64)
    return np.where(rng.random(shape) < 0.5, -x, x)


def test_momenta_with_mantissas_at_the_ends_of_words():
    """Against the oracle to the parity norm, 1e-12 of the largest |R|."""
    rng = np.random.default_rng(61)
    rho, p = W.rest_primitives(GRID)
    q = W.conserved(rho, 0 * rho, 0 * rho, p)
    q[1], q[2] = end_mantissas(rho.shape, rng), end_mantissas(rho.shape, rng)
    q[3] += 0.5 * (q[1] ** 2 + q[2] ** 2) / rho
    cfg, P, _ = pair(GRID, 2, dt=0.001)
    err = rel_err(gpu_rhs(cfg, q), O.rhs(P, q))
    assert np.all(err < 1e-12), err
    shape = (GRID3.nz, GRID3.ny, GRID3.nx)
    rho, p = (np.broadcast_to(f[:, None, :], shape) for f in W.rest_primitives(GRID3.column_grid()))
    q = W.conserved3(rho, 0 * rho, 0 * rho, 0 * rho, p)
    for c in (1, 2, 3):
        q[c] = end_mantissas(shape, rng)
        q[4] += 0.5 * q[c] ** 2 / rho
    cfg, P, _ = pair3(GRID3, 2, dt=0.001)
    err = rel3(gpu_rhs3(cfg, q), O.rhs3(P, q))
    assert np.all(err < 1e-12), err
