"""The work that users of this library have it do, as timed and compared cases.

Each case is one call sequence through the public binding
(paper_2202_11890_gb300.mprk), with the sizes of the repository's workloads
(paper_2202_11890_gb300/workloads.py) or ragged ones inside their ranges:

  step    an instance takes a new state, advances n slow steps and gives the
          result back on the device (mprk_set_state, mprk_step, mprk_get_state)
  static  the allocation-free call on a caller-owned state (mprk_step_static)
  io      independent one-step solves through pinned host buffers (mprk_step_io)
  batch   many uneven instances advanced together (mprk_step_batch)
  served  requests submitted to the server and polled until all are done

exact() evaluates the same slow steps (Algorithm 1 of arXiv 2202.11890 on the
finite-volume scheme of Sec. 2.1 and App. B) with plain torch in float64, whole
arrays at a time.
"""
import math
import random
import time

import numpy as np
import torch

from paper_2202_11890_gb300 import mprk

GAMMA, PR = 1.4, 0.72
MU1, MU2 = 1.0 / 20000.0, 1.0 / 5000.0
G = 0.008140864714
SOUND = 1.05  # above every sound speed plus |u| of the initial states below
FLOPS_2D, FLOPS_3D = 355.7, 759.0  # per cell and stage, from the scheme's formulas as written
DEV = "cuda"


# ---- cases -----------------------------------------------------------------

def _case(name, kind, nx, nS, nB, nF, m, steps, precision="fp64", state="bumps", ny=1, base=0, scheme=0, wall=0,
          x_walls=0, count=1):
    return {"name": name, "kind": kind, "nx": nx, "ny": ny, "nS": nS, "nB": nB, "nF": nF, "m": m, "steps": steps,
            "precision": precision, "state": state, "base": base, "scheme": scheme, "wall": wall, "x_walls": x_walls,
            "count": count}


def listed():
    return [
        # one real-time step of a small grid owned by another framework: latency of 9 launches
        _case("static_64_one_step", "static", 64, 30, 4, 30, 4, 1),
        # the 64 x 64 reference solve, 100 slow steps
        _case("plain_64_run", "step", 64, 30, 4, 30, 4, 100),
        # thermal convection, walls all round, thin cells above the interface
        _case("convection_100x300", "step", 100, 96, 4, 200, 4, 10, state="convection", x_walls=1),
        # an ensemble member fed from and returned to host memory, odd sizes, slip walls
        _case("io_515x389", "io", 515, 187, 11, 191, 2, 1, wall=1, count=4),
        # the single large FP64 solve
        _case("large_2048x1024", "step", 2048, 480, 64, 480, 8, 2, state="fourier"),
        # the fourth-order base on a mid-size grid
        _case("rk4_1024x512", "step", 1024, 240, 32, 240, 4, 1, state="fourier", base=2),
        # the 3-D model
        _case("cube_512x64x200", "step", 512, 96, 8, 96, 4, 1, ny=64),
        # the largest mixed-precision solve
        _case("mixed_4096x2048", "step", 4096, 960, 128, 960, 8, 2, precision="fp32flux", state="fourier"),
        # a mid-size ragged mixed-precision solve
        _case("mixed_321x273", "step", 321, 131, 9, 133, 4, 10, precision="fp32flux"),
        # 256 uneven instances per batched step, both precisions
        _case("batch_256_fp64", "batch", 512, 0, 0, 0, 0, 1, count=256),
        _case("batch_256_fp32flux", "batch", 512, 0, 0, 0, 0, 2, precision="fp32flux", count=256),
        # a burst of requests to the server
        _case("served_24", "served", 1024, 0, 0, 0, 0, 60, precision="fp32flux", count=24),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _rows(rng, nz):
    nB = rng.randint(4, max(4, min(64, nz // 8)))
    nS = max(2, int((nz - nB) * rng.uniform(0.35, 0.65)))
    return nS, nB, max(2, nz - nB - nS)


def draw(rng: random.Random):
    kind = rng.choice(["static", "step", "step", "mixed", "io", "cube", "batch", "served"])
    m = rng.choice([1, 2, 4, 8])
    wall = rng.randint(0, 1)
    if kind == "static":
        nx = _log_int(rng, 32, 512)
        nS, nB, nF = _rows(rng, _log_int(rng, 32, 512))
        c = _case("", "static", nx, nS, nB, nF, m, rng.randint(1, 4), wall=wall, x_walls=rng.randint(0, 1))
    elif kind == "step":
        nx = _log_int(rng, 40, 2048)
        nS, nB, nF = _rows(rng, _log_int(rng, 40, 1024))
        base = rng.choice([0, 0, 0, 1, 2])
        conv = rng.random() < 0.25
        c = _case("", "step", nx, nS, nB, nF, min(m, 4) if base else m, rng.randint(1, 2), base=base, wall=wall,
                  x_walls=1 if conv else rng.randint(0, 1), state="convection" if conv else
                  rng.choice(["bumps", "fourier"]), scheme=1 if rng.random() < 0.15 else 0)
    elif kind == "mixed":
        nx = _log_int(rng, 64, 4096)
        nS, nB, nF = _rows(rng, _log_int(rng, 64, 2048))
        c = _case("", "step", nx, nS, nB, nF, m, rng.randint(1, 2), precision="fp32flux", wall=wall,
                  x_walls=rng.randint(0, 1), state=rng.choice(["bumps", "fourier"]))
    elif kind == "io":
        nx = _log_int(rng, 64, 1024)
        nS, nB, nF = _rows(rng, _log_int(rng, 64, 512))
        c = _case("", "io", nx, nS, nB, nF, min(m, 4), 1, wall=wall, count=rng.randint(2, 4),
                  precision=rng.choice(["fp64", "fp32flux"]))
    elif kind == "cube":
        nS, nB, nF = _rows(rng, _log_int(rng, 32, 200))
        c = _case("", "step", _log_int(rng, 32, 512), nS, nB, nF, min(m, 4), 1, ny=_log_int(rng, 8, 64), wall=wall)
    elif kind == "batch":
        c = _case("", "batch", rng.randint(200, 512), 0, 0, 0, 0, 1, count=_log_int(rng, 8, 200),
                  precision=rng.choice(["fp64", "fp32flux"]))
    else:
        c = _case("", "served", rng.randint(200, 1000), 0, 0, 0, 0, rng.randint(10, 40), precision="fp32flux",
                  count=rng.randint(8, 24))
    del c["name"]
    return c


def _members(case):
    """The single solves of a case: itself, or the uneven instances of a batch
    or of a request stream (sides log-uniform up to nx, rate ratios 2, 4, 8)."""
    if case["kind"] not in ("batch", "served"):
        return [case]
    served = case["kind"] == "served"
    rng = np.random.default_rng(1000 * case["count"] + case["nx"])
    lo = 32 if served else 64
    out = []
    for _ in range(case["count"]):
        nx, nz = (int(round(math.exp(rng.uniform(math.log(lo), math.log(case["nx"]))))) for _ in range(2))
        nB = int(rng.integers(4, 17))
        nS = (nz - nB) // 2
        steps = case["steps"]
        if served:
            steps = max(1, int(round(math.exp(rng.uniform(math.log(max(1, steps / 6)), math.log(steps))))))
        out.append(dict(case, nx=nx, nS=nS, nB=nB, nF=nz - nB - nS, m=int(rng.choice([2, 4, 8])), steps=steps))
    return out


def _spacing(case):
    """(dx, dy, dz1, dz2): x over (-5, 5), square cells; the convection state
    has the depths 7 and 3 of Sec. 5.2 instead."""
    dx = 10.0 / case["nx"]
    if case["state"] == "convection":
        return dx, dx, 7.0 / (case["nS"] + case["nB"]), 3.0 / case["nF"]
    return dx, dx, dx, dx


def _dt(case):
    dx, _, dz1, dz2 = _spacing(case)
    slow = min(dx, dz2) if case["scheme"] == 1 else min(dx, dz1)
    return 0.4 * min(slow, case["m"] * min(dx, dz2)) / SOUND


def _config(case):
    dx, dy, dz1, dz2 = _spacing(case)
    return mprk.mprk_config_default(
        case["nx"], case["nS"], case["nB"], case["nF"], case["m"], dt=_dt(case), dx=dx, dy=dy, dz1=dz1, dz2=dz2,
        ny=case["ny"], base=case["base"], scheme=case["scheme"], wall=case["wall"], x_walls=case["x_walls"],
        precision=mprk.MPRK_FP32FLUX if case["precision"] == "fp32flux" else mprk.MPRK_FP64)


# ---- initial states ----------------------------------------------------------

def _initial(case, seed):
    """[4][nz][nx] (or [5][nz][ny][nx]) float64 on the GPU: the stratified rest
    state with seeded Gaussian bumps or Fourier modes of 1e-2 in density and
    velocity, or the warm and cold bubbles of Sec. 5.2's convection."""
    rng = np.random.default_rng([int(seed), 77])
    nx, ny, n1, nz = case["nx"], case["ny"], case["nS"] + case["nB"], case["nS"] + case["nB"] + case["nF"]
    dx, dy, dz1, dz2 = _spacing(case)
    f = dict(dtype=torch.float64, device=DEV)
    k = torch.arange(nz, **f)
    z = torch.where(k < n1, -(n1 - k - 0.5) * dz1, (k - n1 + 0.5) * dz2).view(nz, 1, 1)
    x = (-5.0 + (torch.arange(nx, **f) + 0.5) * dx).view(1, 1, nx)
    y = ((torch.arange(ny, **f) + 0.5 - 0.5 * ny) * dy).view(1, ny, 1)
    zlo, zhi = -n1 * dz1, (nz - n1) * dz2
    cp = 1.0 / (GAMMA - 1.0)
    dth = torch.zeros((nz, ny, nx), **f)
    drho, u, v, w = (torch.zeros((nz, ny, nx), **f) for _ in range(4))
    if case["state"] == "convection":
        for fluid, zc, rad, amp in ((1, -2.5, 2.5, 1.25), (2, 1.5, 1.0, -7.5)):
            r = torch.sqrt((x - rng.uniform(-0.5, 0.5)) ** 2 + (z - zc) ** 2 + 0.0 * y)
            inside = (r <= rad) & ((k < n1) if fluid == 1 else (k >= n1)).view(nz, 1, 1)
            dth = torch.where(inside, amp * rng.uniform(0.8, 1.0) * (1.0 + torch.cos(math.pi * r)), dth)
    elif case["state"] == "fourier":
        xi, zeta = (x + 5.0) / 10.0, (z - zlo) / (zhi - zlo)
        for field in (drho, u, w):
            for _ in range(10):
                kx, kz = (int(t) for t in rng.integers(1, 9, 2))
                a, b = rng.uniform(0.0, 2.0 * math.pi, 2)
                field += 1e-3 * torch.cos(2.0 * math.pi * kx * xi + a) * torch.cos(math.pi * kz * zeta + b)
    else:
        sig = 4.0 * dx
        for _ in range(4):
            xc, yc, zc = rng.uniform(-5, 5), rng.uniform(-0.5, 0.5) * ny * dy, rng.uniform(zlo, zhi)
            d = rng.normal(size=3)
            d[1] = d[1] if ny > 1 else 0.0
            d /= np.linalg.norm(d)
            ex, ey = (x - xc + 5.0) % 10.0 - 5.0, (y - yc + 0.5 * ny * dy) % (ny * dy) - 0.5 * ny * dy
            env = 1e-2 * torch.exp(-(ex ** 2 + (ey ** 2 if ny > 1 else 0.0) + (z - zc) ** 2) / (2.0 * sig * sig))
            drho += env
            u += d[0] * env
            v += d[1] * env
            w += d[2] * env
    fac = 1.0 + dth / 300.0
    psi = 1.0 - G * z / (cp * fac)
    p = psi ** (GAMMA / (GAMMA - 1.0)) / GAMMA
    rho = psi ** (1.0 / (GAMMA - 1.0)) / fac * (1.0 + drho)
    e = p / (GAMMA - 1.0) + 0.5 * rho * (u * u + v * v + w * w)
    if ny > 1:
        return torch.stack([rho, rho * u, rho * v, rho * w, e]).contiguous()
    return torch.stack([rho, rho * u, rho * w, e]).reshape(4, nz, nx).contiguous()


def _initials(case, seed):
    """The states of a case's solves, in the order of its outputs."""
    if case["kind"] == "io":
        return [_initial(case, 100 * int(seed) + j) for j in range(case["count"])]
    return [_initial(c, 1000 * int(seed) + j) for j, c in enumerate(_members(case))]


# ---- one pass ----------------------------------------------------------------

class _Server:
    def __init__(self):
        self.h = mprk.mprk_server_create(32 << 30)

    def __del__(self):
        mprk.mprk_server_destroy(self.h)


def prepare(case, seed):
    q = _initials(case, seed)
    cfgs = [_config(c) for c in _members(case)]
    s = {"case": case, "kind": case["kind"], "cfgs": cfgs, "steps": [c["steps"] for c in _members(case)]}
    if case["kind"] == "static":
        s["q"] = q[0]
    elif case["kind"] == "io":
        s["inst"] = mprk.Instance(cfgs[0], q[0])
        s["in"] = [t.cpu().pin_memory() for t in q]
        s["out"] = [torch.empty_like(t).pin_memory() for t in s["in"]]
    elif case["kind"] == "served":
        s["q"] = [t.cpu().numpy() for t in q]
        s["out"] = [np.empty_like(t) for t in s["q"]]
        s["server"] = _Server()
    else:
        # the results of all instances lie one after another in one buffer
        torch.cuda.synchronize()
        s["q"] = q
        s["inst"] = [mprk.Instance(c, t) for c, t in zip(cfgs, q)]
        s["flat"] = torch.empty(sum(t.numel() for t in q), dtype=torch.float64, device=DEV)
        s["out"] = [t.view(a.shape) for t, a in zip(torch.split(s["flat"], [t.numel() for t in q]), q)]
    torch.cuda.synchronize()
    return s


def run(s):
    kind = s["kind"]
    if kind == "static":
        out = s["q"].clone()
        mprk.mprk_step_static(s["cfgs"][0], out, s["steps"][0], torch.cuda.current_stream().cuda_stream)
        return out
    if kind == "io":
        mprk.mprk_step_io(s["inst"].h, s["in"], s["out"])
        return s["out"]
    if kind == "served":
        srv = s["server"].h
        waiting = {mprk.mprk_submit(srv, c, q, n): j
                   for j, (c, q, n) in enumerate(zip(s["cfgs"], s["q"], s["steps"]))}
        while waiting:
            for ticket, j in list(waiting.items()):
                status, err, _ = mprk.mprk_poll(srv, ticket, s["out"][j])
                if status == mprk.MPRK_REQ_DONE:
                    if err:
                        raise RuntimeError(f"request {j} failed: {err}")
                    del waiting[ticket]
            time.sleep(2e-4)
        return s["out"]
    for inst, q in zip(s["inst"], s["q"]):
        inst.set_state(q)
    if kind == "batch":
        mprk.mprk_step_batch([i.h for i in s["inst"]], s["steps"][0])
    else:
        s["inst"][0].step(s["steps"][0])
    for inst, out in zip(s["inst"], s["out"]):
        mprk.mprk_get_state(inst.h, out)
    return s["flat"] if kind == "batch" else s["out"][0]


def _stages(base):
    return {0: 2, 1: 3, 2: 4}[base]


def work(case):
    """Each solve's state read and written once, and the scheme's arithmetic:
    the cells of every band times its stages."""
    nbytes = flops = 0.0
    for c in _members(case):
        cells = c["nx"] * c["ny"]
        nc = 5 if c["ny"] > 1 else 4
        st = _stages(c["base"])
        slow = c["m"] * c["nS"] if c["scheme"] == 1 else c["nS"]
        stages = cells * st * (slow + c["m"] * (c["nB"] + c["nF"])) * c["steps"]
        many = c["count"] if c["kind"] == "io" else 1
        nbytes += many * 2.0 * 8.0 * nc * cells * (c["nS"] + c["nB"] + c["nF"])
        flops += many * stages * (FLOPS_3D if c["ny"] > 1 else FLOPS_2D)
    return {"bytes": nbytes, "flops": flops}


# ---- the same steps in plain float64 ------------------------------------------

def exact(case, seed):
    out = [_solve(c, q) for c, q in zip(_members(case) * (case["count"] if case["kind"] == "io" else 1),
                                        _initials(case, seed))]
    if case["kind"] == "io":
        return [t.cpu() for t in out]
    if case["kind"] == "served":
        return [t.cpu().numpy() for t in out]
    return torch.cat([t.reshape(-1) for t in out]) if case["kind"] == "batch" else out[0]


def _tableau(base):
    if base == 1:
        return [[], [1.0], [0.25, 0.25]], [1 / 6, 1 / 6, 2 / 3]
    if base == 2:
        return [[], [0.5], [0.0, 0.5], [0.0, 0.0, 1.0]], [1 / 6, 1 / 3, 1 / 3, 1 / 6]
    return [[], [1.0]], [0.5, 0.5]


def _sum(coef, terms):
    return sum(c * t for c, t in zip(coef, terms) if c != 0.0)


def _solve(case, q):
    """Algorithm 1 with any base: F takes m base steps of dt/m, B restarts the
    base from q_n in every fast substep with the weights b/m, S takes one base
    step and repeats its first stage states afterwards."""
    shape = q.shape
    q = q.reshape(shape[0], shape[1], case["ny"], case["nx"])  # [component][z][y][x]
    A, b = _tableau(case["base"])
    m, dt = case["m"], _dt(case)
    nS, n1 = case["nS"], case["nS"] + case["nB"]
    if case["scheme"] == 1:  # single rate: every row steps like F
        nS = n1 = 0
    for _ in range(case["steps"]):
        fast, acc, slow, first = q[:, n1:], 0.0, [], []
        for sub in range(m):
            R = []
            for a in A:
                Q = torch.cat([q[:, :n1], fast], 1)
                if R:
                    Q[:, nS:n1] += dt * _sum(a, [r[:, nS:n1] for r in R])
                    Q[:, n1:] += (dt / m) * _sum(a, [r[:, n1:] for r in R])
                if sub == 0:
                    if R:
                        Q[:, :nS] += dt * _sum(a, [r[:, :nS] for r in R])
                    first.append(Q[:, :nS].clone())
                else:
                    Q[:, :nS] = first[len(R)]
                R.append(_rhs(case, Q))
            fast = fast + (dt / m) * _sum(b, [r[:, n1:] for r in R])
            acc = acc + _sum(b, [r[:, nS:n1] for r in R])
            if sub == 0:
                slow = q[:, :nS] + dt * _sum(b, [r[:, :nS] for r in R])
        q = torch.cat([slow, q[:, nS:n1] + (dt / m) * acc, fast], 1)
    return q.reshape(shape)


def _pressure(q):
    return (GAMMA - 1.0) * (q[-1] - 0.5 * sum(c * c for c in q[1:-1]) / q[0])


def _lax_friedrichs(L, R, n):
    """Lax-Friedrichs flux along momentum component n, with the largest speed
    of the left, right and Roe-averaged states."""
    F, lam, mom = 0.0, None, range(1, L.shape[0] - 1)
    roe, weight = [0.0] * (len(mom) + 1), 0.0
    for s in (L, R):
        p = _pressure(s)
        un, r = s[n] / s[0], torch.sqrt(s[0])
        f = s * un
        f[n] += p
        f[-1] += p * un
        F = F + 0.5 * f
        speed = un.abs() + torch.sqrt(GAMMA * p / s[0])
        lam = speed if lam is None else torch.maximum(lam, speed)
        for j, c in enumerate(mom):
            roe[j] = roe[j] + s[c] / r
        roe[-1] = roe[-1] + (s[-1] + p) / r
        weight = weight + r
    vel = [t / weight for t in roe[:-1]]
    sound = torch.sqrt((GAMMA - 1.0) * (roe[-1] / weight - 0.5 * sum(t * t for t in vel)))
    return F + 0.5 * torch.maximum(lam, vel[n - 1].abs() + sound) * (L - R)


def _ghosts(a, axis, lo, hi):
    """a with one ghost layer on both ends of axis; lo and hi map the end
    layers to their ghosts, None is periodic."""
    first, last = a.narrow(axis, 0, 1), a.narrow(axis, a.shape[axis] - 1, 1)
    return torch.cat([last if lo is None else lo(first), a, first if hi is None else hi(last)], axis)


def _signed(signs):
    return lambda t: t * torch.tensor(signs, dtype=t.dtype, device=t.device).view(-1, 1, 1, 1)


def _rhs(case, Q):
    """-div(F^I - F^V) + s of every row: the two fluids meet only through the
    interface's bulk fluxes and wall states."""
    n1 = case["nS"] + case["nB"]
    dx, dy, dz1, dz2 = _spacing(case)
    fluids = []
    for rows, dz, mu in ((Q[:, :n1], dz1, MU1), (Q[:, n1:], dz2, MU2)):
        kap = mu / (GAMMA - 1.0) / PR
        vel = rows[1:-1] / rows[0]
        fluids.append((rows, dz, mu, kap, vel, GAMMA * _pressure(rows) / rows[0]))
    (_, _, mua, ka, va, Ta), (_, _, mub, kb, vb, Tb) = fluids
    va, vb, Ta, Tb = va[:, -1:], vb[:, :1], Ta[-1:], Tb[:1]
    shear = 2.0 * mua * mub / (dz2 * mua + dz1 * mub) * (vb - va)[:-1]  # tangential components
    heat = -2.0 * ka * kb / (dz2 * ka + dz1 * kb) * (Tb - Ta)
    walls = (va[:-1] + shear * dz1 / (2.0 * mua), vb[:-1] - shear * dz2 / (2.0 * mub))
    return torch.cat([_fluid_rhs(case, f, up, (dx, dy, f[1]), shear, heat, walls[up])
                      for up, f in enumerate(fluids)], 1)


def _fluid_rhs(case, fluid, up, spacing, shear, heat, uw):
    """One fluid's rows; up: 0 below the interface, 1 above it."""
    q, _, mu, kap, vel, T = fluid
    nd = vel.shape[0]
    axes = {0: 3, nd - 1: 1}  # velocity component -> array axis
    if nd == 3:
        axes[1] = 2
    d = {0: spacing[0], nd - 1: spacing[2]}
    if nd == 3:
        d[1] = spacing[1]
    slip = -1.0 if case["wall"] == 0 else 1.0

    def wall_mirror(c):  # conserved variables: normal momentum odd
        return _signed([-1.0 if j == c + 1 else 1.0 for j in range(nd + 2)])

    def wall_vel(c):  # velocities: normal odd, tangential by the wall's kind
        return _signed([-1.0 if j == c else slip for j in range(nd)])

    def lid_vel(v):  # 2 (wall velocity) - v, the lid at rest normally
        return torch.cat([2.0 * uw, torch.zeros_like(v[:1])]) - v

    def ends(c, wall, lid):
        if c == nd - 1:
            return (wall, lid) if up == 0 else (lid, wall)
        return (wall, wall) if c == 0 and case["x_walls"] else (None, None)

    def central(a, c, lo, hi):
        ext = _ghosts(a, axes[c], lo, hi)
        n = a.shape[axes[c]]
        return ext.narrow(axes[c], 2, n) - ext.narrow(axes[c], 0, n)

    grad = {c: central(vel, c, *ends(c, wall_vel(c), lid_vel)) / (2.0 * d[c]) for c in axes}
    R = torch.zeros_like(q)
    for c, ax in axes.items():
        n = q.shape[ax]
        mirror = ends(c, wall_mirror(c), wall_mirror(c))
        slope = 0.25 * central(q, c, *mirror)
        upper, lower = q + slope, q - slope  # states at a cell's upper and lower face
        up_end = upper.narrow(ax, n - 1, 1) if mirror[0] is None else mirror[0](lower.narrow(ax, 0, 1))
        lo_end = lower.narrow(ax, 0, 1) if mirror[1] is None else mirror[1](upper.narrow(ax, n - 1, 1))
        F = _lax_friedrichs(torch.cat([up_end, upper], ax), torch.cat([lower, lo_end], ax), c + 1)
        # viscous flux from the common face values of the cell pairs
        ev = _ghosts(vel, ax, *ends(c, wall_vel(c), lid_vel))
        same = ends(c, lambda t: t, lambda t: t)
        eT = _ghosts(T[None], ax, *same)[0]
        face = lambda a: (a.narrow(ax, 0, n + 1), a.narrow(ax, 1, n + 1))  # noqa: E731
        vL, vR = face(ev)
        axT = ax - 1
        dT = (eT.narrow(axT, 1, n + 1) - eT.narrow(axT, 0, n + 1)) / d[c]
        mean, dn = 0.5 * (vL + vR), (vR - vL) / d[c]
        dtan = {}
        for t in axes:
            if t != c:
                gL, gR = face(_ghosts(grad[t], ax, *ends(c, wall_vel(c), wall_vel(c))))
                dtan[t] = 0.5 * (gL + gR)
        V = torch.zeros_like(F)
        div = dn[c] + sum(dtan[t][t] for t in dtan)
        for j in range(nd):
            V[j + 1] = mu * (2.0 * dn[c] - 2.0 / 3.0 * div) if j == c else mu * (dtan[j][c] + dn[j])
        V[-1] = sum(mean[j] * V[j + 1] for j in range(nd)) + kap * dT
        if c == nd - 1:  # the interface's bulk fluxes in place of the recipe
            at = V.narrow(ax, n if up == 0 else 0, 1)
            at.zero_()
            at[1:nd] = shear
            at[-1] = (uw * shear).sum(0) - heat
        F = F - V
        R -= (F.narrow(ax, 1, n) - F.narrow(ax, 0, n)) / d[c]
    R[nd] -= G * q[0]
    R[-1] -= G * q[nd]
    return R
