"""The FP64 tile's face fluxes run in 64-bit fixed point where the states of a
face lie in its range (density in [0.5, 4), |momentum| below 0.656, energy in
[1/16, 4), sound speed squared in [0.26, 3.9]) and in double elsewhere. States
across every edge of that range match the oracle's right-hand side, and a face
takes the same form in every tile shape and in the batch kernel.

Tolerance: the parity norm of the FP64 path, 1e-12 of the largest |R| per
component. Both sides round each flux a few dozen times at 2^-53 of its size;
the states below have jumps that make R at least 1e-2 of flux / dx, so the
difference stays below 64 * 2^-53 / 1e-2 = 7e-13."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2202_11890_gb300 import workloads as W
from pairs import oracle_threads, pair, rel_err
from test_gpu_3d import gpu_rhs3, pair3, rel3
from test_gpu_parity import gpu_rhs
from test_gpu_tile_shapes import SHAPES, launch_buckets, load_table

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

GRID = W.Grid(75, 13, 6, 22)  # ragged tiles, Gamma inside a tile


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2202_11890_gb300 import build
    build.build()
    oracle_threads()


def state(kind):
    """Random cell-to-cell variations of 2 % over the rest state, changed so
    that some or all faces leave the fixed-point range."""
    rng = np.random.default_rng(41)
    rho, p = W.rest_primitives(GRID)
    r = [0.02 * rng.uniform(-1, 1, rho.shape) for _ in range(4)]
    rho, p, u, w = rho * (1 + r[0]), p * (1 + r[1]), r[2], r[3]
    # ramps 0 to 1 to 0 over columns 20-50 and rows 8-27, across Gamma and
    # tiles; gentle enough that every reconstructed pressure stays positive
    ramp = [np.minimum(1.0, 1.3 * (1.0 - np.abs(np.linspace(-1, 1, n)))) for n in (20, 31)]
    part = np.zeros(rho.shape)
    part[8:28, 20:51] = np.outer(*ramp)
    if kind == "dense":  # every cell outside
        rho, p = 8.0 * rho, 8.0 * p
    elif kind == "dense patch":  # densities up to 4.4 over the edge 4
        rho, p = rho * 4.3 ** part, p * 2.0 ** part
    elif kind == "thin patch":  # densities down to 0.25, below 0.5
        rho, p = rho * 0.25 ** part, p * 0.4 ** part
    elif kind == "fast patch":  # momenta up to 1, over 0.656
        u, w = u + part * np.sign(r[2]), w - 0.7 * part
    elif kind == "cold patch":  # sound speed squared down to 0.13, energy to 0.2
        p = p * 0.13 ** part
    elif kind == "hot patch":  # sound speed squared up to 4.6, energy to 8
        p = p * 4.5 ** part
    return W.conserved(rho, u, w, p)


KINDS = ["inside", "dense", "dense patch", "thin patch", "fast patch", "cold patch", "hot patch"]


@pytest.mark.parametrize("xwall,wall", [(0, 0), (1, 1)])
@pytest.mark.parametrize("kind", KINDS)
def test_rhs_across_the_range_matches_oracle(kind, xwall, wall):
    q = state(kind)
    cfg, P, _ = pair(GRID, 2, dt=0.001, xwall=xwall, wall=wall)
    err = rel_err(gpu_rhs(cfg, q), O.rhs(P, q))
    assert np.all(err < 1e-12), err


GRID3 = W.Grid3(45, 6, 7, 4, 10)  # ragged tiles, Gamma inside a tile


def state3(kind):
    """As state(), in 3-D: planes 1 to 4 of columns 15-38 and rows 4-17."""
    rng = np.random.default_rng(43)
    rho, p = W.rest_primitives(GRID3.column_grid())
    shape = (GRID3.nz, GRID3.ny, GRID3.nx)
    r = [0.02 * rng.uniform(-1, 1, shape) for _ in range(5)]
    rho, p = rho[:, None, :] * (1 + r[0]), p[:, None, :] * (1 + r[1])
    u, v, w = r[2:]
    rz, ry, rx = [np.minimum(1.0, 1.3 * (1.0 - np.abs(np.linspace(-1, 1, n)))) for n in (14, 6, 24)]
    part = np.zeros(shape)
    part[4:18, :, 15:39] = rz[:, None, None] * ry[None, :, None] * rx
    if kind == "dense":
        rho, p = 8.0 * rho, 8.0 * p
    elif kind == "dense patch":
        rho, p = rho * 4.3 ** part, p * 2.0 ** part
    elif kind == "fast patch":
        u, v, w = u + part, v - 0.8 * part, w + 0.3 * part
    elif kind == "cold patch":
        p = p * 0.2 ** part
    elif kind == "hot patch":
        p = p * 4.5 ** part
    return W.conserved3(rho, u, v, w, p)


@pytest.mark.parametrize("wall,mu1", [(0, W.MU1), (1, 0.1)])
@pytest.mark.parametrize("kind", [k for k in KINDS if k != "thin patch"])
def test_rhs3_across_the_range_matches_oracle(kind, wall, mu1):
    """mu1 = 0.1 puts fluid 1's coefficients beyond the fixed-point form."""
    q = state3(kind)
    cfg, P, _ = pair3(GRID3, 2, dt=0.001, wall=wall, mu1=mu1)
    err = rel3(gpu_rhs3(cfg, q), O.rhs3(P, q))
    assert np.all(err < 1e-12), err


@pytest.mark.parametrize("mu1,mu2", [(0.03, W.MU2), (W.MU1, 0.08), (0.04, 0.04)])
def test_viscosity_across_the_range_matches_oracle(mu1, mu2):
    """Coefficients (8/3) mu / dx around 1, where the fixed-point form ends."""
    q = state("inside")
    cfg, P, _ = pair(GRID, 2, dt=0.001, mu1=mu1, mu2=mu2)
    err = rel_err(gpu_rhs(cfg, q), O.rhs(P, q))
    assert np.all(err < 1e-12), err


@pytest.mark.parametrize("kind", ["dense", "dense patch", "fast patch", "hot patch"])
def test_same_bits_in_every_tile_shape_and_in_a_batch(kind, tmp_path):
    from paper_2202_11890_gb300 import mprk as M
    q = state(kind)
    cfg, _, _ = pair(GRID, 2, dt=0.001)
    try:
        results = []
        for sh in SHAPES:
            load_table(tmp_path, M, launch_buckets(GRID, 2), sh)
            with M.Instance(cfg, q) as inst:
                inst.step(2)
                results.append(inst.state())
        M.mprk_tune_clear()
        with M.Instance(cfg, q) as inst:
            M.mprk_step_batch([inst.h], 2)
            results.append(inst.state())
    finally:
        M.mprk_tune_clear()
    assert np.isfinite(results[0]).all()
    for r in results[1:]:
        assert np.array_equal(results[0], r)


@pytest.mark.parametrize("n1", range(6, 27))
def test_same_bits_wherever_the_interface_meets_a_tile(n1, tmp_path):
    """Tiles away from walls and the interface read their faces without ghosts;
    every distance of the interface (row n1 of 34) from the edges of 8-, 4- and
    2-row tiles gives the same bits, and the oracle's right-hand side."""
    from paper_2202_11890_gb300 import mprk as M
    grid = W.Grid(41, n1 - 4, 4, 34 - n1)
    rng = np.random.default_rng(47)
    rho, p = W.rest_primitives(grid)
    r = [0.02 * rng.uniform(-1, 1, rho.shape) for _ in range(4)]
    q = W.conserved(rho * (1 + r[0]), r[2], r[3], p * (1 + r[1]))
    cfg, P, _ = pair(grid, 2, dt=0.001)
    assert np.all(rel_err(gpu_rhs(cfg, q), O.rhs(P, q)) < 1e-12)
    results = []
    try:
        for sh in SHAPES:
            load_table(tmp_path, M, launch_buckets(grid, 2), sh)
            with M.Instance(cfg, q) as inst:
                inst.step(1)
                results.append(inst.state())
    finally:
        M.mprk_tune_clear()
    assert np.isfinite(results[0]).all()
    for r in results[1:]:
        assert np.array_equal(results[0], r)
