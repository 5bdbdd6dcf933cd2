"""States scattered across the fixed-point range: one face outside takes its row
of 32 faces to the double pass, where the Roe speed is evaluated only where it
can be the largest. The right-hand side matches the oracle and a state gets the
same bits in every tile shape and in a batch.

Tolerance: 1e-12 of the largest |R| per component, the parity norm of the FP64
path: both sides round each flux a few dozen times at 2^-53 of its size, and the
jumps make R at least 1e-2 of flux / dx."""
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


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2202_11890_gb300 import build
    build.build()
    oracle_threads()


def fields(rho, p, n, outside, jump, seed):
    """Cell noise of size `jump` in every variable (n velocities); `outside` of
    the cells get a density below the range."""
    rng = np.random.default_rng(seed)
    r = [jump * rng.uniform(-1, 1, rho.shape) for _ in range(n + 2)]
    rho = np.where(rng.random(rho.shape) < outside, 0.45, 1.0) * rho * (1 + r[0])
    return [rho, p * (1 + r[1])] + r[2:]


@pytest.mark.parametrize("nx", [96, 75, 33])
@pytest.mark.parametrize("outside,jump,scale", [(0.003, 0.02, 1), (0.05, 0.2, 1), (0.3, 0.05, 1), (0.0, 0.25, 8),
                                                (0.0, 0.3, 1)])
def test_rhs_and_bits(nx, outside, jump, scale, tmp_path):
    from paper_2202_11890_gb300 import mprk as M
    g = W.Grid(nx, 13, 6, 22)
    rho, p, u, w = fields(*W.rest_primitives(g), 2, outside, jump, nx)
    q = W.conserved(scale * rho, u, w, scale * p)
    cfg, P, _ = pair(g, 2, dt=0.001)
    err = rel_err(gpu_rhs(cfg, q), O.rhs(P, q))
    assert np.all(err < 1e-12), err
    results = []
    try:
        for sh in SHAPES:
            load_table(tmp_path, M, launch_buckets(g, 2), sh)
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


@pytest.mark.parametrize("outside,jump,scale", [(0.003, 0.02, 1), (0.05, 0.2, 1), (0.3, 0.05, 1), (0.0, 0.25, 8)])
def test_rhs3(outside, jump, scale):
    g = W.Grid3(45, 6, 7, 4, 17)
    shape = (g.nz, g.ny, g.nx)
    rho, p = (np.broadcast_to(f[:, None, :], shape) for f in W.rest_primitives(g.column_grid()))
    rho, p, u, v, w = fields(rho, p, 3, outside, jump, 7)
    q = W.conserved3(scale * rho, u, v, w, scale * p)
    cfg, P, _ = pair3(g, 2, dt=0.001)
    err = rel3(gpu_rhs3(cfg, q), O.rhs3(P, q))
    assert np.all(err < 1e-12), err
