"""Launches of a slow step that overlap at their ends give what the same
launches give one after another (mprk_profile_step), and the state copies and
step completion of four rows per thread handle odd widths and row tails.

Tolerances: FP64 bitwise, since both run the same kernels. The FP32-flux
launches of one wave are compiled apart for the overlap, so the two may
contract float operations differently: 1e-6 per component after three steps, as
between the single and the batched form; a launch that read what the one before
had not written yet would be off by a stage's change, 1e-3."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2202_11890_gb300 import workloads as W
from pairs import oracle_threads, pair, rel_err
from test_gpu_3d import pair3

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2202_11890_gb300 import build
    build.build()
    oracle_threads()


def M():
    from paper_2202_11890_gb300 import mprk
    return mprk


def both(cfg, q, steps):
    """The state after mprk_step and after as many profiled steps."""
    with M().Instance(cfg, q) as a, M().Instance(cfg, q) as b:
        a.step(steps)
        for _ in range(steps):
            M().mprk_profile_step(b.h)
        assert a.status() == 0 and b.status() == 0
        return a.state(), b.state()


@pytest.mark.parametrize("m", [3, 4])
@pytest.mark.parametrize("share", [0.55, 1.0, 1.45])
def test_fp32_flux_launches_of_one_wave(share, m):
    """32 x 16 tiles in about `share` of the SMs' number, between half and one
    and a half of it; ragged columns and rows, Gamma inside a tile."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    rows = 11
    cols = max(1, int(share * sms / rows))
    assert sms <= 2 * rows * cols <= 3 * sms
    g = W.Grid(32 * cols - 13, 72, 9, 16 * rows - 5 - 81)
    q = W.gaussian_bumps(g, 71)
    cfg, P, dt = pair(g, m, q0=q, precision=M().MPRK_FP32FLUX)
    got, apart = both(cfg, q, 3)
    assert np.all(rel_err(got, apart) < 1e-6), rel_err(got, apart)
    ref, _ = O.mprk_step(P, q, 3)
    assert np.all(rel_err(got, ref) < 1e-5), rel_err(got, ref)


@pytest.mark.parametrize("dims,m,base", [((64, 30, 4, 30), 4, 0), ((300, 80, 8, 80), 3, 0), ((700, 150, 20, 171), 2, 0),
                                         ((200, 40, 8, 41), 2, 2)])
def test_fp64_launches(dims, m, base):
    """Every tile shape of the default rule; RK4 last."""
    g = W.Grid(*dims)
    q = W.gaussian_bumps(g, 73)
    cfg, _, _ = pair(g, m, q0=q)
    cfg.base = base
    got, apart = both(cfg, q, 3)
    assert np.isfinite(got).all() and np.array_equal(got, apart)


def test_3d_launches():
    g = W.Grid3(70, 9, 20, 5, 24)
    q = W.gaussian_bumps3(g, 75)
    cfg, _, _ = pair3(g, 3, q0=q)
    got, apart = both(cfg, q, 3)
    assert np.isfinite(got).all() and np.array_equal(got, apart)


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("shift", [0, 1])
def test_odd_width_copies_and_completion(precision, shift):
    """1025 x 701 cells, above the size from which a thread copies four rows,
    with a row tail; shift = 1 moves the caller's buffers off 16-byte bounds."""
    g = W.Grid(1025, 340, 10, 351)
    q = W.gaussian_bumps(g, 77)
    cfg, P, dt = pair(g, 1, q0=q, precision=precision)
    room = torch.zeros(q.size + 1, dtype=torch.float64, device="cuda")
    src = room[shift:shift + q.size].view(q.shape)
    src.copy_(torch.from_numpy(q))
    out = torch.zeros_like(room)
    dst = out[shift:shift + q.size].view(q.shape)
    torch.cuda.synchronize()
    with M().Instance(cfg, q) as inst:
        inst.step(1)
        inst.set_state(src)
        M().mprk_get_state(inst.h, dst)
        inst.sync()
        assert torch.equal(dst, src)
        assert float(out[-1 if shift == 0 else 0]) == 0.0
        inst.step(1)
        got = inst.state()
    with M().Instance(cfg, q) as inst:
        inst.step(1)
        assert np.array_equal(inst.state(), got)
    ref, _ = O.mprk_step(P, q)
    assert np.all(rel_err(got, ref) < (1e-5 if precision else 1e-12))
