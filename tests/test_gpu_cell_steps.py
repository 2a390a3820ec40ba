"""The steps of the cell-parallel march where they can go wrong: grids that
end inside, at and just past a brick on each axis, second neighbours two
cells across a brick face, fewer bricks than blocks and more, and a step
limit inside and between launches."""
import numpy as np
import pytest
import torch

from paper_1502_07303_gb300 import workloads as wl
from parity_util import compare

pytestmark = pytest.mark.gpu

DT = {"f32": torch.float32, "f64": torch.float64}


@pytest.fixture(scope="module")
def fmm():
    if not torch.cuda.is_available():
        pytest.fail("CUDA is required for the gpu tests")
    from paper_1502_07303_gb300 import fmm as _fmm
    return _fmm


def _q(a, dt):
    a = np.asarray(a, np.float64)
    return a.astype(np.float32).astype(np.float64) if dt == "f32" else a


def _dev(a, dt):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=DT[dt], device="cuda")


@pytest.mark.parametrize("dt", ["f64", "f32"])
@pytest.mark.parametrize("shape", [(1, 1, 2), (7, 8, 9), (17, 1, 16), (16, 15, 17), (50, 57, 49)])
def test_first_order_edges(fmm, oracle, dt, shape):
    """Cell by cell the discrete solution, sources in opposite corners."""
    h = 1.0 / max(shape)
    nz, ny, nx = shape
    src = np.unique(np.array([[0, 0, 0], [nx - 1, ny - 1, nz - 1]], np.int64), axis=0)
    F = wl.fourier_speed(shape, wl.draw_fourier_modes(np.random.default_rng(3)), h=h)
    ref = oracle.solve_sources(shape, src, h, speed=_q(F, dt))
    with fmm.Solver(shape, h, dtype=DT[dt], speed=_dev(F, dt), sources=src, schedule=4) as s:
        T, G = s.solve()
    compare(T.cpu().numpy(), G.cpu().numpy(), ref, dt)


@pytest.mark.parametrize("flip", [False, True])
@pytest.mark.parametrize("shape", [(7, 9, 8), (16, 17, 10), (18, 15, 25)])
def test_second_order_edges(fmm, oracle, shape, flip):
    """T = |x|^2 / 2 with slowness |x| from two fixed layers at the low (or,
    mirrored, the high) faces: second-order differences are exact for it, so
    each second neighbour, across a brick face or not, must have been used."""
    h = 1.0 / 24
    Z, Y, X = np.meshgrid(*[(np.arange(n) + 1.0) * h for n in shape], indexing="ij")
    R2 = X * X + Y * Y + Z * Z
    T_ex, F, mask = 0.5 * R2, 1.0 / np.sqrt(R2), np.indices(shape).min(axis=0) < 2
    if flip:
        T_ex, F, mask = (np.ascontiguousarray(a[::-1, ::-1, ::-1]) for a in (T_ex, F, mask))
    T0 = np.where(mask, T_ex, np.inf)
    ref = oracle.march(T0, np.where(mask, oracle.KNOWN_FIX, oracle.FAR).astype(np.uint8), h, speed=F, accuracy=2)
    with fmm.Solver(shape, h, dtype=torch.float64, speed=_dev(F, "f64"), accuracy=2) as s:
        T, G = s.solve_fixed(_dev(T0, "f64"))
    T = T.cpu().numpy()
    compare(T, G.cpu().numpy(), ref, "f64")
    assert np.abs(T - T_ex).max() / T_ex.max() <= 1e-13


@pytest.mark.parametrize("limit", [1, 2, 5, 7])
def test_step_limit(fmm, limit):
    """Launches run 1, 2, 4, ... steps: limits at their ends and inside one;
    the handle then solves in full as if it had not been stopped."""
    shape, h = (20, 20, 20), 1.0 / 20
    src = np.array([[3, 4, 5]], np.int64)
    with fmm.Solver(shape, h, dtype=torch.float64, sources=src, schedule=4) as s:
        full = s.solve()[0].clone()
    with fmm.Solver(shape, h, dtype=torch.float64, sources=src, schedule=4, max_restarts=limit) as s:
        with pytest.raises(fmm.FmmError) as e:
            s.solve()
        assert e.value.code == fmm.FMM_ERR_TIMEOUT
        assert s.stats()["restarts"] == limit
    with fmm.Solver(shape, h, dtype=torch.float64, sources=src, schedule=4) as s:
        assert torch.equal(s.solve()[0], full)
