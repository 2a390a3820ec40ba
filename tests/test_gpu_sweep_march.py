"""The sweep march of a brick where it can go wrong: grids of one to three
bricks per axis with every remainder at the brick edge, with and without a
band width (cells above the bound), fronts that cross a brick in several
octants, and a stopped solve resumed under another schedule."""
import math

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


@pytest.mark.parametrize("dt", ["f64", "f32"])
@pytest.mark.parametrize("schedule", [1, 2, 3])
@pytest.mark.parametrize("shape", [(1, 1, 1), (1, 8, 9), (7, 8, 9), (17, 1, 16), (16, 15, 17), (24, 9, 8)])
def test_brick_edges(fmm, oracle, dt, schedule, shape):
    """Sources in opposite corners and the middle: every octant in one brick."""
    h = 1.0 / max(shape)
    nz, ny, nx = shape
    src = np.unique(np.array([[0, 0, 0], [nx - 1, ny - 1, nz - 1], [nx // 2, 0, nz - 1]], np.int64), axis=0)
    F = wl.fourier_speed(shape, wl.draw_fourier_modes(np.random.default_rng(7)), h=h)
    ref = oracle.solve_sources(shape, src, h, speed=_q(F, dt))
    with fmm.Solver(shape, h, dtype=DT[dt], speed=torch.as_tensor(F, dtype=DT[dt], device="cuda"),
                    sources=src, schedule=schedule) as s:
        T, G = s.solve()
    compare(T.cpu().numpy(), G.cpu().numpy(), ref, dt)


@pytest.mark.parametrize("schedule", [1, 2, 3])
@pytest.mark.parametrize("ahead", [0.0, 1.5])
@pytest.mark.parametrize("width_cells", [2.25, 9.5, math.inf])
def test_bounded_march(fmm, oracle, schedule, ahead, width_cells):
    """Cells above the band (or the look-ahead) stay BAND and are not used."""
    p = wl.random_spheres(shape=(25, 33, 23), count=4, seed=9)
    w = width_cells * p.h
    ref = oracle.solve_reinit(p.phi0, p.h, width=w)
    with fmm.Solver(p.shape, p.h, dtype=torch.float64, schedule=schedule, width=w, ahead=ahead) as s:
        T, G = s.reinit(torch.as_tensor(p.phi0, dtype=torch.float64, device="cuda"))
    compare(T.cpu().numpy(), G.cpu().numpy(), ref, "f64", width=w)


@pytest.mark.parametrize("dt", ["f64", "f32"])
@pytest.mark.parametrize("first,then", [(3, 2), (2, 3)])
def test_stopped_solve_resumes_under_another_schedule(fmm, oracle, dt, first, then):
    p = wl.random_spheres(n=37, count=5, seed=4)
    phi = torch.as_tensor(p.phi0, dtype=DT[dt], device="cuda")
    with fmm.Solver(p.shape, p.h, dtype=DT[dt], schedule=first, stride=1.0, ahead=1.0, max_restarts=5) as s:
        with pytest.raises(fmm.FmmError) as e:
            s.reinit(phi)
        assert e.value.code == fmm.FMM_ERR_TIMEOUT
        image = s.checkpoint()
    with fmm.Solver(p.shape, p.h, dtype=DT[dt], schedule=then, stride=1.0) as s:
        s.restore(image)
        T, G = s.resume()
    compare(T.cpu().numpy(), G.cpu().numpy(), oracle.solve_reinit(_q(p.phi0, dt), p.h), dt)
