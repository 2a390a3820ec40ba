"""Bricks that march again because the bound rose, with a speed field in
double: only the cells next to a newly usable one (or a halo value) are solved,
and the result is the oracle's."""
import numpy as np
import pytest
import torch

from paper_1502_07303_gb300 import workloads as wl
from parity_util import compare

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fmm():
    if not torch.cuda.is_available():
        pytest.fail("CUDA is required for the gpu tests")
    from paper_1502_07303_gb300 import fmm as _fmm
    return _fmm


@pytest.mark.parametrize("prm", [dict(schedule=2), dict(schedule=1, exchange_passes=1), dict(schedule=3, ahead=0.5),
                                 dict(deterministic=True)], ids=["queue", "phased", "ahead", "deterministic"])
@pytest.mark.parametrize("tape", [False, True])
@pytest.mark.parametrize("spacing", [(1.0, 1.0), (1.4, 0.7)])
@pytest.mark.parametrize("stride", [0.5, 3.0])
def test_reopened_bricks(fmm, oracle, prm, tape, spacing, stride):
    shape = (35, 40, 30)
    h = wl.spacing(shape)
    h3 = (h, h * spacing[0], h * spacing[1])
    rng = np.random.default_rng(31)
    F = wl.fourier_speed(shape, wl.draw_fourier_modes(rng), h=h)
    src = wl.random_cells(rng, shape, 5)
    ref = oracle.solve_sources(shape, src, h3, speed=F)
    with fmm.Solver(shape, h3, dtype=torch.float64, speed=torch.as_tensor(F, dtype=torch.float64, device="cuda"),
                    sources=src, stride=stride, record_tape=tape, **prm) as s:
        T, G = s.solve()
        st = s.stats()
    compare(T.cpu().numpy(), G.cpu().numpy(), ref, "f64")
    if prm.get("schedule") == 2 and stride == 0.5:
        # a sweep solves all 512 cells of a brick
        assert st["cell_solves"] < 200 * st["brick_marches"]


@pytest.mark.parametrize("shape", [(1, 8, 9), (17, 1, 16), (16, 15, 17), (35, 40, 30), (64, 57, 66)])
@pytest.mark.parametrize("tape", [False, True])
@pytest.mark.parametrize("sources", [1, 12])
def test_first_march_from_a_list(fmm, oracle, shape, tape, sources):
    """Unequal cells and a speed field in double, default schedule: a brick's
    first march starts from the cells next to BAND cells and halo values."""
    h = 1.0 / max(shape)
    h3 = (h, 1.4 * h, 0.7 * h)
    rng = np.random.default_rng(5)
    F = wl.fourier_speed(shape, wl.draw_fourier_modes(rng), h=h)
    src = wl.random_cells(rng, shape, min(sources, int(np.prod(shape))))
    ref = oracle.solve_sources(shape, src, h3, speed=F)
    with fmm.Solver(shape, h3, dtype=torch.float64, speed=torch.as_tensor(F, dtype=torch.float64, device="cuda"),
                    sources=src, record_tape=tape) as s:
        T, G = s.solve()
    compare(T.cpu().numpy(), G.cpu().numpy(), ref, "f64")


@pytest.mark.parametrize("width_cells", [4.0, np.inf])
def test_level_set_with_speed_and_unequal_cells(fmm, oracle, width_cells):
    p = wl.random_spheres(shape=(41, 50, 37), count=5, seed=12)
    h3 = (p.h, 1.25 * p.h, 0.8 * p.h)
    F = wl.fourier_speed(p.shape, wl.draw_fourier_modes(np.random.default_rng(6)), h=p.h)
    w = width_cells * p.h
    ref = oracle.solve_reinit(p.phi0, h3, speed=F, width=w)
    with fmm.Solver(p.shape, h3, dtype=torch.float64, speed=torch.as_tensor(F, dtype=torch.float64, device="cuda"),
                    width=w) as s:
        T, G = s.reinit(torch.as_tensor(p.phi0, dtype=torch.float64, device="cuda"))
    compare(T.cpu().numpy(), G.cpu().numpy(), ref, "f64", width=w)
