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
