"""The one-launch schedules where most bricks wait for the bound at once: few
CTAs (a scan takes many ring entries per warp), strides far below a cell,
interface values many strides apart, and a batch of grids whose cell sizes
differ by orders of magnitude.  All against the oracle."""
import math

import numpy as np
import pytest
import torch

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


def _layers(shape, h):
    """A level set whose zero set passes through nearly every brick, at a
    distance from the brick's cells that varies from brick to brick."""
    z, y, x = np.indices(shape) * h
    return np.sin(0.37 / h * x + 2.0 * y) * np.cos(0.31 / h * y + z) + 0.7 * np.sin(0.29 / h * z + 1.3 * x) + 0.11


@pytest.fixture(scope="module")
def layers(oracle):
    shape, h = (61, 64, 59), 1.0 / 64
    phi = _layers(shape, h)
    return shape, h, phi, {dt: oracle.solve_reinit(_q(phi, dt), h) for dt in DT}


@pytest.mark.parametrize("dt", ["f64", "f32"])
@pytest.mark.parametrize("schedule", [2, 3])
@pytest.mark.parametrize("ctas", [0, 1, 3, 8])
def test_interface_in_most_bricks(fmm, layers, dt, schedule, ctas):
    shape, h, phi, ref = layers
    with fmm.Solver(shape, h, dtype=DT[dt], schedule=schedule, ctas=ctas, stride=0.05) as s:
        T, G = s.reinit(_dev(phi, dt))
        assert s.stats()["error_flags"] == 0
    compare(T.cpu().numpy(), G.cpu().numpy(), ref[dt], dt)


@pytest.mark.parametrize("ahead", [0.0, 0.4])
@pytest.mark.parametrize("stride", [0.3, 40.0, math.inf])
@pytest.mark.parametrize("ctas", [0, 1, 3])
def test_given_values_many_strides_apart(fmm, oracle, ctas, stride, ahead):
    """One FIX cell in every brick, values up to 100 h apart: every brick but
    the first few waits, and a wide stride releases all of them together."""
    shape, h = (64, 56, 61), 1.0 / 64
    rng = np.random.default_rng(11)
    T0 = np.full(shape, np.inf)
    for k in range(0, shape[0], 8):
        for j in range(0, shape[1], 8):
            for i in range(0, shape[2], 8):
                T0[k + rng.integers(0, min(8, shape[0] - k)), j + rng.integers(0, 8),
                   i + rng.integers(0, min(8, shape[2] - i))] = rng.uniform(0.0, 100.0) * h
    ref = oracle.march(T0, np.where(np.isfinite(T0), oracle.KNOWN_FIX, oracle.FAR).astype(np.uint8), h)
    with fmm.Solver(shape, h, dtype=torch.float64, ctas=ctas, stride=stride, ahead=ahead) as s:
        T, G = s.solve_fixed(_dev(T0, "f64"))
        assert s.stats()["error_flags"] == 0
    compare(T.cpu().numpy(), G.cpu().numpy(), ref, "f64")


@pytest.mark.parametrize("ctas", [0, 1])
def test_batch_of_very_different_cell_sizes(fmm, oracle, ctas):
    """The stride is in units of the smallest cell size: with one fine grid
    the bricks of all others wait."""
    shape = (16, 16, 16)
    hs = [1.0 / 16] * 60 + [1.0 / 500]
    phis = []
    for g, h in enumerate(hs):
        z, y, x = np.indices(shape)
        phis.append((np.sin(0.8 * x + 0.1 * g) + np.cos(0.7 * y) + np.sin(0.6 * z + 0.2 * g) + 0.13) * h)
    with fmm.Batch([shape] * len(hs), hs, dtype=torch.float64, ctas=ctas, stride=0.5) as b:
        Ts, Gs = b.reinit([_dev(p, "f64") for p in phis])
    for p, h, T, G in zip(phis, hs, Ts, Gs):
        compare(T.cpu().numpy(), G.cpu().numpy(), oracle.solve_reinit(p, h), "f64")
