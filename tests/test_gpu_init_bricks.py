"""Interface initialisation where nearly every cell is at the interface (signs
at random): the cell list of a block is full, for one brick per block, a few,
and one per warp, whole grids and batches, and grids that end inside a brick."""
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


def _phi(shape, seed):
    rng = np.random.default_rng(seed)
    a = np.asarray(rng.uniform(0.1, 1.0, shape) * rng.choice([-1.0, 1.0], shape), np.float32).astype(np.float64)
    a.flat[0] = 0.0
    a.flat[-1] = -0.0
    return a


@pytest.mark.parametrize("dt", ["f64", "f32"])
@pytest.mark.parametrize("shape", [(2, 1, 1), (8, 8, 8), (9, 7, 8), (64, 61, 64), (88, 90, 89)])
def test_every_cell_at_the_interface(fmm, oracle, dt, shape):
    phi, h = _phi(shape, 3), 1.0 / max(shape)
    with fmm.Solver(shape, h, dtype=DT[dt]) as s:
        T, G = s.reinit(torch.as_tensor(phi, dtype=DT[dt], device="cuda"))
    compare(T.cpu().numpy(), G.cpu().numpy(), oracle.solve_reinit(phi, h), dt)


@pytest.mark.parametrize("dt", ["f64", "f32"])
@pytest.mark.parametrize("count", [3, 40])
def test_every_cell_at_the_interface_in_a_batch(fmm, oracle, dt, count):
    rng = np.random.default_rng(8)
    shapes = [tuple(int(v) for v in rng.integers(2, 34, 3)) for _ in range(count)]
    hs = [1.0 / max(s) for s in shapes]
    phis = [_phi(s, n) for n, s in enumerate(shapes)]
    with fmm.Batch(shapes, hs, dtype=DT[dt]) as b:
        Ts, Gs = b.reinit([torch.as_tensor(p, dtype=DT[dt], device="cuda") for p in phis])
    for p, h, T, G in zip(phis, hs, Ts, Gs):
        compare(T.cpu().numpy(), G.cpu().numpy(), oracle.solve_reinit(p, h), dt)
