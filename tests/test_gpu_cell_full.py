"""The cell-parallel march with every brick active at once: more active bricks
per block than it has warps, and as few blocks as bricks."""
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


@pytest.mark.parametrize("dt", ["f64", "f32"])
@pytest.mark.parametrize("bucket", [4.0, math.inf])
@pytest.mark.parametrize("shape", [(9, 8, 24), (40, 47, 41), (113, 118, 120)])
def test_a_source_in_every_brick(fmm, oracle, dt, bucket, shape):
    h = 1.0 / max(shape)
    rng = np.random.default_rng(2)
    src = np.array([[min(i + rng.integers(0, 8), shape[2] - 1), min(j + rng.integers(0, 8), shape[1] - 1),
                     min(k + rng.integers(0, 8), shape[0] - 1)]
                    for k in range(0, shape[0], 8) for j in range(0, shape[1], 8) for i in range(0, shape[2], 8)],
                   np.int64)
    ref = oracle.solve_sources(shape, src, h)
    with fmm.Solver(shape, h, dtype=DT[dt], sources=src, schedule=4, bucket=bucket) as s:
        T, G = s.solve()
    compare(T.cpu().numpy(), G.cpu().numpy(), ref, dt)
