"""The per-brick passes of a batch where they can go wrong: grids of one cell,
of one brick exactly, and ending inside a brick in the lower and the upper
half of its layers (a thread holds cells z and z + 4), side by side."""
import numpy as np
import pytest
import torch

from parity_util import compare

pytestmark = pytest.mark.gpu

DT = {"f32": torch.float32, "f64": torch.float64}
SHAPES = [(2, 2, 2), (8, 8, 8), (3, 9, 8), (4, 7, 17), (12, 8, 9), (13, 16, 15), (5, 1, 20)]


@pytest.mark.parametrize("dt", ["f32", "f64"])
def test_ragged_grids(oracle, dt):
    from paper_1502_07303_gb300 import fmm
    phis, hs = [], []
    for n, shape in enumerate(SHAPES):
        h = 1.0 / max(shape)
        z, y, x = np.indices(shape)
        phi = (x + 0.3 * y + 0.2 * z - 0.45 * max(shape) + 0.01 * n + 0.003) * h
        phis.append(phi.astype(np.float32).astype(np.float64) if dt == "f32" else phi)
        hs.append(h)
    with fmm.Batch(SHAPES, hs, dtype=DT[dt]) as b:
        Ts, Gs = b.reinit([torch.as_tensor(p, dtype=DT[dt], device="cuda") for p in phis])
    for phi, h, T, G in zip(phis, hs, Ts, Gs):
        compare(T.cpu().numpy(), G.cpu().numpy(), oracle.solve_reinit(phi, h), dt)
