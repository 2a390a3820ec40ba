"""A stopped solve resumed with a bound below values that its bricks already
hold as KNOWN: the default look-ahead marches a brick to its end, far beyond the
bound, and the resumed schedule starts at the smallest work plus its stride.
Cells above the new bound that fall again must reach their neighbours."""
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


@pytest.fixture(scope="module")
def problem(oracle):
    shape = (48, 41, 56)
    h = wl.spacing(shape)
    rng = np.random.default_rng(17)
    F = wl.fourier_speed(shape, wl.draw_fourier_modes(rng), h=h)
    src = wl.random_cells(rng, shape, 12)
    refs = {dt: oracle.solve_sources(shape, src, h, speed=_q(F, dt)) for dt in DT}
    return shape, h, F, src, refs


THEN = [dict(schedule=2, stride=0.5), dict(schedule=2, stride=3.0), dict(schedule=3, stride=0.5, ahead=0.5),
        dict(schedule=3, stride=2.0, ahead=1.5)]


@pytest.mark.parametrize("dt", ["f64", "f32"])
@pytest.mark.parametrize("stop", [1, 2, 4, 7])
@pytest.mark.parametrize("then", THEN, ids=lambda t: "-".join(f"{v}" for v in t.values()))
def test_resume_below_known_values(fmm, problem, dt, stop, then):
    shape, h, F, src, refs = problem
    speed = torch.as_tensor(F, dtype=DT[dt], device="cuda")
    kw = dict(dtype=DT[dt], speed=speed, sources=src)
    with fmm.Solver(shape, h, schedule=3, stride=1.0, max_restarts=stop, **kw) as s:
        with pytest.raises(fmm.FmmError) as e:
            s.solve()
        assert e.value.code == fmm.FMM_ERR_TIMEOUT
        image = s.checkpoint()
    with fmm.Solver(shape, h, **then, **kw) as s:
        s.restore(image)
        T, G = s.resume()
        assert s.stats()["error_flags"] == 0
    compare(T.cpu().numpy(), G.cpu().numpy(), refs[dt], dt)
