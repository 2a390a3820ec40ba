"""A solve stopped under the phased schedule leaves its pending overlap changes
in the dirty flags, one stopped under a one-launch schedule in the work words:
each resumes under the other."""
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


@pytest.mark.parametrize("dt", ["f64", "f32"])
@pytest.mark.parametrize("stop", [1, 3, 6])
@pytest.mark.parametrize("first,then", [(dict(schedule=1), dict(schedule=2)), (dict(schedule=1), dict(schedule=3)),
                                        (dict(schedule=2), dict(schedule=1)), (dict(schedule=3), dict(schedule=1)),
                                        (dict(schedule=3), dict(deterministic=True)),
                                        (dict(deterministic=True), dict(schedule=3))],
                         ids=["1-2", "1-3", "2-1", "3-1", "3-det", "det-3"])
def test_phased_and_one_launch_images(fmm, oracle, dt, stop, first, then):
    shape = (33, 40, 29)
    h = wl.spacing(shape)
    rng = np.random.default_rng(23)
    F = wl.fourier_speed(shape, wl.draw_fourier_modes(rng), h=h)
    src = wl.random_cells(rng, shape, 5)
    Fq = np.asarray(F, np.float32).astype(np.float64) if dt == "f32" else np.asarray(F, np.float64)
    kw = dict(dtype=DT[dt], speed=torch.as_tensor(F, dtype=DT[dt], device="cuda"), sources=src, stride=1.0,
              exchange_passes=1)
    with fmm.Solver(shape, h, max_restarts=stop, **first, **kw) as s:
        with pytest.raises(fmm.FmmError) as e:
            s.solve()
        assert e.value.code == fmm.FMM_ERR_TIMEOUT
        image = s.checkpoint()
    with fmm.Solver(shape, h, timeout_s=5, **then, **kw) as s:
        s.restore(image)
        T, G = s.resume()
        assert s.stats()["error_flags"] == 0
    compare(T.cpu().numpy(), G.cpu().numpy(), oracle.solve_sources(shape, src, h, speed=Fq), dt)
