"""The double-grid root of Algorithm 11 as a march without a tape computes it
(csrc/fmm_df.cuh, df_root<false>, through fmm_selftest_root_forward) against
exact arithmetic, near ties and with absent axes.

The set and a first root u0 come from float arithmetic: u0 is off by at most
about 3e-7 u (one ulp of the square root's estimate and the rounding of the
discriminant, which is at least q / 2).  The correction c = r / (2 g) is of that
size and carries a relative error of at most about 4e-7 (the reciprocal's
estimate, g, r and the products), so the root is off by 1.2e-13 u.  Where the
float test takes the other set, a shift and a root agree to about 5e-7 and the two
sets' roots differ by a quarter of its square, 6e-14 u.  Together 2e-13 u; 3e-13 u
are allowed, and one rounding of t."""
import ctypes
from decimal import Decimal

import numpy as np
import pytest
import torch

from test_gpu_root import _cases, _exact

pytestmark = pytest.mark.gpu


def _run(lib, m, v1, v2, nd, q):
    dev = lambda a, dt: torch.as_tensor(np.ascontiguousarray(a), dtype=dt, device="cuda")
    args = [dev(a, torch.float64) for a in (m, v1, v2)] + [dev(nd, torch.int32), dev(q, torch.float64)]
    t, k = torch.empty_like(args[0]), torch.empty_like(args[3])
    p = lambda x: ctypes.c_void_p(x.data_ptr())
    assert lib.fmm_selftest_root_forward(*map(p, args), p(t), p(k), len(m), None) == 0
    torch.cuda.synchronize()
    return t.cpu().numpy(), k.cpu().numpy()


@pytest.mark.parametrize("scale", [1.0, 1e-6, 1e9])
@pytest.mark.parametrize("tie", [None, 1e-9, 1e-7, 1e-6])
def test_root_without_a_tape_matches_exact_arithmetic(scale, tie):
    if not torch.cuda.is_available():
        pytest.fail("CUDA is required for the gpu tests")
    from paper_1502_07303_gb300 import fmm
    lib = fmm.load()
    m, v1, v2, nd, q = _cases(4000, seed=77)
    if tie is not None:
        # the second value at the one-value root, or the third at the two-value one
        rng = np.random.default_rng(9)
        s = np.sqrt(q)
        one = rng.random(len(m)) < 0.5
        d1 = np.where(one, s * (1 + rng.uniform(-tie, tie, len(m))), rng.uniform(0.0, 0.95, len(m)) * s)
        u2 = (d1 + np.sqrt(np.maximum(2 * q - d1 ** 2, 0.0))) / 2
        d2 = np.where(one, d1 * rng.uniform(1.0, 2.0, len(m)), u2 * (1 + rng.uniform(-tie, tie, len(m))))
        d2 = np.maximum(d1, d2)
        v1, v2 = m + d1, m + d2
    m, v1, v2, q = m * scale, v1 * scale, v2 * scale, q * scale * scale
    t, k = _run(lib, m, v1, v2, nd, q)
    worst, bad = 0.0, []
    for i in range(len(m)):
        _, te, _, u = _exact(m[i], v1[i], v2[i], int(nd[i]), q[i])
        err = abs(Decimal(float(t[i])) - te) - Decimal("1.2e-16") * te
        worst = max(worst, float(err / u))
        if err > Decimal("3e-13") * u:
            bad.append((i, int(k[i]), float(err / u)))
    print(f"worst {worst:.2e} of u")
    assert not bad, bad[:5]
