"""Double-float multipoles where every pair of a primary has the same direction, so that
the sums of a chunk (x axis, orders m >= 1) or of a lane (z axis, m = 0) reach their
largest size, with either sign.

Tolerance: the sums are good to 2^-36 of the largest weight (1,000 terms), which is 2^-40 of
a sum (at least 28 weights); the connection coefficients amplify that by at most 2^7
against an entry (the ratio of the Gegenbauer polynomials at 1 and 0), 2^-33, which is
less than 1/64 of the entry's FP32 ulp; storing it adds half an ulp.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1709_00086_gb300 as g3  # noqa: E402
from paper_1709_00086_gb300 import catalogs  # noqa: E402

from gpu_util import oracle_alm, to_dev  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lmax", [1, 4, 7, 8, 9, 10])
@pytest.mark.parametrize("axis,sign", [(0, -1), (0, 1), (2, -1), (2, 1)])
def test_pairs_in_one_direction(lmax, axis, sign):
    n = 960  # 30 chunks of 32
    for seed in range(4):
        rng = np.random.default_rng(100 * lmax + seed)
        pos = np.full((n + 1, 3), 64.0, np.float32)
        # exact separations from 2 to 62, in the order of the cells
        pos[1:, axis] += sign * (2.0 + np.arange(n) / 16.0)[::sign].astype(np.float32)
        w = rng.uniform(0.9, 1.0, n + 1).astype(np.float32)
        if axis == 2:  # one lane's pairs alone
            w[1:][np.arange(n) % 32 != 5] = 0.0
        cat = catalogs.Catalog(pos, w, 128.0, 1, 0.0, 63.0, lmax, 1)
        dpos, dwt = to_dev(cat, torch)
        plan = g3.Plan(**cat.params())
        plan.compute(dpos, dwt, n_primary=1, keep_alm=True)
        a, ao = plan.alm(np.array([0])), oracle_alm(cat, np.array([0]))
        for got, ref in ((a.real, ao.real), (a.imag, ao.imag)):
            big = np.abs(ref) > 2.0 ** -4 * np.abs(ao).max()
            ulp = np.spacing(np.abs(ref[big]).astype(np.float32)).astype(np.float64)
            assert (np.abs(got - ref)[big] <= (0.5 + 1 / 64) * ulp).all(), seed
