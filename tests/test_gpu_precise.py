"""Double-float multipoles (G3PCF_F_KEEP_ALM) at every order, for few and many pairs per
bin and for weights of very different size, against the FP64 oracle.

Tolerance: the stored row is FP32 (half an ulp, 6e-8 of an entry at most) and the
double-float sums before it are good to 2^-33 of the largest term, so every entry is
within 1e-7 of the primary's largest.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1709_00086_gb300 as g3  # noqa: E402
from paper_1709_00086_gb300 import catalogs  # noqa: E402

from gpu_util import maxrel, oracle_alm, to_dev  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lmax", range(11))
@pytest.mark.parametrize("n,nbins,los,kind", [
    (40, 3, 1, "plain"),       # chunks of a few pairs
    (3000, 2, 0, "plain"),     # about 1500 pairs per bin: more than 32 chunks
    (700, 5, 2, "spread"),     # weights over twelve decades, either sign
    (700, 5, 1, "zeros"),      # bins whose first chunk has no weight at all
])
def test_double_float_multipoles(lmax, n, nbins, los, kind):
    cat = catalogs.small_case("clustered", n, seed=lmax + n, box=100.0, nbins=nbins, rmin=0.0, rmax=49.0,
                              lmax=lmax, los_mode=los)
    rng = np.random.default_rng(lmax)
    if kind == "spread":
        cat.w[:] = rng.choice([-1.0, 1.0], n) * 10.0 ** rng.uniform(-6.0, 6.0, n)
    elif kind == "zeros":
        cat.w[:] = np.where(rng.random(n) < 0.9, 0.0, cat.w)
    pos, w = to_dev(cat, torch)
    plan = g3.Plan(**cat.params())
    plan.compute(pos, w, keep_alm=True)
    prims = np.array([0, 1, n // 2, n - 1])
    a, ao = plan.alm(prims), oracle_alm(cat, prims)
    for k in range(prims.size):
        assert maxrel(a[k], ao[k]) < 1e-7, k
