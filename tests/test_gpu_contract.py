"""The zeta contractions against the FP64 product of the same multipoles: the plain-FP32
form at the edges of its tiles (32 columns), runs (256 primaries) and row splits, the
tensor-core form at the edges of its k-blocks (64 primaries), accumulation runs (2048) and
of the work items' parts.

Tolerances, entry by entry.  FP32: a run of at most 256 terms, each rounded in the weight
product and in the addition, is within 258 * 2^-24 of sum |w a a'|; the sums of runs
add nothing at that level.  Split BF16: hi + lo leaves 2^-18 of either factor and the
dropped lo lo' another 2^-18; an accumulation run has 3 x 128 MMA steps (K = 16), each
truncating the sum by at most 2^-22.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1709_00086_gb300 as g3  # noqa: E402
from paper_1709_00086_gb300 import catalogs  # noqa: E402

from gpu_util import to_dev  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nbins,lmax", [(1, 0), (3, 2), (16, 1), (11, 2), (32, 0)])
@pytest.mark.parametrize("n", [1, 9, 255, 257, 1025, 2500])
def test_fp32_contraction_edges(nbins, lmax, n):
    cat = catalogs.small_case("uniform", n, seed=n + nbins, box=100.0, nbins=nbins, rmin=0.0, rmax=25.0, lmax=lmax)
    cat.w[::7] *= -1  # weights of either sign
    pos, w = to_dev(cat, torch)
    plan = g3.Plan(**cat.params())
    z, _ = plan.compute(pos, w, fp32_contraction=True, keep_alm=True)
    got = g3.zeta_blocks(z, nbins, lmax)
    a = plan.alm(np.arange(n))  # (n, nbins, nlm), the FP32 rows widened
    wd = cat.w.astype(np.float64)
    for m in range(lmax + 1):
        idx = [l * (l + 1) // 2 + m for l in range(m, lmax + 1)]
        v = a[:, :, idx].transpose(0, 2, 1).reshape(n, -1)  # column (l - m) nbins + b
        want = (wd[:, None] * v).T @ v.conj()
        mag = np.abs(v.real) + np.abs(v.imag)
        bound = 258 * 2.0**-24 * ((np.abs(wd)[:, None] * mag).T @ mag)
        assert np.all(np.abs(got[m] - want) <= bound), m


@pytest.mark.parametrize("sign", [False, True])
@pytest.mark.parametrize("nbins,lmax", [(1, 0), (9, 3), (16, 4)])
@pytest.mark.parametrize("n", [64, 65, 2048, 2049, 4097, 8192, 12353])
def test_tc_contraction_edges(n, nbins, lmax, sign):
    cat = catalogs.small_case("uniform", n, seed=n + nbins, box=100.0, nbins=nbins, rmin=0.0, rmax=9.0, lmax=lmax)
    if sign:
        cat.w[::7] *= -1
    pos, w = to_dev(cat, torch)
    plan = g3.Plan(**cat.params())
    z, _ = plan.compute(pos, w, keep_alm=True)
    got = g3.zeta_blocks(z, nbins, lmax)
    a = plan.alm(np.arange(n))
    wd = cat.w.astype(np.float64)
    for m in range(lmax + 1):
        idx = [l * (l + 1) // 2 + m for l in range(m, lmax + 1)]
        v = a[:, :, idx].transpose(0, 2, 1).reshape(n, -1)
        want = (wd[:, None] * v).T @ v.conj()
        mag = np.abs(v.real) + np.abs(v.imag)
        bound = (3 * 2.0**-18 + 3 * 128 * 2.0**-22) * ((np.abs(wd)[:, None] * mag).T @ mag)
        assert np.all(np.abs(got[m] - want) <= bound), m
