"""The two list formats of the pair stage: direction records (plain forwards) and list
entries (a list budget too small for records).  Both form the same FP32 values in the
same order, so zeta is equal bit for bit; the counts match the FP64 oracle exactly
(integers) also where the bins are so narrow, or the points so close, that the FP32 bin
of a pair is never certain.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1709_00086_gb300 as g3  # noqa: E402
from paper_1709_00086_gb300 import catalogs  # noqa: E402

from gpu_util import oracle_zeta, to_dev  # noqa: E402

pytestmark = pytest.mark.gpu


def _case(los, f64, nbins, lmax, box, rmin, rmax, n=2000, near=False):
    cat = catalogs.small_case("clustered", n, seed=7 * nbins + lmax + los, box=box, nbins=nbins, rmin=rmin,
                              rmax=rmax, lmax=lmax, los_mode=los, dtype=np.float64 if f64 else np.float32)
    if near:  # coincident points, points a rounding apart, points at the box faces
        cat.pos[:40] = cat.pos[40:80]
        cat.pos[80:120] = np.nextafter(cat.pos[120:160], cat.pos.dtype.type(0))
        cat.pos[160:200, 0] = 0
        cat.pos[200:240, 1] = np.nextafter(cat.pos.dtype.type(box), cat.pos.dtype.type(0))
    return cat


@pytest.mark.parametrize("los,f64,nbins,lmax,box,rmin,rmax", [
    (0, False, 10, 10, 333.3, 0.0, 60.0),   # a side that FP32 does not hold
    (0, True, 7, 5, 333.3, 0.0, 60.0),      # FP64 positions, images across the faces
    (1, False, 32, 4, 300.0, 0.0, 80.0),    # five bits of bin
    (1, True, 1, 0, 300.0, 5.0, 80.0),
    (2, False, 17, 6, 300.0, 0.0, 80.0),    # rotated directions
    (2, True, 4, 9, 300.0, 12.5, 80.0),
    (0, False, 8, 3, 1000.0, 50.0, 50.01),  # widths near the FP32 spacing of r
    (0, True, 32, 2, 5000.0, 40.0, 40.5),
])
def test_records_and_entries_are_bit_identical(los, f64, nbins, lmax, box, rmin, rmax):
    cat = _case(los, f64, nbins, lmax, box, rmin, rmax, near=True)
    pos, w = to_dev(cat, torch)
    out = []
    for budget in (0, 1 << 20):
        plan = g3.Plan(**cat.params())
        plan.set_option(g3.OPT_LIST_BYTES, budget)
        z, c = plan.compute(pos, w, fp32_contraction=True)
        out.append((z.cpu().numpy(), c.cpu().numpy(), plan.stats()["list_passes"]))
    assert out[0][2] == 1 and out[1][2] > 1
    _, co = oracle_zeta(cat)
    np.testing.assert_array_equal(out[0][1], co)
    np.testing.assert_array_equal(out[1][1], co)
    np.testing.assert_array_equal(out[0][0], out[1][0])


@pytest.mark.parametrize("n", [1, 2, 32, 33, 65, 257])
def test_partly_filled_chunks(n):
    # every pair in one bin: the last chunk of the bin holds n - 1 pairs modulo 32
    cat = _case(1, False, 1, 4, 100.0, 0.0, 200.0, n=n)
    pos, w = to_dev(cat, torch)
    plan = g3.Plan(**cat.params())
    z, c = plan.compute(pos, w, fp32_contraction=True)
    zo, co = oracle_zeta(cat)
    np.testing.assert_array_equal(c.cpu().numpy(), co)
    # a_lm: FP32 sums of at most 256 terms, each within 2^-24 per operation of ~40
    assert np.abs(z.cpu().numpy() - zo).max() <= 1e-5 * max(np.abs(zo).max(), 1e-300)


@pytest.mark.parametrize("cells", [1, 2, 4])
@pytest.mark.parametrize("los,f64,nbins,lmax,n", [
    (0, False, 10, 4, 2000), (1, True, 32, 3, 1999), (2, False, 7, 5, 2017), (1, False, 1, 2, 33), (2, True, 5, 1, 1),
])
def test_cell_resolutions(cells, los, f64, nbins, lmax, n):
    # about 0.9, 1.9 and 3.9 cells per rmax: the scan places accepted pairs in groups of
    # 32 in the first, from the candidates' lanes in the others
    cat = _case(los, f64, nbins, lmax, 400.0, 0.0, 61.0, n=n, near=n > 240)
    pos, w = to_dev(cat, torch)
    zo, co = oracle_zeta(cat)
    out = []
    for budget in (0, 1 << 20):
        plan = g3.Plan(**cat.params())
        plan.set_option(g3.OPT_CELLS_PER_RMAX, cells)
        plan.set_option(g3.OPT_LIST_BYTES, budget)
        z, c = plan.compute(pos, w, fp32_contraction=True)
        np.testing.assert_array_equal(c.cpu().numpy(), co)
        out.append(z.cpu().numpy())
    np.testing.assert_array_equal(out[0], out[1])
    # FP64 points that FP32 cannot tell apart have no FP32 direction: their bins are NaN
    # here as in the fused kernel, which shares none of this path
    plan = g3.Plan(**cat.params())
    plan.set_option(g3.OPT_PAIR_KERNELS, 1)
    bad = np.isnan(plan.compute(pos, w, fp32_contraction=True)[0].cpu().numpy())
    assert f64 or not bad.any()
    np.testing.assert_array_equal(np.isnan(out[0]), bad)
    # a_lm: at most 2000 / 32 partial sums per lane, ~45 more operations: (63 + 45) 2^-24
    # of sum |w| K_lm; a product of two, K_lm^2 <= (2 lmax + 1) K_00^2
    assert np.abs(np.where(bad, 0, out[0] - zo)).max() <= 1.3e-5 * (2 * lmax + 1) * max(np.abs(zo).max(), 1e-300)
