"""Pairs so close that FP32 positions leave nothing of their separation (FP64 points a few
FP64 ulps apart, also across a box face; FP32 points whose squared separation is below
FP32's range): every kernel takes their direction from the input positions, like the FP64
oracle.  The points are pairs on a grid, alone in the first bin of their partner, so that
bin 0 of a row is one direction.

Tolerance: bin 0 of a row has one term; its FP32 harmonics take at most 45 operations of
2^-24 at lmax = 4, amplified by at most 3 in the Chebyshev form: 1e-5 of the row's largest
entry.  Double-float rows are rounded once to FP32: 1e-7.  Gradients: 1e-6 in double-float
(as everywhere), 1e-5 in FP32.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import oracle  # noqa: E402
import paper_1709_00086_gb300 as g3  # noqa: E402
from paper_1709_00086_gb300 import catalogs  # noqa: E402

from gpu_util import maxrel, oracle_alm, to_dev  # noqa: E402

pytestmark = pytest.mark.gpu
LMAX = 4
KERNELS = {
    "records": (1e-5, False, []),
    "entries": (1e-5, False, [(g3.OPT_LIST_BYTES, 1 << 20)]),
    "fused": (1e-5, False, [(g3.OPT_PAIR_KERNELS, 1)]),
    "monomials": (1e-5, False, [(g3.OPT_BASIS, 1)]),
    "df": (1e-7, True, []),
    "fp32 exact images": (1e-5, True, [(g3.OPT_GRAD_PRECISION, 1)]),
}


def _catalog(los, f64, seed):
    rng = np.random.default_rng(seed)
    box = 300.0
    grid = 20.0 + 35.0 * np.stack(np.meshgrid(*[np.arange(8.0)] * 3, indexing="ij"), axis=-1).reshape(-1, 3)
    a = grid[rng.permutation(512)[:200]] + rng.uniform(-8.0, 8.0, (200, 3))
    if f64:
        step = rng.normal(size=a.shape) * 10.0 ** rng.uniform(-13.0, -5.0, (200, 1))
        b = a + step
        b[:40] = a[:40]
        b[:40, 1] = np.nextafter(a[:40, 1], 0.0)          # one FP64 ulp
        b[(a == b).all(axis=1), 0] += 1e-10
        if los == 0:                                       # across a face, both FP32 box
            a[40:50, 0] = 1e-13 * np.arange(1, 11)
            b[40:50] = a[40:50]
            b[40:50, 0] = box - 1e-12
            b[40:50, 2] += 1e-12
        dtype = np.float64
    else:                                                  # near the corner, r^2 of 1e-44 and less
        a, b = a.astype(np.float32), (a + 0.5).astype(np.float32)
        a[0] = (1e-22, 3e-23, 2e-22)
        b[0] = (3e-22, 1e-23, 5e-23)
        dtype = np.float32
    pos = np.concatenate([a, b]).astype(dtype)
    order = rng.permutation(400)
    w = rng.uniform(0.5, 1.5, 400).astype(np.float32)
    return catalogs.Catalog(np.ascontiguousarray(pos[order]), w, box, 30, 0.0, 60.0, LMAX, los)


@pytest.mark.parametrize("los,f64", [(0, True), (1, True), (2, True), (1, False), (2, False)])
@pytest.mark.parametrize("kernel", list(KERNELS))
@pytest.mark.parametrize("cells", [1, 3])
def test_directions_of_close_pairs(los, f64, kernel, cells):
    tol, keep, options = KERNELS[kernel]
    cat = _catalog(los, f64, 5)
    plan = g3.Plan(**cat.params())
    plan.set_option(g3.OPT_CELLS_PER_RMAX, cells)
    for o, v in options:
        plan.set_option(o, v)
    plan.compute(*to_dev(cat, torch), keep_alm=keep)
    prims = np.arange(cat.n)
    got, ref = plan.alm(prims)[:, 0], oracle_alm(cat, prims)[:, 0]
    assert np.isfinite(got).all()
    top = np.abs(ref).max(axis=1)
    assert (top > 0).sum() >= (390 if f64 else 2)
    assert (np.abs(got - ref).max(axis=1) <= tol * top).all()


@pytest.mark.parametrize("los", [0, 1])
@pytest.mark.parametrize("tol,options", [
    (1e-6, []), (1e-5, [(g3.OPT_GRAD_PRECISION, 1)]), (1e-5, [(g3.OPT_PAIR_KERNELS, 1)]),
])
def test_gradients_of_close_pairs(los, tol, options):
    cat = _catalog(los, True, 6)
    plan = g3.Plan(**cat.params())
    for o, v in options:
        plan.set_option(o, v)
    plan.compute(*to_dev(cat, torch), keep_alm=True)
    rng = np.random.default_rng(7)
    G = rng.normal(size=plan.zsize) + 1j * rng.normal(size=plan.zsize)
    G = np.concatenate([(b + b.conj().T).ravel() for b in oracle.zeta_blocks(G, cat.nbins, cat.lmax)])
    dpos, dw = plan.backward(torch.from_numpy(np.stack([2 * G.real, 2 * G.imag], axis=1)).cuda())
    rpos, rw = oracle.grad(cat.pos, cat.w.astype(np.float64), G, cat.box, cat.nbins, cat.rmin, cat.rmax, cat.lmax,
                           los_mode=los)
    dpos, dw = dpos.cpu().numpy(), dw.cpu().numpy()
    assert maxrel(dw, rw) < tol
    # 1 / r spans eight decades: every point against its own size
    size = np.abs(rpos).max(axis=1)
    assert (np.abs(dpos - rpos).max(axis=1) <= 10 * tol * size + tol * np.median(size)).all()
