"""A captured forward whose pair lists have another chunk size than those the plan sized
its pool for (direction records, 512 bytes a chunk; list entries, 128): it must run the
kernels of the uncaptured call, so rows and zeta are equal bit for bit.
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


@pytest.mark.parametrize("keep_alm,options", [
    (True, []),                               # double-float multipoles
    (True, [(g3.OPT_GRAD_PRECISION, 1)]),     # FP32 multipoles of the exact images
    (False, [(g3.OPT_BASIS, 1)]),             # monomial basis
    (False, [(g3.OPT_LIST_BYTES, 1 << 20)]),  # entries, several passes
])
def test_graph_after_a_plain_forward(keep_alm, options):
    cat = catalogs.small_case("clustered", 3000, seed=3, box=300.0, nbins=6, rmin=0.0, rmax=60.0, lmax=6)
    pos, w = to_dev(cat, torch)
    out = []
    for graph in (False, True):
        plan = g3.Plan(**cat.params())
        if graph:
            plan.compute(pos, w)  # sizes the pool for records
        for opt, value in options:
            plan.set_option(opt, value)
        zr = torch.empty((plan.zsize, 2), dtype=torch.float64, device="cuda")
        cr = torch.empty(cat.nbins, dtype=torch.int64, device="cuda")
        for _ in range(2 if graph else 1):  # capture, replay
            plan.compute(pos, w, keep_alm=keep_alm, graph=graph, out=zr, counts_out=cr)
        out.append((zr.cpu().numpy(), cr.cpu().numpy(), plan.alm(np.arange(0, cat.w.size, 37))))
    for ref, got in zip(*out):
        np.testing.assert_array_equal(got, ref)


@pytest.mark.parametrize("keep_alm,opt", [(False, g3.OPT_BASIS), (True, g3.OPT_GRAD_PRECISION)])
def test_graph_follows_a_changed_option(keep_alm, opt):
    # the same call after the option has changed is a new capture, not a replay of the old one
    cat = catalogs.small_case("clustered", 2000, seed=4, box=300.0, nbins=5, rmin=0.0, rmax=60.0, lmax=5)
    pos, w = to_dev(cat, torch)
    prims = np.arange(0, cat.w.size, 37)
    ref = g3.Plan(**cat.params())
    ref.set_option(opt, 1)
    ref.compute(pos, w, keep_alm=keep_alm)
    plan = g3.Plan(**cat.params())
    zr = torch.empty((plan.zsize, 2), dtype=torch.float64, device="cuda")
    cr = torch.empty(cat.nbins, dtype=torch.int64, device="cuda")
    for value in (0, 0, 1, 1):
        plan.set_option(opt, value)
        plan.compute(pos, w, keep_alm=keep_alm, graph=True, out=zr, counts_out=cr)
    np.testing.assert_array_equal(plan.alm(prims), ref.alm(prims))
