"""The spatial index at the edges of its radix tiles (1,024 keys, 4,096 above 2^18 points)
and of the primaries' compaction, and the list planning of chunked, many-pass and batched
forwards: pair counts against the FP64 oracle (integers, exact)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1709_00086_gb300 as g3  # noqa: E402
from paper_1709_00086_gb300 import catalogs  # noqa: E402

from gpu_util import oracle_zeta, to_dev  # noqa: E402

pytestmark = pytest.mark.gpu


def _counts(cat, n_primary=None, **opts):
    pos, w = to_dev(cat, torch)
    plan = g3.Plan(**cat.params())
    for k, v in opts.items():
        plan.set_option(getattr(g3, k), v)
    _, c = plan.compute(pos, w, n_primary=n_primary, fp32_contraction=True)
    return c.cpu().numpy()


# nc = 1 (one digit of keys), 10 and 200 cells per side (two and three digits)
@pytest.mark.parametrize("n", [1, 1023, 1024, 1025, 3000])
@pytest.mark.parametrize("box,rmax,f64", [(30.0, 20.0, True), (400.0, 40.0, False), (8000.0, 40.0, True)])
def test_counts_at_tile_edges(n, box, rmax, f64):
    cat = catalogs.small_case("uniform", n, seed=n, box=box, nbins=3, rmin=0.0, rmax=rmax, lmax=1, los_mode=1,
                              dtype=np.float64 if f64 else np.float32)
    for n_primary in {n, (n + 1) // 2, min(n, 1024), 0}:
        _, co = oracle_zeta(cat, n_primary=n_primary)
        np.testing.assert_array_equal(_counts(cat, n_primary), co)


@pytest.mark.parametrize("n", [(1 << 18) - 1, (1 << 18) + 1, (1 << 18) + 4097])
def test_counts_around_the_large_sort(n):
    cat = catalogs.small_case("uniform", n, seed=5, box=600.0, nbins=4, rmin=0.0, rmax=30.0, lmax=1)
    _, co = oracle_zeta(cat, n_primary=300)
    np.testing.assert_array_equal(_counts(cat, 300), co)


def test_chunks_and_passes_count_alike():
    # chunks of primaries, each split into passes by a 1 MiB list budget
    cat = catalogs.small_case("clustered", 9000, seed=6, box=300.0, nbins=5, rmin=0.0, rmax=60.0, lmax=2)
    _, co = oracle_zeta(cat)
    np.testing.assert_array_equal(_counts(cat, OPT_CHUNK_ROWS=1024), co)
    np.testing.assert_array_equal(_counts(cat, OPT_CHUNK_ROWS=4096, OPT_LIST_BYTES=1 << 20), co)


def test_batch_counts_with_empty_catalogs():
    cats = catalogs.batched(ncat=6, seed=8, sizes=[0, 1025, 3, 0, 2100, 0], box=400.0)
    plan = g3.Plan(**cats[0].params())
    pos = torch.from_numpy(np.concatenate([c.pos for c in cats])).cuda()
    w = torch.from_numpy(np.concatenate([c.w for c in cats])).cuda()
    _, c = plan.compute_batch(pos, w, np.cumsum([0] + [x.n for x in cats]))
    for k, cat in enumerate(cats):
        _, co = oracle_zeta(cat)
        np.testing.assert_array_equal(c[k].cpu().numpy(), co)
