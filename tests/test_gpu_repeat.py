"""A repeated call needs no more of the device than the plan already holds."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1709_00086_gb300 as g3  # noqa: E402
from paper_1709_00086_gb300 import catalogs  # noqa: E402

from gpu_util import to_dev  # noqa: E402

pytestmark = pytest.mark.gpu


def test_repeat_keeps_the_multipoles_where_other_memory_has_gone():
    # rows of 200,000 primaries at B = lmax = 10: 0.97 GB, more than 0.4 of what is left free
    # before the second call, but held by the plan since the first
    n = 200_000
    rng = np.random.default_rng(1)
    cat = catalogs.Catalog(catalogs.uniform_positions(rng, n, 1000.0, dtype=np.float32), np.ones(n, np.float32),
                           1000.0, 10, 0.0, 12.0, 10, 0)
    pos, w = to_dev(cat, torch)
    plan = g3.Plan(**cat.params())
    out = []
    hold = None
    try:
        for _ in range(2):
            z, _ = plan.compute(pos, w, keep_alm=True)
            out.append((z.cpu().numpy(), plan.alm(np.arange(0, n, 997))))
            if hold is None:
                torch.cuda.empty_cache()
                hold = torch.empty(torch.cuda.mem_get_info()[0] - 2_200_000_000, dtype=torch.uint8, device="cuda")
    finally:
        del hold
        torch.cuda.empty_cache()
    np.testing.assert_array_equal(out[0][0], out[1][0])
    np.testing.assert_array_equal(out[0][1], out[1][1])
