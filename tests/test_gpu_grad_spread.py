"""The primary-weight term of the gradient, dL/dw_i = Re(A_i^H M A_i), where the rows of
multipoles A_i that share a block of the adjoint's matrix product, or the bins of one row,
differ by twelve decades.  Every point that is not a primary lies near one primary, and no
primary lies near another, so that this term is all of dL/dw of a primary; the reference
forms it in FP64 from the rows that the library stores.

Tolerance: with S_c the sum over the bins of sum |M_c| times the row's largest |A| there,
an entry V_c = (M A)_c of W terms is a double-float sum under a head of at most 4 S_c: its
tail gathers W residues of at most 2^-22 S_c (sqrt(W) 2^-24 as a random walk), and each of
its 2 W roundings is 2^-24 of that: below 2^-38 S_c for W <= 220; the row's sum of A_c V_c
adds nothing of that size.  2^-36 of sum |A_c| S_c.
"""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import oracle  # noqa: E402
import paper_1709_00086_gb300 as g3  # noqa: E402
from paper_1709_00086_gb300 import catalogs  # noqa: E402

from gpu_util import to_dev  # noqa: E402

pytestmark = pytest.mark.gpu


def _catalog(kind, nbins, lmax, rng):
    """64 primaries, then 24 secondaries of each; rmax 30, the primaries 70 apart."""
    p = 30.0 + 70.0 * np.stack(np.meshgrid(*[np.arange(4.0)] * 3, indexing="ij"), axis=-1).reshape(-1, 3)
    d = rng.normal(size=(64, 24, 3))
    d /= np.linalg.norm(d, axis=2)[..., None]
    outer = np.arange(24) % 2 == 1
    r = np.where(outer, rng.uniform(18.0, 28.0, (64, 24)), rng.uniform(2.0, 12.0, (64, 24)))
    if kind == "rows":     # light and heavy rows side by side
        w = np.where(np.arange(64)[:, None] % 2 == 0, 1e-6, 1e6)
    else:                  # heavy bins that dL/dzeta leaves out
        w = np.where(outer[None, :], 1e6, 1e-6)
    w = w * rng.uniform(0.5, 1.5, (64, 24))
    pos = np.concatenate([p, (p[:, None] + r[..., None] * d).reshape(-1, 3)]).astype(np.float32)
    return catalogs.Catalog(pos, np.concatenate([np.ones(64), w.ravel()]).astype(np.float32), 300.0, nbins, 0.0,
                            30.0, lmax, 1)


@pytest.mark.parametrize("chunk", [0, 64])
@pytest.mark.parametrize("kind,nbins,lmax", [
    ("rows", 6, 6), ("rows", 5, 10), ("rows", 32, 2), ("rows", 1, 3), ("bins", 6, 6), ("bins", 4, 10), ("bins", 32, 2),
])
def test_rows_and_bins_of_very_different_size(kind, nbins, lmax, chunk):
    rng = np.random.default_rng(nbins + lmax)
    cat = _catalog(kind, nbins, lmax, rng)
    bins = np.arange(nbins) if kind == "rows" else np.arange(nbins // 2)
    G = []
    for m in range(lmax + 1):
        K = nbins * (lmax + 1 - m)
        keep = np.isin(np.arange(K) % nbins, bins)
        b = rng.normal(size=(K, K)) + 1j * rng.normal(size=(K, K))
        G.append(((b + b.conj().T) * np.outer(keep, keep)))
    flat = np.concatenate([b.ravel() for b in G])
    pos, w = to_dev(cat, torch)
    plan = g3.Plan(**cat.params())
    plan.set_option(g3.OPT_CHUNK_ROWS, chunk)
    plan.compute(pos, w, n_primary=64, keep_alm=True)
    a = plan.alm(np.arange(64))
    _, dw = plan.backward(torch.from_numpy(np.stack([2 * flat.real, 2 * flat.imag], axis=1)).cuda())
    dw = dw.cpu().numpy()
    for i in range(64):
        ref = tol = 0.0
        for m in range(lmax + 1):
            M = G[m] + G[m].conj().T
            v = a[i][:, [oracle.lm_index(l, m) for l in range(m, lmax + 1)]].T.reshape(-1)  # (l - m) nbins + b
            ref += np.real(np.conj(v) @ (M @ v))
            big = np.tile((np.abs(v.real) + np.abs(v.imag)).reshape(-1, nbins).max(axis=0), lmax + 1 - m)
            tol += np.sum((np.abs(v.real) + np.abs(v.imag)) * ((np.abs(M.real) + np.abs(M.imag)) @ big))
        assert abs(dw[i] - ref) <= 2.0 ** -36 * tol, i


def test_primary_weight_term_sums_in_fp64():
    # M = 1: V = A exactly, and the term is sum |A|^2 with one rounding of 2^-53 per column and
    # lane (38 of them) and per level of the reduction, as a random walk below 2^-51 of the sum
    rng = np.random.default_rng(3)
    cat = _catalog("bins", 10, 10, rng)
    cat.w[:] = 1.0
    pos, w = to_dev(cat, torch)
    plan = g3.Plan(**cat.params())
    plan.compute(pos, w, n_primary=64, keep_alm=True)
    a = plan.alm(np.arange(64))
    one = np.concatenate([0.5 * np.eye(cat.nbins * (cat.lmax + 1 - m)).ravel() for m in range(cat.lmax + 1)])
    _, dw = plan.backward(torch.from_numpy(np.stack([2 * one, 0 * one], axis=1)).cuda())
    for i, got in enumerate(dw.cpu().numpy()[:64]):
        ref = math.fsum(np.concatenate([a[i].real.ravel() ** 2, a[i].imag.ravel() ** 2]))
        assert abs(got - ref) <= 2.0 ** -51 * ref, i


@pytest.mark.parametrize("lmax", [4, 10])
@pytest.mark.parametrize("kind", ["weights", "inner bin", "light"])
def test_gradients_point_by_point(kind, lmax):
    # weights over twelve decades; a dense clump beside isolated points with dL/dzeta on the
    # innermost bin alone; light points whose rows share blocks with those of a heavy clump.
    # Every point against its own size: the rows of A are FP32 (2^-25 of an entry, amplified by
    # up to 2^7 to a pair's gradient), pairs are rounded to FP32, and one component in a few
    # hundred may cancel tenfold: 1e-4 of the point's own, and 1e-6 of the median's
    n, nbins = 300, 5
    rng = np.random.default_rng(lmax)
    pos = rng.uniform(60.0, 140.0, (n, 3))
    w = rng.uniform(0.5, 1.5, n)
    bins, pick = np.arange(nbins), np.ones(n, bool)
    if kind == "weights":
        w *= 10.0 ** rng.uniform(-6.0, 6.0, n)
    elif kind == "inner bin":
        pos[:200] = 100.0 + 1.5 * rng.normal(size=(200, 3))
        bins = np.arange(1)
    else:
        pick = np.arange(n) % 2 == 0
        pos = np.where(pick[:, None], 60.0, 200.0) + rng.uniform(-9.0, 9.0, (n, 3))
        w *= np.where(pick, 1e-6, 1e6)
    cat = catalogs.Catalog(pos.astype(np.float32), w.astype(np.float32), 300.0, nbins, 0.0, 30.0, lmax, 1)
    G = []
    for m in range(lmax + 1):
        K = nbins * (lmax + 1 - m)
        keep = np.isin(np.arange(K) % nbins, bins)
        b = rng.normal(size=(K, K)) + 1j * rng.normal(size=(K, K))
        G.append(((b + b.conj().T) * np.outer(keep, keep)).ravel())
    G = np.concatenate(G)
    p, wt = to_dev(cat, torch)
    plan = g3.Plan(**cat.params())
    plan.compute(p, wt, keep_alm=True)
    dpos, dw = plan.backward(torch.from_numpy(np.stack([2 * G.real, 2 * G.imag], axis=1)).cuda())
    rpos, rw = oracle.grad(cat.pos.astype(np.float64), cat.w.astype(np.float64), G, cat.box, nbins, 0.0, 30.0, lmax,
                           los_mode=1)
    for got, ref in ((dpos.cpu().numpy(), rpos), (dw.cpu().numpy()[:, None], rw[:, None])):
        size = np.abs(ref[pick]).max(axis=1)
        assert (np.abs(got - ref)[pick].max(axis=1) <= 1e-4 * size + 1e-6 * np.median(size)).all()
