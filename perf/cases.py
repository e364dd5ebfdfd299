"""Measured cases: what a user of this library has it do, through its public entry points.

Every case is one call (or one differentiation step, or one random-catalog correction) on
a seeded synthetic catalog: the recipes and sizes are those of the benchmark, of the tests
and of the workloads in ``paper_1709_00086_gb300/catalogs.py``, or cuts of them at the same
density.  A plan, the catalog's device arrays and, where a program would keep them, the
output buffers are made by ``prepare``; ``run`` is the call itself.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1709_00086_gb300 as g3

LOS_PERIODIC, LOS_OPEN, LOS_RADIAL = 0, 1, 2


def _forward(name, n, box, rmax, nbins, lmax, **kw):
    c = dict(what="forward", n=n, box=box, rmin=0.0, rmax=rmax, nbins=nbins, lmax=lmax,
             los=LOS_PERIODIC, f64=False, clustered=False, ones=False, fp32=False, graph=False,
             primaries=0)
    c.update(kw)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest catalog of the batched workload on its own: launches and latency
        _forward("mock_1k", 1000, 600.0, 150.0, 12, 8),
        # the plain workload: 20,000 uniform points, FP64 positions, unit weights
        _forward("plain_20k", 20000, 1000.0, 200.0, 10, 10, f64=True, ones=True),
        # the same catalog with the plain-FP32 contraction (about 1e-7 instead of 1e-5)
        _forward("plain_20k_fp32", 20000, 1000.0, 200.0, 10, 10, f64=True, ones=True, fp32=True),
        # a survey region with its halo: the first points are primaries, all are
        # secondaries (the sharded run's local step); open box, odd sizes and orders
        _forward("halo_60k", 60013, 517.0, 90.0, 7, 5, rmin=5.0, los=LOS_OPEN, f64=True, clustered=True,
                 primaries=17389),
        # the benchmark's clustered recipe at a tenth of its size and the same density
        _forward("clustered_200k", 200000, 696.0, 200.0, 10, 10, clustered=True),
        # the benchmark's workload: 2,000,000 clustered points, 4e10 pairs
        _forward("clustered_2m", 2000000, 1500.0, 200.0, 10, 10, clustered=True),
        # an observer's survey: open cube, line of sight per primary (a cut of the
        # 50M-point radial workload at a fifth of its density)
        _forward("radial_150k", 150000, 742.0, 200.0, 10, 10, los=LOS_RADIAL, clustered=True),
        # many mocks in one call, replayed from a captured graph (repeated measurements
        # into the same buffers)
        dict(name="mocks_24_graph", what="batch", ncat=24, lo=1000, hi=100000, box=600.0, rmin=0.0, rmax=150.0,
             nbins=12, lmax=8, graph=True, fp32=False),
        # the random-catalog correction: D - R_k and R_k as one batch, averaged on the
        # device, then the isotropic epilogue (negative weights)
        dict(name="randoms_4", what="randoms", n=6000, nrand=4, factor=2, box=500.0, rmin=0.0, rmax=80.0, nbins=8,
             lmax=6, fp32=False),
        # a gradient step on a small catalog (the size the gradient tests use)
        dict(name="grad_2500", what="grad", n=2500, box=250.0, rmin=0.0, rmax=60.0, nbins=8, lmax=6,
             los=LOS_PERIODIC, primaries=0, fp32=False),
        # the differentiation workload at a fifth of its size and the same density
        dict(name="grad_100k", what="grad", n=100000, box=468.0, rmin=0.0, rmax=120.0, nbins=8, lmax=6,
             los=LOS_PERIODIC, primaries=0, fp32=False),
        # a gradient step at the highest order
        dict(name="grad_20k_l10", what="grad", n=20000, box=600.0, rmin=0.0, rmax=120.0, nbins=10, lmax=10,
             los=LOS_OPEN, primaries=0, fp32=False),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    what = rng.choice(["forward", "forward", "forward", "batch", "randoms", "grad"])
    lmax, nbins = rng.randint(4, 10), rng.randint(4, 16)
    rmax = rng.choice([80.0, 120.0, 150.0, 200.0])
    box = round(rmax / rng.uniform(0.12, 0.30), 1)
    cover = 4.0 / 3.0 * math.pi * (rmax / box) ** 3  # a point's neighbours over all points

    def points(lo, hi, most_pairs):
        n = int(_log(rng, lo, hi))
        return min(n, int(math.sqrt(most_pairs / cover))) | 1

    rmin = rng.choice([0.0, 0.0, 5.0, 12.5])
    if what == "forward":
        n = points(1000, 300000, 8e9)
        return _forward("", n, box, rmax, nbins, lmax, rmin=rmin,
                        los=rng.choice([LOS_PERIODIC, LOS_PERIODIC, LOS_OPEN, LOS_RADIAL]),
                        f64=rng.random() < 0.4, clustered=rng.random() < 0.6, ones=rng.random() < 0.3,
                        fp32=rng.random() < 0.25, graph=rng.random() < 0.25,
                        primaries=int(n * rng.uniform(0.1, 0.9)) if rng.random() < 0.3 else 0)
    if what == "batch":
        return dict(what="batch", ncat=rng.randint(3, 40), lo=rng.randint(300, 1500),
                    hi=points(4000, 100000, 4e8), box=box, rmin=rmin, rmax=rmax, nbins=nbins, lmax=lmax,
                    graph=rng.random() < 0.5, fp32=rng.random() < 0.2)
    if what == "randoms":
        return dict(what="randoms", n=points(1000, 20000, 4e7), nrand=rng.randint(1, 6), factor=rng.randint(1, 3),
                    box=box, rmin=rmin, rmax=rmax, nbins=nbins, lmax=lmax, fp32=rng.random() < 0.3)
    n = points(1000, 100000, 1e8)
    return dict(what="grad", n=n, box=box, rmin=rmin, rmax=rmax, nbins=nbins, lmax=lmax,
                los=rng.choice([LOS_PERIODIC, LOS_PERIODIC, LOS_OPEN]),
                primaries=int(n * rng.uniform(0.1, 0.9)) if rng.random() < 0.25 else 0, fp32=rng.random() < 0.3)


# --- inputs ------------------------------------------------------------------


def _into_box(x, box, dtype):
    x = np.mod(x, box).astype(dtype)
    x[(x >= dtype(box)) | (x < 0)] = 0
    return np.ascontiguousarray(x)


def _positions(rng, n, box, clustered, wrap, dtype):
    """Uniform, or 60% uniform and 40% in blobs of width 5 about one centre per 200 points."""
    if not clustered:
        return _into_box(rng.random((n, 3)) * box, box, dtype)
    n_blob = n - int(round(0.6 * n))
    pos = rng.random((n, 3)) * box
    centres = rng.random((max(1, n // 200), 3)) * box
    blob = centres[rng.integers(0, len(centres), n_blob)] + 5.0 * rng.standard_normal((n_blob, 3))
    if not wrap:  # an open box: what leaves it becomes uniform
        out = np.any((blob < 0) | (blob >= box), axis=1)
        blob[out] = rng.random((int(out.sum()), 3)) * box
    at = rng.permutation(n)[:n_blob]
    pos[at] = blob
    return _into_box(pos, box, dtype)


def _weights(rng, n, ones=False):
    return np.ones(n, np.float32) if ones else (0.5 + rng.random(n)).astype(np.float32)


def _offsets(case, rng):
    """Catalog sizes of a batch: log-uniform, the largest and the smallest among them."""
    u = rng.random(case["ncat"])
    u[0], u[-1] = 1.0, 0.0
    sizes = np.exp(np.log(case["lo"]) + u * (np.log(case["hi"]) - np.log(case["lo"]))).astype(np.int64)
    return np.concatenate([[0], np.cumsum(sizes)])


def _zsize(case):
    return sum((case["nbins"] * (case["lmax"] + 1 - m)) ** 2 for m in range(case["lmax"] + 1))


def _arrays(case, seed):
    """Positions, weights, catalog offsets and (for a gradient) dL/dzeta, on the host."""
    rng = np.random.default_rng([seed, 1709])
    box, what = case["box"], case["what"]
    if what == "batch":
        # the sizes are the case's own: another seed draws other points
        offs = _offsets(case, np.random.default_rng(86))
        n = int(offs[-1])
        return _positions(rng, n, box, False, True, np.float32), _weights(rng, n), offs, None
    if what == "randoms":
        n, n_r = case["n"], case["n"] * case["factor"]
        data, w = _positions(rng, n, box, True, True, np.float32), _weights(rng, n)
        alpha = np.float32(np.sum(w, dtype=np.float64) / n_r)
        pos, ws, sizes = [], [], []
        rand = [_positions(rng, n_r, box, False, True, np.float32) for _ in range(case["nrand"])]
        for r in rand:  # D - R_k
            pos += [data, r]
            ws += [w, np.full(n_r, -alpha, np.float32)]
            sizes.append(n + n_r)
        for r in rand:  # R_k
            pos.append(r)
            ws.append(np.full(n_r, alpha, np.float32))
            sizes.append(n_r)
        return np.concatenate(pos), np.concatenate(ws), np.concatenate([[0], np.cumsum(sizes)]), None
    n = case["n"]
    offs = np.array([0, n], np.int64)
    if what == "grad":
        pos = _positions(rng, n, box, True, case["los"] == LOS_PERIODIC, np.float32)
        w = _weights(rng, n)
        gz = rng.standard_normal((_zsize(case), 2))
        return pos, w, offs, gz
    pos = _positions(rng, n, box, case["clustered"], case["los"] == LOS_PERIODIC,
                     np.float64 if case["f64"] else np.float32)
    return pos, _weights(rng, n, case["ones"]), offs, None


def prepare(case, seed):
    pos, w, offs, gz = _arrays(case, seed)
    s = dict(case=case, plan=g3.Plan(nbins=case["nbins"], rmin=case["rmin"], rmax=case["rmax"], lmax=case["lmax"],
                                     box=case["box"], los_mode=case.get("los", LOS_PERIODIC)),
             pos=torch.from_numpy(pos).cuda(), w=torch.from_numpy(w).cuda(), offs=offs, out=None, counts=None)
    if case["what"] == "grad":
        s["pos"].requires_grad_()
        s["w"].requires_grad_()
        s["gz"] = torch.from_numpy(gz).cuda()
    elif case.get("graph"):  # a replayed call writes into the buffers it was captured with
        ncat = len(offs) - 1
        shape = (_zsize(case), 2) if case["what"] == "forward" else (ncat, _zsize(case), 2)
        s["out"] = torch.empty(shape, dtype=torch.float64, device="cuda")
        s["counts"] = torch.empty(shape[:-2] + (case["nbins"],), dtype=torch.int64, device="cuda")
    return s


def run(s):
    case, plan = s["case"], s["plan"]
    if case["what"] == "forward":
        z, counts = plan.compute(s["pos"], s["w"], n_primary=case["primaries"] or None,
                                 fp32_contraction=case["fp32"], graph=case["graph"], out=s["out"],
                                 counts_out=s["counts"])
        return {"zeta": z, "counts": counts}
    if case["what"] == "batch":
        z, counts = plan.compute_batch(s["pos"], s["w"], s["offs"], fp32_contraction=case["fp32"],
                                       graph=case["graph"], out=s["out"], counts_out=s["counts"])
        return {"zeta": z, "counts": counts}
    if case["what"] == "randoms":
        z, counts = plan.compute_batch(s["pos"], s["w"], s["offs"], fp32_contraction=case["fp32"])
        k = case["nrand"]
        mean = [1.0 / k] * k
        field = g3.zeta_combine(z, mean + [0.0] * k, case["nbins"], case["lmax"])
        rand = g3.zeta_combine(z, [0.0] * k + mean, case["nbins"], case["lmax"])
        return {"field": field, "randoms": rand, "counts": counts,
                "isotropic": g3.isotropic(field, case["nbins"], case["lmax"])}
    z = g3.zeta(s["pos"], s["w"], plan, n_primary=case["primaries"] or None, fp32_contraction=case["fp32"])
    dpos, dw = torch.autograd.grad(z, (s["pos"], s["w"]), s["gz"])
    return {"zeta": z.detach(), "dpos": dpos, "dw": dw}


# --- work --------------------------------------------------------------------


def _pairs(case, n, n_primary):
    """Expected ordered pairs: uniform points in the box (clustering adds a percent)."""
    shells = []
    for r in (case["rmin"], case["rmax"]):
        x = r / case["box"]
        v = 4.0 / 3.0 * math.pi * x ** 3
        if case.get("los", LOS_PERIODIC) != LOS_PERIODIC:  # faces, edges and corners of an open cube
            v += -1.5 * math.pi * x ** 4 + 1.6 * x ** 5 - x ** 6 / 6.0
        shells.append(v)
    return float(n) * n_primary * (shells[1] - shells[0])


def work(case):
    lmax, zs = case["lmax"], _zsize(case)
    what = case["what"]
    if what == "batch":
        sizes = np.diff(_offsets(case, np.random.default_rng(86))).tolist()
    elif what == "randoms":
        sizes = ([case["n"] * (1 + case["factor"])] + [case["n"] * case["factor"]]) * case["nrand"]
    else:
        sizes = [case["n"]]
    prim = [case["primaries"] or case["n"]] if what in ("forward", "grad") else sizes
    pairs = sum(_pairs(case, n, p) for n, p in zip(sizes, prim))
    # per pair: separation, unit vector, T_k(z), w (x + iy)^m and one multiply-add per
    # harmonic; per primary 8 flops per complex product of the Hermitian zeta
    per_pair = 14 + 2 * (lmax - 1) + 6 * (lmax - 1) + 2 * (lmax + 1) ** 2
    per_prim = 4 * sum(k * (k + 1) for k in (case["nbins"] * (lmax + 1 - m) for m in range(lmax + 1)))
    flops = pairs * per_pair + sum(prim) * per_prim
    pos_bytes = 24 if case.get("f64") else 12
    nbytes = sum(sizes) * (pos_bytes + 4) + len(sizes) * (16 * zs + 8 * case["nbins"])
    if what == "grad":  # F, its three derivatives per harmonic; V = M A per primary
        flops += pairs * (14 + 8 * (lmax + 1) ** 2) + 2 * sum(prim) * per_prim
        nbytes += sum(sizes) * 16 + 16 * zs
    elif what == "randoms":
        nbytes += 2 * 16 * zs + 8 * (lmax + 1) * case["nbins"] ** 2
    return {"bytes": float(nbytes), "flops": float(flops)}


# --- 64-bit reference --------------------------------------------------------


def _harmonics(u, lmax):
    """Orthonormal Y_lm (Condon-Shortley), m >= 0, of unit vectors (p, 3): (l, m) -> (Re, Im)."""
    x, y, z = u.unbind(-1)
    cr, ci = torch.ones_like(x), torch.zeros_like(x)
    lead = math.sqrt(1.0 / (4.0 * math.pi))
    out = {}
    for m in range(lmax + 1):
        if m > 0:
            cr, ci = cr * x - ci * y, cr * y + ci * x
            lead = -lead * math.sqrt((2.0 * m + 1.0) / (2.0 * m))
        q0, q1 = None, torch.full_like(z, lead)
        for l in range(m, lmax + 1):
            if l == m + 1:
                q0, q1 = q1, math.sqrt(2.0 * m + 3.0) * z * q1
            elif l > m + 1:
                a = math.sqrt((4.0 * l * l - 1.0) / (l * l - m * m))
                b = math.sqrt(((l - 1.0) ** 2 - m * m) / (4.0 * (l - 1.0) ** 2 - 1.0))
                q0, q1 = q1, a * (z * q1 - b * q0)
            out[l, m] = (q1 * cr, q1 * ci)
    return out


def _pair_list(pos, prim, case):
    """Pairs (index into prim, secondary, bin) of the primaries prim, and their separations' images."""
    box, B = case["box"], case["nbins"]
    d = pos[None, :, :] - pos[prim][:, None, :]
    shift = torch.zeros_like(d)
    if case.get("los", LOS_PERIODIC) == LOS_PERIODIC:
        shift = torch.where(d > 0.5 * box, -box, torch.where(d < -0.5 * box, box, 0.0))
        d = d + shift
    r2 = (d[..., 0] * d[..., 0] + d[..., 1] * d[..., 1]) + d[..., 2] * d[..., 2]
    edges = [case["rmin"] + (case["rmax"] - case["rmin"]) * k / B for k in range(B)] + [case["rmax"]]
    e2 = torch.tensor([e * e for e in edges], dtype=torch.float64, device=pos.device)
    b = torch.bucketize(r2, e2, right=True) - 1
    i, j = torch.nonzero((b >= 0) & (b < B) & (r2 > 0), as_tuple=True)
    return i, j, b[i, j], shift[i, j]


def _multipoles(pos, w, prim, case):
    """a_lm of the primaries prim, {m: ((np, K_m) Re, Im)}, columns (l - m) B + b; and the counts."""
    B, lmax = case["nbins"], case["lmax"]
    i, j, b, shift = _pair_list(pos.detach(), prim, case)
    d = pos[j] - pos[prim][i] + shift
    if case.get("los", LOS_PERIODIC) == LOS_RADIAL:  # turn the observer's direction to +z
        n = pos[prim] - 0.5 * case["box"]
        n = (n / n.norm(dim=-1, keepdim=True))[i]
        v = torch.stack([n[:, 1], -n[:, 0], torch.zeros_like(n[:, 0])], -1)
        vd = torch.linalg.cross(v, d)
        d = d + vd + torch.linalg.cross(v, vd) / (1.0 + n[:, 2:])
    Y = _harmonics(d / d.norm(dim=-1, keepdim=True), lmax)
    cell = i * B + b
    wj = w[j]
    a = {}
    for m in range(lmax + 1):
        parts = []
        for part in (0, 1):
            cols = [torch.zeros(len(prim) * B, dtype=torch.float64, device=pos.device)
                    .index_add(0, cell, wj * Y[l, m][part]) for l in range(m, lmax + 1)]
            parts.append(torch.stack([c.view(len(prim), B) for c in cols], 1).reshape(len(prim), -1))
        a[m] = parts
    return a, torch.bincount(b, minlength=B)


def _zeta64(pos, w, case, n_primary, gz=None):
    """zeta (complex128) and counts; with gz, the gradients of sum(gz * zeta) instead of the counts."""
    n, B = len(pos), case["nbins"]
    zeta = counts = 0
    if gz is not None:
        pos, w = pos.requires_grad_(), w.requires_grad_()
    per = max(1, min(n_primary, int(min(2e7 / n, 3e6 / max(1.0, _pairs(case, n, 1))))))
    for p0 in range(0, n_primary, per):
        prim = torch.arange(p0, min(n_primary, p0 + per), device=pos.device)
        a, c = _multipoles(pos, w, prim, case)
        wp = w[prim][:, None]
        blocks = []
        for m, (re, im) in a.items():
            zr = (wp * re).T @ re + (wp * im).T @ im
            zi = (wp * im).T @ re - (wp * re).T @ im
            blocks.append(torch.stack([zr, zi], -1).reshape(-1, 2))
        z = torch.cat(blocks)
        if gz is not None:
            (gz * z).sum().backward()
        zeta, counts = zeta + z.detach(), counts + c
    if gz is not None:
        return zeta, pos.grad, w.grad
    return torch.view_as_complex(zeta), counts


def _isotropic64(z, case):
    B, lmax = case["nbins"], case["lmax"]
    out = torch.zeros((lmax + 1, B, B), dtype=torch.float64, device=z.device)
    off = 0
    for m in range(lmax + 1):
        K = B * (lmax + 1 - m)
        block = z[off:off + K * K].view(K, K).real
        for l in range(m, lmax + 1):
            at = slice((l - m) * B, (l - m + 1) * B)
            out[l] += (1.0 if m == 0 else 2.0) * block[at, at]
        off += K * K
    return out


def exact(case, seed):
    pos, w, offs, gz = _arrays(case, seed)
    sizes = np.diff(offs).tolist()
    prim = [case.get("primaries") or s for s in sizes]
    if sum(float(s) * p for s, p in zip(sizes, prim)) > 6e9:
        return None
    most = 2e7 if case["what"] == "grad" else 2e8
    if sum(_pairs(case, s, p) for s, p in zip(sizes, prim)) * (case["lmax"] + 1) ** 2 / 121.0 > most:
        return None
    pos, w = torch.from_numpy(pos).cuda().double(), torch.from_numpy(w).cuda().double()
    if case["what"] == "grad":
        z, dpos, dw = _zeta64(pos, w, case, prim[0], torch.from_numpy(gz).cuda())
        return {"zeta": z, "dpos": dpos, "dw": dw}
    got = [_zeta64(pos[a:b], w[a:b], case, p) for a, b, p in zip(offs[:-1], offs[1:], prim)]
    if case["what"] == "forward":
        return {"zeta": got[0][0], "counts": got[0][1]}
    z, counts = torch.stack([g[0] for g in got]), torch.stack([g[1] for g in got])
    if case["what"] == "batch":
        return {"zeta": z, "counts": counts}
    k = case["nrand"]
    field = z[:k].sum(0) / k
    return {"field": field, "randoms": z[k:].sum(0) / k, "counts": counts, "isotropic": _isotropic64(field, case)}
