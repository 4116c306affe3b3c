"""Grid densities against the oracle at the edges of the tile pipeline: particle counts
around the staging of 32, ragged and smallest node tiles (8 x 4 x 8 and 8 x 4 x 4), supports
below a node spacing, of a few spacings, and covering whole tiles; grids of one and of
many tiles; single calls and batches of both tile depths."""
import ctypes

import numpy as np
import pytest
import torch

import oracle
from paper_2601_20758_gb300 import _lib as L
from tests.parity import REL, U

pytestmark = pytest.mark.gpu

BOX = ((0.1, 0.05, 0.2), (0.9, 0.95, 0.7))


def _check(got, ref, label):
    """The per-output rule of tests/parity.py. Its headline (1e-5 of any output above 1e-3
    of the peak) is for outputs with many particles: with one particle at a node, 1 - q
    near the support's edge has an absolute error of the peak's rounding."""
    tol = REL * ref["rho"] + 8 * U * ref["wpeak"] + ref["amb"]
    bad = np.nonzero(np.abs(got - ref["rho"]) > tol)[0]
    assert bad.size == 0, f"{label}: {bad.size} outputs outside the tolerance, first {bad[:5]}"


def _params(rule, k, lengths, scope):
    return L.make_params(rule=L.SF_BW_KNN if rule == "knn" else L.SF_BW_FIXED, k=k, fixed_h=lengths,
                         scope=getattr(L, "SF_SCOPE_" + scope))


@pytest.mark.parametrize("dims", [(2, 2, 2), (8, 4, 8), (9, 5, 9), (17, 3, 4), (33, 26, 21)])
@pytest.mark.parametrize("n", [2, 31, 32, 33, 64, 65, 700])
@pytest.mark.parametrize("kernel", ["GAUSS3", "EPAN"])
@pytest.mark.parametrize("reach", ["under", "some", "whole", "knn"])
def test_grid_tiles(dims, n, kernel, reach):
    r = np.random.default_rng(n + dims[0])
    xyz = r.random((n, 3)).astype(np.float32)
    xyz[: n // 3] = (0.5 + 0.003 * r.standard_normal((n // 3, 3))).astype(np.float32)
    scope = "CLIP" if n >= 31 and (n + dims[0]) % 2 else "GLOBAL"
    s = [(BOX[1][a] - BOX[0][a]) / (dims[a] - 1) for a in range(3)]
    f = {"under": 0.3, "some": 2.0, "whole": 40.0, "knn": 0.0}[reach] / (3.0 if kernel == "GAUSS3" else 1.0)
    rule, k = ("knn" if reach == "knn" else "fixed"), min(8, n - 1)
    p = _params(rule, k, tuple(f * v for v in s) if f else (0.0, 0.0, 0.0), scope)
    idx = L.sf_build_index(torch.from_numpy(xyz).cuda())
    nodes = dims[0] * dims[1] * dims[2]
    try:
        L.sf_bandwidths(idx, p)
        if rule == "knn":
            h = torch.empty(n, device="cuda")
            L.sf_get_bandwidths(idx, h)
            ell = oracle.iso_ell(h.cpu().numpy())
        else:
            ell = np.tile(np.float32([f * v for v in s]).astype(np.float64), (n, 1))
        ker = getattr(L, "SF_K_" + kernel)
        grid = torch.empty(nodes, device="cuda")
        mass = L.sf_kde_grid(idx, L.make_box(*BOX), dims, ker, p, grid, want_mass=True)
        pairs = ctypes.c_int64(0)
        L._check("count", L.load().sf_count_support_pairs(idx, ctypes.byref(L.make_box(*BOX)), (ctypes.c_int32 * 3)(*dims),
                                                          ker, ctypes.byref(p), ctypes.byref(pairs), None, None))
        batches = []
        for z in (4, 8):
            t = L.sf_tune()
            t.tile_z, t.items_per_slot = z, 1 + z % 3
            out = [torch.empty(nodes, device="cuda") for _ in range(3)]
            b = L.sf_batch_create(idx, [L.make_box(*BOX)] * 3, [dims] * 3, ker, p, tune=t)
            m = L.sf_batch_run(b, out, want_mass=True)
            torch.cuda.synchronize()
            L.sf_batch_free(b)
            batches.append((out, m))
    finally:
        L.sf_free_index(idx)
    ref = oracle.kde_grid(xyz, ell, BOX, dims, getattr(oracle, kernel), getattr(oracle, "SCOPE_" + scope))
    g = grid.cpu().numpy().astype(np.float64)
    _check(g, ref, f"{dims} {n} {kernel} {reach}")
    cell = s[0] * s[1] * s[2]
    assert abs(mass - g.sum() * cell) <= 1e-12 * abs(mass)
    band = ref["amb"] > 0
    if not band.any():
        assert pairs.value == int(np.sum(ref["pairs"]))
    for out, m in batches:
        for o, mm in zip(out, m):
            o = o.cpu().numpy().astype(np.float64)
            _check(o, ref, f"batch {dims} {n} {kernel} {reach}")
            assert abs(mm - o.sum() * cell) <= 1e-12 * abs(mm)


@pytest.mark.parametrize("kernel", ["GAUSS3", "EPAN"])
@pytest.mark.parametrize("far,width", [(1.0e6, 0.5), (1.0e6, 2.0), (3.0e4, 0.01), (1.0e6, 1.0e-6), (0.0, 0.5)])
def test_node_spacing_below_the_coordinates_rounding(kernel, far, width):
    """A box so narrow in x, so far out, that neighbouring nodes share their nearest float;
    supports below the node spacing in z, of some steps of the coordinates in x."""
    r = np.random.default_rng(int(far) + len(kernel))
    n, dims = 3000, (40, 21, 6)
    ulp = float(np.spacing(np.float32(far + width)))
    xyz = r.random((n, 3)) * np.array([0.0, 10.0, 10.0])
    xyz[:, 0] = far + max(ulp, width / 40) * r.integers(-4, 12, n)
    xyz = xyz.astype(np.float32)
    box = ((far, 0.0, 0.0), (far + width, 10.0, 10.0))
    f = 3.0 if kernel == "GAUSS3" else 1.0
    lengths = (2.3 * max(ulp, width / 40) / f, 0.9 / f, 0.9 / f)
    p = _params("fixed", 8, lengths, "GLOBAL")
    idx = L.sf_build_index(torch.from_numpy(xyz).cuda())
    ker, nodes = getattr(L, "SF_K_" + kernel), dims[0] * dims[1] * dims[2]
    try:
        L.sf_bandwidths(idx, p)
        outs = [torch.empty(nodes, device="cuda") for _ in range(3)]
        L.sf_kde_grid(idx, L.make_box(*box), dims, ker, p, outs[0])
        for z, o in ((4, outs[1]), (8, outs[2])):
            t = L.sf_tune()
            t.tile_z = z
            b = L.sf_batch_create(idx, [L.make_box(*box)], [dims], ker, p, tune=t)
            L.sf_batch_run(b, [o])
            torch.cuda.synchronize()
            L.sf_batch_free(b)
    finally:
        L.sf_free_index(idx)
    ell = np.tile(np.float32(lengths).astype(np.float64), (n, 1))
    ref = oracle.kde_grid(xyz, ell, box, dims, getattr(oracle, kernel), oracle.SCOPE_GLOBAL)
    for o in outs:
        _check(o.cpu().numpy().astype(np.float64), ref, f"{kernel} {far} {width}")
