"""Point densities (DIRECT) against the oracle where a query leaf's work is shared or its
points lie apart: clouds below and above the size from which one warp takes a leaf, with
a thin background around a dense ball, so that leaves of background points have boxes
that cover the ball (over a thousand candidate leaves); every rule, both kernels."""
import numpy as np
import pytest
import torch

import oracle
from paper_2601_20758_gb300 import _lib as L
from tests.parity import density_check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [33, 500, 60_001, 330_000])
@pytest.mark.parametrize("rule,kernel,scope", [("knn", "GAUSS3", "GLOBAL"), ("knn", "EPAN", "CLIP"),
                                               ("fixed", "GAUSS3", "CLIP"), ("fixed", "EPAN", "GLOBAL")])
def test_points_with_wide_leaves(n, rule, kernel, scope):
    r = np.random.default_rng(n)
    thin = 200 if n > 1000 else n // 2
    ball = 0.5 + 0.02 * r.standard_normal((n - thin, 3))
    xyz = np.concatenate([ball, r.random((thin, 3))])[r.permutation(n)].astype(np.float32)
    k = 16
    lengths = (0.004, 0.006, 0.005) if n > 1000 else (0.1, 0.2, 0.15)
    idx = L.sf_build_index(torch.from_numpy(xyz).cuda())
    try:
        p = L.make_params(rule=L.SF_BW_KNN if rule == "knn" else L.SF_BW_FIXED, k=k, fixed_h=lengths,
                          scope=getattr(L, "SF_SCOPE_" + scope))
        L.sf_bandwidths(idx, p)
        if rule == "knn":
            h = torch.empty(n, device="cuda")
            L.sf_get_bandwidths(idx, h)
            ell = oracle.iso_ell(h.cpu().numpy())
        else:
            ell = np.tile(np.float32(lengths).astype(np.float64), (n, 1))
        dens = torch.empty(n, device="cuda")
        ids = torch.empty(n, dtype=torch.int32, device="cuda")
        box = ((0.05, 0.05, 0.05), (0.95, 0.95, 0.95))
        cnt = L.sf_kde_points(idx, L.make_box(*box), None, getattr(L, "SF_K_" + kernel), p, dens, ids)
        torch.cuda.synchronize()
    finally:
        L.sf_free_index(idx)
    inb = oracle.in_box(xyz, box)
    got_ids = ids[:cnt].cpu().numpy()
    assert np.array_equal(got_ids, np.nonzero(inb)[0])
    far = np.abs(xyz[got_ids] - 0.5).max(axis=1) > 0.09
    pick = np.unique(np.concatenate([np.nonzero(far)[0], r.choice(cnt, min(cnt, 300), replace=False)]))
    member = inb if scope == "CLIP" else np.ones(n, bool)
    ref = oracle.density_at(xyz[member], ell[member], xyz[got_ids[pick]].astype(np.float64),
                            getattr(oracle, kernel), 1.0 / member.sum())
    density_check(dens[:cnt].cpu().numpy()[pick], ref, label=f"{rule} {kernel} n={n}")
