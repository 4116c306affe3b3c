"""The estimator's percentile lengths where the order statistics are delicate (few members,
members with equal coordinates, negative coordinates, one statistic per prefix): its grid
against the oracle's, per output."""
import numpy as np
import pytest
import torch

import oracle
from paper_2601_20758_gb300 import _lib as L
from tests.parity import REL, U

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [3, 5, 33, 1000, 20_000])
@pytest.mark.parametrize("cloud", ["negative", "equal", "decades"])
def test_mbe_order_statistics(n, cloud):
    r = np.random.default_rng(n)
    if cloud == "negative":
        xyz, box = 2.0 * r.random((n, 3)) - 1.0, ((-1.0, -1.0, -1.0), (1.0, 1.0, 1.0))
    elif cloud == "equal":  # a few distinct values per axis
        xyz, box = r.integers(0, 7, (n, 3)) / 8.0, ((-0.1, -0.1, -0.1), (1.0, 1.0, 1.0))
    else:
        xyz, box = 10.0 ** (-4.0 * r.random((n, 3))), ((0.0, 0.0, 0.0), (1.0, 1.0, 1.0))
    xyz = xyz.astype(np.float32)
    dims = (13, 9, 11)
    ref = None
    try:
        ref = oracle.mbe(xyz, box, dims, kernel=oracle.GAUSS3)
    except Exception:  # the oracle refuses degenerate spreads
        pass
    idx = L.sf_build_index(torch.from_numpy(xyz).cuda())
    out = torch.empty(dims[0] * dims[1] * dims[2], device="cuda")
    p = L.make_params(rule=L.SF_BW_MBE, scope=L.SF_SCOPE_CLIP)
    try:
        if ref is None:
            with pytest.raises(L.SFError):
                L.sf_kde_grid(idx, L.make_box(*box), dims, L.SF_K_GAUSS3, p, out)
            return
        L.sf_kde_grid(idx, L.make_box(*box), dims, L.SF_K_GAUSS3, p, out)
        torch.cuda.synchronize()
    finally:
        L.sf_free_index(idx)
    f = ref["final"]
    # a length is rounded to float (2^-24) and scaled by a float cube root (2^-22): q changes by
    # at most 2 * 9 * 2^-21.4 at the cutoff, so the sum by less than REL
    tol = REL * f["rho"] + 8 * U * f["wpeak"] + f["amb"]
    assert np.all(np.abs(out.cpu().numpy().astype(np.float64) - f["rho"]) <= tol)
