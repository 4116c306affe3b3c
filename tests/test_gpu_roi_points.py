"""The ROI's points and their number where the call takes another way: boxes around the
whole cloud, most of it, half, a few points and one point (closed faces through points),
on clouds of one leaf, of ragged leaves, and of several index levels; ids, densities and
the clip scope's normaliser against numpy and the oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_2601_20758_gb300 import _lib as L
from tests.parity import REL, U

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 31, 33, 1025, 40_003])
@pytest.mark.parametrize("share", [1.0, 0.99, 0.51, 0.5, 0.49, 0.02, 0.0])
def test_roi_points(n, share):
    r = np.random.default_rng(n)
    xyz = r.random((n, 3)).astype(np.float32)
    xyz[n // 2:] = xyz[r.integers(0, max(1, n // 2), n - n // 2)] if n > 40 else xyz[n // 2:]  # repeated positions
    order = np.sort(xyz[:, 0])
    cut = float(order[min(n - 1, int(share * n))]) if share < 1.0 else 2.0  # a face through a point
    box = ((-0.5, -0.5, -0.5), (cut, 1.5, 1.5))
    inb = oracle.in_box(xyz, box)
    idx = L.sf_build_index(torch.from_numpy(xyz).cuda())
    lengths = (0.05, 0.04, 0.06)
    p = L.make_params(rule=L.SF_BW_FIXED, fixed_h=lengths, scope=L.SF_SCOPE_CLIP)
    dens = torch.full((n + 3,), -5.0, device="cuda")
    ids = torch.full((n + 3,), 77, dtype=torch.int32, device="cuda")
    try:
        q = L.sf_query_workspace(idx, L.make_box(*box), None, L.SF_K_GAUSS3, p, what=L.SF_WS_POINTS)
        cnt = L.sf_kde_points(idx, L.make_box(*box), None, L.SF_K_GAUSS3, p, dens, ids)
        used = L.sf_last_call_workspace()
        torch.cuda.synchronize()
        if cnt > 1:
            short = torch.zeros(cnt - 1, device="cuda")
            with pytest.raises(L.SFError):
                L.sf_kde_points(idx, L.make_box(*box), None, L.SF_K_GAUSS3, p, short, ids)
            assert not short.any()
    finally:
        L.sf_free_index(idx)
    assert cnt == inb.sum() and used <= q
    assert np.array_equal(ids[:cnt].cpu().numpy(), np.nonzero(inb)[0])
    assert bool((dens[cnt:] == -5.0).all()) and bool((ids[cnt:] == 77).all())
    at = r.choice(cnt, min(cnt, 200), replace=False)
    ell = np.tile(np.float32(lengths).astype(np.float64), (cnt, 1))
    ref = oracle.density_at(xyz[inb], ell, xyz[inb][at].astype(np.float64), oracle.GAUSS3, 1.0 / cnt)
    tol = REL * ref["rho"] + 8 * U * ref["wpeak"] + ref["amb"]
    assert np.all(np.abs(dens[:cnt].cpu().numpy()[at].astype(np.float64) - ref["rho"]) <= tol)
