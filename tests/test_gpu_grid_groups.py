"""The grid's walk by groups of neighbouring tiles (2, 4 or 8 to a group from 12,000 tiles on):
whole grids with odd numbers of tiles, so that groups at the ends are partial, against grids
of a few planes of the same nodes, which are walked tile by tile; alone and in a batch whose
ROIs' groups follow one another."""
import numpy as np
import pytest
import torch

from paper_2601_20758_gb300 import _lib as L

pytestmark = pytest.mark.gpu

# tiles of 8 x 4 x 8 nodes: 15 x 25 x 33, 21 x 39 x 31, 35 x 47 x 31 (4-deep tiles: twice in z)
H = (0.02, 0.03, 0.025)
GRIDS = [(117, 99, 262), (165, 153, 243), (273, 187, 246)]


def _cloud():
    r = np.random.default_rng(3)
    p = np.concatenate([r.random((6000, 3)), 0.4 + 0.02 * r.standard_normal((6000, 3))]).astype(np.float32)
    return torch.from_numpy(np.clip(p, 0.0, 1.0)).cuda()


def _planes(idx, kernel, p, dims, grid):
    """Every 8th and the last 3 planes of the grid again, 2 at a time. Their nodes' coordinates
    are the grid's up to FP64 rounding, which FP32 distances may carry across a support's edge:
    there a Gaussian term is e^-4.5 of its largest (two may at one node), an Epanechnikov term
    a rounding of it. A leaf left out is 32 terms of up to the largest."""
    gauss = kernel == L.SF_K_GAUSS3
    largest = (0.0654 if gauss else 0.5969) / (H[0] * H[1] * H[2]) / 12_000
    edge = largest * (2.0 * float(np.exp(-4.5)) if gauss else 1e-5)
    s = 1.0 / (dims[2] - 1)
    grid = grid.reshape(dims[::-1])
    for z in list(range(0, dims[2] - 1, 8)) + [dims[2] - 3, dims[2] - 2]:
        out = torch.empty(dims[0] * dims[1] * 2, device="cuda")
        L.sf_kde_grid(idx, L.make_box((0, 0, z * s), (1, 1, (z + 1) * s)), (dims[0], dims[1], 2), kernel, p, out)
        a, b = grid[z:z + 2], out.reshape(2, dims[1], dims[0])
        assert bool(((a - b).abs() <= 1e-5 * b + edge).all()), (dims, z)
    assert float(grid.max()) > 100.0 * edge


@pytest.mark.parametrize("kernel", ["GAUSS3", "EPAN"])
@pytest.mark.parametrize("scope", ["GLOBAL", "CLIP"])
def test_groups_of_tiles(kernel, scope):
    xyz = _cloud()
    ker = getattr(L, "SF_K_" + kernel)
    p = L.make_params(rule=L.SF_BW_FIXED, scope=L.SF_SCOPE_GLOBAL, fixed_h=H, accel=L.SF_ACCEL_NONE)
    idx = L.sf_build_index(xyz)
    try:
        L.sf_bandwidths(idx, p)
        box = L.make_box((0, 0, 0), (1, 1, 1))
        alone = []
        for dims in GRIDS:
            out = torch.empty(dims[0] * dims[1] * dims[2], device="cuda")
            L.sf_kde_grid(idx, box, dims, ker, p, out)
            _planes(idx, ker, p, dims, out)
            alone.append(out)
        q = L.make_params(rule=L.SF_BW_FIXED, scope=getattr(L, "SF_SCOPE_" + scope), fixed_h=H, accel=L.SF_ACCEL_NONE)
        for z in (4, 8):
            t = L.sf_tune()
            t.tile_z = z
            b = L.sf_batch_create(idx, [box] * 3, GRIDS, ker, q, tune=t)
            outs = [torch.empty_like(o) for o in alone]
            L.sf_batch_run(b, outs)
            torch.cuda.synchronize()
            L.sf_batch_free(b)
            for o, ref in zip(outs, alone):
                assert bool(((o - ref).abs() <= 1e-5 * ref + 1e-6 * ref.max()).all())
    finally:
        L.sf_free_index(idx)
