"""kNN bandwidths bit for bit against the oracle's brute force where the search can go
wrong: list lengths (k on either side of a kernel's range), ragged last leaves, the
smallest clouds, exact ties (lattices, duplicates), many points at one distance from an
isolated one, and distances whose squares leave the FP32 range."""
import numpy as np
import pytest
import torch

import oracle
from paper_2601_20758_gb300 import _lib as L
from paper_2601_20758_gb300 import synth

pytestmark = pytest.mark.gpu


def _clumps(n, r):
    """A tight ball of points far from a thin background: from out there all of the ball is
    at one distance."""
    ball = 0.9 + 1e-5 * r.standard_normal((n // 2, 3))
    thin = r.random((n - n // 2, 3)) * np.array([0.6, 1e-3, 1e-3])
    return np.concatenate([ball, thin])


CLOUDS = {
    "uniform": lambda n, r: r.random((n, 3)),
    "clustered": lambda n, r: synth.plain_cloud(n, seed=5),
    "lattice": lambda n, r: synth.lattice_cloud(int(round(n ** (1 / 3))) + 1, 0.0625)[:n],
    "duplicates": lambda n, r: r.random((max(2, n // 90), 3))[r.integers(0, max(2, n // 90), n)],
    "clumps": _clumps,
    "line": lambda n, r: np.stack([r.random(n) ** 4, np.zeros(n), np.zeros(n)], axis=1),
    "tiny": lambda n, r: 1e-19 * r.random((n, 3)),
    "huge": lambda n, r: 3e18 * r.random((n, 3)),
}


@pytest.mark.parametrize("cloud", sorted(CLOUDS))
@pytest.mark.parametrize("n,k", [(2, 1), (33, 32), (67, 66), (1025, 8), (2500, 34), (2500, 35), (3001, 64),
                                 (3001, 66), (3001, 67), (4099, 256)])
def test_knn_bit_exact(cloud, n, k):
    xyz = np.ascontiguousarray(CLOUDS[cloud](n, np.random.default_rng(11 * n + k)).astype(np.float32))
    n = xyz.shape[0]
    if n <= k:
        pytest.skip("cloud too small")
    idx = L.sf_build_index(torch.from_numpy(xyz).cuda())
    try:
        L.sf_bandwidths(idx, L.make_params(k=k))
        h = torch.empty(n, device="cuda")
        L.sf_get_bandwidths(idx, h)
        torch.cuda.synchronize()
        work = L.sf_knn_work_counts(idx, k)
    finally:
        L.sf_free_index(idx)
    ref, _, _ = oracle.knn(xyz, k)
    assert np.array_equal(h.cpu().numpy().view(np.uint32), np.asarray(ref, dtype=np.float32).view(np.uint32))
    assert work["query_leaves"] == -(-n // 32)


@pytest.mark.parametrize("cloud", sorted(CLOUDS))
@pytest.mark.parametrize("n,k", [(94, 92), (95, 93), (2500, 79), (3001, 92), (3001, 93)])
def test_knn_where_the_longest_lists_begin(cloud, n, k):
    test_knn_bit_exact(cloud, n, k)
