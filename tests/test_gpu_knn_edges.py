"""kNN bandwidths bit for bit where FP32 and FP64 order two points differently across a
power-of-two fraction (the edges of the search's distance bins): the k-th nearest point is
the one whose FP32 squared distance lies on the edge, a farther one's just below it. Alone
(the first bound decides) and with a shell of points that makes the lists overflow. And
where FP32 squares leave its range, next to distances or coordinates of another scale."""
import numpy as np
import pytest
import torch

import oracle
from paper_2601_20758_gb300 import _lib as L

pytestmark = pytest.mark.gpu

F = np.float32


def _d2_f32(q, p):  # the kernel's order, products and sums with one rounding each
    d = (q - p).astype(np.float64)
    xx = (d[:, 0] * d[:, 0]).astype(F).astype(np.float64)
    xy = (d[:, 1] * d[:, 1] + xx).astype(F).astype(np.float64)
    return (d[:, 2] * d[:, 2] + xy).astype(F)


def _d2_f64(q, p):
    d = q.astype(np.float64) - p.astype(np.float64)
    return (d[:, 0] * d[:, 0] + d[:, 1] * d[:, 1]) + d[:, 2] * d[:, 2]


def _swapped(q, edge, r):
    """(a, b): FP32 puts a below the edge and b on it, FP64 puts b nearer."""
    u = r.standard_normal((200_000, 3))
    p = (q + u / np.linalg.norm(u, axis=1)[:, None] * np.sqrt(edge)).astype(F)
    d, e = _d2_f32(q, p), _d2_f64(q, p)
    below, on = d == np.nextafter(F(edge), F(0)), d == F(edge)
    a, b = p[below][np.argmax(e[below])], p[on][np.argmin(e[on])]
    assert _d2_f64(q, a[None])[0] > _d2_f64(q, b[None])[0]
    return a, b


def _check(xyz, k):
    xyz = np.ascontiguousarray(xyz, dtype=F)
    idx = L.sf_build_index(torch.from_numpy(xyz).cuda())
    try:
        L.sf_bandwidths(idx, L.make_params(k=k))
        h = torch.empty(len(xyz), device="cuda")
        L.sf_get_bandwidths(idx, h)
        nbr = torch.empty((len(xyz), k), dtype=torch.int32, device="cuda")
        h2 = torch.empty_like(h)
        L.sf_knn_neighbours(idx, k, nbr, h2)
        torch.cuda.synchronize()
    finally:
        L.sf_free_index(idx)
    ref = np.asarray(oracle.knn(xyz, k)[0], dtype=F)
    assert np.array_equal(h.cpu().numpy().view(np.uint32), ref.view(np.uint32))
    assert np.array_equal(h2.cpu().numpy().view(np.uint32), ref.view(np.uint32))
    far = np.stack([np.sort(_d2_f64(xyz[i], xyz[nbr[i].cpu().numpy()]))[-1] for i in range(0, len(xyz), 97)])
    assert np.array_equal(np.sqrt(far).astype(F), ref[::97])


@pytest.mark.parametrize("k", [1, 2, 8, 33, 64, 70, 200])
@pytest.mark.parametrize("edge", [1.0, 1.25, 1.5, 1.75, 0.0625, 1.0625, 1.4375, 1.00390625])
@pytest.mark.parametrize("shell", [0, 500])
def test_order_across_a_bin_edge(k, edge, shell):
    r = np.random.default_rng(1000 * k + int(256 * edge) + shell)
    for q in (np.zeros(3, F), np.array([0.3137, 0.2719, 0.4141], F)):
        a, b = _swapped(q, edge, r)
        u = r.standard_normal((k + shell, 3))
        u /= np.linalg.norm(u, axis=1)[:, None]
        rad = np.sqrt(edge) * np.concatenate([r.uniform(0.1, 0.6, k - 1), r.uniform(1.01, 1.3, shell), [1.5]])
        xyz = np.concatenate([[q, a, b], (q + u * rad[:, None]).astype(F)]).astype(F)
        xyz = np.ascontiguousarray(xyz[r.permutation(len(xyz))])
        _check(xyz, k)


SCALES = {
    # one point so far out that a scale chosen for it would push the others' squares to zero
    "outlier": lambda r, n: np.concatenate([r.random((n - 1, 3)), [[1e30, 0.0, 0.0]]]),
    "sentinel": lambda r, n: np.concatenate([r.random((n - 1, 3)), [[3e38, 3e38, 3e38]]]),
    "close_pairs": lambda r, n: np.concatenate([1e-12 * r.random((n - 1, 3)), [[1e38, 0.0, 0.0]]]),
    # one axis far from zero against the others' extent: a scale for the extent would overflow it
    "plane": lambda r, n: np.concatenate([2.0 ** -100 * r.random((n, 2)), np.full((n, 1), 2.0)], axis=1),
    "far_plane": lambda r, n: np.concatenate([1e-19 * r.random((n, 2)), np.full((n, 1), 1e30)], axis=1),
    # no scale helps: squares among the smallest floats
    "narrow": lambda r, n: np.concatenate([2.0 ** -64 * r.random((n, 2)), np.full((n, 1), 2.0 ** 126)], axis=1),
}


@pytest.mark.parametrize("cloud", sorted(SCALES))
@pytest.mark.parametrize("k", [1, 8, 64, 100])
def test_scales(cloud, k):
    r = np.random.default_rng(k)
    _check(SCALES[cloud](r, 1500)[r.permutation(1500)], k)


@pytest.mark.parametrize("k", [1, 8, 33, 64, 100])
@pytest.mark.parametrize("each", [2, 9, 40, 60, 150])
@pytest.mark.parametrize("apart", ["exact", "near", "lattice"])
def test_coinciding(each, k, apart):
    """Places that hold several points: the k-th at distance 0, among many at one distance, or
    (near) at distances whose squares FP32 cannot tell from 0."""
    r = np.random.default_rng(each + k)
    n = 3000
    at = r.integers(0, n // each, n)
    if apart == "lattice":
        p = np.stack([at % 7, at // 7 % 7, at // 49], axis=1) * 0.1
    else:
        p = r.random((n // each, 3))[at]
    if apart == "near":
        p[:, 2] = 1e-24 * r.integers(0, 3, n)
    _check(p, k)


@pytest.mark.parametrize("k", [1, 2, 8, 40, 100])
@pytest.mark.parametrize("heavy", [3, 20, 700, 5000])
def test_coinciding_among_close_neighbours(heavy, k):
    """Points at one place among others a rounding of the coordinates away (all within one cell
    of the index's order, so they do not follow one another in it): k-th distances of 0 and
    of one rounding, some at the place, some beside it with too few of their own."""
    r = np.random.default_rng(heavy + k)
    ulp = float(np.spacing(F(0.5)))
    around = 0.5 + ulp * r.integers(-3, 4, (600, 3))
    _check(np.concatenate([np.full((heavy, 3), 0.5), around, r.random((1500, 3))])[r.permutation(heavy + 2100)], k)
