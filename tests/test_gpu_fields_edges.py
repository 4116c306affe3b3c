"""sf_resample_grid and sf_iso_surface at the edges of their kernels: ragged and smallest
grids, nodes on the source box's faces, values that leave the range of the fast paths
(negative, tiny, huge, infinite, NaN, zero), weights and thresholds out of the ordinary."""
from fractions import Fraction

import numpy as np
import pytest
import torch

import oracle
from paper_2601_20758_gb300 import _lib as L

pytestmark = pytest.mark.gpu

FIELDS = {
    "density": lambda r, n: np.exp(4.0 * r.standard_normal(n)),
    "signed": lambda r, n: r.standard_normal(n),
    "tiny": lambda r, n: np.exp(2.0 * r.standard_normal(n)) * 1e-36,
    "huge": lambda r, n: r.random(n) * 3e38,
    "zeros": lambda r, n: np.where(r.random(n) < 0.7, 0.0, r.random(n)),
    "special": lambda r, n: np.where(r.random(n) < 0.02, np.inf, np.where(r.random(n) < 0.02, np.nan, r.random(n))),
}


def _trilinear(src, box, dims, dst_box, dst_dims, weight):
    f = src.astype(np.float64).reshape(dims[2], dims[1], dims[0])
    cell, u, inside = [], [], []
    for k in range(3):
        lo, hi = box[0][k], box[1][k]
        s = (hi - lo) / (dims[k] - 1)
        r = dst_box[0][k] + np.arange(dst_dims[k]) * ((dst_box[1][k] - dst_box[0][k]) / (dst_dims[k] - 1))
        v = (r - lo) * (1.0 / s)
        c = np.clip(np.floor(v).astype(int), 0, dims[k] - 2)
        cell.append(c)
        u.append(v - c)
        inside.append((r >= lo) & (r <= hi))
    out = np.zeros((dst_dims[2], dst_dims[1], dst_dims[0]))
    mag = np.zeros_like(out)
    with np.errstate(all="ignore"):
        for dz in range(2):
            for dy in range(2):
                for dx in range(2):
                    w = (np.where(dz, u[2], 1 - u[2])[:, None, None] * np.where(dy, u[1], 1 - u[1])[None, :, None] *
                         np.where(dx, u[0], 1 - u[0])[None, None, :])
                    g = f[np.ix_(cell[2] + dz, cell[1] + dy, cell[0] + dx)]
                    out += w * g
                    mag += np.abs(w * g)
    ok = inside[2][:, None, None] & inside[1][None, :, None] & inside[0][None, None, :]
    return np.where(ok, weight * out, 0.0).ravel(), np.where(ok, abs(weight) * mag, 0.0).ravel(), int((~ok).sum())


@pytest.mark.parametrize("field", sorted(FIELDS))
@pytest.mark.parametrize("dims,dst,weight", [((2, 2, 2), (2, 2, 2), 1.0), ((7, 5, 9), (33, 9, 17), 1.0),
                                             ((40, 33, 21), (31, 65, 8), -0.37), ((16, 16, 16), (64, 3, 70), 0.0),
                                             ((5, 64, 3), (100, 7, 9), 2e3)])
def test_resample_edges(field, dims, dst, weight):
    r = np.random.default_rng(hash((dims, dst)) % 1000)
    src = FIELDS[field](r, dims[0] * dims[1] * dims[2]).astype(np.float32)
    box = ((-1.0, 0.25, 3.0), (2.0, 0.75, 11.0))
    for dst_box in (box, ((-0.5, 0.3, 2.0), (2.5, 0.7, 9.0))):
        out = torch.full((dst[0] * dst[1] * dst[2],), 7.0, device="cuda")
        n_out = L.sf_resample_grid(torch.from_numpy(src).cuda(), L.make_box(*box), dims, L.make_box(*dst_box), dst,
                                   out, weight=weight, want_outside=True)
        got = out.cpu().numpy()
        weight32 = float(np.float32(weight))
        ref, mag, ref_out = _trilinear(src, box, dims, dst_box, dst, weight32)
        assert n_out == ref_out
        ref32 = ref.astype(np.float32)
        fin = np.isfinite(ref32) & np.isfinite(mag)
        # one rounding to float, of a sum good to 2^-40 of its terms (node positions: 2^-48)
        tol = np.abs(ref) * 2.0 ** -23.9 + mag * 2.0 ** -40 + 2e-45
        assert np.all(np.abs(got.astype(np.float64) - ref)[fin] <= tol[fin])
        assert np.array_equal(np.isnan(got), np.isnan(ref32))
        inf = np.isinf(ref32)
        near_max = np.abs(ref) > 3.4028e38  # on either side of the largest float by its rounding
        assert np.array_equal(got[inf & ~near_max], ref32[inf & ~near_max])


def test_resample_negative_weight_gives_negative_zero():
    # zero times a negative weight is -0, inside the box and outside
    out = torch.full((4 * 4 * 4,), 7.0, device="cuda")
    n_out = L.sf_resample_grid(torch.zeros(27, device="cuda"), L.make_box((0, 0, 0), (1, 1, 1)), (3, 3, 3),
                               L.make_box((0, 0, 0), (1.5, 1, 1)), (4, 4, 4), out, weight=-2.0, want_outside=True)
    got = out.cpu().numpy()
    assert n_out == 16 and not got.any() and np.signbit(got).all()


@pytest.mark.parametrize("dims", [(2, 2, 2), (3, 2, 40), (33, 2, 2), (17, 33, 9), (130, 5, 4), (64, 64, 3)])
@pytest.mark.parametrize("t", [0.5, 0.97, 0.0, -1e300, 1e300, float(np.float32(0.25)), 0.25 + 2.0 ** -40])
def test_iso_edges(dims, t):
    r = np.random.default_rng(dims[0])
    grid = r.random(dims[0] * dims[1] * dims[2]).astype(np.float32)
    grid[r.random(grid.size) < 0.05] = np.float32(0.25)  # values on a threshold
    box = ((0.0, -1.0, 5.0), (2.0, 1.5, 5.5))
    ref = np.asarray(oracle.iso_surface(grid, box, dims, t), dtype=np.float64).reshape(-1, 9)
    d = torch.from_numpy(grid).cuda()
    assert L.sf_iso_surface(d, L.make_box(*box), dims, t) == ref.shape[0]
    tris = torch.full((max(1, ref.shape[0]) + 1, 9), -7.0, device="cuda")
    assert L.sf_iso_surface(d, L.make_box(*box), dims, t, tris) == ref.shape[0]
    got = tris.cpu().numpy()
    assert np.all(got[ref.shape[0]:] == -7.0)
    assert np.allclose(got[:ref.shape[0]], ref, rtol=2.0 ** -22, atol=1e-6)
    if ref.shape[0] > 1:
        short = torch.zeros((ref.shape[0] - 1, 9), device="cuda")
        with pytest.raises(L.SFError):
            L.sf_iso_surface(d, L.make_box(*box), dims, t, short)
        assert not short.any()


@pytest.mark.parametrize("dims", [(131, 127, 83), (3, 700, 900), (1100, 2, 1200)])
def test_iso_large_grid_is_its_slabs(dims):
    """A grid large enough for the longer steps of a warp against slabs of it, which take single
    ones (and which test_iso_edges compares with the oracle): the same triangles in order, up
    to the rounding of the slabs' node coordinates."""
    g = torch.Generator(device="cuda").manual_seed(dims[0])
    f = torch.rand(dims[::-1], generator=g, device="cuda")
    cap = 12 * (dims[0] - 1) * (dims[1] - 1) * (dims[2] - 1)
    t, tris = 0.97, torch.zeros((cap // 4, 9), device="cuda")
    n = L.sf_iso_surface(f.reshape(-1), L.make_box((0, 0, 0), tuple(float(d - 1) for d in dims)), dims, t, tris)
    at = 0
    for z in range(0, dims[2] - 1, 21):
        m = min(22, dims[2] - z)
        part = torch.zeros((cap // 4, 9), device="cuda")
        c = L.sf_iso_surface(f[z:z + m].reshape(-1).contiguous(),
                             L.make_box((0, 0, z), (float(dims[0] - 1), float(dims[1] - 1), float(z + m - 1))),
                             (dims[0], dims[1], m), t, part)
        assert torch.allclose(tris[at:at + c], part[:c], rtol=2.0 ** -22, atol=0.0)
        at += c
    assert at == n > 10_000 and not tris[n:].any()


def test_iso_with_infinities():
    grid = np.array([0.0, 1.0, np.inf, -np.inf, 0.0, 1.0, np.nan, 2.0], dtype=np.float32)
    n = L.sf_iso_surface(torch.from_numpy(grid).cuda(), L.make_box((0, 0, 0), (1, 1, 1)), (2, 2, 2), 0.5)
    inside = grid > 0.5
    corner = [[0, 1, 3, 7], [0, 1, 5, 7], [0, 2, 3, 7], [0, 2, 6, 7], [0, 4, 5, 7], [0, 4, 6, 7]]
    assert n == sum({0: 0, 4: 0, 2: 2}.get(int(inside[c].sum()), 1) for c in corner)


@pytest.mark.parametrize("dst,weight", [((400, 400, 400), 1.0), ((512, 256, 192), 0.7), ((2, 1000, 3000), 1.0),
                                        ((3, 1001, 2000), -3.3), ((17, 900, 700), 1.0)])
def test_resample_is_the_fp64_sum_rounded_once(dst, weight):
    """Every node is the FP64 sum (one fused step a neighbour) rounded to float. Where the
    interval of 2^-43 around it rounds to one float that one; the others are summed again in
    rationals, rounded to FP64 at each step."""
    g = torch.Generator(device="cuda").manual_seed(7)
    dims, box = (61, 67, 59), ((0.0, -1.0, 2.0), (1.0, 1.0, 7.0))
    src = torch.exp(2.0 * torch.randn(dims[::-1], generator=g, device="cuda"))
    dst_box = ((0.0, -0.9, 2.1), (1.0, 1.0, 6.3))
    out = torch.empty(dst[::-1], device="cuda")
    L.sf_resample_grid(src.reshape(-1), L.make_box(*box), dims, L.make_box(*dst_box), dst, out, weight=weight)
    f, cell, u = src.double(), [], []
    for k in range(3):
        s = (box[1][k] - box[0][k]) / (dims[k] - 1)
        r = dst_box[0][k] + torch.arange(dst[k], device="cuda", dtype=torch.float64) * (
            (dst_box[1][k] - dst_box[0][k]) / (dst[k] - 1))
        v = (r - box[0][k]) * (1.0 / s)
        cell.append(v.floor().long().clamp(0, dims[k] - 2))
        u.append(v - cell[k])
    w32 = float(np.float32(weight))
    open_nodes = []
    for z in range(dst[2]):
        val = torch.zeros((dst[1], dst[0]), device="cuda", dtype=torch.float64)
        for dz in range(2):
            plane, wz = f[cell[2][z] + dz], (u[2][z] if dz else 1 - u[2][z])
            for dy in range(2):
                for dx in range(2):
                    w = (u[0] if dx else 1 - u[0])[None, :] * (u[1] if dy else 1 - u[1])[:, None] * wz
                    val += w * plane[cell[1] + dy][:, cell[0] + dx]
        val *= w32
        lo, hi = (val * (1 - 2.0 ** -43)).float(), (val * (1 + 2.0 ** -43)).float()
        assert bool(((out[z] == lo) | (lo != hi)).all())
        open_nodes += [(z, int(y), int(x)) for y, x in torch.nonzero(lo != hi).tolist()]
    assert dst[0] < 400 or len(open_nodes) > 20
    fc, uc, cc = src.cpu().numpy(), [a.cpu().tolist() for a in u], [a.cpu().tolist() for a in cell]
    for z, y, x in open_nodes:
        val = 0.0
        for t in range(8):
            dx, dy, dz = t & 1, t >> 1 & 1, t >> 2
            w = (uc[0][x] if dx else 1.0 - uc[0][x]) * (uc[1][y] if dy else 1.0 - uc[1][y])
            w *= uc[2][z] if dz else 1.0 - uc[2][z]
            val = float(Fraction(w) * Fraction(float(fc[cc[2][z] + dz, cc[1][y] + dy, cc[0][x] + dx])) + Fraction(val))
        assert float(out[z, y, x]) == float(np.float32(w32 * val)), (z, y, x)


def test_resample_weight_of_negative_zero():
    out = torch.full((4 * 4 * 4,), 7.0, device="cuda")
    L.sf_resample_grid(torch.ones(27, device="cuda"), L.make_box((0, 0, 0), (1, 1, 1)), (3, 3, 3),
                       L.make_box((0, 0, 0), (1, 1, 1)), (4, 4, 4), out, weight=-0.0)
    got = out.cpu().numpy()
    assert not got.any() and np.signbit(got).all()


@pytest.mark.parametrize("field", ["density", "signed"])
@pytest.mark.parametrize("dst", [(33, 40, 21), (5, 300, 9), (7, 33, 2), (9, 64, 64), (17, 130, 40), (97, 61, 3),
                                 (65, 200, 120), (2, 129, 17), (4096, 2, 2)])
def test_resample_block_shapes(field, dst):
    """Grids on either side of the rules that shape a block: narrow, just wider than a warp's 8 or
    32 nodes, few columns, few nodes in z."""
    test_resample_edges(field, (19, 23, 29), dst, 1.0)
