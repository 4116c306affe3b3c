"""The framework's measured work: twelve cases through its public entry points.

A case is a dict of plain values. ``prepare`` makes, from the case and a seed
alone, what a user's program holds before the call (the cloud, the resident
index with its bandwidths, the batch plan, the output buffers); ``run`` makes
one pass of calls and returns every output whole; ``work`` states what such a
pass cannot do without; ``exact`` gives the outputs in 64 bits from torch alone.

Clouds: ``plain`` is the half-uniform, half-clustered unit cube of the 100k
workload, ``halo`` the hierarchically clustered cloud with NFW halos of the
large workloads. ROIs are boxes around the most massive halo (around the cube's
centre for plain clouds), moved inside the unit cube.
"""
import math

import torch
import torch.nn.functional as F

from paper_2601_20758_gb300 import _lib as L
from paper_2601_20758_gb300 import synth

KERNELS = {"gauss": L.SF_K_GAUSS3, "epan": L.SF_K_EPAN}
RULES = {"knn": L.SF_BW_KNN, "mbe": L.SF_BW_MBE, "fixed": L.SF_BW_FIXED}
SCOPES = {"global": L.SF_SCOPE_GLOBAL, "clip": L.SF_SCOPE_CLIP}
PRECS = {"fp32": L.SF_PREC_FP32, "tf32": L.SF_PREC_TF32, "bf16": L.SF_PREC_BF16}
MODES = {"direct": L.SF_POINTS_DIRECT, "interp": L.SF_POINTS_INTERP}

MILLION16 = 16_777_216
MILLION67 = 67_108_864


def listed():
    return [
        # A new small cloud: index and per-point bandwidths, before the first view
        # can be drawn (the 100k workload's size and k).
        {"name": "knn_100k", "kind": "knn", "cloud": "plain", "n": 100_000, "k": 32},
        # The same for the cosmology workload: the largest part of its step.
        {"name": "knn_16m", "kind": "knn", "cloud": "halo", "n": MILLION16, "k": 64},
        # One interactive recompute of the 100k workload: the 64^3 grid of the whole
        # cube and the density at every point.
        {"name": "step_100k", "kind": "step", "cloud": "plain", "n": 100_000, "k": 32, "edge": 1.0,
         "nx": 64, "ny": 64, "nz": 64, "kernel": "gauss", "scope": "global", "mode": "direct"},
        # The widest ROI of the cosmology workload's nested sequence: grid and point densities.
        {"name": "step_16m", "kind": "step", "cloud": "halo", "n": MILLION16, "k": 64, "edge": 1.0,
         "nx": 128, "ny": 128, "nz": 128, "kernel": "gauss", "scope": "global", "mode": "direct"},
        # A zoomed view of the large workload: supports of many node spacings.
        {"name": "grid_zoom_67m", "kind": "grid", "cloud": "halo", "n": MILLION67, "k": 64, "rule": "knn",
         "edge": 0.05, "nx": 256, "ny": 256, "nz": 256, "kernel": "gauss", "scope": "global", "prec": "fp32"},
        # The zoomed-out view of a large cloud: many particles per node, supports of
        # about a node spacing (a billion points at 256^3 are 64 to a node, here 32).
        {"name": "grid_cube_67m", "kind": "grid", "cloud": "halo", "n": MILLION67, "k": 64, "rule": "knn",
         "edge": 1.0, "nx": 128, "ny": 128, "nz": 128, "kernel": "gauss", "scope": "global", "prec": "fp32"},
        # Plain KDE with one smoothing length per axis over a ragged box, particles of
        # the box only: a user's own lengths with the Epanechnikov kernel.
        {"name": "grid_fixed_1m", "kind": "grid", "cloud": "plain", "n": 1_000_003, "k": 32, "rule": "fixed",
         "edge": 0.83, "nx": 97, "ny": 131, "nz": 61, "kernel": "epan", "scope": "clip", "prec": "fp32"},
        # A view of the serving stream that asks for the BF16 tensor-core grid.
        {"name": "grid_bf16_16m", "kind": "grid", "cloud": "halo", "n": MILLION16, "k": 64, "rule": "knn",
         "edge": 0.1, "nx": 192, "ny": 192, "nz": 192, "kernel": "gauss", "scope": "global", "prec": "bf16"},
        # The paper's own estimator on one ROI (percentile lengths, pilot, adaptive
        # lengths, final grid).
        {"name": "mbe_16m", "kind": "grid", "cloud": "halo", "n": MILLION16, "k": 64, "rule": "mbe",
         "edge": 0.37, "nx": 128, "ny": 128, "nz": 128, "kernel": "epan", "scope": "clip", "prec": "fp32"},
        # The batched workload: 64 uneven ROIs in one planned execution.
        {"name": "batch_16m", "kind": "batch", "cloud": "halo", "n": MILLION16, "k": 64, "rois": 64,
         "gmin": 32, "gmax": 256, "kernel": "gauss", "scope": "global"},
        # The selection of a view: the points above the 90th density percentile and
        # the surface of the volume they lie in.
        {"name": "select_4m", "kind": "select", "n": 4_194_304, "n_total": MILLION16, "percentile": 90.0,
         "nx": 192, "ny": 192, "nz": 192},
        # A small pan answered from the view cache: a finished grid read at new nodes.
        {"name": "resample_96", "kind": "resample", "sx": 128, "sy": 128, "sz": 128, "nx": 96, "ny": 96,
         "nz": 96, "edge": 0.75},
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _cloud_draw(rng, lo, hi):
    n = int(_log(rng, lo, hi))
    k = rng.choice([8, 16, 32, 33, 48, 64])
    return {"cloud": "plain" if n < 2_000_000 and rng.random() < 0.5 else "halo", "n": n, "k": k}


def _edge_draw(rng, n, lo):
    """A box edge that leaves a few hundred particles of a sparse cloud inside."""
    return _log(rng, max(lo, min(0.9, (2000.0 / n) ** (1.0 / 3.0))), 1.0)


def _dims_draw(rng, lo, hi):
    g = _log(rng, lo, hi)
    d = [max(lo, min(hi, int(g * rng.uniform(0.7, 1.4)))) for _ in range(3)]
    return {"nx": d[0], "ny": d[1], "nz": d[2]}


def draw(rng):
    kind = rng.choice(["knn", "step", "grid", "grid", "mbe", "batch", "select", "resample"])
    if kind == "knn":
        return {"kind": "knn", **_cloud_draw(rng, 20_000, MILLION16)}
    if kind == "step":
        cloud = _cloud_draw(rng, 50_000, MILLION16)
        return {"kind": "step", **cloud, "edge": _edge_draw(rng, cloud["n"], 0.1),
                **_dims_draw(rng, 24, 160), "kernel": rng.choice(["gauss", "gauss", "epan"]),
                "scope": rng.choice(["global", "global", "clip"]),
                "mode": rng.choice(["direct", "direct", "interp"])}
    if kind == "grid" and rng.random() < 0.2:
        return {"kind": "grid", "cloud": "plain", "n": int(_log(rng, 50_000, 2_000_000)), "k": 32,
                "rule": "fixed", "edge": rng.uniform(0.3, 1.0), **_dims_draw(rng, 32, 160),
                "kernel": rng.choice(["gauss", "epan"]), "scope": rng.choice(["global", "clip"]),
                "prec": "fp32"}
    if kind == "grid":
        kernel = rng.choice(["gauss", "gauss", "gauss", "epan"])
        cloud = _cloud_draw(rng, 100_000, MILLION67)
        return {"kind": "grid", **cloud, "rule": "knn",
                "edge": _edge_draw(rng, cloud["n"], 0.01), **_dims_draw(rng, 32, 256), "kernel": kernel,
                "scope": rng.choice(["global", "global", "clip"]),
                "prec": rng.choice(["fp32", "fp32", "tf32", "bf16"]) if kernel == "gauss" else "fp32"}
    if kind == "mbe":
        cloud = _cloud_draw(rng, 100_000, MILLION16)
        return {"kind": "grid", **cloud, "rule": "mbe",
                "edge": _edge_draw(rng, cloud["n"], 0.1), **_dims_draw(rng, 32, 128), "kernel": "epan",
                "scope": "clip", "prec": "fp32"}
    if kind == "batch":
        gmin = int(_log(rng, 24, 64))
        return {"kind": "batch", **_cloud_draw(rng, 200_000, MILLION16), "rois": int(_log(rng, 4, 64)),
                "gmin": gmin, "gmax": int(_log(rng, gmin + 1, 192)),
                "kernel": rng.choice(["gauss", "gauss", "epan"]), "scope": rng.choice(["global", "global", "clip"])}
    if kind == "select":
        n = int(_log(rng, 30_000, 8_000_000))
        return {"kind": "select", "n": n, "n_total": int(n * _log(rng, 1.0, 8.0)) + 1,
                "percentile": rng.uniform(75.0, 99.5), **_dims_draw(rng, 48, 224)}
    s = _dims_draw(rng, 48, 192)
    return {"kind": "resample", "sx": s["nx"], "sy": s["ny"], "sz": s["nz"], **_dims_draw(rng, 48, 256),
            "edge": rng.uniform(0.05, 1.0)}


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
class _Held:
    """An index (and a plan over it), released with the state that holds it."""

    def __init__(self, idx):
        self.idx, self.plan = idx, None

    def __del__(self):
        if self.plan is not None:
            L.sf_batch_free(self.plan)
        L.sf_free_index(self.idx)


def _cloud(case, seed):
    if case["cloud"] == "plain":
        return torch.from_numpy(synth.plain_cloud(case["n"], seed=1000 + seed)).cuda(), (0.5, 0.5, 0.5)
    xyz, centre = synth.large_cloud_device(case["n"], seed=1000 + seed)
    torch.cuda.empty_cache()  # the generator's temporaries back to the device
    return xyz, tuple(float(c) for c in centre)


def _box(centre, edge):
    lo = [min(max(c - edge / 2, 0.0), 1.0 - edge) for c in centre]
    return lo, [v + edge for v in lo]


def _dims(case):
    return case["nx"], case["ny"], case["nz"]


def _lengths(case):
    """The fixed lengths: a few node spacings, another on each axis (at least two mean
    distances between particles)."""
    most = 2.0 * case["n"] ** (-1.0 / 3.0)
    f = {"epan": (5.0, 6.0, 3.5), "gauss": (1.8, 2.2, 1.4)}[case["kernel"]]
    return tuple(max(f[i] * case["edge"] / (d - 1), most * (1.0 if case["kernel"] == "epan" else 0.4))
                 for i, d in enumerate(_dims(case)))


def _params(case):
    rule = case.get("rule", "knn")
    p = L.make_params(rule=RULES[rule], k=case["k"], scope=SCOPES[case.get("scope", "global")],
                      fixed_h=_lengths(case) if rule == "fixed" else (0.0, 0.0, 0.0))
    p.prec = PRECS[case.get("prec", "fp32")]
    return p


def _rois(case, xyz, seed):
    """Uneven boxes about points of the cloud, with grids of uneven edges."""
    at = torch.randint(case["n"], (case["rois"],), generator=torch.Generator().manual_seed(77 + seed))
    u = torch.rand((case["rois"], 4), generator=torch.Generator().manual_seed(77), dtype=torch.float64).tolist()
    centres = xyz[at.to(xyz.device)].double().tolist()
    boxes, dims = [], []
    for c, v in zip(centres, u):
        edge = math.exp(math.log(0.02) * v[0])
        boxes.append(_box(c, edge))
        e = case["gmin"] * (case["gmax"] / case["gmin"]) ** v[1]
        dims.append((int(e), max(2, int(e * (0.8 + 0.4 * v[2]))), max(2, int(e * (0.8 + 0.4 * v[3])))))
    return boxes, [tuple(min(case["gmax"], d) for d in dd) for dd in dims]


def _field(dims, g):
    """A smooth positive field over several decades (x fastest), as a density grid is."""
    coarse = [max(3, d // 32) for d in dims]
    r = torch.randn((1, 1, coarse[2], coarse[1], coarse[0]), generator=g, device="cuda")
    f = F.interpolate(r, size=(dims[2], dims[1], dims[0]), mode="trilinear", align_corners=True)
    return torch.exp(2.0 * f)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "resample":
        g = torch.Generator(device="cuda").manual_seed(31 + seed)
        src = (case["sx"], case["sy"], case["sz"])
        off = torch.rand(3, generator=torch.Generator().manual_seed(31 + seed), dtype=torch.float64).tolist()
        lo = [o * (1.0 - case["edge"]) for o in off]
        hi = [v + case["edge"] for v in lo]
        out = torch.empty(case["nx"] * case["ny"] * case["nz"], device="cuda")
        return {"kind": kind, "src": _field(src, g).reshape(-1), "src_dims": src, "dims": _dims(case),
                "src_box": L.make_box((0.0, 0.0, 0.0), (1.0, 1.0, 1.0)), "box": L.make_box(lo, hi),
                "roi": (lo, hi), "out": out}
    if kind == "select":
        g = torch.Generator(device="cuda").manual_seed(53 + seed)
        dims, n, total = _dims(case), case["n"], case["n_total"]
        grid = _field(dims, g)
        where = 2.0 * torch.rand((1, n, 1, 1, 3), generator=g, device="cuda") - 1.0
        dens = F.grid_sample(grid, where, align_corners=True).reshape(-1).contiguous()
        step = total / n  # ascending original indices, unevenly spread
        ids = ((torch.arange(n, device="cuda", dtype=torch.float64) +
                torch.rand(n, generator=g, device="cuda", dtype=torch.float64) * (1.0 - 1.0 / step)) * step)
        ids = torch.minimum(ids.long(), torch.tensor(total - 1, device="cuda")).to(torch.int32)
        nodes = dims[0] * dims[1] * dims[2]
        return {"kind": kind, "grid": grid.reshape(-1).contiguous(), "dims": dims, "dens": dens, "ids": ids,
                "n": n, "n_total": total, "percentile": case["percentile"],
                "box": L.make_box((0.1, 0.2, 0.3), (0.6, 0.7, 0.8)),
                "mask": torch.empty(total, dtype=torch.uint8, device="cuda"),
                "sel": torch.zeros(n, dtype=torch.int32, device="cuda"),
                "tris": torch.zeros((nodes // 2, 9), device="cuda")}
    xyz, centre = _cloud(case, seed)
    if kind == "knn":
        return {"kind": kind, "xyz": xyz, "params": _params(case), "h": torch.empty(case["n"], device="cuda")}
    held = _Held(L.sf_build_index(xyz))
    p = _params(case)
    L.sf_bandwidths(held.idx, p)
    state = {"kind": kind, "held": held, "idx": held.idx, "params": p, "kernel": KERNELS[case["kernel"]]}
    if kind == "batch":
        boxes, dims = _rois(case, xyz, seed)
        try:
            held.plan = L.sf_batch_create(held.idx, [L.make_box(*b) for b in boxes], dims, state["kernel"], p)
        finally:
            torch.cuda.synchronize()
        state["plan"] = held.plan
        state["outs"] = [torch.empty(d[0] * d[1] * d[2], device="cuda") for d in dims]
        return state
    roi = _box(centre, case["edge"])
    dims = _dims(case)
    state.update(box=L.make_box(*roi), dims=dims, grid=torch.empty(dims[0] * dims[1] * dims[2], device="cuda"))
    if kind == "step":
        q = L.sf_params.from_buffer_copy(p)
        q.points_mode = MODES[case["mode"]]
        state.update(points_params=q, dens=torch.zeros(case["n"], device="cuda"),
                     ids=torch.zeros(case["n"], dtype=torch.int32, device="cuda"))
    torch.cuda.synchronize()
    return state


# ---------------------------------------------------------------------------
# One pass
# ---------------------------------------------------------------------------
def run(state):
    kind = state["kind"]
    if kind == "knn":
        idx = L.sf_build_index(state["xyz"])
        try:
            L.sf_bandwidths(idx, state["params"])
            L.sf_get_bandwidths(idx, state["h"])
        finally:
            L.sf_free_index(idx)
        return {"h": state["h"]}
    if kind == "grid":
        L.sf_kde_grid(state["idx"], state["box"], state["dims"], state["kernel"], state["params"], state["grid"])
        return {"grid": state["grid"]}
    if kind == "step":
        L.sf_kde_grid(state["idx"], state["box"], state["dims"], state["kernel"], state["params"], state["grid"])
        n = L.sf_kde_points(state["idx"], state["box"], state["dims"], state["kernel"], state["points_params"],
                            state["dens"], state["ids"])
        return {"grid": state["grid"], "dens": state["dens"], "ids": state["ids"], "count": n}
    if kind == "batch":
        L.sf_batch_run(state["plan"], state["outs"])
        return {"grids": state["outs"]}
    if kind == "select":
        nsel, t = L.sf_select(None, state["dens"], state["ids"], state["n"], state["n_total"],
                              percentile=state["percentile"], d_mask=state["mask"], d_sel_ids=state["sel"])
        nt = L.sf_iso_surface(state["grid"], state["box"], state["dims"], t, state["tris"])
        return {"mask": state["mask"], "sel": state["sel"], "threshold": t, "tris": state["tris"], "counts": [nsel, nt]}
    L.sf_resample_grid(state["src"], state["src_box"], state["src_dims"], state["box"], state["dims"], state["out"])
    return {"out": state["out"]}


# ---------------------------------------------------------------------------
# What a pass cannot do without
# ---------------------------------------------------------------------------
def _pairs(case, outputs):
    """In-support pairs: a support that holds k neighbours within h holds about k (R/h)^3
    particles within R, so each output has that many terms; fixed lengths: the
    particles of the box in one support."""
    if case.get("rule") == "fixed":
        hx, hy, hz = _lengths(case)
        r = 3.0 if case["kernel"] == "gauss" else 1.0
        return outputs * case["n"] * min(1.0, 4.19 * r ** 3 * hx * hy * hz)
    if case.get("rule") == "mbe":
        return outputs * 300.0  # lengths of at most five node spacings
    return outputs * case["k"] * (27.0 if case["kernel"] == "gauss" else 1.0)


def work(case):
    kind = case["kind"]
    if kind == "knn":
        return {"bytes": 16.0 * case["n"], "flops": 8.0 * case["k"] * case["n"]}
    if kind == "resample":
        out = case["nx"] * case["ny"] * case["nz"]
        read = min(1.0, (case["edge"] + 0.02) ** 3) * case["sx"] * case["sy"] * case["sz"]
        return {"bytes": 4.0 * (out + read), "flops": 24.0 * out}
    if kind == "select":
        nodes = case["nx"] * case["ny"] * case["nz"]
        left = 1.0 - case["percentile"] / 100.0
        tris = 6.0 * nodes ** (2.0 / 3.0) * 4.0
        return {"bytes": case["n"] * (8.0 + 4.0 * left) + case["n_total"] + 4.0 * nodes + 36.0 * tris,
                "flops": 6.0 * nodes}
    if kind == "batch":
        mean = (case["gmax"] ** 3 - case["gmin"] ** 3) / (3.0 * math.log(case["gmax"] / case["gmin"]))
        nodes = case["rois"] * mean
        return {"bytes": 4.0 * nodes + 16.0 * case["n"], "flops": 13.0 * _pairs(case, nodes)}
    nodes = case["nx"] * case["ny"] * case["nz"]
    inside = case["n"] * case["edge"] ** 2  # the clouds are clustered about the ROI's centre
    w = {"bytes": 4.0 * nodes + 16.0 * inside, "flops": 13.0 * _pairs(case, nodes)}
    if kind == "step":
        w["bytes"] += 8.0 * inside
        w["flops"] += 13.0 * _pairs(case, inside) if case["mode"] == "direct" else 14.0 * inside
    return w


# ---------------------------------------------------------------------------
# 64-bit values
# ---------------------------------------------------------------------------
_P3 = math.erf(3.0 / math.sqrt(2.0)) - math.sqrt(2.0 / math.pi) * 3.0 * math.exp(-4.5)


def _exact_h(xyz, k):
    """Distance to the k-th nearest other point, rounded to float as the rule states."""
    x = xyz.double()
    out = []
    for a in x.split(2048):
        d2 = sum((a[:, i, None] - x[None, :, i]).square() for i in range(3))
        out.append(torch.topk(d2, k + 1, dim=1, largest=False, sorted=True).values[:, k])
    return torch.cat(out).sqrt().float()


def _exact_density(at, y, ell, kernel, neff):
    """Kernel sums at the positions ``at`` [m, 3] over the particles y [n, 3] with lengths
    ell [n, 3], pair by pair."""
    cut, norm = (9.0, 1.0 / ((2.0 * math.pi) ** 1.5 * _P3)) if kernel == "gauss" else (1.0, 15.0 / (8.0 * math.pi))
    c = norm / ell.prod(dim=1) / neff
    rl = 1.0 / ell
    out = []
    for a in at.split(max(1, (1 << 27) // max(1, y.shape[0]))):
        q = sum(((a[:, i, None] - y[None, :, i]) * rl[None, :, i]).square() for i in range(3))
        w = torch.exp(-0.5 * q) if kernel == "gauss" else 1.0 - q
        out.append((w.masked_fill_(q >= cut, 0.0) * c).sum(dim=1))
    return torch.cat(out)


def _axes(roi, dims):
    return [roi[0][i] + torch.arange(dims[i], device="cuda", dtype=torch.float64) *
            ((roi[1][i] - roi[0][i]) / (dims[i] - 1)) for i in range(3)]


def _nodes(roi, dims):
    z, y, x = torch.meshgrid(*reversed(_axes(roi, dims)), indexing="ij")
    return torch.stack([x.reshape(-1), y.reshape(-1), z.reshape(-1)], dim=1)


def _exact_window(roi, dims, y, h, kernel, neff):
    """The grid of one smoothing length per axis: every particle added to the nodes of
    its support's box (a window of the same size for all)."""
    cut, r, norm = (9.0, 3.0, 1.0 / ((2.0 * math.pi) ** 1.5 * _P3)) if kernel == "gauss" else (1.0, 1.0, 15.0 / (8.0 * math.pi))
    s = [(roi[1][i] - roi[0][i]) / (dims[i] - 1) for i in range(3)]
    first = torch.stack([torch.floor((y[:, i] - r * h[i] - roi[0][i]) / s[i]) for i in range(3)], dim=1).long()
    off = [torch.arange(int(2 * r * h[i] / s[i]) + 3, device="cuda") for i in range(3)]
    out = torch.zeros(dims[0] * dims[1] * dims[2], device="cuda", dtype=torch.float64)
    per = off[0].numel() * off[1].numel() * off[2].numel()
    for a in range(0, y.shape[0], max(1, (1 << 26) // per)):
        b = min(y.shape[0], a + max(1, (1 << 26) // per))
        node = [first[a:b, i, None] + off[i] for i in range(3)]
        q = [((roi[0][i] + node[i].double() * s[i] - y[a:b, i, None]) / h[i]).square() for i in range(3)]
        ok = [(node[i] >= 0) & (node[i] < dims[i]) for i in range(3)]
        qq = q[2][:, :, None, None] + q[1][:, None, :, None] + q[0][:, None, None, :]
        keep = (qq < cut) & ok[2][:, :, None, None] & ok[1][:, None, :, None] & ok[0][:, None, None, :]
        w = torch.exp(-0.5 * qq) if kernel == "gauss" else 1.0 - qq
        at = (node[2][:, :, None, None] * dims[1] + node[1][:, None, :, None]) * dims[0] + node[0][:, None, None, :]
        out.index_add_(0, at[keep], w[keep])
    return out * (norm / (h[0] * h[1] * h[2]) / neff)


def _trilinear(grid, roi, dims, at):
    """A grid (x fastest) read at positions inside its box."""
    f = grid.double().reshape(dims[2], dims[1], dims[0])
    cell, t = [], []
    for i in range(3):
        v = (at[:, i] - roi[0][i]) * (1.0 / ((roi[1][i] - roi[0][i]) / (dims[i] - 1)))
        c = v.floor().long().clamp(0, dims[i] - 2)
        cell.append(c)
        t.append(v - c)
    out = torch.zeros_like(at[:, 0])
    for dz in range(2):
        for dy in range(2):
            for dx in range(2):
                w = (t[0] if dx else 1 - t[0]) * (t[1] if dy else 1 - t[1]) * (t[2] if dz else 1 - t[2])
                out += w * f[cell[2] + dz, cell[1] + dy, cell[0] + dx]
    return out


def _exact_tris(grid, roi, dims, t):
    """The surface where the field, linear on the six tetrahedra about each cell's main
    diagonal, passes t: triangles by cell, tetrahedron and case, outward."""
    f = grid.double().reshape(dims[2], dims[1], dims[0])
    lo = torch.tensor(roi[0], device="cuda", dtype=torch.float64)
    s = torch.tensor([(roi[1][i] - roi[0][i]) / (dims[i] - 1) for i in range(3)], device="cuda", dtype=torch.float64)
    inside = f > t
    corner = [[0, 1, 3, 7], [0, 1, 5, 7], [0, 2, 3, 7], [0, 2, 6, 7], [0, 4, 5, 7], [0, 4, 6, 7]]

    def at(v, m):
        return v[m >> 2: dims[2] - 1 + (m >> 2), (m >> 1) & 1: dims[1] - 1 + ((m >> 1) & 1), m & 1: dims[0] - 1 + (m & 1)]

    keys, tris = [], []
    for o, cs in enumerate(corner):
        nin = sum(at(inside, m).int() for m in cs)
        iz, iy, ix = torch.nonzero((nin > 0) & (nin < 4), as_tuple=True)
        key = ((iz * (dims[1] - 1) + iy) * (dims[0] - 1) + ix) * 12 + 2 * o
        m = torch.tensor(cs, device="cuda")
        ijk = torch.stack([ix[:, None] + (m & 1), iy[:, None] + ((m >> 1) & 1), iz[:, None] + (m >> 2)], dim=2)
        P = lo + ijk.double() * s
        v = f[ijk[..., 2], ijk[..., 1], ijk[..., 0]]
        ins = v > t
        cnt = ins.sum(dim=1)
        cen = (P * ins[..., None]).sum(dim=1) / cnt[:, None]

        def cross(r, a, b):
            fa, fb = v[r, a], v[r, b]
            return P[r, a] + ((t - fa) / (fb - fa))[:, None] * (P[r, b] - P[r, a])

        def put(r, k, tri):
            n = torch.linalg.cross(tri[:, 1] - tri[:, 0], tri[:, 2] - tri[:, 0])
            flip = (n * (tri[:, 0] - cen[r])).sum(dim=1) < 0
            tri = torch.where(flip[:, None, None], tri[:, [0, 2, 1]], tri)
            keys.append(k)
            tris.append(tri)

        rows = torch.arange(cnt.numel(), device="cuda")
        r = rows[cnt != 2]
        lone = (ins[r] == (cnt[r] == 1)[:, None]).int().argmax(dim=1)
        rest = torch.tensor([[1, 2, 3], [0, 2, 3], [0, 1, 3], [0, 1, 2]], device="cuda")[lone]
        put(r, key[r], torch.stack([cross(r, lone, rest[:, j]) for j in range(3)], dim=1))
        r = rows[cnt == 2]
        order = torch.argsort((~ins[r]).int(), dim=1, stable=True)  # inside corners first, each in order
        a, b, c, d = (order[:, j] for j in range(4))
        put(r, key[r], torch.stack([cross(r, a, c), cross(r, a, d), cross(r, b, d)], dim=1))
        put(r, key[r] + 1, torch.stack([cross(r, a, c), cross(r, b, d), cross(r, b, c)], dim=1))
    return torch.cat(tris)[torch.argsort(torch.cat(keys))].reshape(-1, 9)


def _fill(v, rows):
    """As the call leaves a buffer of that many rows: zeros after the last row written."""
    out = torch.zeros((rows,) + tuple(v.shape[1:]), dtype=v.dtype, device=v.device)
    out[:v.shape[0]] = v
    return out


def exact(case, seed):
    kind = case["kind"]
    if kind == "resample":
        st = prepare(case, seed)
        at = _nodes(st["roi"], st["dims"])
        return {"out": _trilinear(st["src"], ((0.0,) * 3, (1.0,) * 3), st["src_dims"], at)}
    if kind == "select":
        st = prepare(case, seed)
        rank = min(max(1, math.ceil(case["percentile"] / 100.0 * case["n"])), case["n"])
        t = float(torch.sort(st["dens"]).values[rank - 1])
        keep = st["dens"] > t
        mask = torch.zeros(case["n_total"], dtype=torch.uint8, device="cuda")
        mask[st["ids"][keep].long()] = 1
        tris = _exact_tris(st["grid"], ((0.1, 0.2, 0.3), (0.6, 0.7, 0.8)), st["dims"], t)
        counts = [int(keep.sum()), tris.shape[0]]
        return {"mask": mask, "sel": _fill(st["ids"][keep], case["n"]), "threshold": t,
                "tris": _fill(tris, st["tris"].shape[0]), "counts": counts}
    if kind == "batch" or case["n"] > 2_100_000:
        return None
    if kind == "knn":
        return {"h": _exact_h(_cloud(case, seed)[0], case["k"]).double()} if case["n"] <= 200_000 else None
    dims, roi, kernel = _dims(case), None, case["kernel"]
    nodes = dims[0] * dims[1] * dims[2]
    rule = case.get("rule", "knn")
    fp32 = case.get("prec", "fp32") == "fp32"
    if rule != "fixed" and (not fp32 or case["n"] > 200_000 or case["n"] * nodes > 4e10):
        return None
    xyz, centre = _cloud(case, seed)
    roi = _box(centre, case["edge"])
    x = xyz.double()
    lo, hi = (torch.tensor(v, device="cuda", dtype=torch.float64) for v in roi)
    inb = ((x >= lo) & (x <= hi)).all(dim=1)
    member = inb if case["scope"] == "clip" else torch.ones_like(inb)
    y, neff = x[member], float(member.sum())
    if rule == "fixed":
        return {"grid": _exact_window(roi, dims, y, _lengths(case), kernel, neff)}
    at = _nodes(roi, dims)
    if rule == "mbe":
        nb = y.shape[0]
        spread = torch.sort(y, dim=0).values
        pct = []
        for q in (0.2, 0.8):
            pos = q * (nb - 1)
            i = int(math.floor(pos))
            pct.append(spread[i] + (pos - i) * (spread[min(i + 1, nb - 1)] - spread[i]))
        ell = 2.0 * (pct[1] - pct[0]) / math.log(nb)
        pilot = _exact_density(at, y, ell.expand(nb, 3), kernel, neff)
        pden = _trilinear(pilot, roi, dims, y)
        cap = torch.tensor([5.0 * (roi[1][i] - roi[0][i]) / (dims[i] - 1) for i in range(3)], device="cuda",
                           dtype=torch.float64)
        each = torch.minimum(ell * (pden.mean() / pden).pow(1.0 / 3.0)[:, None], cap)
        return {"grid": _exact_density(at, y, each, kernel, neff)}
    h = _exact_h(xyz, case["k"]).double()
    ell = h[member][:, None].expand(-1, 3)
    grid = _exact_density(at, y, ell, kernel, neff)
    if kind == "grid":
        return {"grid": grid}
    pts = x[inb]
    dens = _exact_density(pts, y, ell, kernel, neff) if case["mode"] == "direct" else _trilinear(grid, roi, dims, pts)
    return {"grid": grid, "dens": _fill(dens, case["n"]), "ids": _fill(torch.nonzero(inb)[:, 0].int(), case["n"]),
            "count": pts.shape[0]}
