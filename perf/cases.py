"""The framework's measured workloads: what a user has it compute, through its
public entry points, from the smallest call to the largest.

Inputs are seeded AIS-like fixes made on the GPU with the recipe of the
`workloads` package (vessels on waypoint lanes at 5-20 kn with a fix every
10 s, port clusters, a uniform background), as absolute projected metres with
a large false origin or as (lon, lat) degrees.  A case names its kind:

  density   one density on a grid (grid): every kernel and path a user selects
  batch     many densities of different sizes in one call (grid_batched)
  fit       one step of the bandwidth fit: the density, its LSCV loss with the
            loss's cotangent and direct partials, and the density's adjoint
            (grid, lscv_grid, grid_backward: the calls of autograd.lscv_loss)
  backward  the adjoint of a density for a given cotangent (grid_backward)
  binned    the paper's count-matrix estimator (grid_binned)
  simplify  Douglas-Peucker compression of the trajectories (dp_simplify)
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2004_13653_gb300 as kde

FALSE_ORIGIN = (13_545_000.0, 3_652_000.0)  # magnitude of projected coordinates, metres
REF_LON, REF_LAT = 121.68185, 31.3456       # centre of the (lon, lat) box, degrees
EARTH_RADIUS = 6371008.8
WGS84_A, WGS84_E2 = 6378137.0, 0.00669437999014
KNOT = 1852.0 / 3600.0
GAUSS_REACH = 6.0       # bandwidths beyond which a Gaussian term is below 2^-24 of its peak
EXACT_REACH = 10.0      # bandwidths beyond which it is below 2^-72: nothing in 64 bits
EXACT_FLOPS = 6e12      # matrix work of exact() that stays within seconds in FP64

KERNELS = ("uniform", "triangular", "epanechnikov", "quartic", "triweight", "tricube", "cosine")


def listed():
    return [
        # a quick look at a few vessels: 2,000 fixes on a 64 x 64 grid; latency and launches
        dict(name="gauss_2k_64sq", kind="density", kernel="gaussian", path="auto", n=2_000, nx=64,
             ny=64, box=20_000.0, h=200.0, mix="lanes", weighted=False, lonlat=False),
        # one region's day of lane traffic on the usual 1024 x 1024 grid
        dict(name="gauss_1m_1024sq", kind="density", kernel="gaussian", path="auto", n=1_000_000,
             nx=1024, ny=1024, box=50_000.0, h=150.0, mix="lanes", weighted=False, lonlat=False),
        # the flagship: 20M raw (lon, lat) fixes, projected in the call, on 4096 x 4096
        dict(name="gauss_20m_4096sq_lonlat", kind="density", kernel="gaussian", path="auto",
             n=20_000_000, nx=4096, ny=4096, box=100_000.0, h=100.0, mix="mixture",
             weighted=False, lonlat=True),
        # a smooth overview map: weighted fixes, a bandwidth of tens of cells, a ragged grid
        dict(name="gauss_wide_300k_777x1111", kind="density", kernel="gaussian", path="auto",
             n=300_007, nx=777, ny=1111, box=40_000.0, h=2000.0, mix="mixture", weighted=True,
             lonlat=False),
        # the same lane traffic with a compact kernel over a few cells
        dict(name="epan_1m_1024sq", kind="density", kernel="epanechnikov", path="auto",
             n=1_000_000, nx=1024, ny=1024, box=50_000.0, h=150.0, mix="lanes", weighted=False,
             lonlat=False),
        # a compact kernel over a wide support, weighted, ragged grid
        dict(name="quartic_wide_1m_1000x900", kind="density", kernel="quartic", path="auto",
             n=1_000_003, nx=1000, ny=900, box=50_000.0, h=2000.0, mix="mixture", weighted=True,
             lonlat=False),
        # the FP32 path, for callers who want FP32 factors and sums throughout
        dict(name="simt_gauss_1m_512sq", kind="density", kernel="gaussian", path="simt",
             n=1_000_000, nx=512, ny=512, box=50_000.0, h=300.0, mix="lanes", weighted=True,
             lonlat=False),
        # 24 regions of mixed size, Gaussian and Epanechnikov, in one call
        dict(name="batch_24", kind="batch", count=24, n_lo=10_000, n_hi=2_000_000, side_lo=7,
             side_hi=11, layout=7),
        # one step of the bandwidth fit on thinned lane traffic
        dict(name="fit_1470k_1024sq", kind="fit", n=1_470_000, nx=1024, ny=1024, box=50_000.0,
             h=150.0),
        # gradients of a smooth map for a cotangent from elsewhere
        dict(name="backward_wide_500k_1024sq", kind="backward", n=500_000, nx=1024, ny=1024,
             box=50_000.0, h=800.0, mix="lanes"),
        # the paper's own estimator on the flagship's fixes, gaps interpolated
        dict(name="binned_20m_4096sq", kind="binned", kernel="gaussian", n=20_000_000, nx=4096,
             ny=4096, box=100_000.0, h=100.0, fixes=500, mix="mixture"),
        # thinning 4,000 tracks of 500 fixes at 10 m before anything else
        dict(name="simplify_2m_eps10", kind="simplify", n=2_000_000, box=50_000.0, fixes=500,
             eps=10.0),
    ]


def draw(rng):
    def log_between(a, b):
        return math.exp(rng.uniform(math.log(a), math.log(b)))

    def sides(a, b):
        nx, ny = int(log_between(a, b)), int(log_between(a, b))
        if rng.random() < 0.4:  # the square powers of two most users take
            nx = ny = 2 ** round(math.log2(nx))
        return nx, ny

    kind = rng.choice(["density"] * 5 + ["batch", "fit", "backward", "binned", "simplify"])
    mix = rng.choice(["lanes", "mixture"])
    box = log_between(10_000.0, 100_000.0)
    if kind == "batch":
        return dict(kind=kind, count=rng.randint(2, 24), n_lo=10_000, n_hi=2_000_000, side_lo=7,
                    side_hi=11, layout=rng.randrange(1 << 20))
    if kind == "simplify":
        return dict(kind=kind, n=int(log_between(5e3, 2e6)), box=box,
                    fixes=int(log_between(40, 6000)), eps=log_between(1.0, 200.0))
    if kind == "binned":
        nx, ny = sides(128, 4096)
        return dict(kind=kind, kernel=rng.choice(KERNELS + ("gaussian",)),
                    n=int(log_between(1e4, 2e7)), nx=nx, ny=ny, box=box,
                    h=box / max(nx, ny) * log_between(2.0, 10.0), fixes=int(log_between(50, 2000)),
                    mix=mix)
    if kind == "fit":
        nx, ny = sides(128, 1024)
        return dict(kind=kind, n=int(log_between(2e4, 1.47e6)), nx=nx, ny=ny, box=box,
                    h=box / max(nx, ny) * log_between(1.0, 5.0))
    if kind == "backward":
        nx, ny = sides(128, 1024)
        return dict(kind=kind, n=int(log_between(1e4, 1e6)), nx=nx, ny=ny, box=box,
                    h=box / max(nx, ny) * log_between(1.0, 30.0), mix=mix)
    family = rng.choice(["gaussian", "gaussian", "compact", "compact", "radial", "simt"])
    nx, ny = sides(64, 4096)
    n = int(log_between(2e3, 2e7))
    cells = log_between(1.0, 60.0)
    if family == "simt":
        n = max(2000, min(n, int(1e12 / (nx * ny))))
    elif family != "gaussian":
        cells = min(cells, max(1.0, math.sqrt(2e10 / n) / 2))
    kernel = ("gaussian" if family == "gaussian" else
              rng.choice(KERNELS + ("gaussian",)) if family == "simt" else rng.choice(KERNELS))
    return dict(kind=kind, kernel="radial_" + kernel if family == "radial" else kernel,
                path="simt" if family == "simt" else "auto", n=n, nx=nx, ny=ny, box=box,
                h=box / max(nx, ny) * cells, mix=mix, weighted=rng.random() < 0.5,
                lonlat=rng.random() < 0.25)


# ------------------------------------------------------------------ inputs

def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _uniform(g, lo, hi, *shape):
    return torch.rand(*shape, dtype=torch.float64, device="cuda", generator=g) * (hi - lo) + lo


def _normal(g, sigma, *shape):
    return torch.randn(*shape, dtype=torch.float64, device="cuda", generator=g) * sigma


def _lanes(g, n, box, lanes, fixes=500):
    """n fixes of vessels on `lanes` waypoint chains, `fixes` in a row per vessel."""
    n_traj = max(1, -(-n // fixes))
    k = 6
    a = _uniform(g, 0.0, 2.0 * math.pi, lanes)
    d = torch.stack([a.cos(), a.sin()], -1)
    c = 0.5 * box + _uniform(g, -0.2, 0.2, lanes, 2) * box
    t = torch.linspace(-0.55, 0.55, k, dtype=torch.float64, device="cuda") * box
    perp = torch.stack([-d[:, 1], d[:, 0]], -1)
    way = c[:, None] + t[None, :, None] * d[:, None] + perp[:, None] * _normal(g, 0.08 * box, lanes, k, 1)
    way = way.clamp(0.02 * box, 0.98 * box)
    seg = way[:, 1:] - way[:, :-1]
    length = seg.norm(dim=-1)
    cum = torch.cat([torch.zeros_like(length[:, :1]), length.cumsum(1)], 1)
    lane = torch.randint(0, lanes, (n_traj,), device="cuda", generator=g)
    speed = _uniform(g, 5.0, 20.0, n_traj) * KNOT * 10.0
    turn = torch.where(torch.rand(n_traj, device="cuda", generator=g) < 0.5, -1.0, 1.0).double()
    s = _uniform(g, 0.0, 2.0 * box, n_traj)[:, None] + (turn * speed)[:, None] * torch.arange(
        fixes, dtype=torch.float64, device="cuda")
    total = cum[lane, -1][:, None]
    s = torch.remainder(s, 2.0 * total)
    s = torch.where(s > total, 2.0 * total - s, s)
    xy = torch.zeros(n_traj, fixes, 2, dtype=torch.float64, device="cuda")
    for q in range(k - 1):
        inside = (s >= cum[lane, q][:, None]) & ((s < cum[lane, q + 1][:, None]) | (q == k - 2))
        f = ((s - cum[lane, q][:, None]) / length[lane, q].clamp_min(1e-9)[:, None])[..., None]
        xy = torch.where(inside[..., None], way[lane, q][:, None] + f * seg[lane, q][:, None], xy)
    across = way[:, -1] - way[:, 0]
    across = torch.stack([-across[:, 1], across[:, 0]], -1) / across.norm(dim=-1, keepdim=True).clamp_min(1e-9)
    xy += (across[lane] * _normal(g, 60.0, n_traj, 1))[:, None]
    return (xy + _normal(g, 20.0, n_traj, fixes, 2)).reshape(-1, 2)[:n]


def _local(g, n, box, mix, fixes=500):
    """Local metres inside the box, and the number of leading fixes that form tracks."""
    if mix == "lanes":
        return _lanes(g, n, box, 8, fixes), n
    n_port, n_uni = n // 5, n // 10
    n_lane = n - n_port - n_uni
    ports = _uniform(g, 0.1 * box, 0.9 * box, 20, 2)
    at = torch.randint(0, 20, (n_port,), device="cuda", generator=g)
    return torch.cat([_lanes(g, n_lane, box, 12, fixes), ports[at] + _normal(g, 0.005 * box, n_port, 2),
                      _uniform(g, 0.0, box, n_uni, 2)]), n_lane


def _metres(local):
    return (local + torch.tensor(FALSE_ORIGIN, dtype=torch.float64, device="cuda")).contiguous()


def _offsets(n_track, n, fixes):
    """Trajectory bounds: tracks of `fixes`, then every other fix on its own."""
    tracks = torch.arange(0, n_track, fixes, dtype=torch.int64, device="cuda")
    return torch.cat([tracks, torch.arange(n_track, n + 1, dtype=torch.int64, device="cuda")])


def _weights(g, n, weighted):
    if weighted:
        return torch.rand(n, device="cuda", generator=g) * 1.5 + 0.5
    return torch.ones(n, device="cuda")


def _instances(case):
    """The geometry of a batch: part of the case, the same for every seed."""
    rng = np.random.default_rng(case["layout"])
    out = []
    for _ in range(case["count"]):
        n = int(math.exp(rng.uniform(math.log(case["n_lo"]), math.log(case["n_hi"]))))
        side = 2 ** int(rng.integers(case["side_lo"], case["side_hi"] + 1))
        out.append(dict(n=n, nx=side, ny=side, h=float(rng.uniform(50.0, 800.0)),
                        kernel="gaussian" if rng.random() < 0.5 else "epanechnikov",
                        box=float(rng.uniform(10_000.0, 100_000.0))))
    return out


def _cell(case):
    return case["box"] / max(case["nx"], case["ny"])


def prepare(case, seed):
    g = _generator(seed)
    kind = case["kind"]
    if kind == "batch":
        insts = []
        for c in _instances(case):
            xy, _ = _local(g, c["n"], c["box"], "mixture")
            insts.append(dict(points=_metres(xy), weights=_weights(g, c["n"], False),
                              origin=FALSE_ORIGIN, cell=_cell(c), nx=c["nx"], ny=c["ny"],
                              h=c["h"], kernel=c["kernel"]))
        return dict(kind=kind, insts=insts)
    n, box = case["n"], case["box"]
    if kind == "simplify":
        xy, n_track = _local(g, n, box, "lanes", case["fixes"])
        return dict(kind=kind, points=_metres(xy), offsets=_offsets(n_track, n, case["fixes"]),
                    eps=case["eps"])
    st = dict(kind=kind, nx=case["nx"], ny=case["ny"], cell=_cell(case), h=case["h"],
              origin=FALSE_ORIGIN)
    xy, n_track = _local(g, n, box, case.get("mix", "lanes"), case.get("fixes", 500))
    if kind == "binned":
        st.update(points=_metres(xy), offsets=_offsets(n_track, n, case["fixes"]),
                  kernel=case["kernel"])
    elif kind == "fit":
        # how many raw fixes each thinned one stands for, normalised as the fit does
        w = 1.0 + torch.rand(n, device="cuda", generator=g)
        st.update(points=_metres(xy), weights=w * (n / w.sum()))
    elif kind == "backward":
        st.update(points=_metres(xy), weights=_weights(g, n, True),
                  cotangent=torch.randn(case["ny"], case["nx"], device="cuda", generator=g))
    else:
        st.update(kernel=case["kernel"], path=case["path"], opts={},
                  weights=_weights(g, n, case["weighted"]))
        if case["lonlat"]:
            k_lat = 180.0 / (math.pi * EARTH_RADIUS)
            k_lon = k_lat / math.cos(math.radians(REF_LAT))
            scale = torch.tensor([k_lon, k_lat], dtype=torch.float64, device="cuda")
            corner = torch.tensor([[REF_LON - 0.5 * box * k_lon, REF_LAT - 0.5 * box * k_lat]],
                                  dtype=torch.float64, device="cuda")
            st["points"] = (xy * scale + corner).contiguous()
            st["origin"] = tuple(kde.project_mercator(corner, REF_LAT)[0].tolist())
            st["opts"] = dict(flags=kde.FLAG_LONLAT, lat0_deg=REF_LAT)
        else:
            st["points"] = _metres(xy)
    return st


def run(state):
    s, kind = state, state["kind"]
    if kind == "density":
        return kde.grid(s["points"], s["weights"], s["origin"], s["cell"], s["nx"], s["ny"], s["h"],
                        s["kernel"], path=s["path"], **s["opts"])
    if kind == "batch":
        return kde.grid_batched(s["insts"])
    if kind == "fit":
        at = (s["points"], s["weights"], s["origin"], s["cell"], s["nx"], s["ny"], s["h"])
        F = kde.grid(*at, "gaussian", path="tc_split16", flags=kde.FLAG_SKIP_ZERO)
        loss, G, w_direct, xy_direct, h_direct = kde.lscv_grid(F, *at)
        gxy, gw, gh = kde.grid_backward(*at, G)
        return {"density": F, "loss": loss, "cotangent": G,
                "direct": {"points": xy_direct, "weights": w_direct, "h": h_direct},
                "adjoint": {"points": gxy, "weights": gw, "h": gh}}
    if kind == "backward":
        gxy, gw, gh = kde.grid_backward(s["points"], s["weights"], s["origin"], s["cell"], s["nx"],
                                        s["ny"], s["h"], s["cotangent"])
        return {"points": gxy, "weights": gw, "h": gh}
    if kind == "binned":
        density, counts, _ = kde.grid_binned(s["points"], s["offsets"], s["origin"], s["cell"],
                                             s["nx"], s["ny"], s["h"], s["kernel"], count=False)
        return {"density": density, "counts": counts}
    keep, kept, kept_offsets, levels = kde.dp_simplify(s["points"], s["offsets"], s["eps"])
    # as many rows as there were fixes, zeros after the kept ones: a fixed shape for what follows
    kept = torch.nn.functional.pad(kept, (0, 0, 0, s["points"].shape[0] - kept.shape[0]))
    return {"keep": keep, "points": kept, "offsets": kept_offsets, "levels": levels}


# -------------------------------------------------------------------- work

def _window(case, reach_cells):
    """Cells of one point's support, at most the grid."""
    return (min(case["nx"], 2.0 * reach_cells + 1.0) * min(case["ny"], 2.0 * reach_cells + 1.0))


def _density_work(case):
    reach = GAUSS_REACH if case["kernel"] == "gaussian" else 1.0
    n, cells = case["n"], case["nx"] * case["ny"]
    # one multiply-add per point and cell within its support; two factors per
    # row and column are left out
    return {"bytes": 20.0 * n + 4.0 * cells,
            "flops": 2.0 * n * _window(case, reach * case["h"] / _cell(case))}


def work(case):
    kind = case["kind"]
    if kind == "density":
        return _density_work(case)
    if kind == "batch":
        parts = [_density_work(c) for c in _instances(case)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    n = case["n"]
    if kind == "simplify":
        # fixes in; the mask and about half of the fixes out; the cross product
        # (7 operations) of each fix at each of about log2(fixes) levels
        return {"bytes": 16.0 * n + n + 8.0 * n,
                "flops": 7.0 * n * max(1.0, math.log2(case["fixes"]))}
    cells = case["nx"] * case["ny"]
    if kind == "binned":
        a = min(127.0, (4.0 if case["kernel"] == "gaussian" else 1.0) * case["h"] / _cell(case))
        return {"bytes": 16.0 * n + 8.0 * cells, "flops": 4.0 * n + 4.0 * cells * (2.0 * a + 1.0)}
    window = _window(case, GAUSS_REACH * case["h"] / _cell(case))
    if kind == "backward":  # two products per cell of a point's support
        return {"bytes": 20.0 * n + 4.0 * cells + 12.0 * n, "flops": 4.0 * n * window}
    # the density, its adjoint, and the loss's own terms per point and cell
    return {"bytes": 20.0 * n + 24.0 * n + 8.0 * cells, "flops": 6.0 * n * window + 100.0 * n + 4.0 * cells}


# ------------------------------------------------------------------- exact

def _factor(kernel, s):
    """k(s) of a Table 1 kernel with its constant, FP64."""
    a = s.abs()
    if kernel == "gaussian":
        return torch.exp(-0.5 * s * s) / math.sqrt(2.0 * math.pi)
    v = {"uniform": lambda: torch.full_like(s, 0.5), "triangular": lambda: 1.0 - a,
         "epanechnikov": lambda: 0.75 * (1.0 - s * s),
         "quartic": lambda: 15.0 / 16.0 * (1.0 - s * s) ** 2,
         "triweight": lambda: 35.0 / 32.0 * (1.0 - s * s) ** 3,
         "tricube": lambda: 70.0 / 81.0 * (1.0 - a ** 3) ** 3,
         "cosine": lambda: math.pi / 4.0 * torch.cos(0.5 * math.pi * s)}[kernel]()
    return torch.where(a <= 1.0, v, torch.zeros_like(v))


def _radial_factor(kernel, r):
    """K of a radial kernel at radius r (in bandwidths), FP64."""
    c = {"uniform": 1.0 / math.pi, "triangular": 3.0 / math.pi, "epanechnikov": 2.0 / math.pi,
         "quartic": 3.0 / math.pi, "triweight": 4.0 / math.pi, "tricube": 220.0 / (81.0 * math.pi),
         "cosine": math.pi / (4.0 * math.pi - 8.0)}[kernel]
    v = {"uniform": lambda: torch.ones_like(r), "triangular": lambda: 1.0 - r,
         "epanechnikov": lambda: 1.0 - r * r, "quartic": lambda: (1.0 - r * r) ** 2,
         "triweight": lambda: (1.0 - r * r) ** 3, "tricube": lambda: (1.0 - r ** 3) ** 3,
         "cosine": lambda: torch.cos(0.5 * math.pi * r)}[kernel]()
    return torch.where(r <= 1.0, c * v, torch.zeros_like(v))


def _tiles(xy, nx, ny, cell, reach, side):
    """Groups of points by tile of `side` cells, each with the cells within its
    reach: (indices, first column, end, first row, end)."""
    lo = -reach - cell  # points beyond it reach no cell centre
    ok = (xy[:, 0] > lo) & (xy[:, 1] > lo) & (xy[:, 0] < nx * cell - lo) & (xy[:, 1] < ny * cell - lo)
    tx = (nx + side - 1) // side
    bx = (xy[:, 0] / (cell * side)).floor().clamp(0, tx - 1).long()
    by = (xy[:, 1] / (cell * side)).floor().clamp(0, (ny + side - 1) // side - 1).long()
    key = torch.where(ok, by * tx + bx, torch.full_like(bx, -1))
    key, order = key.sort()
    tiles, counts = key.unique_consecutive(return_counts=True)
    r, at = int(math.ceil(reach / cell)) + 2, 0
    for tile, count in zip(tiles.tolist(), counts.tolist()):
        if tile >= 0:
            i0, j0 = (tile % tx) * side, (tile // tx) * side
            for b in range(at, at + count, 65536):
                yield (order[b:min(b + 65536, at + count)], max(0, i0 - r), min(nx, i0 + side + r),
                       max(0, j0 - r), min(ny, j0 + side + r))
        at += count


def _tile_work(n, nx, ny, cell, reach, side):
    span = side + 2.0 * (reach / cell + 2.0)
    return 2.0 * n * min(nx, span) * min(ny, span)


def _centres(a, b, cell):
    return (torch.arange(a, b, dtype=torch.float64, device="cuda") + 0.5) * cell


def _exact_density(xy, w, nx, ny, cell, h, kernel):
    """The direct sum over points, FP64, on points relative to the grid's corner."""
    n = xy.shape[0]
    out = torch.zeros(ny, nx, dtype=torch.float64, device="cuda")
    if kernel.startswith("radial_"):
        reach = h
        if n * (16 + 2 * reach / cell + 4) ** 2 > 3e9:
            return None
        for at, i0, i1, j0, j1 in _tiles(xy, nx, ny, cell, reach, 16):
            for part in at.split(max(1, (1 << 26) // ((i1 - i0) * (j1 - j0)))):
                dx = (_centres(i0, i1, cell)[None] - xy[part, :1]) / h
                dy = (_centres(j0, j1, cell)[None] - xy[part, 1:]) / h
                r = (dx[:, None, :] ** 2 + dy[:, :, None] ** 2).sqrt()
                out[j0:j1, i0:i1] += (w[part][:, None, None] * _radial_factor(kernel[7:], r)).sum(0)
        return out / (n * h * h)
    reach = (EXACT_REACH if kernel == "gaussian" else 1.0) * h
    side = 256 if n > 100_000 else 1024
    if _tile_work(n, nx, ny, cell, reach, side) > EXACT_FLOPS:
        return None
    for at, i0, i1, j0, j1 in _tiles(xy, nx, ny, cell, reach, side):
        A = _factor(kernel, (_centres(i0, i1, cell)[None] - xy[at, :1]) / h)
        B = _factor(kernel, (_centres(j0, j1, cell)[None] - xy[at, 1:]) / h) * w[at][:, None]
        out[j0:j1, i0:i1] += B.T @ A
    return out / (n * h * h)


def _exact_adjoint(xy, w, cell, h, G):
    """Gradients of sum(G F) for the Gaussian density F: points, weights, h."""
    n, (ny, nx) = xy.shape[0], G.shape
    gxy, gw = torch.zeros_like(xy), torch.zeros_like(w)
    gh = torch.zeros((), dtype=torch.float64, device="cuda")
    c = 1.0 / (n * h * h)
    for at, i0, i1, j0, j1 in _tiles(xy, nx, ny, cell, EXACT_REACH * h, 256):
        s = (_centres(i0, i1, cell)[None] - xy[at, :1]) / h
        t = (_centres(j0, j1, cell)[None] - xy[at, 1:]) / h
        A, B, T = _factor("gaussian", s), _factor("gaussian", t), G[j0:j1, i0:i1]
        U, V = B @ T, A @ T.T  # over the rows, over the columns
        f = (A * U).sum(1)
        gw[at] = c * f
        gxy[at, 0] = c * w[at] / h * (s * A * U).sum(1)
        gxy[at, 1] = c * w[at] / h * (t * B * V).sum(1)
        q = (s * s * A * U).sum(1) + (t * t * B * V).sum(1)
        gh += (c * w[at] / h * (q - 2.0 * f)).sum()
    return gxy, gw, gh


def _exact_fit(xy, w, nx, ny, cell, h0):
    """The density, the grid LSCV loss, its partials and the adjoint, FP64."""
    n = xy.shape[0]
    F = _exact_density(xy, w, nx, ny, cell, h0, "gaussian").requires_grad_(True)
    xy, w = xy.clone().requires_grad_(True), w.clone().requires_grad_(True)
    h = torch.tensor(h0, dtype=torch.float64, device="cuda", requires_grad=True)
    f = xy / cell - 0.5
    i = f.detach().floor()
    a = f - i
    loo = torch.zeros_like(w)
    for q in (0, 1):
        for p in (0, 1):
            ii, jj = i[:, 0] + p, i[:, 1] + q
            ok = (ii >= 0) & (jj >= 0) & (ii < nx) & (jj < ny)
            at = (jj.clamp(0, ny - 1) * nx + ii.clamp(0, nx - 1)).long()
            ww = (a[:, 0] if p else 1.0 - a[:, 0]) * (a[:, 1] if q else 1.0 - a[:, 1])
            r2 = (((ii + 0.5) * cell - xy[:, 0]) ** 2 + ((jj + 0.5) * cell - xy[:, 1]) ** 2) / h ** 2
            own = w * torch.exp(-0.5 * r2) / (2.0 * math.pi * n * h * h)
            loo = loo + torch.where(ok, ww * (F.reshape(-1)[at] - own), torch.zeros_like(ww))
    loss = cell * cell * (F * F).sum() - 2.0 / n * (w * loo).sum()
    G, gxy, gw, gh = torch.autograd.grad(loss, (F, xy, w, h))
    axy, aw, ah = _exact_adjoint(xy.detach(), w.detach(), cell, h0, G)
    return {"density": F.detach(), "loss": loss.detach(), "cotangent": G,
            "direct": {"points": gxy, "weights": gw, "h": gh},
            "adjoint": {"points": axy, "weights": aw, "h": ah}}


def _exact_mercator(lonlat):
    """Eq. 1-4 at the standard latitude, FP64."""
    phi0, e = math.radians(REF_LAT), math.sqrt(WGS84_E2)
    r0 = WGS84_A * math.cos(phi0) / math.sqrt(1.0 - WGS84_E2 * math.sin(phi0) ** 2)
    phi = torch.deg2rad(lonlat[:, 1])
    es = e * torch.sin(phi)
    q = torch.log(torch.tan(0.25 * math.pi + 0.5 * phi)) + 0.5 * e * torch.log((1.0 - es) / (1.0 + es))
    return torch.stack([torch.deg2rad(lonlat[:, 0]) * r0, q * r0], -1)


def _exact_binned(counts, nx, ny, cell, h, kernel, n):
    """The count matrix convolved with the kernel's stencil, FP64."""
    a = min(127, math.ceil(4.0 * h / cell) if kernel == "gaussian" else math.floor(h / cell))
    t = torch.arange(-a, a + 1, dtype=torch.float64, device="cuda") * cell / h
    k = _factor(kernel, t)
    out = torch.zeros(ny, nx, dtype=torch.float64, device="cuda")
    rows = torch.zeros_like(out)
    for s in range(-a, a + 1):
        lo, hi = max(0, s), min(nx, nx + s)
        if lo < hi:
            rows[:, lo:hi] += k[s + a] * counts[:, lo - s:hi - s]
    for s in range(-a, a + 1):
        lo, hi = max(0, s), min(ny, ny + s)
        if lo < hi:
            out[lo:hi] += k[s + a] * rows[lo - s:hi - s]
    return out / (n * h * h)


def _exact_counts(points, offsets, origin, cell, nx, ny):
    """The count matrix with the gaps between a track's fixes filled linearly."""
    ij = ((points - torch.tensor(origin, dtype=torch.float64, device="cuda")) / cell).floor()
    ok = (ij >= 0).all(1) & (ij[:, 0] < nx) & (ij[:, 1] < ny)
    counts = torch.zeros(ny * nx, dtype=torch.float64, device="cuda")

    def add(at):
        if at.shape[0]:
            counts.add_(torch.bincount((at[:, 1] * nx + at[:, 0]).long(), minlength=ny * nx))

    add(ij[ok])
    same = torch.ones(points.shape[0], dtype=torch.bool, device="cuda")
    same[offsets[1:] - 1] = False  # the last fix of a track has no next
    pair = torch.nonzero(same[:-1] & ok[:-1] & ok[1:])[:, 0]
    d = ij[pair + 1] - ij[pair]
    steps = d.abs().amax(1)
    c = 1
    while pair.numel():
        more = steps > c
        pair, d, steps = pair[more], d[more], steps[more]
        add((ij[pair] + (c / steps)[:, None] * d + 0.5).floor())
        c += 1
    return counts.reshape(ny, nx)


def exact(case, seed):
    kind = case["kind"]
    if kind == "simplify":
        return None  # whole numbers and copies of the input
    st = prepare(case, seed)
    if kind == "batch":
        return [_exact_density(d["points"] - torch.tensor(d["origin"], dtype=torch.float64, device="cuda"),
                               d["weights"].double(), d["nx"], d["ny"], d["cell"], d["h"], d["kernel"])
                for d in st["insts"]]
    pts = st["points"].detach()
    if case.get("lonlat"):
        pts = _exact_mercator(pts)
    nx, ny, cell = st["nx"], st["ny"], st["cell"]
    if kind == "binned":
        counts = _exact_counts(pts, st["offsets"], st["origin"], cell, nx, ny)
        return {"density": _exact_binned(counts, nx, ny, cell, st["h"], st["kernel"], case["n"]),
                "counts": None}
    xy = pts - torch.tensor(st["origin"], dtype=torch.float64, device="cuda")
    w = st["weights"].detach().double()
    if kind == "density":
        return _exact_density(xy, w, nx, ny, cell, st["h"], st["kernel"])
    if 3 * _tile_work(case["n"], nx, ny, cell, EXACT_REACH * case["h"], 256) > 1.5 * EXACT_FLOPS:
        return None
    if kind == "fit":
        return _exact_fit(xy, w, nx, ny, cell, case["h"])
    gxy, gw, gh = _exact_adjoint(xy, w, cell, st["h"], st["cotangent"].double())
    return {"points": gxy, "weights": gw, "h": gh}
