"""The adjoint's window form in groups of sorted points: against the FP64 oracle
and against the one-point form (which a workspace without room for the sort
still takes), at the edges of the groups, the bins, the thread tiles (window
half-widths 12, 28 and 44) and the grid."""
import ctypes

import numpy as np
import pytest

import oracle
import workloads
from kde_testutil import TOL_GRAD, rel_linf

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2004_13653_gb300 as kde  # noqa: E402

# two FP32 evaluations of sums of up to 96 x 96 products each: 2 sqrt(2 x 96)
# roundings of 2^-24 relative to the largest value, with a margin of six
SAME = 1e-5


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    kde.load(build_if_stale=True)


def dev(a, dt):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=dt, device="cuda")


def backward(wl, w, G, workspace=None, want_w=True):
    pts, grad = dev(wl.xy, torch.float64), dev(G, torch.float32)
    wt = None if w is None else dev(w, torch.float32)
    gxy = torch.full((wl.n, 2), float("nan"), device="cuda")
    gw = torch.full((wl.n,), float("nan"), device="cuda")
    gh = ctypes.c_double(0.0)
    a = kde.make_args(pts, wt, wl.origin, wl.cell, wl.nx, wl.ny, wl.h, "gaussian", grad)
    o = kde.make_opts("simt", 0, torch.cuda.current_stream(), workspace)
    kde.check(kde.load().kde_grid_backward(
        ctypes.byref(a), grad.data_ptr(), gxy.data_ptr(), gw.data_ptr() if want_w else None,
        ctypes.byref(gh), ctypes.byref(o)))
    return gxy.cpu().numpy(), gw.cpu().numpy(), gh.value


def one_point_workspace(wl):
    """What the call needs without the sort: 20 bytes per padded point, 16 per
    point of FP64 terms, the tables."""
    pad = (wl.n + 511) // 512 * 512
    size = 1024 + 20 * pad + 16 * wl.n + 8 * (wl.nx + wl.ny) + 10 * 256
    return torch.empty(size, dtype=torch.uint8, device="cuda")


@pytest.mark.parametrize("n,nx,ny,h_cells", [
    (16384, 96, 80, 1.3),     # R = 12: the smallest thread tile
    (16385, 97, 81, 1.4),     # R = 13: one cell more
    (20000, 160, 120, 3.3),   # R = 28
    (20001, 161, 121, 3.4),   # R = 29
    (17000, 256, 203, 5.3),   # R = 44: the largest window
    (17000, 256, 203, 5.4),   # R = 45: one point at a time
    (30000, 40, 9, 2.0),      # windows wider than the grid, hundreds of points per bin
    (16400, 3, 500, 1.0),
])
def test_matches_one_point_form_and_oracle(n, nx, ny, h_cells):
    wl = workloads.random_points(31, n, 10.0 * max(nx, ny), 10.0, nx, ny, 10.0 * h_cells,
                                 oracle.GAUSSIAN)
    wl.w[::5] *= -1.0
    G = np.random.default_rng(1).normal(0, 1, (ny, nx))
    gxy, gw, gh = backward(wl, wl.w, G)
    sxy, sw, sh = backward(wl, wl.w, G, workspace=one_point_workspace(wl))
    assert rel_linf(gxy, sxy) <= SAME and rel_linf(gw, sw) <= SAME
    assert gh == pytest.approx(sh, rel=1e-4)
    sel = np.random.default_rng(2).choice(n, 300, replace=False)
    sub = wl.xy[sel]
    rw, rxy, _ = oracle.kde_vjp_gauss(sub, wl.w[sel], wl.origin, wl.cell, nx, ny, wl.h, G)
    scale = len(sel) / n  # the density's 1/N
    assert rel_linf(gw[sel], rw * scale) <= TOL_GRAD
    assert rel_linf(gxy[sel], rxy * scale) <= TOL_GRAD


def test_clusters_empty_bins_far_points_and_missing_outputs():
    """Bins with 1, 64, 65 and thousands of points, points out of every cell's
    reach (exact zeros), unit weights, no weight gradient."""
    rng = np.random.default_rng(7)
    parts = [np.full((64, 2), 405.0) + rng.random((64, 2)), np.full((65, 2), 885.0) + rng.random((65, 2)),
             np.array([[1200.0, 300.0]]), rng.normal(700.0, 30.0, (16500, 2)),
             np.array([[-900.0, 100.0], [5000.0, 700.0], [100.0, 9e5]])]
    local = np.concatenate(parts)
    n = len(local)
    wl = workloads.Workload("clusters", local, np.ones(n, np.float32), 1280.0, 10.0, 128, 110, 20.0,
                            oracle.GAUSSIAN, np.array([0, n]), 0)
    G = rng.normal(0, 1, (110, 128))
    gxy, gw, gh = backward(wl, None, G)
    sxy, sw, sh = backward(wl, None, G, workspace=one_point_workspace(wl))
    assert not gxy[-3:].any() and not gw[-3:].any()
    assert rel_linf(gxy, sxy) <= SAME and rel_linf(gw, sw) <= SAME
    assert gh == pytest.approx(sh, rel=1e-4)
    again = backward(wl, None, G)
    np.testing.assert_array_equal(again[0], gxy)
    assert again[2] == gh
    nxy, nw, _ = backward(wl, None, G, want_w=False)
    np.testing.assert_array_equal(nxy, gxy)
    assert np.isnan(nw).all()


def own_window(local, w, cell, h, G, n):
    """FP64 gradients of the points, each over the cells within 10 bandwidths; G: one row."""
    span = int(np.ceil(10 * h / cell))
    i = np.floor(local[:, 0] / cell).astype(np.int64)[:, None] + np.arange(-span, span + 1)
    g = np.where((i >= 0) & (i < len(G)), G[np.clip(i, 0, len(G) - 1)], 0.0)
    s = ((i + 0.5) * cell - local[:, :1]) / h
    t = (0.5 * cell - local[:, 1:]) / h
    f = np.exp(-0.5 * (s * s + t * t)) * g / (2 * np.pi * n * h * h)
    return (np.stack([(s * f).sum(1), (t * f).sum(1)], 1) * w[:, None] / h, f.sum(1))


@pytest.mark.parametrize("nx,cell,h", [(3_000_000, 7.3, 0.9), (34_000_000, 7.3, 0.9),
                                       (34_000_000, 10.0, 20.0), (100_000_000, 10.0, 3.0)])
def test_long_axes(nx, cell, h):
    """The sort's FP32 bin keys are several cells off at the far end of a long axis."""
    n = 16384
    rng = np.random.default_rng(nx)
    local = np.stack([(nx - rng.random(n) * 0.02 * nx) * cell, rng.random(n) * cell], 1)
    w = (rng.random(n) + 0.5).astype(np.float32)
    wl = workloads.Workload("long", local, w, nx * cell, cell, nx, 1, h, oracle.GAUSSIAN,
                            np.array([0, n]), 0)
    G = rng.standard_normal(nx, dtype=np.float32)
    gxy, gw, _ = backward(wl, w, G[None])
    at = wl.xy - np.asarray(wl.origin)
    rxy, rw = own_window(at, w.astype(np.float64), cell, h, G.astype(np.float64), n)
    assert rel_linf(gw, rw) <= TOL_GRAD
    assert rel_linf(gxy, rxy) <= TOL_GRAD


@pytest.mark.parametrize("value", [float("inf"), float("-inf"), float("nan")])
@pytest.mark.parametrize("h_cells", [0.6, 1.4, 3.3, 5.3])
def test_non_finite_cotangent_cells(value, h_cells):
    """Such a cell reaches the points whose own window holds it, no others."""
    n, nx, ny = 20000, 130, 117
    wl = workloads.random_points(33, n, 10.0 * nx, 10.0, nx, ny, 10.0 * h_cells, oracle.GAUSSIAN)
    G = np.random.default_rng(3).normal(0, 1, (ny, nx))
    clean = backward(wl, wl.w, G)
    G[40, 51] = value
    gxy, gw, _ = backward(wl, wl.w, G)
    sxy, sw, _ = backward(wl, wl.w, G, workspace=one_point_workspace(wl))
    hit = ~np.isfinite(sw)
    assert 0 < hit.sum() < n
    np.testing.assert_array_equal(~np.isfinite(gw), hit)
    np.testing.assert_array_equal(np.isfinite(gxy), np.isfinite(sxy))
    assert rel_linf(gw[~hit], clean[1][~hit]) <= SAME
    assert rel_linf(gxy[~hit], clean[0][~hit]) <= SAME


@pytest.mark.parametrize("nx,h_cells", [(3_000_000, 1.0), (34_000_000, 1.5), (34_000_000, 3.0)])
def test_long_axes_with_points_in_clusters(nx, h_cells):
    """As above, with enough points in a bin for groups of them."""
    n, cell, per = 16384, 7.3, 64
    rng = np.random.default_rng(nx)
    at = np.repeat(nx - rng.integers(0, nx // 50, n // per), per)
    local = np.stack([(at + rng.random(n) * 4.0) * cell, rng.random(n) * cell], 1)
    w = (rng.random(n) + 0.5).astype(np.float32)
    wl = workloads.Workload("long", local, w, nx * cell, cell, nx, 1, h_cells * cell,
                            oracle.GAUSSIAN, np.array([0, n]), 0)
    G = rng.standard_normal(nx, dtype=np.float32)
    gxy, gw, _ = backward(wl, w, G[None])
    rxy, rw = own_window(wl.xy - np.asarray(wl.origin), w.astype(np.float64), cell, wl.h,
                         G.astype(np.float64), n)
    assert rel_linf(gw, rw) <= TOL_GRAD
    assert rel_linf(gxy, rxy) <= TOL_GRAD


@pytest.mark.parametrize("n,side,h_cells,sorts", [
    (16383, 300, 2.0, False), (16384, 1024, 1.0, True), (16384, 300, 2.0, True),
    (20011, 128, 3.0, True), (16400, 2048, 5.3, True),
    (20000, 100, 0.75, False), (20000, 100, 0.76, True),  # windows of 16 and of 18 cells
    (65535, 900, 2.0, True), (65536, 900, 2.0, False),    # 5.1 points a bin
    (65536, 640, 2.0, True), (70000, 900, 3.25, False), (70000, 900, 3.3, True),
])
def test_bins_with_few_points(n, side, h_cells, sorts):
    """Points spread evenly, 0.25 to 78 a bin: bins without a group, points left over
    beside groups, and the lines of the rule that sorts the points at all."""
    wl = workloads.random_points(34, n, 10.0 * side, 10.0, side, side, 10.0 * h_cells,
                                 oracle.GAUSSIAN)
    G = np.random.default_rng(4).normal(0, 1, (side, side))
    before = kde.launch_count()
    gxy, gw, gh = backward(wl, wl.w, G)
    launches = kde.launch_count() - before
    sxy, sw, sh = backward(wl, wl.w, G, workspace=one_point_workspace(wl))
    assert (launches > kde.launch_count() - before - launches) == sorts
    assert rel_linf(gxy, sxy) <= SAME and rel_linf(gw, sw) <= SAME
    assert gh == pytest.approx(sh, rel=1e-4)


@pytest.mark.parametrize("h_cells", [3.3, 5.3])
def test_error_no_larger_than_one_point_form(h_cells):
    """Rms over 20,000 points, a statistic that repeats to a few percent: sums of W
    terms added from the small ones to the large ones round less than in order."""
    n, nx, ny = 20000, 190, 170
    wl = workloads.random_points(35, n, 10.0 * ny, 10.0, nx, ny, 10.0 * h_cells, oracle.GAUSSIAN)
    G = np.random.default_rng(5).normal(0, 1, (ny, nx)).astype(np.float32)
    at = wl.xy - np.asarray(wl.origin)
    s = ((np.arange(nx) + 0.5) * wl.cell - at[:, :1]) / wl.h
    t = ((np.arange(ny) + 0.5) * wl.cell - at[:, 1:]) / wl.h
    A, B = np.exp(-0.5 * s * s), np.exp(-0.5 * t * t)
    U = A @ G.T.astype(np.float64)  # over the columns
    V = B @ G.astype(np.float64)
    c = 1.0 / (2 * np.pi * n * wl.h ** 2)
    rw = c * (B * U).sum(1)
    rxy = c * wl.w[:, None].astype(np.float64) / wl.h * np.stack([(s * A * V).sum(1), (t * B * U).sum(1)], 1)
    gxy, gw, _ = backward(wl, wl.w, G)
    sxy, sw, _ = backward(wl, wl.w, G, workspace=one_point_workspace(wl))
    for got, one, ref in ((gxy, sxy, rxy), (gw, sw, rw)):
        assert np.sqrt(((got - ref) ** 2).mean()) <= 0.95 * np.sqrt(((one - ref) ** 2).mean())
