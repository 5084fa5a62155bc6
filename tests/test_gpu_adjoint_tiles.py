"""The adjoint's contractions over the cells near each tile of sorted points:
against the window form and the oracle at the edges of the tiles (128 points),
the accumulators (32 to 256 cells), the 16- and 64-cell steps and the grid, and
against the contractions over the whole grid, which a workspace without room
for the sort still takes."""
import ctypes

import numpy as np
import pytest

import oracle
import workloads
from kde_testutil import TOL_GRAD, rel_linf

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2004_13653_gb300 as kde  # noqa: E402

# split-FP16 (22 bits, the tensor core's truncating FP32 sums over at most 20
# steps of 16 cells: 20 x 2^-24 of the largest) against FP32, with a margin
SAME = 1e-5


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    kde.load(build_if_stale=True)


def backward(wl, G, path, workspace=None):
    pts = torch.as_tensor(np.ascontiguousarray(wl.xy), dtype=torch.float64, device="cuda")
    w = torch.as_tensor(wl.w, dtype=torch.float32, device="cuda")
    grad = torch.as_tensor(G, dtype=torch.float32, device="cuda")
    gxy = torch.full((wl.n, 2), float("nan"), device="cuda")
    gw = torch.full((wl.n,), float("nan"), device="cuda")
    gh = ctypes.c_double(0.0)
    a = kde.make_args(pts, w, wl.origin, wl.cell, wl.nx, wl.ny, wl.h, "gaussian", grad)
    o = kde.make_opts(path, 0, torch.cuda.current_stream(), workspace)
    kde.check(kde.load().kde_grid_backward(ctypes.byref(a), grad.data_ptr(), gxy.data_ptr(),
                                           gw.data_ptr(), ctypes.byref(gh), ctypes.byref(o)))
    return gxy.cpu().numpy(), gw.cpu().numpy(), gh.value


def whole_grid_workspace(wl):
    pad = (wl.n + 511) // 512 * 512
    up = lambda v, q: (v + q - 1) // q  # noqa: E731
    tiles = 65536 * (up(wl.nx, 256) * up(wl.ny, 64) + up(wl.ny, 256) * up(wl.nx, 64))
    size = 1024 + 20 * pad + 16 * wl.n + 8 * (wl.nx + wl.ny) + tiles + 12 * 256
    return torch.empty(size, dtype=torch.uint8, device="cuda")


@pytest.mark.parametrize("n,nx,ny,h_cells", [
    (4096, 500, 333, 3.0),
    (4097, 257, 511, 7.0),     # one column past a 256-cell accumulator
    (5000, 255, 320, 2.0),
    (6001, 1030, 70, 5.0),     # windows taller than the grid
    (9000, 700, 650, 16.4),    # windows of two accumulators
    (9001, 900, 820, 33.0),    # and of three
])
def test_matches_window_form_and_whole_grid(n, nx, ny, h_cells):
    wl = workloads.random_points(51, n, 10.0 * max(nx, ny), 10.0, nx, ny, 10.0 * h_cells,
                                 oracle.GAUSSIAN)
    wl.w[::7] *= -1.0
    G = np.random.default_rng(1).normal(0, 1, (ny, nx)).astype(np.float32)
    gxy, gw, gh = backward(wl, G, "tc_split16")
    dxy, dw, dh = backward(wl, G, "tc_split16", whole_grid_workspace(wl))
    sxy, sw, sh = backward(wl, G, "simt")
    for xy, w in ((dxy, dw), (sxy, sw)):
        assert rel_linf(gxy, xy) <= SAME and rel_linf(gw, w) <= SAME
    assert gh == pytest.approx(sh, rel=1e-3) and dh == pytest.approx(sh, rel=1e-3)
    sel = np.random.default_rng(2).choice(n, 200, replace=False)
    rw, rxy, _ = oracle.kde_vjp_gauss(wl.xy[sel], wl.w[sel], wl.origin, wl.cell, nx, ny, wl.h, G)
    assert rel_linf(gw[sel], rw * len(sel) / n) <= TOL_GRAD
    assert rel_linf(gxy[sel], rxy * len(sel) / n) <= TOL_GRAD


def test_clusters_and_points_out_of_reach():
    """A dense cluster (many tiles in one bin), a thin background (tiles across
    many bins) and points no cell reaches: exact zeros."""
    rng = np.random.default_rng(7)
    local = np.concatenate([rng.normal(3000.0, 40.0, (3000, 2)), rng.uniform(0, 6000, (2000, 2)),
                            np.array([[-9000.0, 100.0], [5000.0, 90000.0]])])
    n = len(local)
    wl = workloads.Workload("clusters", local, np.ones(n, np.float32), 6000.0, 10.0, 600, 590, 80.0,
                            oracle.GAUSSIAN, np.array([0, n]), 0)
    G = rng.normal(0, 1, (590, 600)).astype(np.float32)
    gxy, gw, gh = backward(wl, G, "tc_split16")
    sxy, sw, sh = backward(wl, G, "simt")
    assert not gxy[-2:].any() and not gw[-2:].any()
    assert rel_linf(gxy, sxy) <= SAME and rel_linf(gw, sw) <= SAME
    assert gh == pytest.approx(sh, rel=1e-3)
    again = backward(wl, G, "tc_split16")
    np.testing.assert_array_equal(again[0], gxy)
    np.testing.assert_array_equal(again[1], gw)
    assert again[2] == gh
