"""Small Gaussian densities in one launch: against the FP64 oracle at the edges
of the tiles, the batches, the clusters and the rule that takes them there, and
what the general path does beside the arithmetic: status words, (lon, lat)
input, weights of any sign and size, streams and capture."""
import numpy as np
import pytest

import oracle
import workloads
from kde_testutil import TOL_FP32, rel_linf

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2004_13653_gb300 as kde  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    kde.load(build_if_stale=True)


def dev(wl):
    return (torch.as_tensor(np.ascontiguousarray(wl.xy), dtype=torch.float64, device="cuda"),
            torch.as_tensor(wl.w, dtype=torch.float32, device="cuda"))


def density(wl, **kw):
    pts, w = dev(wl)
    return kde.grid(pts, w, wl.origin, wl.cell, wl.nx, wl.ny, wl.h, "gaussian", **kw)


def one_launch(wl):
    before = kde.launch_count()
    density(wl)
    return kde.launch_count() - before == 1


@pytest.mark.parametrize("n,nx,ny,h_cells,small", [
    (1, 16, 16, 2.0, True), (31, 17, 15, 1.0, True), (33, 1, 40, 3.0, True),
    (255, 64, 64, 0.6, True), (257, 64, 64, 0.6, True), (2048, 65, 63, 5.0, True),
    (2049, 150, 149, 2.0, True), (16384, 60, 61, 4.0, True),
    (16385, 60, 61, 4.0, False),      # one point more
    (6000, 100, 100, 3.0, True),      # 6e7 pairs
    (6000, 101, 100, 3.0, False),
])
def test_matches_oracle(n, nx, ny, h_cells, small):
    wl = workloads.random_points(60 + n, n, 12.0 * max(nx, ny), 12.0, nx, ny, 12.0 * h_cells,
                                 oracle.GAUSSIAN)
    wl.w[::4] *= -0.25
    assert one_launch(wl) == small
    F = density(wl).cpu().numpy()
    ref = oracle.kde_grid(wl.xy, wl.w, wl.origin, wl.cell, nx, ny, wl.h, oracle.GAUSSIAN)
    assert rel_linf(F, ref) <= (TOL_FP32 if small else 1e-5)
    np.testing.assert_array_equal(density(wl).cpu().numpy(), F)


@pytest.mark.parametrize("scale", [1e-30, 1e30, 3e37])
def test_weights_of_any_size(scale):
    wl = workloads.random_points(71, 3000, 600.0, 10.0, 64, 64, 40.0, oracle.GAUSSIAN)
    wl.w *= np.float32(scale)
    F = density(wl).cpu().numpy()
    ref = oracle.kde_grid(wl.xy, wl.w, wl.origin, wl.cell, 64, 64, wl.h, oracle.GAUSSIAN)
    assert rel_linf(F, ref) <= TOL_FP32


def test_status_lonlat_plain_call_and_capture():
    wl = workloads.random_points(72, 2000, 20_000.0, 312.5, 64, 64, 700.0, oracle.GAUSSIAN)
    ll, _, lat0 = wl.lonlat()
    xy = oracle.mercator(ll, lat0)
    origin = tuple(xy.min(axis=0))
    pts = torch.as_tensor(np.ascontiguousarray(ll), dtype=torch.float64, device="cuda")
    F = kde.grid(pts, None, origin, wl.cell, 64, 64, wl.h, "gaussian",
                 flags=kde.FLAG_LONLAT | kde.FLAG_SYNC, lat0_deg=lat0).cpu().numpy()
    ref = oracle.kde_grid(xy, np.ones(2000, np.float32), origin, wl.cell, 64, 64, wl.h,
                          oracle.GAUSSIAN)
    assert rel_linf(F, ref) <= TOL_FP32
    pts, w = dev(wl)
    out = torch.empty((64, 64), device="cuda")
    kde.grid_simple(pts, w, wl.origin, wl.cell, 64, 64, wl.h, "gaussian", out)
    plain = density(wl).cpu().numpy()
    np.testing.assert_array_equal(out.cpu().numpy(), plain)
    host = kde.grid(np.ascontiguousarray(wl.xy), wl.w, wl.origin, wl.cell, 64, 64, wl.h, "gaussian")
    assert rel_linf(host, plain) <= 1e-5  # host buffers take the general path
    g, st = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    st.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(st), torch.cuda.graph(g, stream=st):
        kde.grid(pts, w, wl.origin, wl.cell, 64, 64, wl.h, "gaussian", out=out, stream=st)
    out.zero_()
    g.replay()
    torch.cuda.synchronize()
    np.testing.assert_array_equal(out.cpu().numpy(), plain)
    pts[77, 0] = float("nan")
    with pytest.raises(kde.KDEError) as e:
        kde.grid(pts, w, wl.origin, wl.cell, 64, 64, wl.h, "gaussian", flags=kde.FLAG_SYNC)
    assert e.value.code == kde.KDE_EDATA


@pytest.mark.parametrize("n,h,scale,signs", [
    (2000, 0.02, 3e38, 1),    # overflows near the points: infinities there, numbers elsewhere
    (2000, 0.02, 3e38, 2),    # the same with weights of both signs: sums that cancel
    (50, 0.01, 1e38, 1),      # 1 / (2 pi n h^2) times the weight overflows by itself
    (16384, 1e-3, 1e37, 1),
])
def test_only_results_that_overflow_are_infinite(n, h, scale, signs):
    """Weights near the largest FP32 number and small bandwidths, as the general path
    has them: an infinity where the density overflows, its value (or zero) elsewhere."""
    wl = workloads.random_points(73, n, 40.0 * h, h, 40, 40, 1.3 * h, oracle.GAUSSIAN)
    wl.local[:, 0] *= 0.4  # the far columns are out of every point's reach
    wl.w = (wl.w * np.float32(scale / np.abs(wl.w).max())).astype(np.float32)
    if signs == 2:
        wl.w[::2] *= -1.0
    assert one_launch(wl)
    F = density(wl).cpu().numpy()
    ref = oracle.kde_grid(wl.xy, wl.w, wl.origin, wl.cell, 40, 40, wl.h, oracle.GAUSSIAN)
    top = float(np.finfo(np.float32).max)
    sure = np.abs(np.abs(ref) / top - 1.0) > 1e-5  # FP32 decides at the edge
    assert (np.abs(ref) > top).any() == (signs == 1) and (np.abs(ref) < top).any()
    assert not np.isnan(F).any()
    big = (np.abs(ref) > top) & sure
    np.testing.assert_array_equal(F[big], np.sign(ref[big]) * np.inf)
    rest = (np.abs(ref) < top) & sure
    assert np.isfinite(F[rest]).all()
    # as the FP32 path, relative to the largest value there is (signs: to that of |w|)
    peak = np.abs(ref).max() if signs == 1 else oracle.kde_grid(
        wl.xy, np.abs(wl.w), wl.origin, wl.cell, 40, 40, wl.h, oracle.GAUSSIAN).max()
    assert np.abs(F[rest] - ref[rest]).max() <= TOL_FP32 * peak


@pytest.mark.parametrize("n,nx,ny,small", [
    (2600, 1, 3600, True),        # 1.5e8 pairs of the 225 tiles' cells
    (2605, 1, 3600, False),
    (2605, 3600, 1, False),
    (16384, 1, 3600, False),
    (3, 1024, 1024, True),        # 4096 tiles
    (3, 1024, 1025, False),
    (1, 2048, 2048, False),
])
def test_rule_counts_whole_tiles(n, nx, ny, small):
    wl = workloads.random_points(80 + n, n, 12.0 * max(nx, ny), 12.0, nx, ny, 30.0,
                                 oracle.GAUSSIAN)
    if min(nx, ny) == 1:  # onto the grid's one row or column
        wl.local[:, 1 if ny == 1 else 0] *= 1.0 / 3600
    assert one_launch(wl) == small
    F = density(wl).cpu().numpy()
    cells = np.random.default_rng(n).integers(0, nx * ny, 2000)
    cells[0] = int(F.argmax())
    ref = oracle.kde_cells(wl.xy, wl.w, wl.origin, wl.cell, nx, ny, wl.h, oracle.GAUSSIAN, cells)
    assert rel_linf(F.reshape(-1)[cells], ref) <= (TOL_FP32 if small else 1e-5)
