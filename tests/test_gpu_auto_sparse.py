"""AUTO's choice of the block-sparse contraction for Gaussian densities: the
call must stay within split-FP16's 1e-5 of the FP64 oracle and agree with the
dense contraction (path="tc_split16") to the rounding of the sums, over ragged
grids, signed and missing weights, points outside the grid, host buffers and
batches that mix dense, block-sparse and compact instances; it must still run
where only the dense plan's workspace is there, and under graph capture."""
import numpy as np
import pytest

import oracle
import workloads
from kde_testutil import TOL_SPLIT, rel_linf

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2004_13653_gb300 as kde  # noqa: E402

# both contractions sum the same nonzero products: each is within 1e-6 of the
# sum by the drain's bound (12 truncated steps of 2^-24 per 64 sorted points,
# 48 per 256 in input order)
SAME = 4e-6


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    kde.load(build_if_stale=True)


def case(n, nx, ny, h_cells, seed=900):
    """A box one tenth wider than the grid on every side, cells of 20 m."""
    wl = workloads.random_points(seed, n, 20.0 * max(nx, ny), 20.0, nx, ny, 20.0 * h_cells,
                                 oracle.GAUSSIAN)
    return wl


def on_device(wl, weights="own"):
    pts = torch.as_tensor(np.ascontiguousarray(wl.xy), dtype=torch.float64, device="cuda")
    w = None if weights is None else torch.as_tensor(wl.w, dtype=torch.float32, device="cuda")
    return pts, w


def density(wl, pts, w, **kw):
    return kde.grid(pts, w, wl.origin, wl.cell, wl.nx, wl.ny, wl.h, "gaussian", **kw)


def launches(fn):
    before = kde.launch_count()
    fn()
    torch.cuda.synchronize()
    return kde.launch_count() - before


@pytest.mark.parametrize("n,nx,ny,h_cells", [
    (60_000, 1500, 1300, 1.0),    # ragged tiles, reach far inside a tile
    (60_001, 2049, 513, 3.3),     # one column and one row past a tile
    (200_000, 1024, 1024, 12.0),  # reach of 91 cells: two or three tiles a point
])
@pytest.mark.parametrize("weights", ["own", "signed", None])
def test_matches_dense_and_oracle(n, nx, ny, h_cells, weights):
    wl = case(n, nx, ny, h_cells)
    if weights == "signed":
        wl.w[::3] *= -0.4
    pts, w = on_device(wl, weights)
    auto_launches = launches(lambda: density(wl, pts, w))
    F = density(wl, pts, w, flags=kde.FLAG_SYNC).cpu().numpy()
    assert auto_launches > launches(lambda: density(wl, pts, w, path="tc_split16")), \
        "this case is meant to take the block-sparse contraction"
    D = density(wl, pts, w, path="tc_split16", flags=kde.FLAG_SYNC).cpu().numpy()
    assert rel_linf(F, D) <= SAME
    cells = np.unique(np.concatenate([
        np.random.default_rng(5).integers(0, nx * ny, 400), [0, nx - 1, nx * ny - 1],
        [int(np.argmax(np.abs(F)))]]))
    ref = oracle.kde_cells(wl.xy, wl.w if w is not None else np.ones(n, np.float32), wl.origin,
                           wl.cell, nx, ny, wl.h, oracle.GAUSSIAN, cells)
    assert rel_linf(F.reshape(-1)[cells], ref) <= TOL_SPLIT


def test_wide_bandwidth_and_small_grids_stay_dense():
    # (at most 6e7 point-cell pairs of at most 16384 points go to neither)
    for wl in (case(40_000, 300, 280, 40.0), case(20_000, 64, 64, 0.6), case(500, 900, 900, 2.0)):
        pts, w = on_device(wl)
        a = density(wl, pts, w).cpu().numpy()
        d = density(wl, pts, w, path="tc_split16").cpu().numpy()
        np.testing.assert_array_equal(a, d)


def test_dense_workspace_and_named_tilings_are_enough():
    """A caller's workspace sized for the dense plan, and any named part of
    the tiling, give the dense contraction bit for bit (400,000 points: the
    pieces' partials then need more than the dense splits')."""
    wl = case(400_000, 1024, 1024, 3.0)
    pts, w = on_device(wl)
    D = density(wl, pts, w, path="tc_split16").cpu().numpy()
    args = (pts, w, wl.origin, wl.cell, wl.nx, wl.ny, wl.h, "gaussian")
    out = torch.empty((wl.ny, wl.nx), device="cuda")
    small = kde.workspace_size(*args, out, path="tc_split16")
    assert kde.workspace_size(*args, out) > small
    ws = torch.empty(small, dtype=torch.uint8, device="cuda")
    np.testing.assert_array_equal(density(wl, pts, w, workspace=ws).cpu().numpy(), D)
    np.testing.assert_array_equal(density(wl, pts, w, k_chunk=256).cpu().numpy(), D)
    ws = torch.empty(kde.workspace_size(*args, out), dtype=torch.uint8, device="cuda")
    S = density(wl, pts, w).cpu().numpy()
    np.testing.assert_array_equal(density(wl, pts, w, workspace=ws).cpu().numpy(), S)


def test_host_buffers_and_capture():
    wl = case(60_001, 2049, 513, 3.3)
    pts, w = on_device(wl)
    F = density(wl, pts, w).cpu().numpy()
    np.testing.assert_array_equal(density(wl, np.ascontiguousarray(wl.xy), wl.w), F)
    out = torch.empty((wl.ny, wl.nx), device="cuda")
    g, st = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    st.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(st), torch.cuda.graph(g, stream=st):
        density(wl, pts, w, out=out, stream=st)
    out.zero_()
    g.replay()
    torch.cuda.synchronize()
    np.testing.assert_array_equal(out.cpu().numpy(), F)


def test_batch_mixes_dense_sparse_and_compact():
    wls = [case(50_000, 1300, 1100, 2.0, 910), case(30_000, 250, 260, 30.0, 911),
           case(40_000, 700, 650, 2.5, 912), case(70_000, 900, 1500, 4.0, 913),
           case(3_000, 128, 128, 3.0, 914)]
    kernels = ["gaussian", "gaussian", "epanechnikov", "gaussian", "gaussian"]
    insts = []
    for wl, k in zip(wls, kernels):
        pts, w = on_device(wl)
        insts.append(dict(points=pts, weights=w, origin=wl.origin, cell=wl.cell, nx=wl.nx,
                          ny=wl.ny, h=wl.h, kernel=k))
    outs = [o.cpu().numpy() for o in kde.grid_batched(insts, flags=kde.FLAG_SYNC)]
    again = [o.cpu().numpy() for o in kde.grid_batched(insts, flags=kde.FLAG_SYNC)]
    for wl, k, F, G in zip(wls, kernels, outs, again):
        np.testing.assert_array_equal(F, G)
        cells = np.random.default_rng(6).integers(0, wl.nx * wl.ny, 300)
        cells = np.unique(np.append(cells, int(np.argmax(F))))
        ref = oracle.kde_cells(wl.xy, wl.w, wl.origin, wl.cell, wl.nx, wl.ny, wl.h,
                               getattr(oracle, k.upper()), cells)
        assert rel_linf(F.reshape(-1)[cells], ref) <= (TOL_SPLIT if k == "gaussian" else 1e-6)
