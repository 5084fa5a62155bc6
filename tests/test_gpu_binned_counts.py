"""The binned estimator's counting where its FP32 cell index, its integer gap
filling and its trajectory-end bits hand over to the FP64 and searching forms:
the counts must equal the oracle's exactly, whichever form runs."""
import ctypes

import numpy as np
import pytest

import oracle
import workloads

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2004_13653_gb300 as kde  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    kde.load(build_if_stale=True)


def counts(xy, off, origin, cell, nx, ny):
    pts = torch.as_tensor(np.ascontiguousarray(xy), device="cuda")
    o = None if off is None else torch.as_tensor(np.asarray(off, np.int64), device="cuda")
    _, C, added = kde.grid_binned(pts, o, origin, cell, nx, ny, 2.0 * cell, "uniform", 1)
    return C.cpu().numpy(), added


def check(xy, off, origin, cell, nx, ny):
    C, added = counts(xy, off, origin, cell, nx, ny)
    ref, ref_added = oracle.count_matrix(xy, np.array([0, len(xy)]) if off is None else off,
                                         origin, cell, nx, ny)
    np.testing.assert_array_equal(C, ref)
    assert added == ref_added


@pytest.mark.parametrize("n", [1, 31, 32, 33, 511, 512, 513, 4097])
@pytest.mark.parametrize("lens", [1, 3, 40])
def test_warp_and_trajectory_edges(n, lens):
    """Fix counts around a round, a warp's share and a block's; trajectories
    that end inside, at and across them."""
    rng = np.random.default_rng(n)
    xy = np.cumsum(rng.normal(size=(n, 2)) * 30.0, axis=0) + 5000.0
    off = np.unique(np.append(np.arange(0, n, lens), n))
    check(xy, off, (3000.0, 3100.0), 7.3, 500, 450)
    check(xy, None, (3000.0, 3100.0), 7.3, 500, 450)


@pytest.mark.parametrize("cell", [1e-31, 1e-6, 1.0 / 3.0, 1e7, 1e31])
def test_cell_magnitudes(cell):
    """Cells outside FP32's range, quotients beyond 2^21 and exact multiples of
    the cell."""
    rng = np.random.default_rng(3)
    k = rng.integers(0, 40, (400, 2)).astype(np.float64)
    xy = np.concatenate([k[:200] * cell, (k[200:] + rng.random((200, 2))) * cell,
                         rng.normal(size=(20, 2)) * 1e9 * cell])
    check(xy, None, (0.0, 0.0), cell, 40, 37)


@pytest.mark.parametrize("move", [(6, 3), (6, -3), (10, 5), (12, 6), (7, 7), (9, 0), (0, -11),
                                  (100, 50), (99, 66), (30, -45), (1 << 18, 3), (300001, 150000)])
def test_gaps(move):
    """Moves whose minor step hits exact halves (ties, with c / c_max exact and
    not), diagonal and straight moves, and moves evaluated in FP64."""
    di, dj = move
    nx, ny = abs(di) + 3, abs(dj) + 3
    if nx * ny > 2 ** 22:  # a band of rows around the start is enough
        ny = 2 ** 22 // nx
        dj = ny - 3
    i0, j0 = (1 if di >= 0 else nx - 2), (1 if dj >= 0 else ny - 2)
    xy = np.array([[i0 + 0.5, j0 + 0.5], [i0 + di + 0.5, j0 + dj + 0.5],
                   [i0 + 0.5, j0 + 0.5]])
    check(xy, None, (0.0, 0.0), 1.0, nx, ny)


def raw_counts(pts, off, n, cell, nx, ny, workspace):
    out = torch.empty((ny, nx), device="cuda")
    C = torch.empty((ny, nx), dtype=torch.int32, device="cuda")
    org = (ctypes.c_double * 2)(0.0, 0.0)
    o = kde.make_opts("auto", kde.FLAG_SYNC, torch.cuda.current_stream(), workspace)
    kde.check(kde.load().kde_grid_binned(
        pts.data_ptr(), off.data_ptr(), off.numel() - 1, n, ctypes.byref(org), cell, nx, ny,
        2.0 * cell, 0, 1, 1, C.data_ptr(), out.data_ptr(), None, ctypes.byref(o)))
    return C.cpu().numpy()


@pytest.mark.parametrize("regular", [True, False])
def test_without_scratch_for_the_ends_and_offsets_that_fall(regular):
    """A workspace that holds the row buffer only, and offsets that do not rise
    (no result is defined for them, but every form gives the same)."""
    rng = np.random.default_rng(8)
    n, nx, ny = 10000, 20, 18
    xy = torch.as_tensor(np.cumsum(rng.normal(size=(n, 2)), axis=0) + 9.0, device="cuda")
    off = np.unique(np.append(rng.integers(0, n, 900), [0, n]))
    if not regular:
        off[40], off[200] = off[41] + 5, off[100]
    off = torch.as_tensor(off, device="cuda")
    a = raw_counts(xy, off, n, 1.0, nx, ny, None)
    # 9 x 8 cells: 288 bytes of rows, 1252 of end bits; the workspace of the one without them
    b = raw_counts(xy, off, n, 2.5, 9, 8, None)
    c = raw_counts(xy, off, n, 2.5, 9, 8, torch.empty(256 + 512, dtype=torch.uint8, device="cuda"))
    np.testing.assert_array_equal(b, c)
    if regular:
        ref, _ = oracle.count_matrix(xy.cpu().numpy(), off.cpu().numpy(), (0.0, 0.0), 1.0, nx, ny)
        np.testing.assert_array_equal(a, ref)
