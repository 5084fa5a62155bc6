"""The direct sum's running sums in tensor memory and its point splits: one tile
of points and one more, ragged tiles of cells, every count of splits that a call
may take, cells far larger than the bandwidth, and a workspace for two splits
only, against the FP64 oracle at the path's 1e-6."""
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


def run(wl, kid, **kw):
    pts = torch.as_tensor(np.ascontiguousarray(wl.xy), dtype=torch.float64, device="cuda")
    w = torch.as_tensor(wl.w, dtype=torch.float32, device="cuda")
    return kde.grid(pts, w, wl.origin, wl.cell, wl.nx, wl.ny, wl.h, kid, path="simt",
                    flags=kde.FLAG_SYNC, **kw).cpu().numpy()


@pytest.mark.parametrize("kid", [oracle.GAUSSIAN, oracle.COSINE], ids=["gaussian", "cosine"])
@pytest.mark.parametrize("n,nx,ny,h_cells", [
    (1, 129, 65, 9.0), (256, 128, 64, 9.0), (257, 127, 63, 9.0), (513, 130, 66, 30.0),
    (20_000, 140, 70, 3.0), (9_000, 40, 30, 0.3)])
def test_tiles_and_splits(n, nx, ny, h_cells, kid):
    wl = workloads.random_points(950, n, 10.0 * max(nx, ny), 10.0, nx, ny, 10.0 * h_cells, kid)
    ref = oracle.kde_grid(wl.xy, wl.w, wl.origin, wl.cell, nx, ny, wl.h, kid)
    for kw in ({}, dict(split_k=1), dict(split_k=5)):
        assert rel_linf(run(wl, kid, **kw), ref) <= TOL_FP32


def test_workspace_for_two_splits():
    wl = workloads.random_points(951, 30_000, 1300.0, 10.0, 130, 70, 50.0, oracle.GAUSSIAN)
    pts = torch.as_tensor(np.ascontiguousarray(wl.xy), dtype=torch.float64, device="cuda")
    w = torch.as_tensor(wl.w, dtype=torch.float32, device="cuda")
    args = (pts, w, wl.origin, wl.cell, wl.nx, wl.ny, wl.h, "gaussian")
    full = kde.workspace_size(*args, torch.empty(wl.ny, wl.nx, device="cuda"), path="simt")
    two = kde.workspace_size(*args, torch.empty(wl.ny, wl.nx, device="cuda"), path="simt",
                             split_k=2)
    assert two < full
    ref = oracle.kde_grid(wl.xy, wl.w, wl.origin, wl.cell, wl.nx, wl.ny, wl.h, oracle.GAUSSIAN)
    for size in (full, two):
        ws = torch.empty(size, dtype=torch.uint8, device="cuda")
        assert rel_linf(run(wl, oracle.GAUSSIAN, workspace=ws), ref) <= TOL_FP32
