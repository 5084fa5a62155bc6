"""The cutoff path's work items: sort-bin sides on both sides of each line, heavy
blocks sliced and whole, more items than the CTAs that take them, and grids that
are mostly blocks without a point, against the FP64 oracle at the path's 1e-6."""
import numpy as np
import pytest

import oracle
import workloads
from kde_testutil import TOL_FP32, rel_linf, sample_cells

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2004_13653_gb300 as kde  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    kde.load(build_if_stale=True)


@pytest.mark.parametrize("kid", [oracle.QUARTIC, oracle.RADIAL + oracle.EPANECHNIKOV],
                         ids=["quartic", "radial_epanechnikov"])
@pytest.mark.parametrize("n,nx,ny,h_cells", [
    (270_000, 181, 163, 4.0),    # 4-cell bins
    (262_143, 181, 163, 4.0),    # one point short of them: 8-cell bins
    (40_000, 250, 190, 6.5),     # few blocks: heavy ones sliced beyond 6 cells
    (40_000, 700, 690, 6.5),     # many: whole
    (30_000, 170, 130, 12.0),    # 8-cell bins
    (30_000, 170, 130, 12.01),   # 16-cell bins
    (900, 2100, 1900, 1.0),      # 15,708 blocks, most of them empty
])
def test_items(n, nx, ny, h_cells, kid):
    wl = workloads.random_points(940, n, 10.0 * max(nx, ny), 10.0, nx, ny, 10.0 * h_cells,
                                 kid % oracle.RADIAL)
    rng = np.random.default_rng(941)  # a third of the points within a few blocks
    wl.local[: n // 3] = np.array([4.0 * nx, 6.0 * ny]) + rng.normal(0.0, 60.0, (n // 3, 2))
    F = kde.grid(torch.as_tensor(np.ascontiguousarray(wl.xy), dtype=torch.float64, device="cuda"),
                 torch.as_tensor(wl.w, dtype=torch.float32, device="cuda"), wl.origin, wl.cell,
                 nx, ny, wl.h, kid, flags=kde.FLAG_SYNC,
                 out=torch.full((ny, nx), np.nan, device="cuda")).cpu().numpy()
    assert np.isfinite(F).all()
    cells = sample_cells(F, 400, seed=942)
    ref = oracle.kde_cells(wl.xy, wl.w, wl.origin, wl.cell, nx, ny, wl.h, kid, cells)
    assert rel_linf(F.reshape(-1)[cells], ref) <= TOL_FP32
    # cells that no point comes near are exactly zero, and all others were written
    ci = np.floor(wl.local / 10.0).astype(np.int64)
    r = int(np.ceil(h_cells)) + 1
    count = np.zeros((ny + 1, nx + 1), np.int64)
    lo, hi = np.clip(ci - r, 0, (nx, ny)), np.clip(ci + r + 1, 0, (nx, ny))
    for (a, b), s in (((lo[:, 1], lo[:, 0]), 1), ((hi[:, 1], hi[:, 0]), 1),
                      ((lo[:, 1], hi[:, 0]), -1), ((hi[:, 1], lo[:, 0]), -1)):
        np.add.at(count, (a, b), s)
    near = count.cumsum(0).cumsum(1)[:ny, :nx] > 0
    assert (F[~near] == 0.0).all()


@pytest.mark.parametrize("h_cells", [0.02, 0.3, 0.75])
def test_supports_below_a_cell_near_the_origin(h_cells):
    """Offsets from a block's first cell are up to 16 / h_cells bandwidths, of
    which a point's own cell leaves less than one: FP32 must not round the
    former (1e-6 bounds the result, whose slope per bandwidth is up to 1.5)."""
    rng = np.random.default_rng(943)
    nx, ny = 40, 37
    wl = workloads.random_points(944, 4000, 400.0, 10.0, nx, ny, 10.0 * h_cells, oracle.QUARTIC)
    cell = rng.integers(0, (nx, ny), (4000, 2))
    wl.local[:] = 10.0 * (cell + 0.5 + rng.uniform(-1.0, 1.0, (4000, 2)) * h_cells)
    F = kde.grid(torch.as_tensor(np.ascontiguousarray(wl.xy), dtype=torch.float64, device="cuda"),
                 torch.as_tensor(wl.w, dtype=torch.float32, device="cuda"), wl.origin, wl.cell,
                 nx, ny, wl.h, oracle.QUARTIC, flags=kde.FLAG_SYNC).cpu().numpy()
    ref = oracle.kde_grid(wl.xy, wl.w, wl.origin, wl.cell, nx, ny, wl.h, oracle.QUARTIC)
    cells = np.flatnonzero(ref.reshape(-1) > 0.01 * ref.max())
    err = np.abs(F.reshape(-1)[cells] - ref.reshape(-1)[cells]) / ref.reshape(-1)[cells]
    # a factor near the support's edge is steep relative to its value: 1% of the
    # maximum still leaves u's error amplified by at most 2 * 1.5 / sqrt(0.01)
    assert err.max() <= 30 * 2.0 ** -22
