"""Centring and scaling on pairs of FP32 numbers, and the FP64 form behind it:
densities of points at every magnitude the two hand over at, against the
oracle, and (lon, lat) input against the projected one."""
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


def cuda(a, dtype):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=dtype, device="cuda")


@pytest.mark.parametrize("n", [1, 63, 64, 65, 511, 512, 513, 2049])
def test_point_counts_around_a_warp_and_the_padding(n):
    wl = workloads.random_points(40 + n, n, 800.0, 10.0, 70, 66, 45.0, oracle.EPANECHNIKOV)
    F = kde.grid(cuda(wl.xy, torch.float64), cuda(wl.w, torch.float32), wl.origin, wl.cell, wl.nx,
                 wl.ny, wl.h, "epanechnikov", path="simt").cpu().numpy()
    ref = oracle.kde_grid(wl.xy, wl.w, wl.origin, wl.cell, wl.nx, wl.ny, wl.h, oracle.EPANECHNIKOV)
    assert rel_linf(F, ref) <= TOL_FP32 if ref.any() else not F.any()


@pytest.mark.parametrize("scale", [1e-25, 1e-17, 1.0, 1e15, 1e25])
def test_magnitudes(scale):
    """Units so small or large that the differences or the scale 1 / h leave
    the FP32-pair form's range; points on the origin itself; far points."""
    rng = np.random.default_rng(4)
    xy = rng.uniform(0.0, 400.0, (300, 2))
    xy[:3] = 0.0
    xy[3] = [1e60, 5.0]
    xy *= scale
    w = np.ones(len(xy), np.float32)
    args = ((0.0, 0.0), 10.0 * scale, 40, 40, 30.0 * scale)
    F = kde.grid(cuda(xy, torch.float64), cuda(w, torch.float32), *args, "quartic",
                 path="simt").cpu().numpy()
    ref = oracle.kde_grid(xy, w, *args, oracle.QUARTIC)
    if np.max(ref) < 3e38 and np.max(ref) > 1e-37:
        assert rel_linf(F, ref) <= TOL_FP32
    else:  # the density itself is outside FP32's range
        assert not F.any() or np.isinf(F).any()


def test_lonlat_matches_projected_metres_inside_and_outside_the_series():
    """Latitudes up to two degrees from the standard one: the series near it,
    the closed form beyond.  10 cm of position are 1e-3 bandwidths, far above
    the projection's 1e-6 m, so the two densities agree to FP32's rounding."""
    rng = np.random.default_rng(5)
    lat0 = 31.3
    ll = np.stack([121.7 + rng.uniform(-2, 2, 4000), lat0 + rng.uniform(-2, 2, 4000)], 1)
    xy = oracle.mercator(ll, lat0)
    origin = tuple(xy.min(axis=0))
    cell = float((xy.max(axis=0) - xy.min(axis=0)).max() / 200)
    w = np.ones(len(ll), np.float32)
    F = kde.grid(cuda(ll, torch.float64), cuda(w, torch.float32), origin, cell, 200, 200,
                 4.0 * cell, "quartic", path="simt", flags=kde.FLAG_LONLAT,
                 lat0_deg=lat0).cpu().numpy()
    ref = oracle.kde_grid(xy, w, origin, cell, 200, 200, 4.0 * cell, oracle.QUARTIC)
    assert rel_linf(F, ref) <= TOL_FP32


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
def test_non_finite_points_are_reported(bad):
    xy = np.random.default_rng(6).uniform(0, 100, (200, 2))
    xy[130, 1] = bad
    with pytest.raises(kde.KDEError) as e:
        kde.grid(cuda(xy, torch.float64), None, (0.0, 0.0), 10.0, 10, 10, 20.0, "quartic",
                 path="simt", flags=kde.FLAG_SYNC)
    assert e.value.code == kde.KDE_EDATA


@pytest.mark.parametrize("h", [1e-6, 3e-9, 1e-12, 1e-17])
@pytest.mark.parametrize("far", [1e28, -1e30])
def test_points_too_far_for_fp32_are_only_far(h, far):
    """A finite coordinate whose offset in bandwidths is past FP32's range: the point
    is out of every cell's reach, not bad data."""
    rng = np.random.default_rng(7)
    xy = rng.uniform(0.0, 40.0 * h, (300, 2))
    xy[11] = [far, 5.0 * h]
    xy[12] = [5.0 * h, far]
    w = np.ones(len(xy), np.float32)
    args = ((0.0, 0.0), h, 40, 40, 3.0 * h)
    F = kde.grid(cuda(xy, torch.float64), cuda(w, torch.float32), *args, "quartic",
                 flags=kde.FLAG_SYNC).cpu().numpy()
    ref = oracle.kde_grid(xy, w, *args, oracle.QUARTIC)
    assert rel_linf(F, ref) <= TOL_FP32


def test_far_end_of_a_long_axis_in_fp64():
    """1e8 bandwidths from the origin, points in the last tenth of the cells, each in
    reach of its own only.  The position and the cell's centre keep 2^-49 of 1e8 each,
    after two FP64 products each with a rounded factor; the kernel's slope is at most 2."""
    nx, cell, h = 30_000_000, 1.0, 0.3
    rng = np.random.default_rng(8)
    at = rng.choice(nx // 10, 3000, replace=False) + nx - nx // 10
    u = rng.uniform(-0.9, 0.9, 3000)
    xy = np.stack([(at + 0.5) * cell - u * h, np.full(3000, 0.5 * cell)], 1)
    u = ((at + 0.5) * cell - xy[:, 0]) / h  # as the FP64 coordinate has it
    F = kde.grid(cuda(xy, torch.float64), None, (0.0, 0.0), cell, nx, 1, h, "epanechnikov")
    got = F[0, torch.as_tensor(at, device="cuda")].cpu().numpy().astype(np.float64)
    ref = 0.75 ** 2 * (1.0 - u * u) / (3000 * h * h)
    assert int((F != 0).sum()) == 3000
    assert rel_linf(got, ref) <= 2 * (nx * cell / h) * (2 * 2.0 ** -49 + 4 * 2.0 ** -53) + 2.0 ** -22


def test_cell_tables_of_long_sides_and_many_instances():
    """Tables longer than the launch's blocks fill in one go (1.2M cells for one
    instance, 4864 for each of 256)."""
    rng = np.random.default_rng(9)
    nx = 3_000_001
    xy = np.stack([rng.uniform(0.0, nx, 5000), rng.uniform(0.0, 1.0, 5000)], 1)
    F = kde.grid(cuda(xy, torch.float64), None, (0.0, 0.0), 1.0, nx, 1, 2.0, "quartic").cpu().numpy()
    cells = np.unique(np.clip(xy[:, 0].astype(np.int64)[:, None] + [-1, 0, 1], 0, nx - 1))
    ref = oracle.kde_cells(xy, None, (0.0, 0.0), 1.0, nx, 1, 2.0, oracle.QUARTIC, cells)
    # an offset of at most one keeps 2^-48 of 1.5e6 and FP32's rounding
    assert rel_linf(F[0, cells], ref) <= TOL_FP32
    insts = []
    for k in range(256):
        side = 20011 if k == 200 else 16 + k % 5
        at = rng.uniform(0.0, 1.0, (300, 2)) * [side, 9]
        insts.append(dict(points=cuda(at, torch.float64), weights=None, origin=(0.0, 0.0), cell=1.0,
                          nx=side, ny=9, h=2.5, kernel="quartic"))
    out = kde.grid_batched(insts)
    for k in (0, 199, 200, 201, 255):
        q = insts[k]
        ref = oracle.kde_grid(q["points"].cpu().numpy(), None, q["origin"], 1.0, q["nx"], 9, 2.5,
                              oracle.QUARTIC)
        assert rel_linf(out[k].cpu().numpy(), ref) <= TOL_FP32
