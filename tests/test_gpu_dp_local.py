"""Douglas-Peucker trajectories processed whole in one CTA (with FP32 brackets
of the cross products) beside those of the level-synchronous kernel: the keep
masks must equal the oracle's sequential FP64 recursion bit for bit."""
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


def check(xy, lens, eps):
    offsets = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    xy = np.ascontiguousarray(xy, dtype=np.float64)
    keep, out, out_off, its = kde.dp_simplify(torch.as_tensor(xy, device="cuda"),
                                              torch.as_tensor(offsets, device="cuda"), eps)
    ref = oracle.douglas_peucker(xy, offsets, eps).astype(np.uint8)
    np.testing.assert_array_equal(keep.cpu().numpy(), ref)
    np.testing.assert_array_equal(out.cpu().numpy(), xy[ref.astype(bool)])
    np.testing.assert_array_equal(out_off.cpu().numpy(),
                                  np.concatenate([[0], np.cumsum(ref)])[offsets])
    return its


def walks(rng, lens, step, origin):
    return np.concatenate([np.cumsum(rng.normal(size=(n, 2)) * step, axis=0) + origin
                           for n in lens])


@pytest.mark.parametrize("lens", [
    [2, 3, 4, 31, 32, 33, 127, 128, 129, 511, 512, 513],  # lane, warp and CTA remainders
    [512] * 5 + [513] * 5,          # the smallest shared-memory size and one point above it
    [40] * 300 + [2000, 11000],            # short tracks and one that only the level kernel takes
    [9727, 9728, 9729, 9730],       # the largest shared-memory size and beyond
    [1] * 400 + [0] * 50 + [700],
])
@pytest.mark.parametrize("eps", [0.0, 3.0, 60.0])
def test_lengths(lens, eps):
    rng = np.random.default_rng(21)
    check(walks(rng, lens, 20.0, np.array(workloads.FALSE_ORIGIN)), lens, eps)


@pytest.mark.parametrize("scale", [1e-30, 1e-12, 1.0, 1e9, 1e25])
def test_magnitudes(scale):
    """Coordinates whose FP32 products underflow or overflow: the brackets then
    decide nothing and every point is evaluated in FP64."""
    rng = np.random.default_rng(22)
    lens = [200, 64, 3]
    check(walks(rng, lens, scale, np.zeros(2)), lens, 2.0 * scale)


def test_ties_and_flat_tracks():
    """Exact ties (zigzags on a grid), collinear runs, repeated points, closed
    loops: the first of equal points is the split."""
    i = np.arange(600, dtype=np.float64)
    zig = np.stack([i, (i % 2) * 8.0], 1)
    line = np.stack([i, 2.0 * i], 1)
    same = np.repeat(np.array([[5.0, 7.0]]), 100, axis=0)
    t = np.arange(256) * (2 * np.pi / 256)
    loop = np.stack([100 * np.cos(t), 100 * np.sin(t)], 1)
    loop = np.vstack([loop, loop[:1]])
    parts = [zig, line, same, loop, np.repeat(zig[:50], 4, axis=0)]
    xy = np.vstack(parts) + np.array([4096.0, 8192.0])
    for eps in (0.0, 4.0, 7.999, 8.0):
        check(xy, [len(p) for p in parts], eps)


@pytest.mark.parametrize("eps", [1e-7, 4.0, 7.999, 8.0])
def test_long_segments_shared_by_warps(eps):
    """Tracks whose top levels have fewer segments than the CTA has warps: ties over
    the whole track, ends of the track as the split, flat and closed tracks."""
    i = np.arange(9000, dtype=np.float64)
    zig = np.stack([i, (i % 2) * 8.0], 1)
    line = np.stack([i, 2.0 * i], 1)
    plateau = np.stack([i[:3000], np.where((i[:3000] > 100) & (i[:3000] < 2900), 50.0, 0.0)], 1)
    late = np.stack([i[:5000], np.exp((i[:5000] - 4999.0) / 40.0) * 3000.0], 1)
    t = np.arange(4000) * (2 * np.pi / 4000)
    loop = np.stack([1000 * np.cos(t), 1000 * np.sin(t)], 1)
    loop = np.vstack([loop, loop[:1]])
    same = np.repeat(np.array([[5.0, 7.0]]), 2000, axis=0)
    for parts in ([zig], [line], [plateau, late], [loop, same], [zig[:700], late, plateau, line[:1500]]):
        check(np.vstack(parts) + np.array([4096.0, 8192.0]), [len(q) for q in parts], eps)


@pytest.mark.parametrize("lens", [[640], [641], [960, 961], [3000], [9728], [9728] * 3 + [40] * 50])
@pytest.mark.parametrize("eps", [0.5, 30.0, 500.0])
def test_lengths_of_single_tracks(lens, eps):
    """Every number of warps a CTA can have and of segments a level can have."""
    rng = np.random.default_rng(23)
    check(walks(rng, lens, 20.0, np.array(workloads.FALSE_ORIGIN)), lens, eps)
