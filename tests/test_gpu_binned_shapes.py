"""The binned estimator where its passes change form with the size: fixes per warp
and the trajectory-end bits (from 2^17 fixes on), rows of up to 128 columns a warp
each, one or four columns per thread of the column pass.  Counts equal the oracle's
exactly, the convolution is within the rounding of its two FP32 sums."""
import numpy as np
import pytest

import oracle
from kde_testutil import rel_linf

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2004_13653_gb300 as kde  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    kde.load(build_if_stale=True)


def binned(xy, off, cell, nx, ny, h, window, kernel="gaussian"):
    pts = torch.as_tensor(np.ascontiguousarray(xy), device="cuda")
    o = None if off is None else torch.as_tensor(np.asarray(off, np.int64), device="cuda")
    out, C, added = kde.grid_binned(pts, o, (0.0, 0.0), cell, nx, ny, h, kernel, window)
    return out.cpu().numpy(), C.cpu().numpy(), added


@pytest.mark.parametrize("n", [131071, 131072, 311295, 622592, 700001])
@pytest.mark.parametrize("form", ["short", "long", "one", "irregular"])
def test_counts_around_the_bits_and_the_rounds(n, form):
    rng = np.random.default_rng(n)
    xy = np.cumsum(rng.normal(size=(n, 2)) * 3.0, axis=0)
    xy = np.abs((xy + 1000.0) % 3000.0 - 20.0)  # jumps across the grid now and then
    off = {"short": np.append(np.arange(0, n, 3), n), "long": np.append(np.arange(0, n, 1000), n),
           "one": None, "irregular": np.array([0, 500, 400, 90000, n])}[form]
    _, C, added = binned(xy, off, 7.3, 400, 391, 20.0, 5)
    if form == "irregular":  # not an input with a meaning, but one that may not fault
        assert C.sum() - added == ((xy < [400 * 7.3, 391 * 7.3]) & (xy >= 0)).all(1).sum()
        return
    ref, ref_added = oracle.count_matrix(xy, np.array([0, n]) if off is None else off, (0.0, 0.0),
                                         7.3, 400, 391)
    np.testing.assert_array_equal(C, ref)
    assert added == ref_added


def separable(M, cell, h, window):
    """Eq. 7's stencil as a row and a column pass, FP64."""
    a = window // 2
    k = oracle.kernel_1d(oracle.GAUSSIAN, np.arange(-a, a + 1) * cell / h)
    for axis in (0, 1):
        P = np.pad(M, [(a, a) if q == axis else (0, 0) for q in (0, 1)])
        m = M.shape[axis]
        M = sum(k[u] * (P[u:u + m] if axis == 0 else P[:, u:u + m]) for u in range(window))
    return M


@pytest.mark.parametrize("nx,ny", [(1, 700), (20, 3000), (32, 900), (33, 900), (127, 130), (128, 64),
                                   (129, 65), (512, 7), (513, 9), (1500, 1), (1300, 1090),
                                   (40, 9001)])
@pytest.mark.parametrize("window", [1, 3, 97, 255])
def test_convolution_at_the_edges_of_its_forms(nx, ny, window):
    rng = np.random.default_rng(nx * 7 + window)
    n, cell = 3000, 2.0
    xy = rng.random((n, 2)) * [nx * cell, ny * cell]
    h = cell * max(window, 3) / 8.0
    out, C, _ = binned(xy, np.arange(n + 1), cell, nx, ny, h, window)
    ref = separable(C.astype(np.float64), cell, h, window) / (n * h * h)
    # sums of positive terms: 2 x 255 roundings of 2^-24, and the coefficients'
    assert rel_linf(out, ref) <= 4e-5
