"""What the kernels behind the bin sort do with its bin starts after it timed out:
the starts can then be anything, and nothing may be written past a list or read
past a buffer.  The starts are written here; no sort runs."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2004_13653_gb300 as kde  # noqa: E402

M, NBINS, GROUP, FEW, FAR = 2048, 7, 64, 12, 1024
ENTRIES = M // GROUP + NBINS + 2


@pytest.fixture(scope="module")
def lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return kde.load(build_if_stale=True)


def listed(lib, starts, failed):
    start = torch.as_tensor(np.asarray(starts, dtype=np.uint32).view(np.int32), device="cuda")
    groups = torch.full((ENTRIES, 4), -7, dtype=torch.int32, device="cuda")
    singles = torch.full((M,), -7, dtype=torch.int32, device="cuda")
    counters = torch.full((3,), -7, dtype=torch.int32, device="cuda")
    kde.check(lib.kde_diag_adjoint_list(start.data_ptr(), NBINS, M, failed, groups.data_ptr(),
                                        singles.data_ptr(), counters.data_ptr(), None))
    return groups.cpu().numpy(), singles.cpu().numpy(), counters.cpu().numpy()


@pytest.mark.parametrize("starts", [
    [0, 0, 1, 65, 129, 194, 194, 500],    # 0, 1, 64, 64, 65, 0, 306 points, 1548 beyond reach
    [3, 14, 26, 101, 177, 177, 188, 2047],  # 11, 12, 64 + 11, 64 + 12, 0, 11, 1859, 1 beyond
    [0, 0, 0, 0, 0, 0, 0, 0],              # 2048 beyond
])
def test_adjoint_groups_of_rising_starts(lib, starts):
    groups, singles, counters = listed(lib, starts, 0)
    want, alone = [], []
    for b, (a, e) in enumerate(zip(starts, starts[1:] + [M])):
        most = GROUP if b < NBINS else FAR
        for k in range(a, e, most):
            if b < NBINS and e - k < FEW:
                alone += range(k, e)
            else:
                want.append((b, k, min(most, e - k), 0))
    assert counters.tolist() == [len(want), 0, len(alone)]
    assert sorted(map(tuple, groups[:len(want)].tolist())) == want
    assert sorted(singles[:len(alone)].tolist()) == alone
    assert (groups[len(want):] == -7).all() and (singles[len(alone):] == -7).all()


@pytest.mark.parametrize("starts", [[2048, 0, 2048, 0, 2048, 0, 2048, 0], [5, 4, 3, 2, 1, 0, 0, 2048],
                                    [0, 2 ** 32 - 1, 0, 2 ** 31, 7, 600, 1, 2 ** 31 + 5]])
def test_adjoint_lists_nothing_after_a_timed_out_sort(lib, starts):
    groups, singles, counters = listed(lib, starts, 1)
    assert counters.tolist() == [0, 0, 0]
    assert (groups == -7).all() and (singles == -7).all()


@pytest.mark.parametrize("side", [32, 128, 256])
@pytest.mark.parametrize("starts", [[0, 2, 2, 5, 6], [2 ** 31, 3, 2 ** 32 - 1, 2 ** 31 + 2, 1],
                                    [6, 2 ** 31, 0, 2 ** 32 - 6, 5], [0, 7, 2 ** 30, 2, 2 ** 31 - 1]])
def test_reduces_read_no_piece_outside_their_buffer(lib, side, starts):
    pieces, nx, ny = 6, 2 * side - 3, 2 * side - 5  # 2 x 2 tiles
    rng = np.random.default_rng(side)
    part = rng.integers(-50, 50, (pieces, side, side)).astype(np.float32)  # sums are exact
    buf = np.stack([part, np.zeros_like(part)], -1) if side == 32 else part
    buf = torch.as_tensor(buf, device="cuda")
    begin = torch.as_tensor(np.asarray(starts, dtype=np.uint32).view(np.int32), device="cuda")
    out = torch.full((ny, nx), 1000.0, device="cuda")
    kde.check(lib.kde_diag_piece_reduce(begin.data_ptr(), buf.data_ptr(), pieces, side, nx, ny,
                                        out.data_ptr(), None))
    got = out.cpu().numpy()
    for t in range(4):
        a, b = min(starts[t], pieces), min(starts[t + 1], pieces)
        y, x = side * (t // 2), side * (t % 2)
        h, w = min(side, ny - y), min(side, nx - x)
        want = part[a:max(a, b)].sum(0)[:h, :w]
        if side == 32 and b - a == 1:
            want = np.full((h, w), 1000.0)
        np.testing.assert_array_equal(got[y:y + h, x:x + w], want)
