"""What the kernels behind the bin sort do with its bin starts after it timed out:
the starts can then be anything, and nothing may be written past a list or read
past a buffer.  The starts are written here; no sort runs."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2004_13653_gb300 as kde  # noqa: E402

M, NBINS, GROUP = 512, 7, 64
ENTRIES = M // GROUP + NBINS + 2


@pytest.fixture(scope="module")
def lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return kde.load(build_if_stale=True)


def listed(lib, starts, failed):
    start = torch.as_tensor(np.asarray(starts, dtype=np.uint32).view(np.int32), device="cuda")
    groups = torch.full((ENTRIES, 4), -7, dtype=torch.int32, device="cuda")
    counters = torch.full((2,), -7, dtype=torch.int32, device="cuda")
    kde.check(lib.kde_diag_adjoint_list(start.data_ptr(), NBINS, M, failed, groups.data_ptr(),
                                        counters.data_ptr(), None))
    return groups.cpu().numpy(), counters.cpu().numpy()


def test_adjoint_groups_of_rising_starts(lib):
    starts = [0, 0, 1, 65, 129, 194, 194, 500]  # 0, 1, 64, 64, 65, 0, 306 points, 12 beyond reach
    groups, counters = listed(lib, starts, 0)
    ends = starts[1:] + [M]
    want = [(b, a + k, min(GROUP, e - a - k), 0) for b, (a, e) in enumerate(zip(starts, ends))
            for k in range(0, e - a, GROUP)]
    assert counters.tolist() == [len(want), 0]
    assert sorted(map(tuple, groups[:len(want)].tolist())) == want
    assert (groups[len(want):] == -7).all()


@pytest.mark.parametrize("starts", [[512, 0, 512, 0, 512, 0, 512, 0], [5, 4, 3, 2, 1, 0, 0, 512],
                                    [0, 2 ** 32 - 1, 0, 2 ** 31, 7, 600, 1, 2 ** 31 + 5]])
def test_adjoint_lists_nothing_after_a_timed_out_sort(lib, starts):
    groups, counters = listed(lib, starts, 1)
    assert counters.tolist() == [0, 0]
    assert (groups == -7).all()
