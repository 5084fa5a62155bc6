"""The compact kernels' gather on 32 x 32-cell tiles (product kernels, supports
of more than 16 cells, dense points; their radial variants stay in 16 x 16
blocks at the same sizes): every kernel and its radial variant against the FP64 oracle at the cutoff path's 1e-6, on ragged grids around the
tile's side, tiles of one piece and of many, points outside the grid, signed
weights; the same results in a batch, under graph capture and again; and the
16 x 16-cell blocks where the workspace holds no more."""
import dataclasses

import numpy as np
import pytest

import oracle
import workloads
from kde_testutil import TOL_FP32, clear_of_support_edge, rel_linf

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2004_13653_gb300 as kde  # noqa: E402

COMPACT = [k for k in range(8) if k != oracle.GAUSSIAN]


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    kde.load(build_if_stale=True)


def case(n, nx, ny, h_cells, kid, seed=930):
    """Half of the points in a box one tenth wider than the grid, half of them
    within a few cells of its middle (more than one piece for the tiles there)."""
    wl = workloads.random_points(seed, n, 10.0 * max(nx, ny), 10.0, nx, ny, 10.0 * h_cells,
                                 kid % oracle.RADIAL)
    rng = np.random.default_rng(seed)
    at = np.array([5.0 * nx, 5.0 * ny])
    wl.local[: n // 2] = at + rng.normal(0.0, 30.0, (n // 2, 2))
    return wl


def args(wl):
    return (torch.as_tensor(np.ascontiguousarray(wl.xy), dtype=torch.float64, device="cuda"),
            torch.as_tensor(wl.w, dtype=torch.float32, device="cuda"), wl.origin, wl.cell, wl.nx,
            wl.ny, wl.h)


def oracle_grid(wl, kid, w=None):
    return oracle.kde_grid(wl.xy, wl.w if w is None else w, wl.origin, wl.cell, wl.nx, wl.ny, wl.h,
                           kid)


@pytest.mark.parametrize("radial", [False, True], ids=["product", "radial"])
@pytest.mark.parametrize("kid", COMPACT, ids=[oracle.KERNEL_NAMES[k] for k in COMPACT])
def test_kernels_on_a_ragged_grid(kid, radial):
    k = kid + (oracle.RADIAL if radial else 0)
    wl = case(130_001, 65, 33, 17.0, k)
    if kid == oracle.UNIFORM:  # in parts: the radial check holds every pair
        parts = [clear_of_support_edge(dataclasses.replace(wl, local=wl.local[i::16], w=wl.w[i::16]),
                                       radial=radial) for i in range(16)]
        wl = dataclasses.replace(wl, local=np.concatenate([q.local for q in parts]),
                                 w=np.concatenate([q.w for q in parts]))
    F = kde.grid(*args(wl), k, flags=kde.FLAG_SYNC).cpu().numpy()
    assert rel_linf(F, oracle_grid(wl, k)) <= TOL_FP32


@pytest.mark.parametrize("n,nx,ny,h_cells", [
    (300_000, 31, 63, 16.01),   # just past the line; one tile across
    (130_000, 64, 32, 40.0),    # whole tiles
    (61_000, 33, 257, 300.0),   # every point reaches every tile
])
def test_signed_weights_around_the_tile(n, nx, ny, h_cells):
    wl = case(n, nx, ny, h_cells, oracle.QUARTIC, seed=931)
    w = wl.w.copy()
    w[::3] *= -0.5
    a = list(args(wl))
    a[1] = torch.as_tensor(w, dtype=torch.float32, device="cuda")
    F = kde.grid(*a, oracle.QUARTIC, flags=kde.FLAG_SYNC).cpu().numpy()
    assert rel_linf(F, oracle_grid(wl, oracle.QUARTIC, w)) <= TOL_FP32


def test_same_in_a_batch_under_capture_and_again():
    wls = [case(150_000, 96, 70, 20.0, oracle.TRIWEIGHT, seed=932),
           case(3000, 50, 40, 4.0, oracle.EPANECHNIKOV, seed=933),
           case(90_000, 300, 280, 18.0, oracle.EPANECHNIKOV, seed=934)]
    kids = ["triweight", "epanechnikov", "epanechnikov"]
    alone = [kde.grid(*args(w), k) for w, k in zip(wls, kids)]
    names = ("points", "weights", "origin", "cell", "nx", "ny", "h", "kernel")
    insts = [dict(zip(names, args(w) + (k,))) for w, k in zip(wls, kids)]
    for F, G in zip(alone, kde.grid_batched(insts)):
        assert torch.equal(F, G)
    a, out = args(wls[0]), torch.empty_like(alone[0])
    g, st = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    st.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(st), torch.cuda.graph(g, stream=st):
        kde.grid(*a, kids[0], out=out, stream=st)
    out.zero_()
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(out, alone[0])


def test_smaller_workspace_takes_the_blocks():
    wl = case(200_000, 256, 256, 20.0, oracle.EPANECHNIKOV, seed=935)
    a = args(wl)
    out = torch.empty(wl.ny, wl.nx, device="cuda")
    full = kde.workspace_size(*a, "epanechnikov", out)
    # the pieces' partial tiles alone take 200,000 x 16 / 512 x 8 KB = 51 MB
    for size in (full, full - (2 << 20)):
        ws = torch.empty(size, dtype=torch.uint8, device="cuda")
        F = kde.grid(*a, "epanechnikov", workspace=ws, flags=kde.FLAG_SYNC).cpu().numpy()
        cells = np.random.default_rng(7).integers(0, wl.nx * wl.ny, 300)
        ref = oracle.kde_cells(wl.xy, wl.w, wl.origin, wl.cell, wl.nx, wl.ny, wl.h,
                               oracle.EPANECHNIKOV, np.unique(cells))
        assert rel_linf(F.reshape(-1)[np.unique(cells)], ref) <= TOL_FP32


def test_more_than_1024_tiles():
    """35 x 34 tiles: the work list of several launches."""
    wl = case(800_000, 1100, 1060, 17.0, oracle.QUARTIC, seed=936)
    F = kde.grid(*args(wl), oracle.QUARTIC, flags=kde.FLAG_SYNC).cpu().numpy()
    cells = np.random.default_rng(8).integers(0, wl.nx * wl.ny, 400)
    cells = np.unique(np.append(cells, int(np.argmax(F))))
    ref = oracle.kde_cells(wl.xy, wl.w, wl.origin, wl.cell, wl.nx, wl.ny, wl.h, oracle.QUARTIC,
                           cells)
    assert rel_linf(F.reshape(-1)[cells], ref) <= TOL_FP32


@pytest.mark.parametrize("gauss", [(60_000, 1500, 1300, 1.0), (20_000, 256, 256, 40.0)],
                         ids=["block_sparse", "dense"])
def test_beside_a_contraction(gauss):
    """On the side stream of a batch with a Gaussian: the bits of a call alone."""
    n, nx, ny, h_cells = gauss
    wls = [case(150_000, 96, 70, 20.0, oracle.TRIWEIGHT, seed=937),
           workloads.random_points(938, n, 20.0 * max(nx, ny), 20.0, nx, ny, 20.0 * h_cells,
                                   oracle.GAUSSIAN),
           case(90_000, 300, 280, 18.0, oracle.EPANECHNIKOV, seed=939)]
    kids = ["triweight", "gaussian", "epanechnikov"]
    names = ("points", "weights", "origin", "cell", "nx", "ny", "h", "kernel")
    insts = [dict(zip(names, args(w) + (k,))) for w, k in zip(wls, kids)]
    for _ in range(2):
        out = kde.grid_batched(insts)
        for k in (0, 2):
            assert torch.equal(out[k], kde.grid(*args(wls[k]), kids[k]))
