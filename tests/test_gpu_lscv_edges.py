"""The LSCV loss's point terms at and beyond the grid's edges, against the FP64 oracle:
a point's cell is found in 32 bits, and points far outside must stay outside."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2004_13653_gb300 as kde  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    kde.load(build_if_stale=True)


@pytest.mark.parametrize("nx,ny", [(1, 1), (1, 9), (37, 1), (37, 21)])
def test_points_on_and_far_beyond_every_edge(nx, ny):
    cell, h = 2.0, 5.0
    rng = np.random.default_rng(nx)
    inside = rng.uniform(0.0, 1.0, (40, 2)) * [nx * cell, ny * cell]
    x = np.array([-3e12, -5e9, -2.0, -1.0, -0.5, 0.0, 1.0, nx * cell - 1.0, nx * cell,
                  nx * cell + 1.0, nx * cell + 2.0, 5e9, 3e12])
    y = np.array([-3e12, -1.0, -0.5, 1.0, ny * cell - 1.0, ny * cell + 0.5, 5e9, 3e12])
    xy = np.concatenate([inside, np.stack(np.meshgrid(x, y), -1).reshape(-1, 2)])
    w = rng.uniform(0.5, 1.5, len(xy)).astype(np.float32)
    F = rng.uniform(0.5, 1.0, (ny, nx)).astype(np.float32)
    pts = torch.as_tensor(xy, device="cuda")
    loss, G, gw, gxy, _ = kde.lscv_grid(torch.as_tensor(F, device="cuda"), pts,
                                        torch.as_tensor(w, device="cuda"), (0.0, 0.0), cell, nx, ny, h)
    ref = oracle.lscv_loss(F.astype(np.float64), xy, w, (0.0, 0.0), cell, nx, ny, h)
    # FP64 sums of terms of one size; positions to 2^-46
    assert float(loss) == pytest.approx(ref, rel=1e-9)
    refG = oracle.lscv_cotangent(F.astype(np.float64), xy, w, (0.0, 0.0), cell, nx, ny)
    np.testing.assert_allclose(G.cpu().numpy(), refG, rtol=1e-6, atol=1e-6 * np.abs(refG).max())
    out = (xy[:, 0] < -cell) | (xy[:, 1] < -cell) | (xy[:, 0] > (nx + 1) * cell) | \
        (xy[:, 1] > (ny + 1) * cell)
    assert out.any() and not gw.cpu().numpy()[out].any() and not gxy.cpu().numpy()[out].any()
