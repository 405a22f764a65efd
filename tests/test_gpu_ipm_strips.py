"""Every cell of a pass is mapped once, however its fetches are dealt out to strips: grids of a
few cells to either side of the largest pass in strips, refinement levels, an affine lens
whose map is 1 / |det| in every pixel that the grid covers."""
import numpy as np
import pytest
import torch

from paper_2211_00354_gb300 import lens, synth

pytestmark = pytest.mark.gpu


def T(a):
    return torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


def affine(ks, g):
    # one star without mass: y = ((1 - ks - g) x1, (1 - ks + g) x2)
    return lens.LensFMM(T([[0.0, 0.0]]), T([0.0]), ks, g, p=4, leaf_size=4, target_box=(-5, 5, -5, 5))


@pytest.mark.parametrize("ks,g", [(0.0, 0.0), (0.9, 0.05)])
@pytest.mark.parametrize("nx,ny", [(1, 1), (7, 5), (40, 33), (333, 101), (1000, 997), (2000, 2001),
                                   (2508, 2508), (2509, 2509)])
def test_affine_map(ks, g, nx, ny):
    h = 9.0 / max(nx, ny)
    grid = synth.Grid(x0=-4.5, y0=-4.5, h=h, nx=nx, ny=ny)
    a, b = 1 - ks - g, 1 - ks + g
    # a window that holds the whole image of the grid, and no cell cut by its edge
    u = sorted((-4.5 * a, (-4.5 + nx * h) * a)), sorted((-4.5 * b, (-4.5 + ny * h) * b))
    pad = 0.1 * (u[0][1] - u[0][0]), 0.1 * (u[1][1] - u[1][0])
    box = (u[0][0] - pad[0], u[0][1] + pad[0], u[1][0] - pad[1], u[1][1] + pad[1])
    # at least 64 pixels for 4096 cells a pixel, so that it is one pass
    npx = max(12, int(np.ceil(np.sqrt(nx * ny / 64.0))))
    with affine(ks, g) as P:
        mp, st = P.ipm_map(grid, box, npx, npx)
    assert st["chunks"] == 1 and st["cells"] == nx * ny
    # each cell's fractions sum to 1, float32 sums of a thread's few thousand cells
    np.testing.assert_allclose(st["area_in_map"], nx * ny * h * h, rtol=1e-6)
    mp = mp.cpu().numpy()
    pu, pv = (box[1] - box[0]) / npx, (box[3] - box[2]) / npx
    np.testing.assert_allclose(mp.sum() * pu * pv, nx * ny * h * h, rtol=1e-5)
    # pixels wholly inside the grid's image; at most ~100 float32 additions each
    lo = [int(np.ceil((u[k][0] - box[2 * k]) / p + 0.01)) for k, p in ((0, pu), (1, pv))]
    hi = [int(np.floor((u[k][1] - box[2 * k]) / p - 0.01)) for k, p in ((0, pu), (1, pv))]
    inner = mp[lo[1]:hi[1], lo[0]:hi[0]]
    assert inner.size > 0
    np.testing.assert_allclose(inner, 1.0 / abs(a * b), rtol=2e-5)


@pytest.mark.parametrize("nx", [20, 300, 1100])
def test_refined_levels(nx):
    # every cell is over the cap of one pixel and split twice
    grid = synth.Grid(x0=-4.0, y0=-4.0, h=8.0 / nx, nx=nx, ny=nx)
    npx = int(1.5 * nx)
    with affine(0.0, 0.0) as P:
        mp, st = P.ipm_map(grid, (-5, 5, -5, 5), npx, npx, bbox_cap=1, refine_levels=2)
    assert st["cells_refined"] > 0
    total = st["area_in_map"] + st["area_outside"] + st["area_dropped"] + st["area_degenerate"]
    np.testing.assert_allclose(total, 64.0, rtol=1e-5)
