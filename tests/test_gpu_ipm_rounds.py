"""The map kernel's rounds of 32 cells on affine lenses (a massless star):
grids whose cell counts straddle the warp, the chunk and the fetch sizes, with
cells of one or two pixels, small boxes and large boxes, against the oracle's
scalar IPM of the exact corners."""
import numpy as np
import pytest
import torch

import oracle
from paper_2211_00354_gb300 import lens, synth

pytestmark = pytest.mark.gpu


def T(a):
    return torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


def affine_map(nx, ny, ks, g, h, half, npix):
    grid = synth.Grid(x0=-0.5 * nx * h + 0.13 * h, y0=-0.5 * ny * h - 0.21 * h, h=h, nx=nx, ny=ny)
    R = max(abs(grid.x0), abs(grid.y0), nx * h, ny * h)
    with lens.LensFMM(T([[0.0, 0.0]]), T([0.0]), ks, g, p=4, leaf_size=4, prec=lens.FP64,
                      target_box=(-R, R, -R, R)) as P:
        mp, st = P.ipm_map(grid, (-half, half, -half, half), npix, npix)
    return grid, mp.cpu().numpy(), st


# (kappa_s, gamma): cells of 0.02 x 0.4, 0.7 x 2.1, 8.4 x 8.4 pixels (pixel 0.1, h below)
@pytest.mark.parametrize("ks,g,h", [(0.525, 0.425, 0.04), (0.5, 0.25, 0.28), (-3.0, 0.0, 0.21)])
@pytest.mark.parametrize("nx,ny", [(1, 1), (31, 3), (33, 2), (257, 65), (64, 128)])
def test_affine_cells_match_the_oracle(ks, g, h, nx, ny):
    grid, mp, st = affine_map(nx, ny, ks, g, h, 2.0, 40)
    y = grid.corners() * np.array([1 - ks - g, 1 - ks + g])
    ref, st_ref = oracle.ipm_map(y, grid.h, (-2.0, 2.0, -2.0, 2.0), 40, 40)
    # a float32 corner carries 2^-24 of a pixel; the thinnest cells here have
    # an area of 0.008 pixel^2, so a fraction is good to ~1e-5 and a pixel's
    # sum to 1e-4 of the largest with room for its few hundred terms
    np.testing.assert_allclose(mp, ref, rtol=1e-4, atol=1e-4 * np.abs(ref).max())
    assert st["area_in_map"] == pytest.approx(st_ref["area_in_map"], rel=1e-5,
                                              abs=1e-5 * st_ref["area_total"])


@pytest.mark.parametrize("nx,ny", [(1100, 1200), (2600, 2600), (3400, 3300)])
def test_large_grids_cover_every_pixel_once(nx, ny):
    # fetches of one, several and the most chunks; at most 64 cells a pixel
    # between flushes drift by up to 64 2^-25, and as much again for the fractions
    ks, g = 0.2, 0.3
    h = 8.0 / nx
    _, mp, st = affine_map(nx, ny, ks, g, h, 1.0, 200)
    np.testing.assert_allclose(mp, 1.0 / ((1 - ks - g) * (1 - ks + g)), rtol=4e-6)
    led = st["area_in_map"] + st["area_outside"] + st["area_dropped"] + st["area_degenerate"]
    assert abs(led - st["area_total"]) <= 1e-6 * st["area_total"]
