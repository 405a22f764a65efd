"""Float32-bulk grid deflections (2 x 2 blocks of rays a thread): odd, narrow
and one-row grids, leaves of few and of many rays, near fields longer than
one staging, W boxes, bands of rows, equal and unequal masses."""
import numpy as np
import pytest
import torch

import oracle
from paper_2211_00354_gb300 import lens, synth

pytestmark = pytest.mark.gpu


def T(a):
    return torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


FIELDS = {
    "equal": lambda: synth.config_uniform(seed=5, n=1500, kappa_star=0.4, kappa_s=0.1, gamma=0.2),
    "unequal": lambda: synth.config_uniform(seed=6, n=1500, kappa_star=0.4, kappa_s=0.1, gamma=0.2,
                                            mass_range=(0.5, 1.5)),
    "clustered": lambda: synth.c3_clustered(seed=7, n_clusters=12, per_cluster=200),
}


@pytest.mark.parametrize("field,leaf", [("equal", 4), ("equal", 128), ("unequal", 16),
                                        ("clustered", 8), ("clustered", 64)])
@pytest.mark.parametrize("nx,ny", [(1, 1), (1, 40), (40, 1), (6, 7), (64, 65), (255, 30)])
def test_grid_blocks_match_the_oracle_in_any_band(field, leaf, nx, ny):
    f = FIELDS[field]()
    h = 12.0 / max(nx, ny)
    grid = synth.Grid(x0=-5.7, y0=-6.1, h=h, nx=nx, ny=ny)
    box = (grid.x0, grid.x0 + nx * h, grid.y0, grid.y0 + ny * h)
    with lens.LensFMM(T(f.stars), T(f.masses), f.kappa_s, f.gamma, p=24, leaf_size=leaf,
                      prec=lens.FP32_BULK, target_box=box) as P:
        # a band's first row starts other 2 x 2 blocks
        bands = {row0: P.deflect_grid(grid, row0=row0).cpu().numpy() for row0 in (0, ny // 2, ny)}
    x = grid.corners()
    ref = oracle.deflect(f.stars, f.masses, f.kappa_s, f.gamma, x.reshape(-1, 2)).reshape(x.shape)
    # a float32 term m / |d| carries a few 2^-24, a sum of eight up to eight more
    # of its absolute terms; the groups add up without rounding
    d = x[:, :, None, :] - f.stars[None, None]
    bound = 16 * 2.0 ** -24 * (f.masses / np.hypot(d[..., 0], d[..., 1])).sum(-1)
    for row0, y in bands.items():
        assert y.shape == x[row0:].shape
        assert np.all(np.hypot(*np.moveaxis(y - ref[row0:], -1, 0)) <= bound[row0:])
