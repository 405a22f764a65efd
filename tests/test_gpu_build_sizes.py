"""Plan builds over the sizes at which the tree's scans change form (one block
up to 32768 entries, then the general scan) and the read-backs of an almost
empty tree; maps on both sides of the grid size up to which the rows of a chunk
are taken without asking for the free memory."""
import numpy as np
import pytest
import torch

import oracle
from paper_2211_00354_gb300 import lens, synth

pytestmark = pytest.mark.gpu


def T(a):
    return torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


@pytest.mark.parametrize("prec", [lens.FP32_BULK, lens.FP64])
@pytest.mark.parametrize("n,leaf", [(1, 1), (2, 1), (5, 1), (300, 300), (3000, 2), (26000, 2),
                                    (27500, 2), (29000, 2), (150000, 2)])
def test_trees_of_all_sizes_match_the_oracle(prec, n, leaf):
    f = synth.config_uniform(seed=n, n=n, kappa_star=0.3, kappa_s=0.1, gamma=0.2,
                             mass_range=(0.5, 1.5))
    L = float(np.abs(f.stars).max()) + 0.5
    x = synth.random_rays(7, 200, (-L, -L), (L, L))
    with lens.LensFMM(T(f.stars), T(f.masses), f.kappa_s, f.gamma, p=40, leaf_size=leaf, prec=prec,
                      target_box=(-L, L, -L, L)) as P:
        info = P.info()
        y = P.deflect(T(x)).cpu().numpy()
    print(n, info["n_boxes"], info["n_active_leaves"], info["n_active_boxes"])
    if n == 3000:
        assert info["n_boxes"] < 32768
    if n == 150000:
        assert min(info["n_active_leaves"], info["n_active_boxes"]) > 32768
    ref = oracle.deflect(f.stars, f.masses, f.kappa_s, f.gamma, x)
    r = np.hypot(x[:, None, 0] - f.stars[None, :, 0], x[:, None, 1] - f.stars[None, :, 1])
    # float32 terms of a few 2^-24 each; order 40 leaves 10 * 0.547^41 of a term
    eps = 16 * 2.0 ** -24 if prec == lens.FP32_BULK else 1e-9
    assert np.all(np.hypot(*(y - ref).T) <= eps * (f.masses / r).sum(1))


@pytest.mark.parametrize("nx", [1, 2048, 2049])
def test_maps_of_grids_about_the_memory_query(nx):
    # y = diag(0.45, 1.05) x exactly; the grid's image covers the map
    ks, g = 0.25, 0.3
    h = 12.0 / nx
    grid = synth.Grid(x0=-6.0, y0=-6.0, h=h, nx=nx, ny=nx)
    with lens.LensFMM(T([[0.0, 0.0]]), T([0.0]), ks, g, p=4, leaf_size=4, prec=lens.FP32_BULK,
                      target_box=(-6, 6, -6, 6)) as P:
        mp, st = P.ipm_map(grid, (-1.0, 1.0, -2.0, 2.0), 64, 80)
    # float32 fractions of up to ~(0.031/0.0026)(0.05/0.0062) = 97 cells a pixel:
    # 97 roundings of 2^-24 at most
    np.testing.assert_allclose(mp.cpu().numpy(), 1 / (0.45 * 1.05), rtol=97 * 2.0 ** -24 + 2e-6)
    assert st["cells"] == nx * nx
