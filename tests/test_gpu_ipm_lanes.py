"""Chunks of 4, 8, 16 and 32 cells a warp: a map in one pass against bands of rows whose
cells make shorter chunks, and a refined map against the oracle's totals."""
import numpy as np
import pytest
import torch

from paper_2211_00354_gb300 import lens, synth

pytestmark = pytest.mark.gpu


def T(a):
    return torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


@pytest.fixture(scope="module")
def whole():
    f = synth.config_uniform(seed=3, n=400, kappa_star=0.4, kappa_s=0.0, gamma=0.2)
    n = 700
    grid = synth.Grid(x0=-5.0, y0=-5.0, h=10.0 / n, nx=n, ny=n)
    P = lens.LensFMM(T(f.stars), T(f.masses), f.kappa_s, f.gamma, p=16, leaf_size=8,
                     prec=lens.FP32_BULK, target_box=(-5, 5, -5, 5))
    mp, st = P.ipm_map(grid, (-2.0, 2.0, -2.0, 2.0), 90, 90, bbox_cap=64)
    yield P, grid, mp.cpu().numpy(), st
    P.close()


@pytest.mark.parametrize("rows", [1, 7, 28, 56, 112, 223, 699])
def test_bands_of_any_chunk_agree(whole, rows):
    P, grid, mp, st = whole
    m2, s2 = P.ipm_map(grid, (-2.0, 2.0, -2.0, 2.0), 90, 90, bbox_cap=64,
                       max_cells_per_chunk=rows * grid.nx)
    m2 = m2.cpu().numpy()
    # float32 additions in another order, as between chunkings before
    np.testing.assert_allclose(m2, mp, rtol=2e-6, atol=1e-6 * np.abs(mp).max())
    for k in ("cells", "cells_dropped", "cells_degenerate", "cells_ext"):
        assert s2[k] == st[k]
    for k in ("area_in_map", "area_outside", "area_dropped"):
        assert s2[k] == pytest.approx(st[k], rel=1e-6, abs=1e-6 * st["area_total"])


@pytest.mark.parametrize("levels", [0, 1, 2, 3])
def test_refined_ledger_adds_up(whole, levels):
    P, grid, mp, st = whole
    m2, s2 = P.ipm_map(grid, (-2.0, 2.0, -2.0, 2.0), 90, 90, bbox_cap=6, refine_levels=levels)
    led = sum(s2[k] for k in ("area_in_map", "area_outside", "area_dropped", "area_degenerate"))
    assert abs(led - s2["area_total"]) <= 1e-6 * s2["area_total"]
    pix = (4.0 / 90) ** 2
    assert abs(float(m2.sum()) * pix - s2["area_in_map"]) <= 2e-6 * s2["area_total"]
