"""Ill-conditioned cells, a lane a cell: point lenses whose folded cells reach boxes of a
few pixels, of hundreds and beyond the size a lane takes, with and without a cap, in
queues of less than a warp and of many, against the oracle's scalar apportionment."""
import numpy as np
import pytest
import torch

import oracle
from paper_2211_00354_gb300 import lens, synth

pytestmark = pytest.mark.gpu


def T(a):
    return torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


@pytest.mark.parametrize("nstar,ncell", [(1, 24), (1, 120), (40, 90), (40, 400)])
@pytest.mark.parametrize("npix", [7, 60, 500, 1500])
@pytest.mark.parametrize("cap", [0, 64])
def test_folded_cells_of_all_sizes(nstar, ncell, npix, cap):
    rng = np.random.default_rng(nstar)
    st = rng.uniform(-1.5, 1.5, (nstar, 2))
    m = np.full(nstar, 1.0 / nstar)
    h = 4.0 / ncell
    grid = synth.Grid(x0=-2.0, y0=-2.0, h=h, nx=ncell, ny=ncell)
    box = (-1.0, 1.0, -1.0, 1.0)
    y = oracle.deflect(st, m, 0.2, 0.3, grid.corners().reshape(-1, 2)).reshape(ncell + 1, ncell + 1, 2)
    ref, rs = oracle.ipm_map(y, h, box, npix, npix, bbox_cap=cap)
    with lens.LensFMM(T(st), T(m), 0.2, 0.3, p=40, leaf_size=8, prec=lens.FP64,
                      target_box=(-2, 2, -2, 2)) as P:
        mp, s = P.ipm_map(grid, box, npix, npix, bbox_cap=cap)
    mp = mp.cpu().numpy()
    print(nstar, ncell, npix, cap, {k: v for k, v in s.items() if "cell" in k})
    # the mean error of a map the repository's tests allow (the difference arrays leave
    # float32 roundings of a row's sums in all of its pixels), and that of its peaks
    assert np.abs(mp - ref).sum() <= 1e-3 * np.abs(ref).sum()
    assert np.abs(mp - ref).max() <= 2e-2 * np.abs(ref).max()
    for k in ("area_in_map", "area_outside", "area_dropped", "area_degenerate"):
        assert s[k] == pytest.approx(rs[k], rel=1e-5, abs=2e-6 * rs["area_total"])


@pytest.mark.parametrize("npix", [50, 800])
def test_long_queues_agree_with_short_ones(npix):
    # one chunk (a queue of thousands, several cells a warp) against bands of a few
    # rows (a cell a warp): the same cells, the same fractions, other orders of
    # float32 additions
    rng = np.random.default_rng(3)
    st = rng.uniform(-2, 2, (3000, 2))
    m = np.full(3000, 1.5e-3)
    n = 3000
    grid = synth.Grid(x0=-2.0, y0=-2.0, h=4.0 / n, nx=n, ny=n)
    box = (-0.7, 0.7, -0.7, 0.7)
    with lens.LensFMM(T(st), T(m), 0.0, 0.3, p=16, leaf_size=8, prec=lens.FP32_BULK,
                      target_box=(-2, 2, -2, 2)) as P:
        a, sa = P.ipm_map(grid, box, npix, npix, bbox_cap=64)
        b, sb = P.ipm_map(grid, box, npix, npix, bbox_cap=64, max_cells_per_chunk=40 * n)
    print({k: v for k, v in sa.items() if "cells" in k})
    assert sa["cells_ext"] == sb["cells_ext"] > 2432
    a, b = a.cpu().numpy(), b.cpu().numpy()
    # ~1e4 additions of 2^-24 a pixel at the coarser map, in random order
    assert np.linalg.norm(a - b) <= 1e-5 * np.linalg.norm(b)
    assert np.abs(a - b).max() <= 1e-4 * np.abs(b).max()
    for k in ("area_in_map", "area_outside", "area_dropped", "area_degenerate"):
        assert sa[k] == pytest.approx(sb[k], rel=1e-6, abs=1e-6 * sa["area_total"])
