"""Values at the ends of the integer-pipe conversions: offsets that are zero or far
below float32's normal range, masses that are zero or subnormal in float32, cells
on the root box's edges, negative zero; a field in both precisions over rays, a grid
and a map."""
import numpy as np
import pytest
import torch

import oracle
from paper_2211_00354_gb300 import lens, synth

pytestmark = pytest.mark.gpu


def T(a):
    return torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


def field(scale):
    # a dyadic lattice: stars on box corners and centres at every level, some
    # moved by amounts that vanish in float32 or in the box
    g = np.arange(-8, 9) * 0.5
    st = np.stack(np.meshgrid(g, g), axis=-1).reshape(-1, 2)
    st[st == 0.0] = -0.0
    st[::3] += 0.125
    st[1::7] += 2.0 ** -40
    st[2::11, 0] = 2.0 ** -80
    st[3::13, 1] = -1e-45
    m = np.full(len(st), 1.0)
    m[::5], m[1::5], m[2::5] = 0.0, 1e-41, 1.0 + 2.0 ** -24
    m[3::5] = 1.0 + 2.0 ** -23 + 2.0 ** -24  # ties: one to even below, one above
    # a scale for the lengths (masses go with their square)
    return st * scale, m * scale * scale


@pytest.mark.parametrize("prec", [lens.FP32_BULK, lens.FP64])
@pytest.mark.parametrize("scale", [1.0, 2.0 ** -12, 2.0 ** 20, 3.7e3])
def test_offsets_and_masses_at_the_ends_of_float32(prec, scale):
    st, m = field(scale)
    L = 4.25 * scale
    x = synth.random_rays(1, 1500, (-L, -L), (L, L))
    x[0] = (0.0, -0.0)
    x[1] = (2.0 ** -70 * scale, -2.0 ** -100 * scale)
    x[2:40] = st[5:43] + 2.0 ** -9 * scale
    r = np.hypot(x[:, None, 0] - st[None, :, 0], x[:, None, 1] - st[None, :, 1])
    x = x[r.min(1) > 1e-6 * scale]
    r = np.hypot(x[:, None, 0] - st[None, :, 0], x[:, None, 1] - st[None, :, 1])
    n = 64
    grid = synth.Grid(x0=-L, y0=-L, h=2 * L / n, nx=n, ny=n)
    with lens.LensFMM(T(st), T(m), 0.1, 0.2, p=40, leaf_size=4, prec=prec,
                      target_box=(-L, L, -L, L)) as P:
        y = P.deflect(T(x)).cpu().numpy()
        yg = P.deflect_grid(grid).cpu().numpy().reshape(-1, 2)
    # float32 terms of a few 2^-24 each, 2^-24 for a mass; a mass below
    # float32's normal range may go to zero
    eps = 16 * 2.0 ** -24 if prec == lens.FP32_BULK else 1e-10
    ref = oracle.deflect(st, m, 0.1, 0.2, x)
    assert np.all(np.hypot(*(y - ref).T) <= eps * (m / r).sum(1) + 1e-30)
    c = grid.corners().reshape(-1, 2)
    rg = np.hypot(c[:, None, 0] - st[None, :, 0], c[:, None, 1] - st[None, :, 1])
    ok = rg.min(1) > 1e-6 * scale
    refg = oracle.deflect(st, m, 0.1, 0.2, c[ok])
    assert np.all(np.hypot(*(yg[ok] - refg).T) <= eps * (m / rg[ok]).sum(1) + 1e-30)
