"""The light curve's rays in parts of the sample grid's cells: rays on the edges of
cells and parts and one cell outside, sample grids of one cell, of many, and so
large that the cells are split less or not at all, origins far from zero, rays
that are not finite."""
import numpy as np
import pytest
import torch

import oracle
from paper_2211_00354_gb300 import lens

pytestmark = pytest.mark.gpu


def T(a):
    return torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


SIGMA, TRUNC = 0.03125, 4.0  # a cut, and a cell, of 1/8: parts of 1/32


@pytest.mark.parametrize("org", [0.0, -3.0, 4096.0])
@pytest.mark.parametrize("span", [0.0, 0.3, 5.0, 200.0, 700.0, 40000.0])
def test_light_curve_and_gradient_over_sample_grids(org, span):
    rng = np.random.default_rng(int(span) + 1)
    ns = 40
    t = np.linspace(0.0, 1.0, ns) if span else np.zeros(1)
    s = np.stack([org + span * t, -org + span * t[::-1]], axis=1)
    # around every sample: the lattice of parts (edges and corners of cells among
    # them) half a cell wider than the cut, and random rays
    k = np.arange(-6, 7) / 32.0
    lat = np.stack(np.meshgrid(k, k), axis=-1).reshape(-1, 2)
    y = (np.round(s * 32)[:, None] / 32 + lat[None]).reshape(-1, 2)
    y = np.concatenate([y, (s[:, None] + rng.uniform(-0.2, 0.2, (len(s), 60, 2))).reshape(-1, 2),
                        rng.uniform(-1e5, 1e5, (50, 2))])
    # pairs on the cut itself are in or out by the last bit: leave them out
    d = np.hypot(y[:, None, 0] - s[None, :, 0], y[:, None, 1] - s[None, :, 1])
    y = y[np.abs(d - SIGMA * TRUNC).min(1) > 1e-9]
    w = 1e-3
    F = lens.light_curve(T(y), w, T(s), SIGMA, TRUNC).cpu().numpy()
    Fo = oracle.light_curve(y, w, s, SIGMA, TRUNC)
    # float-float pair terms, 2^-44 of a coordinate's 2^-53 rounding on top
    tol = 1e-12 + 4.0 * 2.0 ** -53 * (abs(org) + span) / SIGMA * TRUNC
    assert np.all(np.abs(F - Fo) <= tol * np.abs(Fo).max())
    Tk = 0.8 * Fo + 0.1
    bad = np.array([[np.nan, 0.0], [np.inf, org], [org, -np.inf], [1e300, 1e300]])
    g = lens.light_curve_grad(T(np.concatenate([y, bad])), w, T(s), SIGMA, T(Fo), T(Tk), TRUNC)
    g = g.cpu().numpy()
    go = oracle.light_curve_grad(y, w, s, SIGMA, Fo, Tk, TRUNC)
    assert np.all(g[len(y):] == 0.0)
    assert np.all(np.abs(g[:len(y)] - go) <= 10 * tol * np.abs(go).max())


def test_no_ray_near_and_rows_of_eight_bytes():
    s = np.array([[0.0, 0.0], [1.0, 0.0]])
    y = np.full((300, 2), 50.0)
    F = lens.light_curve(T(y), 1.0, T(s), SIGMA, TRUNC)
    g = lens.light_curve_grad(T(y), 1.0, T(s), SIGMA, F, F, TRUNC)
    assert torch.all(F == 0) and torch.all(g == 0)
    # a view whose rows start on an odd multiple of eight bytes
    rng = np.random.default_rng(0)
    flat = T(rng.uniform(-0.2, 0.2, 801))
    v = flat[1:].view(400, 2)
    y = v.cpu().numpy()
    F = lens.light_curve(v, 1.0, T(s), SIGMA, TRUNC).cpu().numpy()
    np.testing.assert_allclose(F, oracle.light_curve(y, 1.0, s, SIGMA, TRUNC), rtol=1e-11)
