"""Calls too small for the forms made for large ones: a finite source of a few pixels on
small maps (one pass up to 2^16 pixels and R = 4), and the light curve's gradient of few
rays (taken as they come up to 4096), on both sides of each line."""
import math

import numpy as np
import pytest
import torch

import oracle
from paper_2211_00354_gb300 import lens

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ny,nx", [(256, 256), (256, 257), (16, 16), (300, 400)])
@pytest.mark.parametrize("sigma,trunc", [(0.3, 3.0), (0.8, 5.0), (1.0, 5.0)])  # R = 0, 4, 5
def test_small_sources(ny, nx, sigma, trunc):
    rng = np.random.default_rng(ny + nx)
    m = 0.1 + 10.0 * rng.random((ny, nx))
    R, cut = int(math.floor(trunc * sigma)), (trunc * sigma) ** 2
    num, den = np.zeros_like(m), np.zeros_like(m)
    for dy in range(-R, R + 1):
        ys, yd = slice(max(0, -dy), ny - max(0, dy)), slice(max(0, dy), ny - max(0, -dy))
        for dx in range(-R, R + 1):
            if dx * dx + dy * dy > cut:
                continue
            w = math.exp(-(dx * dx + dy * dy) / (2.0 * sigma * sigma))
            xs, xd = slice(max(0, -dx), nx - max(0, dx)), slice(max(0, dx), nx - max(0, -dx))
            num[ys, xs] += w * m[yd, xd]
            den[ys, xs] += w
    got = lens.map_source(torch.tensor(m, device="cuda"), sigma, trunc).cpu().numpy()
    # positive sums of at most ~100 float-float terms, 2^-47 each
    np.testing.assert_allclose(got, num / den, rtol=128 * 2.0 ** -47)


@pytest.mark.parametrize("n", [1, 31, 4095, 4096, 4097])
def test_gradient_of_few_rays(n):
    rng = np.random.default_rng(n)
    y = rng.uniform(-1.2, 1.2, (n, 2))
    y[0] = 0.0
    t = np.linspace(-0.9, 0.9, 60)
    s = np.stack([t, 0.4 * t], axis=1)
    Fo = oracle.light_curve(y, 1e-3, s, 0.05)
    T = lambda a: torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")
    g = lens.light_curve_grad(T(y), 1e-3, T(s), 0.05, T(Fo), T(0.8 * Fo + 0.1)).cpu().numpy()
    go = oracle.light_curve_grad(y, 1e-3, s, 0.05, Fo, 0.8 * Fo + 0.1)
    # float-float pairs: 2^-44 of the terms summed for a ray (they cancel at y = 0)
    d = y[:, None] - s[None]
    G = 1e-3 / (2 * np.pi * 0.05 ** 2) * np.exp(-(d ** 2).sum(2) / (2 * 0.05 ** 2))
    S = (np.abs(2 * (0.2 * Fo - 0.1)) * G * np.hypot(d[..., 0], d[..., 1])).sum(1) / 0.05 ** 2
    assert np.all(np.abs(g - go).max(1) <= 60 * 2.0 ** -44 * S + 1e-300)
    far = np.abs(y[:, 1] - 0.4 * y[:, 0]) > 0.4  # beyond 6 sigma of the track
    assert np.all(g[far] == 0.0)
