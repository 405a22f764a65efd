"""The float64 pair sums' reciprocal over its whole range: one star of mass 1 at the origin,
no smooth field, so that a ray (d, 0) gets y = (-1/d, 0) through 1/d^2."""
import numpy as np
import pytest
import torch

from paper_2211_00354_gb300 import lens

pytestmark = pytest.mark.gpu


def T(a):
    return torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


def test_within_an_ulp_over_mantissas_and_exponents():
    rng = np.random.default_rng(1)
    k = np.arange(-511, 511)  # d^2 from the least normal number to beyond the range's upper end, 2^1021
    mant = 1.0 + rng.integers(0, 2 ** 25, (len(k), 64)) * 2.0 ** -25  # 26 bits: d^2 is exact
    mant[:, 0], mant[:, 1] = 1.0, 2.0 - 2.0 ** -25
    mant[:, 2], mant[:, 3] = 1.0 + 2.0 ** -20, 1.0 + 2.0 ** -21 - 2.0 ** -25  # about the coarse step
    d = np.ldexp(mant, k[:, None]).ravel()
    x = T(np.stack([d, np.zeros_like(d)], 1))
    y = lens.direct_deflect(T([[0.0, 0.0]]), T([1.0]), 1.0, 0.0, x).cpu().numpy()
    assert np.all(y[:, 1] == 0)
    # an ulp (2^-52 at most) for 1/d^2, half an ulp for its product with d; d^2 and the
    # lens equation round nothing
    rel = np.longdouble(y[:, 0]) * np.longdouble(d) + 1
    assert np.abs(rel).max() <= 1.5 * 2.0 ** -52


@pytest.mark.parametrize("d", [1e-152, 2e-154, 1.5e-154, 1e-170, 0.0])
def test_rays_where_the_squared_distance_ends(d):
    stars, masses = T([[0.0, 0.0], [3.0, 1.0]]), T([2.0, 1.0])
    x = T([[d, 0.0]])
    far = np.array([3.0, 1.0]) / 10.0
    with lens.LensFMM(stars, masses, 0.0, 0.0, p=8, leaf_size=4, prec=lens.FP64,
                      target_box=(-4, 4, -4, 4)) as P:
        got = [P.deflect(x).cpu().numpy()[0], lens.direct_deflect(stars, masses, 0, 0, x).cpu().numpy()[0]]
    # 2 / d where d^2 is a normal number, nothing where it is 0
    own = 2.0 / d if d * d > 0 else 0.0
    for y in got:
        np.testing.assert_allclose(y, [d + far[0] - own, far[1]], rtol=1e-14)
