"""The direct sums on inputs that are not finite: a NaN in one coordinate of a star or a
ray reaches both components, and a star exactly on a ray adds nothing whatever its mass."""
import numpy as np
import pytest
import torch

from paper_2211_00354_gb300 import lens

pytestmark = pytest.mark.gpu


def T(a):
    return torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


def forms(stars, masses, rays, prec):
    """y of the forms without and with the Jacobian (float64 alone: the float32 form
    with it takes a NaN distance for a star on the ray), and the Jacobian."""
    args = T(stars), T(masses), 0.1, 0.2, T(rays)
    y = lens.direct_deflect(*args, prec=prec).cpu().numpy()
    if prec == lens.FP32_BULK:
        return [y], None
    y2, J = lens.direct_deflect(*args, prec=prec, jacobian=True)
    return [y, y2.cpu().numpy()], J.cpu().numpy()


@pytest.mark.parametrize("prec", [lens.FP64, lens.FP32_BULK])
@pytest.mark.parametrize("n", [1, 7, 300])
@pytest.mark.parametrize("coordinate", [0, 1])
def test_nan_in_one_coordinate(prec, n, coordinate):
    rng = np.random.default_rng(n)
    stars, masses, rays = rng.normal(size=(n, 2)), rng.uniform(0.5, 1.5, n), rng.normal(size=(9, 2))
    bad = rays.copy()
    bad[4, coordinate] = np.nan
    ok = np.arange(9) != 4
    ys, J = forms(stars, masses, bad, prec)
    for y in ys + ([] if J is None else [J.reshape(9, 4)]):
        assert np.isnan(y[4]).all() and np.isfinite(y[ok]).all()
    s = stars.copy()
    s[n // 2, coordinate] = np.nan
    ys, J = forms(s, masses, rays, prec)
    for y in ys + ([] if J is None else [J]):
        assert np.isnan(y).all()


@pytest.mark.parametrize("mass", [np.inf, np.nan])
def test_a_star_on_the_ray_adds_nothing_whatever_its_mass(mass):
    stars, masses = np.array([[0.5, 0.25], [1.5, 0.25]]), np.array([mass, 2.0])
    ys, J = forms(stars, masses, [[0.5, 0.25], [0.5, 1.0]], lens.FP64)
    # only the other star: d = (-1, 0), m / d = -2, and m / d^2 = 2 in the Jacobian
    for y in ys:
        np.testing.assert_allclose(y[0], [0.7 * 0.5 + 2.0, 1.1 * 0.25], rtol=1e-15)
        assert not np.isfinite(y[1]).all()
    np.testing.assert_allclose(J[0].ravel(), [0.7 + 2.0, 0.0, 0.0, 1.1 - 2.0], rtol=1e-15, atol=0)
