"""The potential's near field of millions of stars at distances of 2^-490: the sum of the
squared distances' exponents is beyond 32 bits."""
import numpy as np
import pytest
import torch

from paper_2211_00354_gb300 import lens

pytestmark = pytest.mark.gpu


def T(a):
    return torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


@pytest.mark.parametrize("power", [-490, 0])
def test_many_stars_next_to_a_large_leaf(power):
    # a strip of stars along the middle of the right-hand side of the box [0, 1/2]^2 of
    # the unit square: all of its leaves touch that box, one leaf, where the rays are
    n = 2_400_000
    rng = np.random.default_rng(1)
    s = np.stack([0.5 + rng.uniform(1e-6, 1e-5, n), rng.uniform(0.01, 0.49, n)], 1)
    s = np.concatenate([s, [[0.0, 0.0], [1.0, 1.0]]])  # the tree's corners
    x = np.array([[0.25, 0.25], [0.375, 0.125], [0.3, 0.45]])
    m = 2.0 ** -20
    scale = 2.0 ** power
    with lens.LensFMM(T(s * scale), T(np.full(len(s), m)), 0.0, 0.0, p=16, leaf_size=1024,
                      prec=lens.FP64, target_box=tuple(scale * np.array([0.25, 0.375, 0.125, 0.45]))) as P:
        i = P.info()
        assert i["n_active_leaves"] == 1 and i["u_stars"] > n
        psi = P.potential(T(x * scale)).cpu().numpy()
    d = x[:, None] - s[None]
    want = m * (0.5 * np.log((d * d).sum(-1)) + power * np.log(2.0)).sum(1)
    # exponents exact, one rounding of a product of mantissas a star
    np.testing.assert_allclose(psi, want, rtol=0, atol=4 * 2.0 ** -53 * n * m + 1e-12 * np.abs(want).max())
