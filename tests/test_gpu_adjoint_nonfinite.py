"""The float64 adjoint where a ray's gradient is not finite: the star that the ray lies on
takes nothing from it, every other star does."""
import numpy as np
import pytest
import torch

from paper_2211_00354_gb300 import lens

pytestmark = pytest.mark.gpu


def T(a):
    return torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan])
@pytest.mark.parametrize("m", [2, 130])
def test_the_star_on_the_ray_takes_nothing(value, m):
    rng = np.random.default_rng(m)
    stars, masses = np.array([[0.5, 0.25], [1.5, -0.75], [-0.5, 0.5]]), np.array([1.0, 2.0, 0.5])
    rays, gy = rng.uniform(-1, 1, (m, 2)), rng.normal(size=(m, 2))
    rays[m // 2] = stars[0]
    gy[m // 2] = 0.0
    with lens.LensFMM(T(stars), T(masses), 0.0, 0.1, p=8, leaf_size=4, prec=lens.FP64,
                      target_box=(-2, 2, -2, 2)) as P:  # one leaf: pairs alone
        want = [t.cpu().numpy() for t in P.adjoint(T(rays), T(gy))]
        gy[m // 2] = value
        gxy, gm, _ = (t.cpu().numpy() for t in P.adjoint(T(rays), T(gy)))
    np.testing.assert_allclose(gxy[0], want[0][0], rtol=1e-13)
    np.testing.assert_allclose(gm[0], want[1][0], rtol=1e-13)
    assert not np.isfinite(gxy[1:]).any() and not np.isfinite(gm[1:]).any()
