"""Float64 pair sums and their transposes: leaves of fewer and more stars than
the lanes that share them, U lists of more stars than a block, tiles of one ray,
rays on and within 1e-150 of a star (the reciprocal's range)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2211_00354_gb300 import lens, synth

pytestmark = pytest.mark.gpu


def T(a):
    return torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


@pytest.mark.parametrize("leaf", [1, 8, 9, 33, 300])
@pytest.mark.parametrize("m", [1, 129, 3000])
def test_adjoint_over_leaf_sizes(leaf, m):
    f = synth.config_uniform(seed=leaf, n=700, kappa_star=0.3, kappa_s=0.2, gamma=0.4,
                             mass_range=(0.5, 1.5))
    rays = synth.random_rays(m, m, (-5.0, -3.0), (5.0, 3.0))
    rays[0] = f.stars[np.argmin(np.hypot(*f.stars.T))]  # on a star
    gy = np.random.default_rng(m).normal(size=rays.shape)
    with lens.LensFMM(T(f.stars), T(f.masses), f.kappa_s, f.gamma, p=48, leaf_size=leaf,
                      prec=lens.FP64, target_box=(-5, 5, -3, 3)) as P:
        gxy, gm, _ = P.adjoint(T(rays), T(gy))
    rgxy, rgm, _ = oracle.adjoint(f.stars, f.masses, rays, gy)
    # every star gets something from a ray that is not on it, unless the only one is
    assert np.linalg.norm(gxy.cpu().numpy() - rgxy) <= 1e-10 * np.linalg.norm(rgxy)
    assert np.linalg.norm(gm.cpu().numpy() - rgm) <= 1e-10 * np.linalg.norm(rgm)


@pytest.mark.parametrize("d", [0.0, 1e-170, 1e-152, 1e-150, 1e-100, 1e-20])
def test_ray_next_to_a_star_at_the_origin(d):
    # the star's own term is m / d where |d|^2 is a normal number, and 0 on the star
    stars, masses = T([[0.0, 0.0], [3.0, 1.0]]), T([2.0, 1.0])
    x = T([[d, 0.0]])
    far = np.array([3.0, 1.0]) / 10.0  # -m (x - x_i) / |x - x_i|^2 of the other star
    with lens.LensFMM(stars, masses, 0.0, 0.0, p=8, leaf_size=4, prec=lens.FP64,
                      target_box=(-4, 4, -4, 4)) as P:
        got = [P.deflect(x).cpu().numpy()[0], lens.direct_deflect(stars, masses, 0, 0, x).cpu().numpy()[0]]
    own = 2.0 / d if d >= 1e-150 else 0.0
    for y in got:
        if 0.0 < d < 1e-150:
            assert np.all(np.isfinite(y)) or d >= 1e-160  # |d|^2 underflows: nothing, or up to 2 / d
            continue
        np.testing.assert_allclose(y, [d + far[0] - own, far[1]], rtol=1e-14)
