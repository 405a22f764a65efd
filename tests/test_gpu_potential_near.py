"""The potential's near field: equal and unequal masses, leaves whose U lists
exceed one run of mantissa products, W boxes below and above the size summed
directly, one ray and many, rays on a star and so near it that the squared
distance is subnormal or vanishes."""
import math

import numpy as np
import pytest
import torch

import oracle
from paper_2211_00354_gb300 import lens, synth

pytestmark = pytest.mark.gpu


def T(a):
    return torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


def scale(stars, masses, x):
    d = np.hypot(x[:, None, 0] - stars[None, :, 0], x[:, None, 1] - stars[None, :, 1])
    return np.sum(masses * (1.0 + np.abs(np.log(np.where(d > 1e-200, d, 1.0)))), axis=1)


@pytest.mark.parametrize("equal", [True, False])
@pytest.mark.parametrize("leaf,clusters", [(2, 8), (12, 8), (60, 8), (200, 0), (1024, 0)])
@pytest.mark.parametrize("m", [1, 37, 2000])
def test_potential_near_field(equal, leaf, clusters, m):
    rng = np.random.default_rng(leaf)
    if clusters:
        f = synth.c3_clustered(seed=leaf, n_clusters=clusters, per_cluster=250)
        stars, box = f.stars, (-9.0, 9.0, -7.0, 7.0)
    else:
        stars, box = synth.uniform_disk(rng, 4000, 8.0), (-6.0, 6.0, -5.0, 5.0)
    masses = np.full(len(stars), 0.7) if equal else rng.lognormal(0.0, 1.0, len(stars))
    x = np.stack([rng.uniform(box[0], box[1], m), rng.uniform(box[2], box[3], m)], axis=1)
    inside = np.flatnonzero((np.abs(stars[:, 0]) < box[1]) & (np.abs(stars[:, 1]) < box[3]))
    x[0] = stars[inside[0]] if len(inside) else x[0]  # on a star: it adds nothing
    with lens.LensFMM(T(stars), T(masses), 0.1, 0.2, p=48, leaf_size=leaf, prec=lens.FP64,
                      target_box=box) as P:
        psi = P.potential(T(x)).cpu().numpy()
    ref = oracle.potential(stars, masses, 0.1, 0.2, x)
    assert np.max(np.abs(psi - ref) / scale(stars, masses, x)) < 1e-12


@pytest.mark.parametrize("d", [0.0, 1e-170, 3e-160, 1e-150, 1e-30])
@pytest.mark.parametrize("masses", [(2.0, 2.0), (2.0, 1.0)])
def test_potential_next_to_a_star_at_the_origin(d, masses):
    with lens.LensFMM(T([[0.0, 0.0], [3.0, 1.0]]), T(masses), 0.0, 0.0, p=8, leaf_size=4,
                      prec=lens.FP64, target_box=(-4, 4, -4, 4)) as P:
        psi = P.potential(T([[d, 0.0]])).item()
    want = masses[1] * 0.5 * math.log(10.0)
    if d * d > 0.0:
        want += masses[0] * 0.5 * math.log(d * d)
    assert psi == pytest.approx(want, rel=1e-14)
