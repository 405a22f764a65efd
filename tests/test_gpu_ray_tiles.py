"""Arbitrary rays in small tiles without a size read back: counts at the edges of
a tile and of the one-block offsets, fields with and without W boxes, both
precisions, and a ray outside the target region wherever it stands."""
import numpy as np
import pytest
import torch

import oracle
from paper_2211_00354_gb300 import lens, synth

pytestmark = pytest.mark.gpu


def T(a):
    return torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


@pytest.mark.parametrize("prec", [lens.FP32_BULK, lens.FP64])
@pytest.mark.parametrize("field,leaf", [("uniform", 8), ("uniform", 600), ("clustered", 8)])
@pytest.mark.parametrize("m", [1, 31, 127, 128, 129, 257, 4000])
def test_rays_match_the_oracle(prec, field, leaf, m):
    if field == "uniform":
        f = synth.config_uniform(seed=1, n=1200, kappa_star=0.4, kappa_s=0.1, gamma=0.2,
                                 mass_range=(0.5, 1.5))
    else:
        f = synth.c3_clustered(seed=2, n_clusters=10, per_cluster=150)
    x = synth.random_rays(m, m, (-7.0, -5.0), (7.0, 5.0))
    with lens.LensFMM(T(f.stars), T(f.masses), f.kappa_s, f.gamma, p=40, leaf_size=leaf, prec=prec,
                      target_box=(-7, 7, -5, 5)) as P:
        y, J = (t.cpu().numpy() for t in P.deflect(T(x), jacobian=True))
        y2 = P.deflect(T(x)).cpu().numpy()
    ref, Jref = oracle.deflect(f.stars, f.masses, f.kappa_s, f.gamma, x, jacobian=True)
    d = x[:, None, :] - f.stars[None]
    r = np.hypot(d[..., 0], d[..., 1])
    # float32 terms: a few 2^-24 each, up to eight more in a partial sum; the
    # order-40 expansions and float64 are far below that
    eps = 16 * 2.0 ** -24 if prec == lens.FP32_BULK else 1e-10
    b1, b2 = eps * (f.masses / r).sum(1), 2 * eps * (f.masses / r ** 2).sum(1)
    for v in (y, y2):
        assert np.all(np.hypot(*(v - ref).T) <= b1)
    assert np.all(np.abs(J.reshape(m, 4) - Jref.reshape(m, 4)).max(1) <= b2)


@pytest.mark.parametrize("prec", [lens.FP32_BULK, lens.FP64])
@pytest.mark.parametrize("bad", [0, 700, 1499])
@pytest.mark.parametrize("value", [1e6, np.nan, np.inf])
def test_a_ray_outside_is_refused_and_the_plan_goes_on(prec, bad, value):
    f = synth.config_uniform(seed=3, n=400, kappa_star=0.3, kappa_s=0.0, gamma=0.1)
    x = synth.random_rays(4, 1500, (-3.0, -3.0), (3.0, 3.0))
    z = x.copy()
    z[bad, bad % 2] = value
    with lens.LensFMM(T(f.stars), T(f.masses), f.kappa_s, f.gamma, p=24, leaf_size=8, prec=prec,
                      target_box=(-3, 3, -3, 3)) as P:
        want = P.deflect(T(x))
        for call in (P.deflect, P.potential, lambda r: P.adjoint(r, torch.ones_like(r))):
            with pytest.raises(lens.LensError) as ei:
                call(T(z))
            assert ei.value.status == lens.LENS_EDOMAIN
            assert torch.equal(P.deflect(T(x)), want)


def test_more_leaves_than_one_block_scans():
    # over 16384 active leaves: the offsets by the general scans
    f = synth.config_uniform(seed=5, n=60000, kappa_star=0.4, kappa_s=0.0, gamma=0.0)
    R = np.hypot(*f.stars.T).max()
    x = synth.random_rays(6, 3000, (-0.6 * R, -0.6 * R), (0.6 * R, 0.6 * R))
    with lens.LensFMM(T(f.stars), T(f.masses), 0.0, 0.0, p=24, leaf_size=2,
                      prec=lens.FP64) as P:
        assert P.info()["n_active_leaves"] > 16384
        y = P.deflect(T(x)).cpu().numpy()
    ref = oracle.deflect(f.stars, f.masses, 0.0, 0.0, x)
    d = x[:, None, :] - f.stars[None]
    assert np.all(np.hypot(*(y - ref).T) <= 1e-6 * (f.masses / np.hypot(d[..., 0], d[..., 1])).sum(1))
