"""The float32 adjoint on either side of the number of rays from which its tiles are twice
as large, with a last tile of few rays, against the sums over all pairs in float64."""
import numpy as np
import pytest
import torch

from paper_2211_00354_gb300 import lens, synth

pytestmark = pytest.mark.gpu


def T(a):
    return torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


@pytest.mark.parametrize("m", [2 ** 19 - 1, 2 ** 19, 2 ** 19 + 77])
@pytest.mark.parametrize("leaf", [8, 300])
def test_large_tiles_match_the_pair_sums(m, leaf):
    f = synth.config_uniform(seed=4, n=300, kappa_star=0.3, kappa_s=0.2, gamma=0.4, mass_range=(0.5, 1.5))
    S, M = T(f.stars), T(f.masses)
    x = T(synth.random_rays(m % 1000, m, (-5.0, -3.0), (5.0, 3.0)))
    gy = T(np.random.default_rng(7).normal(size=(m, 2)))
    with lens.LensFMM(S, M, f.kappa_s, f.gamma, p=40, leaf_size=leaf, prec=lens.FP32_BULK,
                      target_box=(-5, 5, -3, 3)) as P:
        gxy, gm, _ = P.adjoint(x, gy)
    # dL/dm = -sum g.d/|d|^2, dL/dx = sum m (g/|d|^2 - 2 d (g.d)/|d|^4)
    rm, rx = torch.zeros_like(M), torch.zeros_like(S)
    bm, bx = torch.zeros_like(M), torch.zeros_like(M)
    for a in range(0, m, 1 << 16):
        d = x[a:a + (1 << 16), None] - S[None]
        g = gy[a:a + (1 << 16), None]
        i = 1.0 / (d * d).sum(-1)
        gd = (g * d).sum(-1) * i
        rm -= gd.sum(0)
        rx += (g * i[..., None] - 2 * d * (gd * i)[..., None]).sum(0)
        n = g.norm(dim=-1)
        bm += (n * i.sqrt()).sum(0)
        bx += (n * i).sum(0)
    rx *= M[:, None]
    # float32 terms: a few 2^-24 of their size each, compensated sums; order 40 is far below
    eps = 16 * 2.0 ** -24
    assert torch.all((gm - rm).abs() <= eps * bm)
    assert torch.all((gxy - rx).norm(dim=1) <= eps * M * bx)
