"""The transposed operators at expansion orders about the sizes of a warp and of a
block's groups, and ray tiles that are not whole, against the oracle's gradient in
both precisions; stars on rays; U lists of a few and of many stars."""
import numpy as np
import pytest
import torch

import oracle
from paper_2211_00354_gb300 import lens, synth

pytestmark = pytest.mark.gpu


def T(a):
    return torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


def check(st, m, x, gy, p, leaf, prec, L):
    with lens.LensFMM(T(st), T(m), 0.1, 0.2, p=p, leaf_size=leaf, prec=prec,
                      target_box=(-L, L, -L, L)) as P:
        gxy, gm, _ = (t.cpu().numpy() for t in P.adjoint(T(x), T(gy)))
    rxy, rm, _ = oracle.adjoint(st, m, x, gy)
    d = np.hypot(x[:, None, 0] - st[None, :, 0], x[:, None, 1] - st[None, :, 1])
    d = np.where(d > 0, d, np.inf)
    c = np.hypot(gy[:, 0], gy[:, 1])[:, None]
    S1, S2 = (c / d).sum(0), m * (c / d ** 2).sum(0)
    # series truncated after order p, ratio sqrt2 / (4 - sqrt2), and their derivative;
    # in float32 a few 2^-24 of a term, up to 128 of them in a lane's partial
    # sum of moments of up to p products each
    rho = np.sqrt(2) / (4 - np.sqrt(2))
    eps = (128 + p) * 2.0 ** -24 if prec == lens.FP32_BULK else 1e-12
    b1 = 4 * rho ** (p + 1) / (1 - rho) + eps
    b2 = 16 * (p + 2) * rho ** p / (1 - rho) ** 2 + eps * (p + 2)
    assert np.all(np.abs(gm - rm) <= b1 * S1 + 1e-300)
    assert np.all(np.hypot(*(gxy - rxy).T) <= b2 * S2 + 1e-300)


@pytest.mark.parametrize("prec", [lens.FP32_BULK, lens.FP64])
@pytest.mark.parametrize("p", [1, 2, 3, 24, 30, 31, 32, 42, 43, 63, 64])
def test_orders(prec, p):
    rng = np.random.default_rng(p)
    st = rng.uniform(-6, 6, (900, 2))
    m = rng.uniform(0.5, 1.5, len(st))
    x = synth.random_rays(p, 3000, (-6, -6), (6, 6))
    check(st, m, x, rng.normal(size=x.shape), p, 4, prec, 6.0)


@pytest.mark.parametrize("prec", [lens.FP32_BULK, lens.FP64])
@pytest.mark.parametrize("n,leaf", [(1, 1), (3, 16), (40, 64), (900, 16), (3000, 300)])
@pytest.mark.parametrize("nr", [1, 2, 7, 8, 9, 127, 128, 129, 1000])
def test_tiles(prec, n, leaf, nr):
    rng = np.random.default_rng(n + nr)
    st = rng.uniform(-3, 3, (n, 2))
    m = rng.uniform(0.5, 1.5, n)
    x = synth.random_rays(nr, nr, (-3, -3), (3, 3))
    x[0] = st[0]  # on a star: no term
    check(st, m, x, rng.normal(size=x.shape), 40, leaf, prec, 3.1)
