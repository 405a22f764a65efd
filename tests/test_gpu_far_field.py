"""The far field's translations (M2L, P2L, L2L) at expansion orders about the sizes of
a warp and of a block's groups, with a warp a box and a block a box (a small target
region), on trees whose V lists are full, cut by the target region, and one-sided."""
import numpy as np
import pytest
import torch

import oracle
from paper_2211_00354_gb300 import lens, synth

pytestmark = pytest.mark.gpu


def T(a):
    return torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


@pytest.mark.parametrize("p", [1, 2, 3, 4, 15, 24, 30, 31, 32, 33, 42, 43, 63, 64])
@pytest.mark.parametrize("kind", ["uniform", "clustered", "line", "corner"])
def test_expansions_of_every_order_match_the_direct_sum(kind, p):
    rng = np.random.default_rng(p)
    box = (-6.0, 6.0, -6.0, 6.0)
    if kind == "clustered":
        cen = rng.uniform(-5, 5, (12, 2))
        st = (cen[:, None, :] + rng.normal(0, 0.1, (12, 100, 2))).reshape(-1, 2)
    elif kind == "line":
        st = np.stack([rng.uniform(-6, 6, 800), np.full(800, 0.3)], axis=1)
    else:
        st = rng.uniform(-6, 6, (1500, 2))
        if kind == "corner":
            box = (4.0, 6.0, -6.0, -3.5)
    m = rng.uniform(0.5, 1.5, len(st))
    x = synth.random_rays(p, 1500, (box[0], box[2]), (box[1], box[3]))
    with lens.LensFMM(T(st), T(m), 0.1, 0.2, p=p, leaf_size=4, prec=lens.FP64, target_box=box) as P:
        y = P.deflect(T(x)).cpu().numpy()
    ref = oracle.deflect(st, m, 0.1, 0.2, x)
    S = (m / np.hypot(x[:, None, 0] - st[None, :, 0], x[:, None, 1] - st[None, :, 1])).sum(1)
    # one truncation of the multipole and one of the local series, each a
    # geometric tail of ratio sqrt2 / (4 - sqrt2) (the nearest V offset); the
    # distance to the box centre against that to the star gives the factor
    rho = np.sqrt(2) / (4 - np.sqrt(2))
    bound = 4 * rho ** (p + 1) / (1 - rho) + 1e-13
    assert np.all(np.hypot(*(y - ref).T) <= bound * S)
