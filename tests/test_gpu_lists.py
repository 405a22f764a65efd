"""Interaction lists of a warp a box, and a small region's local expansions by chains of
ancestors: trees of one box, of few and of many active boxes, on both sides of the
number up to which a region counts as small, graded trees with coarse neighbours in several
places and deep descents, targets at the root's edge and corner and outside the stars."""
import numpy as np
import pytest
import torch

import oracle
from paper_2211_00354_gb300 import lens, synth

pytestmark = pytest.mark.gpu


def T(a):
    return torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


def stars_of(kind, rng):
    if kind == "uniform":
        return rng.uniform(-6, 6, (2500, 2))
    if kind == "graded":  # ever finer towards a corner and a point
        r = 6.0 * 0.97 ** np.arange(700)
        t = rng.uniform(0, 2 * np.pi, 700)
        a = np.stack([r * np.cos(t), r * np.sin(t)], axis=1)
        return np.concatenate([a * 0.5 + 2.9, rng.uniform(-6, 6, (300, 2)), -6 + a[:300] ** 2 / 20])
    if kind == "graded to a radius":
        r = 6.0 * 0.98 ** np.arange(700)  # down to 4e-6, ~0.02 of that apart
        t = rng.uniform(0, 2 * np.pi, 700)
        a = np.stack([r * np.cos(t), r * np.sin(t)], axis=1)
        return np.concatenate([a * 0.5 + 2.9, rng.uniform(-6, 6, (300, 2)),
                               -6 + rng.uniform(0, 0.02, (300, 2))])
    if kind == "hole":  # fine around, nothing inside
        r, t = rng.uniform(3.0, 3.05, 2500), rng.uniform(0, 2 * np.pi, 2500)
        return np.stack([r * np.cos(t), r * np.sin(t)], axis=1)
    return np.array([[0.25, -0.5]])


@pytest.mark.parametrize("kind", ["uniform", "graded", "graded to a radius", "hole", "single"])
@pytest.mark.parametrize("box", [(-6, 6, -6, 6), (2.5, 3.2, 2.5, 3.2), (-6, -5.5, -6, 6),
                                 (-0.4, 0.4, -0.4, 0.4), (9.0, 12.0, -1.0, 1.0)])
@pytest.mark.parametrize("leaf", [2, 20])
def test_deflections_and_gradients_over_lists(kind, box, leaf):
    rng = np.random.default_rng(5)
    st = stars_of(kind, rng)
    m = rng.uniform(0.5, 1.5, len(st))
    x = synth.random_rays(leaf, 800, (box[0], box[2]), (box[1], box[3]))
    gy = rng.normal(size=x.shape)
    # more stars than a leaf takes in a box of the deepest level (28): refused
    lo = np.minimum(st.min(0), (box[0], box[2]))
    hi = np.maximum(st.max(0), (box[1], box[3]))
    size = (hi - lo).max() * (1.0 + 1e-6)
    q = np.floor((st - (0.5 * (lo + hi) - 0.5 * size)) * (2.0 ** 28 / size)).astype(np.int64)
    if np.unique(q[:, 0] * 2 ** 28 + q[:, 1], return_counts=True)[1].max() > leaf:
        with pytest.raises(lens.LensError) as ei:
            lens.LensFMM(T(st), T(m), 0.1, 0.2, p=40, leaf_size=leaf, prec=lens.FP64, target_box=box)
        assert ei.value.status == lens.LENS_EDEPTH
        return
    with lens.LensFMM(T(st), T(m), 0.1, 0.2, p=40, leaf_size=leaf, prec=lens.FP64, target_box=box) as P:
        info = P.info()
        y = P.deflect(T(x)).cpu().numpy()
        gxy, gm, _ = (t.cpu().numpy() for t in P.adjoint(T(x), T(gy)))
    print(kind, box, leaf, info["n_active_boxes"], info["n_v"], info["n_x"], info["n_u"], info["n_w"])
    d = np.hypot(x[:, None, 0] - st[None, :, 0], x[:, None, 1] - st[None, :, 1])
    ref = oracle.deflect(st, m, 0.1, 0.2, x)
    # order 40 leaves 10 * 0.547^41 of a term, and (p + 2) times that of its derivative
    assert np.all(np.hypot(*(y - ref).T) <= 1e-9 * (m / d).sum(1))
    rxy, rm, _ = oracle.adjoint(st, m, x, gy)
    c = np.hypot(gy[:, 0], gy[:, 1])[:, None]
    assert np.all(np.abs(gm - rm) <= 1e-9 * (c / d).sum(0))
    assert np.all(np.hypot(*(gxy - rxy).T) <= 1e-7 * m * (c / d ** 2).sum(0))
