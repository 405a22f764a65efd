"""Fields about the size up to which one block sorts the stars, and about its
threads: uniform, clustered (boxes deeper than the sorted bits: the keys are sorted
again in full) and with coincident stars; order and deflections."""
import numpy as np
import pytest
import torch

import oracle
from paper_2211_00354_gb300 import lens, synth

pytestmark = pytest.mark.gpu


def T(a):
    return torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


@pytest.mark.parametrize("kind", ["uniform", "clustered", "pairs", "line"])
@pytest.mark.parametrize("n", [1, 2, 31, 33, 1023, 1024, 1025, 4097, 8191, 8192, 8193])
def test_fields_about_the_block_sort(kind, n):
    rng = np.random.default_rng(n)
    if kind == "uniform":
        st = rng.uniform(-5, 5, (n, 2))
    elif kind == "clustered":
        st = rng.uniform(-5, 5, (n, 2))
        st[: n // 2] = 1.0 + rng.normal(0, 1e-6, (n // 2, 2))
    elif kind == "pairs":
        st = rng.uniform(-5, 5, (n, 2))
        st[: n // 2] = st[n - n // 2:]
    else:
        st = np.stack([np.linspace(-5, 5, n), np.zeros(n)], axis=1)
    m = rng.uniform(0.5, 1.5, n)
    x = synth.random_rays(n, 150, (-5, -5), (5, 5))
    # more stars than a leaf takes in one box of the deepest level (28) of the root,
    # the target region and a millionth: refused, whichever way the stars are sorted
    size = 11.0 * (1.0 + 1e-6)
    q = np.floor((st + 0.5 * size) * (2.0 ** 28 / size)).astype(np.int64)
    if np.unique(q[:, 0] * 2 ** 28 + q[:, 1], return_counts=True)[1].max() > 4:
        with pytest.raises(lens.LensError) as ei:
            lens.LensFMM(T(st), T(m), 0.1, 0.2, p=40, leaf_size=4, prec=lens.FP64,
                         target_box=(-5.5, 5.5, -5.5, 5.5))
        assert ei.value.status == lens.LENS_EDEPTH
        return
    with lens.LensFMM(T(st), T(m), 0.1, 0.2, p=40, leaf_size=4, prec=lens.FP64,
                      target_box=(-5.5, 5.5, -5.5, 5.5)) as P:
        y = P.deflect(T(x)).cpu().numpy()
        gy = torch.ones((len(x), 2), dtype=torch.float64, device="cuda")
        gm = P.adjoint(T(x), gy)[1].cpu().numpy()
    ref = oracle.deflect(st, m, 0.1, 0.2, x)
    d = np.hypot(x[:, None, 0] - st[None, :, 0], x[:, None, 1] - st[None, :, 1])
    # order 40 leaves 10 * 0.547^41 of a term
    assert np.all(np.hypot(*(y - ref).T) <= 1e-9 * (m / d).sum(1))
    # the gradient comes back in the caller's order of the stars
    rm = oracle.adjoint(st, m, x, np.ones((len(x), 2)))[1]
    assert np.all(np.abs(gm - rm) <= 1e-9 * np.sqrt(2) * (1 / d).sum(0))
