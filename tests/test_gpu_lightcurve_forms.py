"""The light-curve gradient's two forms, the rays in the order of the samples' cells and as
they come: the same for every ray but for the order of a cell's samples (which varies by
itself), on either side of the line between them, and the second form where the memory for
the order is not to be had."""
import os
import subprocess
import sys

import numpy as np
import pytest
import torch

from paper_2211_00354_gb300 import lens

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def T(a):
    return torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


@pytest.mark.parametrize("ns", [1, 8, 9, 10, 60, 500])
@pytest.mark.parametrize("m", [4097, 20_001])
@pytest.mark.parametrize("sigma,trunc", [(0.5, 4.0), (0.05, 6.0), (0.002, 5.0)])
def test_every_ray_gets_the_same(ns, m, sigma, trunc):
    rng = np.random.default_rng(ns)
    smp, F = T(rng.uniform(-1, 1, (ns, 2))), T(rng.uniform(0.5, 2, ns))
    y = rng.uniform(-1.5, 1.5, (m, 2))
    y[:ns] = smp.cpu().numpy()[:m] + 0.3 * sigma  # some near the samples whatever sigma is
    y[7], y[8], y[9] = np.nan, [np.inf, 0.0], [1e300, -1e300]
    y = T(y)
    args = 0.01, smp, sigma, F, 0.5 * F
    got = lens.light_curve_grad(y, *args, trunc=trunc)
    # up to 4096 rays always go as they come
    want = torch.cat([lens.light_curve_grad(y[a:a + 4096].contiguous(), *args, trunc=trunc)
                      for a in range(0, m, 4096)])
    # float-float sums of the same terms: 2^-46 of their sizes an addition
    q = ((y[:, None] - smp[None]) ** 2).sum(-1)
    size = torch.where(q <= (1.01 * trunc * sigma) ** 2, (-q / (2 * sigma ** 2)).exp() * q.sqrt(), 0.0) * F
    bound = size.sum(1) * 0.01 / (2 * np.pi * sigma ** 4) * ns * 2.0 ** -46
    assert torch.all((got - want).abs() <= bound[:, None]) and want.abs().max() > 0


# 5e5 rays near 300 samples in a few cells: 22 MB for the order of the gradient's rays
CHILD = r"""
import sys
sys.path.insert(0, %r)
import numpy as np, torch
from paper_2211_00354_gb300 import lens
rng = np.random.default_rng(1)
T = lambda a: torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")
smp, F = T(rng.uniform(-1, 1, (300, 2))), T(rng.uniform(0.5, 2, 300))
y = T(rng.uniform(-1, 1, (500_000, 2)))
np.save(sys.argv[1], lens.light_curve_grad(y, 0.01, smp, 0.2, F, 0.5 * F, trunc=4.0).cpu().numpy())
""" % ROOT


def test_without_the_memory_for_the_order(tmp_path):
    got = []
    for fault in ("", "memory@%d" % (12 << 20)):
        path = str(tmp_path / ("g%d.npy" % len(got)))
        out = subprocess.run([sys.executable, "-c", CHILD, path], env=dict(os.environ, LENS_FAULT=fault),
                             capture_output=True, text=True, timeout=300)
        assert out.returncode == 0, out.stdout + out.stderr
        got.append(np.load(path))
    # as above, 300 terms of at most 2 |F - T| w / (2 pi sigma^2) exp(-1/2) / sigma each
    term = 2 * 1.0 * 0.01 / (2 * np.pi * 0.2 ** 2) * np.exp(-0.5) / 0.2
    assert np.abs(got[0] - got[1]).max() <= 300 * 300 * term * 2.0 ** -46
    assert np.abs(got[0]).max() > term
