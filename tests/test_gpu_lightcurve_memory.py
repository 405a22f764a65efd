"""The light curve and its gradient where the memory for their ray orders is not to be
had: the pool as a device of few bytes (LENS_FAULT=memory@BYTES, in a child process)."""
import os
import subprocess
import sys

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# 5e5 rays near 400 samples strewn over 500 x 500 cells: 4e6 parts and their 96 MB of
# counters, 6 MB with whole cells; ray positions 16 MB
CHILD = r"""
import sys
sys.path.insert(0, %r)
import numpy as np, torch
from paper_2211_00354_gb300 import lens
rng = np.random.default_rng(1)
T = lambda a: torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")
smp = rng.uniform(-25, 25, (400, 2))
y = T(rng.uniform(-25, 25, (500_000, 2)))
args = y, 0.01, T(smp), 0.02
F = lens.light_curve(*args, trunc=5.0)
g = lens.light_curve_grad(*args, F, 0.5 * F, trunc=5.0)
np.savez(sys.argv[1], F=F.cpu().numpy(), g=g.cpu().numpy(), near=(g != 0).any(1).sum().item())
""" % ROOT


def run(path, **env):
    out = subprocess.run([sys.executable, "-c", CHILD, path], env=dict(os.environ, **env),
                         capture_output=True, text=True, timeout=300)
    assert out.returncode == 0, out.stdout + out.stderr
    return np.load(path)


@pytest.mark.parametrize("megabytes", [64, 30])
def test_few_bytes_give_the_same(tmp_path, megabytes):
    want = run(str(tmp_path / "a.npz"))
    got = run(str(tmp_path / "b.npz"), LENS_FAULT="memory@%d" % (megabytes << 20))
    assert want["near"] > 1000
    # the order of the sums alone differs: float-float terms (2^-48) of a sample's
    # few rays
    np.testing.assert_allclose(got["F"], want["F"], rtol=1e-12)
    size = np.abs(want["g"]).max()
    np.testing.assert_allclose(got["g"], want["g"], rtol=0, atol=1e-12 * size)
