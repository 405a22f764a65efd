"""Maps on a device of few bytes (LENS_FAULT=memory@BYTES, in a child process): a grid that
is small enough to be taken at once is taken in chunks where that leaves too little for
the map's accumulators, the refinement's queue or its levels."""
import os
import subprocess
import sys

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# 1500^2 cells: 45 MB of corners and queue
CHILD = r"""
import sys
sys.path.insert(0, %r)
import numpy as np, torch
from paper_2211_00354_gb300 import lens, synth
f = synth.config_uniform(seed=3, n=1000, kappa_star=0.4, kappa_s=0.0, gamma=0.2)
T = lambda a: torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")
grid = synth.Grid(x0=-7.5, y0=-7.5, h=0.01, nx=1500, ny=1500)
npx, refine = int(sys.argv[2]), int(sys.argv[3])
with lens.LensFMM(T(f.stars), T(f.masses), 0.0, 0.2, p=16, leaf_size=16,
                  target_box=(-7.5, 7.5, -7.5, 7.5)) as P:
    mp, st = P.ipm_map(grid, (-4, 4, -4, 4), npx, npx, bbox_cap=16 if refine else 0, refine_levels=refine)
np.savez(sys.argv[1], mp=mp.cpu().numpy(), chunks=st["chunks"], refined=st["cells_refined"], cells=st["cells"],
         area=[st[k] for k in ("area_in_map", "area_outside", "area_dropped", "area_degenerate")])
""" % ROOT


def run(path, npx, refine, **env):
    out = subprocess.run([sys.executable, "-c", CHILD, path, str(npx), str(refine)],
                         env=dict(os.environ, **env), capture_output=True, text=True, timeout=300)
    assert out.returncode == 0, out.stdout + out.stderr
    return np.load(path)


# 2000^2 pixels: 32 MB of accumulators; refinement: 9 MB of queue, then the levels
# (which of the buffers is refused from 54 MB up depends on the plan's size and the field)
@pytest.mark.parametrize("npx,refine,megabytes", [(2000, 0, 65), (400, 2, 53), (400, 2, 55), (400, 2, 56),
                                                  (400, 2, 57), (2000, 0, 500)])
def test_few_bytes_give_the_same_map(tmp_path, npx, refine, megabytes):
    want = run(str(tmp_path / "a.npz"), npx, refine)
    got = run(str(tmp_path / "b.npz"), npx, refine, LENS_FAULT="memory@%d" % (megabytes << 20))
    assert want["chunks"] == 1
    if megabytes in (53, 65, 500):
        assert (got["chunks"] > 1) == (megabytes < 500)
    assert got["refined"] == want["refined"] and (want["refined"] > 0) == (refine > 0)
    np.testing.assert_allclose(got["area"], want["area"], rtol=1e-5, atol=1e-6 * want["area"].sum())
    # float32 additions in another order: at most 64 or so a pixel, 2^-24 each
    assert np.abs(got["mp"] - want["mp"]).sum() <= 64 * 2.0 ** -24 * want["mp"].sum()
