"""Grid deflections into a buffer on any multiple of eight bytes: the same bits."""
import ctypes

import numpy as np
import pytest
import torch

from paper_2211_00354_gb300 import lens, synth

pytestmark = pytest.mark.gpu


def T(a):
    return torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


@pytest.mark.parametrize("prec", [lens.FP32_BULK, lens.FP64])
@pytest.mark.parametrize("jacobian", [False, True])
@pytest.mark.parametrize("nx,ny", [(1, 1), (37, 20), (64, 65)])
def test_any_multiple_of_eight_bytes(prec, jacobian, nx, ny):
    f = synth.config_uniform(seed=5, n=700, kappa_star=0.4, kappa_s=0.1, gamma=0.2, mass_range=(0.5, 1.5))
    h = 8.0 / max(nx, ny)
    grid = synth.Grid(x0=-4.0, y0=-4.0, h=h, nx=nx, ny=ny)
    box = (grid.x0, grid.x0 + nx * h, grid.y0, grid.y0 + ny * h)
    k = (nx + 1) * (ny + 1)
    L, g = lens.load(), lens.grid_struct(grid)
    got = []
    with lens.LensFMM(T(f.stars), T(f.masses), f.kappa_s, f.gamma, p=16, leaf_size=16, prec=prec,
                      target_box=box) as P:
        for shift in (0, 1):  # in float64 values from a 16-byte boundary
            y = torch.full((2 * k + 3,), -7.5, dtype=torch.float64, device="cuda")
            J = torch.full((4 * k + 3,), -7.5, dtype=torch.float64, device="cuda")
            assert y.data_ptr() % 16 == 0 and J.data_ptr() % 16 == 0
            assert L.lens_deflect_grid(P._handle, ctypes.byref(g), 0, ny + 1, y.data_ptr() + 8 * shift,
                                       J.data_ptr() + 8 * shift if jacobian else None,
                                       torch.cuda.current_stream().cuda_stream) == lens.LENS_OK
            torch.cuda.synchronize()
            got.append((y[shift:shift + 2 * k], J[shift:shift + 4 * k]))
            # nothing beside it
            assert torch.all(torch.cat([y[:shift], y[shift + 2 * k:]]) == -7.5)
    assert torch.equal(got[0][0], got[1][0]) and torch.equal(got[0][1], got[1][1])
