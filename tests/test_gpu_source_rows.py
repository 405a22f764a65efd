"""Finite source by row sums: disks of no, few and many pixels, maps smaller
than the disk, odd widths, a ring of row sums that wraps, and the radius beyond
which the one-pass kernel runs, against a plain float64 sum over the disk."""
import math

import pytest
import torch

from paper_2211_00354_gb300 import lens

pytestmark = pytest.mark.gpu


def plain(m, sigma, trunc):
    R, cut = int(math.floor(trunc * sigma)), trunc * trunc * sigma * sigma
    ny, nx = m.shape
    num, den = torch.zeros_like(m), torch.zeros_like(m)
    for dy in range(-min(R, ny - 1), min(R, ny - 1) + 1):
        ys, yd = slice(max(0, -dy), ny - max(0, dy)), slice(max(0, dy), ny - max(0, -dy))
        for dx in range(-min(R, nx - 1), min(R, nx - 1) + 1):
            if dx * dx + dy * dy > cut:
                continue
            w = math.exp(-(dx * dx + dy * dy) / (2.0 * sigma * sigma))
            xs, xd = slice(max(0, -dx), nx - max(0, dx)), slice(max(0, dx), nx - max(0, -dx))
            num[ys, xs] += w * m[yd, xd]
            den[ys, xs] += w
    return num / den


@pytest.mark.parametrize("ny,nx,sigma,trunc", [
    (1, 1, 2.0, 3.0), (3, 300, 4.0, 6.0), (257, 2, 3.0, 5.0), (64, 129, 0.3, 2.0),
    (65, 127, 0.5, 4.0), (200, 131, 2.0, 4.5), (40, 256, 12.0, 5.0),
    (40, 30, 64.0, 4.0),     # R = 256, the largest of the two-pass form
    (40, 30, 64.25, 4.0),    # R = 257: the one-pass kernel
])
def test_source_matches_a_plain_sum(ny, nx, sigma, trunc):
    g = torch.Generator("cuda").manual_seed(ny + nx)
    m = 0.1 + 10.0 * torch.rand((ny, nx), generator=g, dtype=torch.float64, device="cuda")
    R = int(math.floor(trunc * sigma))
    # a positive sum of at most ~3 R float-float terms a chain, 2^-47 each
    torch.testing.assert_close(lens.map_source(m, sigma, trunc), plain(m, sigma, trunc),
                               rtol=(3 * R + 8) * 2.0 ** -47, atol=0.0)


def test_ring_wraps():
    # ~93 half-widths of 2500 columns: a ring of 232 rows, filled 32 output rows at a time
    g = torch.Generator("cuda").manual_seed(3)
    m = 0.1 + 10.0 * torch.rand((300, 2500), generator=g, dtype=torch.float64, device="cuda")
    got = lens.map_source(m, 20.0, 5.0)
    # the same map upside down takes other rows through other slots
    torch.testing.assert_close(lens.map_source(m.flip(0).contiguous(), 20.0, 5.0).flip(0), got,
                               rtol=310 * 2.0 ** -47, atol=0.0)
    # a window whose disks lie in the map, by the plain sum
    sub = m[20:221 + 20, 900:1101]
    w = plain(sub, 20.0, 5.0)[100, 100]
    assert abs(got[120, 1000].item() / w.item() - 1) <= 310 * 2.0 ** -47


def test_non_finite_pixels_spoil_their_disk_only():
    m = torch.ones((60, 70), dtype=torch.float64, device="cuda")
    m[30, 40] = math.nan
    out = lens.map_source(m, 2.0, 3.0)
    y, x = torch.meshgrid(torch.arange(60.0), torch.arange(70.0), indexing="ij")
    disk = ((y - 30) ** 2 + (x - 40) ** 2 <= 36.0).cuda()
    assert torch.equal(torch.isnan(out), disk)
