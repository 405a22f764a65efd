"""The bound on the tiles of a call's rays, on the host: never below the count of any
distribution over the leaves, reached by the worst one, and m for tiles of one ray (so that
a potential call is refused by its number of rays alone)."""
import itertools
import subprocess

import pytest

from paper_2211_00354_gb300 import _build

MAIN = r"""
#include <cstdio>
#include "lens_internal.h"
int main() {
  long long m, nl;
  int tile;
  while (std::scanf("%lld %lld %d", &m, &nl, &tile) == 3)
    std::printf("%lld\n", (long long)lens::ray_tiles_max(m, nl, tile));
}
"""


@pytest.fixture(scope="module")
def bound(tmp_path_factory):
    d = tmp_path_factory.mktemp("tiles")
    (d / "main.cu").write_text(MAIN)
    subprocess.run([_build.nvcc(), *_build.NVCC_FLAGS, "-I", _build.CSRC, "-o", str(d / "main"),
                    str(d / "main.cu")], check=True)

    def f(cases):
        out = subprocess.run([str(d / "main")], input="".join("%d %d %d\n" % c for c in cases),
                             capture_output=True, text=True, check=True).stdout
        return [int(v) for v in out.split()]
    return f


def worst(m, nl, tile):
    """The most tiles: one ray in each leaf that can have one, then whole tiles more."""
    k = min(m, nl)
    return k + (m - k) // tile


def test_small_counts_against_every_distribution(bound):
    cases = [(m, nl, t) for m in range(1, 8) for nl in range(1, 4) for t in (1, 2, 3)]
    for (m, nl, t), b in zip(cases, bound(cases)):
        most = max(sum((c + t - 1) // t for c in cs)
                   for cs in itertools.product(range(m + 1), repeat=nl) if sum(cs) == m)
        assert b == most == worst(m, nl, t)


def test_large_counts(bound):
    top = 2 ** 31 - 2
    cases = [(top, 10 ** 6, 1), (1_100_000_000, 1_100_000_000, 1), (top, 10 ** 8, 128), (top, 1, 256),
             (10 ** 6, 10 ** 8, 128), (129, 7, 128)]
    got = bound(cases)
    assert got == [worst(*c) for c in cases]
    assert got[0] == top and got[1] == 1_100_000_000
