"""A call whose scratch is refused part of the way returns once its stream is idle:
no kernel of it can store into the host words that a later call takes."""
import contextlib

import numpy as np
import pytest
import torch

from paper_2211_00354_gb300 import lens, synth

pytestmark = pytest.mark.gpu


class Refusing:
    """torch's allocator, refusing the k-th allocation (from 0) after arm(k), none after arm(-1)."""

    def __init__(self):
        self.left = -1

        def alloc(size, stream, ctx):
            self.left -= 1
            return None if self.left == -1 else lens._torch_alloc(size, stream, ctx)

        self.cb = lens.ALLOC_FN(alloc)
        self.struct = lens.lens_allocator(self.cb, lens._FREE_CB, None)

    def arm(self, k):
        self.left = k


@contextlib.contextmanager
def behind_a_long_kernel():
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        torch.cuda._sleep(20_000_000)  # ~10 ms: the call's own kernels are all behind it
    yield s
    s.synchronize()


def T(a):
    return torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


@pytest.mark.parametrize("n,leaf", [(300, 8), (60_000, 2)])
def test_calls_with_rays(monkeypatch, n, leaf):
    f = synth.config_uniform(seed=1, n=n, kappa_star=0.3, kappa_s=0.0, gamma=0.1)
    R = 0.5 * np.hypot(*f.stars.T).max()
    x = T(synth.random_rays(2, 3000, (-R, -R), (R, R)))
    gy = torch.ones_like(x)
    a = Refusing()
    monkeypatch.setattr(lens, "TORCH_ALLOCATOR", a.struct)
    with lens.LensFMM(T(f.stars), T(f.masses), 0.0, 0.1, p=16, leaf_size=leaf, target_box=(-R, R, -R, R),
                      use_torch_allocator=True) as P:
        P.deflect(x)
        torch.cuda.synchronize()
        for call in (lambda s: P.deflect(x, stream=s), lambda s: P.potential(x, stream=s),
                     lambda s: P.adjoint(x, gy, stream=s)):
            for k in range(40):
                with behind_a_long_kernel() as s:
                    a.arm(k)
                    try:
                        call(s)
                        break  # fewer allocations than that
                    except lens.LensError as e:
                        assert e.status == lens.LENS_ENOMEM
                        # (the first allocations come before anything is launched)
                        assert k < 3 or s.query()
                    finally:
                        a.arm(-1)
            assert 4 <= k < 39
            call(None)
