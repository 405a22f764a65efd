"""A call refused for a ray outside the target region: its stream is idle and its
outputs hold what they held, on the default stream and on another one."""
import numpy as np
import pytest
import torch

from paper_2211_00354_gb300 import lens, synth

pytestmark = pytest.mark.gpu

MARK = -7.5  # no output has this value throughout


def T(a):
    return torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


@pytest.mark.parametrize("side", [False, True])
@pytest.mark.parametrize("prec", [lens.FP32_BULK, lens.FP64])
@pytest.mark.parametrize("m,n,leaf", [(1, 300, 8), (300_000, 300, 512), (20_000, 60_000, 2)])
def test_outputs_are_left_alone_and_the_stream_is_idle(m, n, leaf, prec, side):
    f = synth.config_uniform(seed=m, n=n, kappa_star=0.3, kappa_s=0.0, gamma=0.1)
    R = 0.5 * np.hypot(*f.stars.T).max()
    x = synth.random_rays(2, m, (-R, -R), (R, R))
    x[m // 2, 0] = 3 * R
    x, gy = T(x), torch.ones((m, 2), dtype=torch.float64, device="cuda")
    L = lens.load()
    with lens.LensFMM(T(f.stars), T(f.masses), 0.0, 0.1, p=16, leaf_size=leaf, prec=prec,
                      target_box=(-R, R, -R, R)) as P:
        if n == 60_000:
            assert P.info()["n_active_leaves"] > 16384  # the offsets by the general scans
        outs = {k: torch.full(s, MARK, dtype=torch.float64, device="cuda")
                for k, s in dict(y=(m, 2), jac=(m, 4), psi=(m,), gxy=(n, 2), gm=(n,), gkg=(2,)).items()}
        o = {k: v.data_ptr() for k, v in outs.items()}
        torch.cuda.synchronize()
        stream = torch.cuda.Stream() if side else torch.cuda.current_stream()
        s, h, r = stream.cuda_stream, P._handle, x.data_ptr()
        for call in (lambda: L.lens_deflect(h, r, m, o["y"], None, s),
                     lambda: L.lens_deflect(h, r, m, o["y"], o["jac"], s),
                     lambda: L.lens_potential(h, r, m, o["psi"], s),
                     lambda: L.lens_deflect_adjoint(h, r, m, gy.data_ptr(), o["gxy"], o["gm"], o["gkg"], s)):
            assert call() == lens.LENS_EDOMAIN
            assert stream.query()
    torch.cuda.synchronize()
    assert torch.equal(outs.pop("gkg"), torch.zeros(2, dtype=torch.float64, device="cuda"))
    for k, v in outs.items():
        assert torch.all(v == MARK), k
