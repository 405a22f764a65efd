"""Calls from threads that come and go: the end of one waits for no other stream's work,
and threads alive at once do not share their host words."""
import threading

import numpy as np
import pytest
import torch

from paper_2211_00354_gb300 import lens, synth

pytestmark = pytest.mark.gpu


def T(a):
    return torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


@pytest.fixture
def field():
    f = synth.config_uniform(seed=1, n=2000, kappa_star=0.4, kappa_s=0.0, gamma=0.1)
    return T(f.stars), T(f.masses)


def test_the_end_of_a_thread_waits_for_no_other_stream(field):
    x = T(synth.random_rays(1, 2000, (-3.0, -3.0), (3.0, 3.0)))
    with lens.LensFMM(*field, 0.0, 0.1, p=16, leaf_size=16, target_box=(-3, 3, -3, 3)) as P:
        want = P.deflect(x)
        busy, mine = torch.cuda.Stream(), torch.cuda.Stream()
        torch.cuda.synchronize()

        def work():
            with torch.cuda.stream(mine):
                P.deflect(x)

        for _ in range(2):
            with torch.cuda.stream(busy):
                torch.cuda._sleep(400_000_000)  # ~200 ms, a few calls are over long before
            t = threading.Thread(target=work)
            t.start()
            t.join()
            with torch.cuda.stream(mine):
                y = P.deflect(x)
            mine.synchronize()
            assert not busy.query()
            assert torch.equal(y, want)
            torch.cuda.synchronize()


def test_threads_at_once_and_one_after_another(field):
    rays = [T(synth.random_rays(k, 500 + 100 * k, (-3.0, -3.0), (3.0, 3.0))) for k in range(6)]
    bad = T([[1e3, 0.0]])

    def run(k, out):
        with torch.cuda.stream(torch.cuda.Stream()):
            for _ in range(30):
                with lens.LensFMM(*field, 0.0, 0.1, p=16, leaf_size=16, target_box=(-3, 3, -3, 3)) as P:
                    out[k] = P.deflect(rays[k])
                    with pytest.raises(lens.LensError):
                        P.deflect(bad)
            torch.cuda.current_stream().synchronize()

    want = [None] * 6
    for k in range(6):
        run(k, want)
    torch.cuda.synchronize()
    for _ in range(2):
        got = [None] * 6
        ts = [threading.Thread(target=run, args=(k, got)) for k in range(6)]
        [t.start() for t in ts]
        [t.join() for t in ts]
        for a, b in zip(got, want):
            assert torch.equal(a, b)
