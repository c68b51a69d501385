"""Idle device blocks kept between calls: solves from two host threads on two streams, each taking blocks the other
released, give the results they give alone; the idle blocks return to the device on request."""
import threading

import numpy as np
import pytest

from paper_1810_06760_gb300 import workloads as W
from tests.helpers import gpu_setup

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fga():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1810_06760_gb300 import build, fga as F
    build.build()
    F.lib()
    return F


def test_two_threads_share_idle_blocks(fga):
    import torch
    cases = [W.smooth(nq=4, np_=4, ny=24, nsteps=24, n_samples=12, rx_side=5, snap_side=6, grid_n=17),
             W.smooth(nq=4, np_=4, ny=26, nsteps=20, n_samples=9, rx_side=6, snap_side=7, grid_n=17, k=48.0)]
    setups = [gpu_setup(w, 0) for w in cases]

    def solve(i):
        w, (model, desc, keep) = cases[i], setups[i]
        u, s = fga.solve(model, desc, w.dt, w.nsteps, w.times, rw=w.rw, rx_axes=w.rx_axes, snap_axes=w.snap_axes)
        return u, s

    alone = [[t.cpu().numpy() for t in solve(i)] for i in range(2)]
    torch.cuda.synchronize()
    got, errors = [[], []], []

    def work(i):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                for r in range(6):
                    got[i].append([t.cpu().numpy() for t in solve((i + r) % 2)])
        except Exception as e:   # reported by the main thread
            errors.append(e)

    threads = [threading.Thread(target=work, args=(i,)) for i in range(2)]
    [t.start() for t in threads]
    [t.join() for t in threads]
    assert not errors, errors
    for i in range(2):
        for r, (u, s) in enumerate(got[i]):
            np.testing.assert_array_equal(u, alone[(i + r) % 2][0])
            np.testing.assert_array_equal(s, alone[(i + r) % 2][1])


def test_idle_blocks_are_given_back(fga):
    import torch
    w = W.smooth(nq=8, np_=6, ny=24, nsteps=8, n_samples=8, rx_side=8, snap_side=0, grid_n=17)
    model, desc, keep = gpu_setup(w, 0)
    for _ in range(2):
        fga.solve(model, desc, w.dt, w.nsteps, w.times, rw=w.rw, rx_axes=w.rx_axes)
    torch.cuda.synchronize()
    held = torch.cuda.mem_get_info()[0]
    fga.set_device_memory_limit(0)
    # the solve's beam set and its sorted copy alone are 2 x 196 B x 442,368 beams = 173 MB
    assert torch.cuda.mem_get_info()[0] - held > 150 * 10 ** 6
