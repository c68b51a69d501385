"""Sums of a window's samples under a bound on the library's device memory: where the partial sums of many samples (or
many tiles) do not fit, fewer are taken per launch, with the same result.  The bounds leave room for the beam set and the
records and for a part of the partial sums, whose full size is 256 MB."""
import numpy as np
import pytest

from paper_1810_06760_gb300 import workloads as W
from tests.test_gpu_cells import fga  # noqa: F401
from tests.helpers import gpu_setup

pytestmark = pytest.mark.gpu


# records of 32,000 beams x samples: 184 MB (points, FP32), 184 MB (FP64), 61 MB and 5 MB (planes)
@pytest.mark.parametrize("kind,prec,n_times,room", [("points", 0, 120, 310e6), ("points", 1, 60, 330e6),
                                                    ((60, 50), 0, 40, 180e6), ((300, 290), 0, 3, 120e6)])
def test_sums_fit_a_memory_bound(fga, kind, prec, n_times, room):  # noqa: F811
    import torch
    w = W.smooth(nq=4, np_=5, ny=24, nsteps=8, grid_n=33)
    times = w.T * np.arange(1, n_times + 1) / n_times
    model, desc, keep = gpu_setup(w, prec)
    if kind == "points":
        rx = dict(rx=torch.as_tensor(np.random.default_rng(5).uniform(0.0, 1.0, (2500, 3)), device="cuda"))
    else:
        rx = dict(rx_axes=tuple((np.arange(n) + 0.5) / n for n in kind) + (np.array([0.5]),))
    u, _ = fga.solve(model, desc, w.dt, w.nsteps, times, rw=w.rw, **rx)
    fga.set_device_memory_limit(fga.device_memory_in_use() + room)
    try:
        v, _ = fga.solve(model, desc, w.dt, w.nsteps, times, rw=w.rw, **rx)
    finally:
        fga.set_device_memory_limit(0)
    assert float(u.abs().max()) > 0 and torch.equal(u, v)
