"""Reverse mode of a small beam set under a bound on the library's memory: the reverse step's scratch (two states a thread)
grows with the beams, up to the 14 MB of all resident threads, and the gradient does not depend on the bound."""
import numpy as np
import pytest

from paper_1810_06760_gb300 import workloads as W
from tests.test_gpu_cells import fga  # noqa: F401
from tests.helpers import gpu_setup

pytestmark = pytest.mark.gpu


def test_small_gradient_fits_a_small_bound(fga):  # noqa: F811
    import torch
    w = W.smooth(nq=2, np_=3, ny=16, nsteps=8, n_samples=3, grid_n=9)
    model, desc, keep = gpu_setup(w, 0)
    rng = np.random.default_rng(1)
    rx = torch.as_tensor(rng.uniform(0.2, 0.8, (9, 3)), device="cuda")
    ub = torch.as_tensor(rng.standard_normal((3, 9, 3, 2)) @ np.array([1, 1j]), device="cuda").to(torch.complex64)
    grads = []
    for room in (0, 10e6):
        if room:
            fga.set_device_memory_limit(fga.device_memory_in_use() + room)
        try:
            grads.append(fga.solve_vjp(model, desc, w.dt, w.nsteps, w.times, rx, ub, rw=w.rw, checkpoint_every=4))
        finally:
            fga.set_device_memory_limit(0)
    for a, b in zip(*grads):
        a, b = a.cpu().numpy(), b.cpu().numpy()
        assert np.any(a)
        # node cotangents are added with atomics: rounding of the order
        assert np.linalg.norm(a - b) <= 1e-5 * np.linalg.norm(a)
