"""Receiver planes on the tensor cores against the FP32 point sum (another kernel) at the same points: tile edges of
both axes (quarters of 1 to 6 points, one to several tiles, ragged ones), spacings coarse enough to stop the factor
recurrences, planes whose partial sums are taken in several groups of tiles, and all samples of a window in one
launch.  Tolerance: the FP32 parity bar of a Gaussian sum, 1e-4 (the two kernels' own errors are 2e-6 and 5e-6)."""
import numpy as np
import pytest

from paper_1810_06760_gb300 import workloads as W
from tests.helpers import gpu_setup, rel_l2

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


@pytest.fixture(scope="module")
def beams(fga):
    w = W.smooth(nq=4, np_=5, ny=24, grid_n=33)
    model, desc, keep = gpu_setup(w, 0)
    b = fga.decompose(model, desc)
    fga.propagate(model, b, w.dt, 40)
    return w, b, (model, desc, keep)


def _points(axes):
    return np.stack(np.meshgrid(*axes, indexing="ij"), -1).reshape(-1, 3)


@pytest.mark.parametrize("n0,n1,lo,hi", [(1, 1, 0.4, 0.4), (1, 20, 0.0, 1.0), (3, 4, 0.2, 0.8), (5, 5, 0.0, 1.0),
                                         (24, 20, 0.0, 1.0), (25, 21, 0.0, 1.0), (17, 13, -1.0, 3.0), (6, 9, -6.0, 7.0),
                                         (300, 290, 0.0, 1.0)])
def test_plane_matches_points(fga, beams, n0, n1, lo, hi):
    import torch
    w, b, _ = beams
    axes = (np.linspace(lo, hi, n0), np.linspace(lo, hi, n1), np.array([0.45]))
    u = fga.reconstruct_lattice(b, axes, rw=w.rw).cpu().numpy().reshape(-1, 3)
    v = fga.reconstruct(b, torch.as_tensor(_points(axes), device="cuda"), rw=w.rw).cpu().numpy()
    assert np.linalg.norm(v) > 0 and rel_l2(u, v) <= 1e-4


@pytest.mark.parametrize("n0,n1,n_times", [(20, 20, 37), (16, 16, 1), (7, 23, 90)])
def test_samples_of_a_window_match_points(fga, n0, n1, n_times):
    import torch
    w = W.smooth(nq=4, np_=4, ny=24, nsteps=40, n_samples=n_times, grid_n=33)
    model, desc, keep = gpu_setup(w, 0)
    axes = tuple((np.arange(n) + 0.5) / n for n in (n0, n1)) + (np.array([0.3]),)
    u, _ = fga.solve(model, desc, w.dt, w.nsteps, w.times, rw=w.rw, rx_axes=axes)
    v, _ = fga.solve(model, desc, w.dt, w.nsteps, w.times, torch.as_tensor(_points(axes), device="cuda"), rw=w.rw)
    u, v = u.cpu().numpy().reshape(n_times, -1), v.cpu().numpy().reshape(n_times, -1)
    assert max(rel_l2(a, b) for a, b in zip(u, v)) <= 1e-4
