"""Volume lattices on the tensor cores against the FP32 point sum (another kernel) at the same points: tile edges of
every axis, odd row counts, components as rows (few points per plane) and as columns, axes with and without
uniform spacing, single-plane lattices outside the plane kernel.  Tolerance: the FP32 parity bar, 1e-4 (the
kernels' own errors are up to 5e-5 in this sum's FP32 accumulation, and 2e-6)."""
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


@pytest.mark.parametrize("uniform", [True, False])
@pytest.mark.parametrize("shape", [(1, 1, 2), (5, 6, 7), (33, 9, 16), (7, 3, 2), (32, 8, 17), (61, 13, 5), (3, 50, 1), (40, 130, 1),
                                   (2, 1, 40)])
def test_volume_matches_points(fga, beams, shape, uniform):
    import torch
    w, b, _ = beams
    axes = []
    for d, n in enumerate(shape):
        a = np.linspace(0.1, 0.9, n) if n > 1 else np.array([0.45])
        axes.append(a if uniform else np.sort(a + 0.3 / max(n, 4) * np.sin(3.0 * np.arange(n) + d)))
    u = fga.reconstruct_lattice(b, axes, rw=w.rw).cpu().numpy().reshape(-1, 3)
    x = np.stack(np.meshgrid(*axes, indexing="ij"), -1).reshape(-1, 3)
    v = fga.reconstruct(b, torch.as_tensor(x, device="cuda"), rw=w.rw).cpu().numpy()
    assert np.linalg.norm(v) > 0 and rel_l2(u, v) <= 1e-4
