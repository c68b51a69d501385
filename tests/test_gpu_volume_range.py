"""The factor recurrences of the volume lattices' kernel where their numbers are extreme.

Amplitudes: the sum is linear, and a scaling of the data by a power of two changes no rounding in it, so the sums of
2^s f are 2^s times those of f bit for bit, on a lattice coarse enough that runs of points start far outside the beams."""
import dataclasses

import numpy as np
import pytest

from paper_1810_06760_gb300 import workloads as W
from tests.test_gpu_cells import fga  # noqa: F401
from tests.helpers import gpu_setup, rel_l2

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(8, 16, 8), (9, 8, 2)])   # components as columns and as rows
@pytest.mark.parametrize("s", [40, 100])
def test_volume_scales_with_the_data(fga, shape, s):  # noqa: F811
    w = W.smooth(nq=4, np_=5, ny=24, grid_n=33)
    axes = [0.1375 * np.arange(n) for n in shape]         # 1.1 / sqrt(k)
    out = []
    for scale in (0, s):
        model, desc, keep = gpu_setup(dataclasses.replace(w, f=np.ldexp(w.f.real, scale) + 1j * np.ldexp(w.f.imag, scale)), 0)
        b = fga.decompose(model, desc)
        fga.propagate(model, b, w.dt, 40)
        out.append(fga.reconstruct_lattice(b, axes, rw=w.rw).cpu().numpy())
    assert np.abs(out[0]).max() > 0
    np.testing.assert_array_equal(out[1].view(np.float32), np.ldexp(out[0].view(np.float32), s))


@pytest.mark.parametrize("shape", [(32, 8, 8), (8, 12, 10)])
def test_coarse_volume_reaching_far_from_the_beams(fga, shape):  # noqa: F811
    """Spacings at which the ratio of a run's neighbours overflows for beams at the far end of the tile: against the
    FP32 point sum (another kernel) at the same points, at the FP32 parity bar, 1e-4."""
    import torch
    w = W.smooth(nq=4, np_=5, ny=24, grid_n=33)
    model, desc, keep = gpu_setup(w, 0)
    b = fga.decompose(model, desc)
    axes = [0.9 - h * np.arange(n)[::-1] for n, h in zip(shape, (0.22, 0.5, 0.3))]
    u = fga.reconstruct_lattice(b, axes, rw=w.rw).cpu().numpy().reshape(-1, 3)
    x = np.stack(np.meshgrid(*axes, indexing="ij"), -1).reshape(-1, 3)
    v = fga.reconstruct(b, torch.as_tensor(x, device="cuda"), rw=w.rw).cpu().numpy()
    assert np.linalg.norm(v) > 0 and rel_l2(u, v) <= 1e-4
