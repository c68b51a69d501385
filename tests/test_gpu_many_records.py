"""Volume-lattice sum of more than 2^31 / 12 beam records: record offsets pass 32 bits.  186.6 M beams of all four classes
start at one point with nearly one direction (their contributions add up instead of cancelling), so that the records
beyond the 178.9 M-th carry several per cent of the sum.  Against the point sum (another kernel) at the same points.
Tolerance 5e-3: the lattice kernel's FP32 accumulation truncates, 3e-8 a step and 58,000 steps an item here."""
import dataclasses

import numpy as np
import pytest

from paper_1810_06760_gb300 import workloads as W
from tests.test_gpu_cells import fga  # noqa: F401
from tests.helpers import gpu_setup, rel_l2

pytestmark = pytest.mark.gpu


def test_volume_sum_beyond_32_bit_offsets(fga):  # noqa: F811
    import torch
    if torch.cuda.mem_get_info()[0] < 120e9:
        pytest.skip("needs 60 GB of device memory")
    w = W.smooth(nq=1, np_=360, ny=24, grid_n=17)
    p = w.mesh.p0 + 0.5 * (w.mesh.np_ - 1) * w.mesh.dp    # the packet's direction
    dp = np.full(3, 0.2 / 360)
    w = dataclasses.replace(w, mesh=dataclasses.replace(w.mesh, p0=p - 0.1 + 0.5 * dp, dp=dp))
    assert 4 * w.mesh.M * 12 > 2 ** 31
    model, desc, keep = gpu_setup(w, 0)
    b = fga.decompose(model, desc)
    try:
        axes = [c + 0.02 * np.arange(-n, n + 1) for c, n in zip(w.mesh.q0, (1, 2, 1))]
        u = fga.reconstruct_lattice(b, axes, rw=w.rw).cpu().numpy().reshape(-1, 3)
        x = np.stack(np.meshgrid(*axes, indexing="ij"), -1).reshape(-1, 3)
        v = fga.reconstruct(b, torch.as_tensor(x, device="cuda"), rw=w.rw).cpu().numpy()
    finally:
        b.close()
    assert np.linalg.norm(v) > 0 and rel_l2(u, v) <= 5e-3
