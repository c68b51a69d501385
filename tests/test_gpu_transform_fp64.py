"""FP64 wave-packet transform at every width of its tiles (8 J columns, J from 2 to 9 by the number of pairs per axis) and
beyond one tile, rows and terms that are no multiples of 32 and 16, against the direct sums in numpy.  Tolerance: phases
of up to 50 rad rounded to 2^-53 and sums of at most 70 terms in three stages, 1e-13."""
import numpy as np
import pytest

from paper_1810_06760_gb300 import workloads as W
from tests.helpers import rel_l2
from tests.test_gpu_cells import fga  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nq,np_,ny", [(1, 1, (1, 1, 1)), (5, 4, (33, 31, 32)), (5, 6, (1, 70, 3)), (6, 6, (5, 2, 65)),
                                       (6, 8, (16, 17, 15)), (7, 8, (9, 8, 7)), (4, 16, (20, 3, 11)), (9, 8, (13, 14, 12)),
                                       (10, 10, (7, 5, 6))])
def test_fp64_transform_tile_widths(fga, nq, np_, ny):  # noqa: F811
    import torch
    rng = np.random.default_rng(nq * 100 + np_)
    k = 24.0
    f = rng.normal(size=tuple(ny) + (3,)) + 1j * rng.normal(size=tuple(ny) + (3,))
    y0, dy = np.array([0.1, -0.2, 0.3]), np.array([0.02, 0.03, 0.025])
    mesh = W.MeshSpec(nq, np.array([0.2, -0.1, 0.4]), np.array([0.07, 0.05, 0.06]), np_, np.array([-0.6, 0.2, 0.1]),
                      np.array([0.2, 0.15, 0.1]))
    desc = fga.init_desc(k, torch.as_tensor(f, device="cuda"), None, y0, dy, mesh, (0,), fga.PREC_FP64)
    got = fga.transform(desc).cpu().numpy()
    ref = f
    for a in range(3):
        q = np.repeat(mesh.q0[a] + mesh.dq[a] * np.arange(nq), np_)
        p = np.tile(mesh.p0[a] + mesh.dp[a] * np.arange(np_), nq)
        d = (y0[a] + dy[a] * np.arange(ny[a]))[None] - q[:, None]
        ref = np.moveaxis(np.tensordot(np.exp(-1j * k * p[:, None] * d - 0.5 * k * d * d), ref, axes=(1, a)), 0, a)
    assert rel_l2(got, ref * np.prod(dy)) <= 1e-13
