"""Tensor-core wave-packet transform at the edges of its tiles (128 rows, 64 columns, K blocks of 32) against the
direct sums in numpy: single points, uneven axes, 64 and 65 columns, K of one block, two and a ragged third.
Tolerance: three FP16-split stages of 2^-22 per product and FP32 accumulation over at most 70 terms: 1e-5."""
import numpy as np
import pytest

from paper_1810_06760_gb300 import workloads as W
from tests.helpers import rel_l2

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


@pytest.mark.parametrize("nq,np_,ny", [(1, 1, (1, 1, 1)), (2, 4, (33, 31, 32)), (8, 8, (1, 70, 3)), (13, 5, (5, 2, 65)),
                                       (3, 43, (9, 8, 7)), (1, 3, (64, 64, 2))])
def test_transform_tile_edges(fga, nq, np_, ny):
    import torch
    rng = np.random.default_rng(nq * 100 + np_)
    k = 24.0
    f = rng.normal(size=tuple(ny) + (3,)) + 1j * rng.normal(size=tuple(ny) + (3,))
    y0, dy = np.array([0.1, -0.2, 0.3]), np.array([0.02, 0.03, 0.025])
    mesh = W.MeshSpec(nq, np.array([0.2, -0.1, 0.4]), np.array([0.07, 0.05, 0.06]), np_, np.array([-0.6, 0.2, 0.1]),
                      np.array([0.2, 0.15, 0.1]))
    desc = fga.init_desc(k, torch.as_tensor(f, device="cuda"), None, y0, dy, mesh, (0,), fga.PREC_FP32)
    got = fga.transform(desc).cpu().numpy()
    ref = f
    for a in range(3):
        q = np.repeat(mesh.q0[a] + mesh.dq[a] * np.arange(nq), np_)
        p = np.tile(mesh.p0[a] + mesh.dp[a] * np.arange(np_), nq)
        d = (y0[a] + dy[a] * np.arange(ny[a]))[None] - q[:, None]
        ref = np.moveaxis(np.tensordot(np.exp(-1j * k * p[:, None] * d - 0.5 * k * d * d), ref, axes=(1, a)), 0, a)
    assert rel_l2(got, ref * np.prod(dy)) <= 1e-5
