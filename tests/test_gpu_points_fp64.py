"""FP64 Gaussian sum at points (table-driven sine, cosine and exponential) against the allocation-free sum, another
kernel with the library's functions: point counts around a tile of 32 and around the powers of two that share its lanes, ragged beam counts, phases below and far above a
turn, windows beyond the range of exponents the tables take (am < -700) and phases beyond theirs.  Tolerance: the
phases round to |ph| 2^-53 in either kernel (1e-14 at 100 rad; 1e-9 at 1e7 rad), sums of some thousand terms that cancel
by up to a factor of ten: 1e-12, and 1e-7 for the largest phases."""
import dataclasses

import numpy as np
import pytest

from paper_1810_06760_gb300 import workloads as W
from tests.helpers import gpu_setup, rel_l2
from tests.test_gpu_cells import fga  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 2, 5, 12, 33, 500])
@pytest.mark.parametrize("nq,np_,k,rw,pscale,tol", [(1, 1, 64.0, None, 1.0, 1e-12), (3, 3, 128.0, None, 1.0, 1e-12),
                                                   (4, 5, 16.0, 0.2, 1.0, 1e-12), (3, 4, 2000.0, 1.0, 1.0, 1e-12),
                                                   (2, 3, 64.0, None, 1e6, 1e-7)])
def test_fp64_points_match_library_functions(fga, n, nq, np_, k, rw, pscale, tol):  # noqa: F811
    import torch
    w = W.smooth(nq=nq, np_=np_, ny=24, k=min(k, 128.0), grid=False)
    mesh = dataclasses.replace(w.mesh, p0=w.mesh.p0 * pscale, dp=w.mesh.dp * pscale)
    if pscale > 1.0:
        mesh = dataclasses.replace(mesh, q0=w.mesh.q0, dq=w.mesh.dq)
    w = dataclasses.replace(w, k=k, mesh=mesh)
    model, desc, keep = gpu_setup(w, 1)
    b = fga.decompose(model, desc)
    if pscale == 1.0:
        fga.propagate(model, b, w.dt, 20)
    pts = 0.5 + 0.4 * (W.random_points(n, 0.0, 1.0, 3) - 0.5)
    x = torch.as_tensor(pts, device="cuda")
    u = fga.reconstruct(b, x, rw=rw or w.rw)
    v = torch.empty_like(u)
    fga.reconstruct_noalloc(b, x, v, rw=rw or w.rw)
    u, v = u.cpu().numpy(), v.cpu().numpy()
    assert np.isfinite(u.view(np.float64)).all() and (n < 33 or np.any(v))   # a few points may lie in no window
    assert rel_l2(u, v) <= tol if np.any(v) else not np.any(u)
