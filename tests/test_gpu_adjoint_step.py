"""FP32 reverse steps on grid media (one kernel per class and step, threads striding over the beams) against the
FP64 stage kernels: grids of two nodes, uneven axes, beams that leave the grid (clamped sampling), ragged class
blocks, more beams in a class than threads in flight, steps with and without samples, the sample at the last step,
checkpoint lengths that do not divide the steps.  Tolerance: the FP32 bar of the gradient, 1e-4 relative L2 (the
FP32 rounding of the trajectory, 2e-5, amplified by k |x - Q| in the phase derivatives)."""
import numpy as np
import pytest

from paper_1810_06760_gb300 import workloads as W
from tests.helpers import rel_l2
from tests.test_gpu_cells import _fields, fga  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,ext,nq,np_,classes,nsteps,every", [
    ((2, 2, 2), 1.0, 3, 3, (0, 1, 2, 3), 20, 20),
    ((3, 17, 5), 0.6, 3, 5, (3,), 13, 5),
    ((40, 9, 33), 1.2, 4, 4, (0, 2), 17, 8),
    ((33, 32, 2), 0.3, 7, 6, (1, 2), 9, 4),          # 74,088 beams a class
])
def test_fp32_step_matches_fp64(fga, shape, ext, nq, np_, classes, nsteps, every):  # noqa: F811
    import torch
    origin = (0.5 - 0.5 * ext,) * 3
    h = tuple(ext / (n - 1) for n in shape)
    gp, gs = _fields(shape, 2.0, h, origin), _fields(shape, 1.2, h, origin)
    model = fga.Model("grid", grid_p=torch.as_tensor(gp, device="cuda"), grid_s=torch.as_tensor(gs, device="cuda"),
                      origin=origin, spacing=h)
    w = W.smooth(nq=nq, np_=np_, ny=16, grid=False, k=16.0)
    f = torch.as_tensor(w.f, device="cuda")
    dt = 0.01
    T = dt * nsteps
    times = np.array([0.13 * T, 0.14 * T, 0.6 * T, T])
    rng = np.random.default_rng(nsteps)
    rx = torch.as_tensor(np.array([0.35, 0.45, 0.55]) + 0.25 * (2 * rng.random((19, 3)) - 1), device="cuda")
    ub = torch.as_tensor(rng.standard_normal((4, 19, 3, 2)) @ np.array([1, 1j]), device="cuda")
    g = []
    for prec in (0, 1):
        desc = fga.init_desc(w.k, f, None, w.y0, w.dy, w.mesh, classes, prec)
        g.append(fga.solve_vjp(model, desc, dt, nsteps, times, rx, ub.to(torch.complex128 if prec else torch.complex64),
                               checkpoint_every=every))
        torch.cuda.synchronize()
    for s in (0, 1):
        a, b = g[0][s].cpu().numpy(), g[1][s].cpu().numpy()
        used = any((c >= 2) == bool(s) for c in classes)
        assert np.any(b) == used
        if used:
            assert rel_l2(a, b) <= 1e-4
        else:
            assert not np.any(a)
