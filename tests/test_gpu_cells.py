"""FP32 propagation on grid media (the kernel that keeps each beam's grid cell in shared memory) against the
FP64 general kernel on the same beams: grids of two nodes, uneven axes, beams that leave the grid (clamped
sampling) and steps that cross several cells, ragged class blocks and class subsets.  Tolerance: the FP32
parity bar of the library, 1e-4 (rounding of 40 steps: 2e-6 per field, times the Jacobian's growth)."""
import numpy as np
import pytest

from paper_1810_06760_gb300 import workloads as W
from tests.helpers import rel_l2

pytestmark = pytest.mark.gpu

GROUPS = {"Q": slice(0, 3), "P": slice(3, 6), "dzQ": slice(6, 24), "dzP": slice(24, 42), "a": slice(42, 46)}


@pytest.fixture(scope="module")
def fga():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1810_06760_gb300 import build, fga as F
    build.build()
    F.lib()
    return F


def _fields(shape, c0, h, origin):
    """c0 + 0.1 sum_d sin(a_d x_d + d) with exact derivatives on an uneven node grid."""
    a = np.array([2.0, 1.5, 2.5])
    ax = [origin[d] + h[d] * np.arange(shape[d]) for d in range(3)]
    X = np.meshgrid(*ax, indexing="ij")
    out = np.zeros(tuple(shape) + (10,))
    out[..., 0] = c0
    for d, hess in zip(range(3), (4, 7, 9)):
        ph = a[d] * X[d] + d
        out[..., 0] += 0.1 * np.sin(ph)
        out[..., 1 + d] = 0.1 * a[d] * np.cos(ph)
        out[..., hess] = -0.1 * a[d] ** 2 * np.sin(ph)
    return out.astype(np.float32)


@pytest.mark.parametrize("classes", [(0, 1, 2, 3), (3,), (0, 2)])
@pytest.mark.parametrize("shape,ext", [((2, 2, 2), 1.0), ((3, 17, 5), 0.6), ((40, 9, 33), 1.2), ((65, 64, 2), 0.3)])
def test_fp32_cells_match_fp64(fga, shape, ext, classes):
    import torch
    origin = (0.5 - 0.5 * ext,) * 3
    h = tuple(ext / (n - 1) for n in shape)
    gp, gs = _fields(shape, 2.0, h, origin), _fields(shape, 1.2, h, origin)
    model = fga.Model("grid", grid_p=torch.as_tensor(gp, device="cuda"), grid_s=torch.as_tensor(gs, device="cuda"),
                      origin=origin, spacing=h)
    torch.cuda.synchronize()
    w = W.smooth(nq=3, np_=5, ny=16, grid=False)        # 3,375 beams per class: a ragged last block
    f = torch.as_tensor(w.f, device="cuda")
    st = []
    for prec in (0, 1):
        beams = fga.decompose(model, fga.init_desc(w.k, f, None, w.y0, w.dy, w.mesh, classes, prec))
        fga.propagate(model, beams, 0.01, 39)
        fga.propagate(model, beams, -0.004, 1)
        s, meta = beams.export()
        st.append(s)
    for name, sl in GROUPS.items():
        assert rel_l2(st[0][:, sl], st[1][:, sl]) <= 1e-4, name
