"""The selection's tiles (1024 mesh points, all classes at once) against the beams of an unselected decomposition,
filtered here: meshes of less than a tile, a ragged last tile and many tiles, class subsets, an initial velocity, one
node on an axis.  The threshold lies in the middle of the widest gap of |psi| near the wanted quantile, so that rounding
cannot move a beam across it.  Tolerance of the states: the same formulas in another kernel, a few ulp (1e-6 in FP32,
1e-14 in FP64, relative L2)."""
import numpy as np
import pytest

from paper_1810_06760_gb300 import workloads as W
from tests.helpers import rel_l2
from tests.test_gpu_cells import fga  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("nq,np_,classes,v0,quantile", [(2, 3, (1,), False, 0.5), (3, 4, (0, 1, 2, 3), True, 0.9),
                                                       (5, 1, (0, 3), False, 0.3), (4, 5, (2, 3), True, 0.99)])
def test_selected_tiles(fga, nq, np_, classes, v0, quantile, prec):  # noqa: F811
    import torch
    w = W.smooth(nq=nq, np_=np_, ny=16, grid=False, k=16.0)
    model = fga.model_from_medium(w.medium, "cuda")
    f = torch.as_tensor(w.f, device="cuda")
    g = torch.as_tensor(8j * w.f[::-1].copy(), device="cuda") if v0 else None
    full = fga.decompose(model, fga.init_desc(w.k, f, g, w.y0, w.dy, w.mesh, classes, prec))
    st, meta, ids, _, _ = full.export_all()
    mag = np.sqrt((st[:, 42:46] ** 2).sum(1))
    rel = np.sort(mag / mag.max())
    lo = int(quantile * (rel.size - 2))
    win = slice(lo, min(lo + 20, rel.size - 1))
    i = lo + int(np.argmax(np.diff(np.log(np.maximum(rel, 1e-30)))[win]))
    eps = float(np.sqrt(rel[i] * rel[i + 1]))
    keep = mag / mag.max() > eps
    sel = fga.decompose(model, fga.init_desc(w.k, f, g, w.y0, w.dy, w.mesh, classes, prec, psi_rel_min=eps))
    st2, meta2, ids2, _, _ = sel.export_all()
    assert 0 < keep.sum() < keep.size
    assert np.array_equal(ids2, ids[keep]) and np.array_equal(meta2, meta[keep])
    for sl in (slice(0, 3), slice(3, 6), slice(6, 42), slice(42, 46)):
        assert rel_l2(st2[:, sl], st[keep][:, sl]) <= (1e-14 if prec else 1e-6)
