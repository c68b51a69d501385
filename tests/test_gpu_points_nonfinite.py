"""Point sums of a beam set in which a few beams' amplitudes or propagation vectors are infinite, NaN or as large as
a float goes: only the points within those beams' windows are affected, the others are the sums of the rest.  FP32 and
FP64; tolerances of sums that are only grouped otherwise, 1e-5 and 1e-12."""
import numpy as np
import pytest

from paper_1810_06760_gb300 import workloads as W
from tests.test_gpu_cells import fga  # noqa: F401
from tests.helpers import gpu_setup, rel_l2

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 37, 3000])
@pytest.mark.parametrize("prec", [0, 1])
def test_points_outside_a_bad_beams_window(fga, prec, n):  # noqa: F811
    import torch
    w = W.smooth(nq=4, np_=4, ny=24, grid_n=17)
    model, desc, keep = gpu_setup(w, prec)
    b = fga.decompose(model, desc)
    k, wt, _ = fga.beams_params(b)
    st, meta = b.export()
    bad = np.arange(3, st.shape[0], st.shape[0] // 24)
    rng = np.random.default_rng(2)
    for i, j in enumerate(bad):
        field = (42, 43, 3 + i % 3)[i % 3]               # Re a, Im a, a component of P
        st[j, field] = (np.inf, np.nan, -np.inf, 3e38)[i % 4]
    st[bad, 0:3] += rng.uniform(-0.2, 0.2, (len(bad), 3))
    x = rng.uniform(-0.6, 1.5, (n, 3))
    near = (np.linalg.norm(x[:, None] - st[None, bad, 0:3], axis=-1) <= w.rw * (1 + 1e-5)).any(1)
    x[0] = x[near][0] if n > 1 else x[0]
    near = (np.linalg.norm(x[:, None] - st[None, bad, 0:3], axis=-1) <= w.rw * (1 + 1e-5)).any(1)
    good = np.setdiff1d(np.arange(st.shape[0]), bad)
    u, v = (fga.reconstruct(fga.beams_import(st[s], meta[s], k, wt, prec), torch.as_tensor(x, device="cuda"), rw=w.rw).cpu()
            .numpy() for s in (np.arange(st.shape[0]), good))
    assert np.isfinite(v).all()
    if n > 1:
        assert near.any() and (~near).any() and not np.isfinite(u[near]).all()
        assert np.linalg.norm(v[~near]) > 0
    assert np.isfinite(u[~near]).all()
    assert rel_l2(u[~near], v[~near]) <= (1e-5 if prec == 0 else 1e-12)
