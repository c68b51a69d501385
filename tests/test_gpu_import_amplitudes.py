"""A P beam has one amplitude.  The slot of the second one of an imported P beam takes no part in the propagation and is
exported as it came, in every medium and precision; an S beam's second amplitude does change."""
import numpy as np
import pytest

from paper_1810_06760_gb300 import workloads as W
from tests.test_gpu_cells import fga  # noqa: F401
from tests.helpers import gpu_setup

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("medium", ["const", "sine", "grid"])
@pytest.mark.parametrize("prec", [0, 1])
def test_second_amplitude_of_p_beams(fga, medium, prec):  # noqa: F811
    w = W.smooth(nq=2, np_=3, ny=16, grid_n=17, grid=medium == "grid")
    model, desc, keep = gpu_setup(w, prec)
    beams = fga.decompose(model, desc)
    k, wt, _ = fga.beams_params(beams)
    st, meta = beams.export()
    st[:, 44:46] = np.array([1.0, 2.0]) * (1.0 + np.arange(st.shape[0]) % 8)[:, None]   # exact in FP32
    if medium == "const":
        model = fga.Model("const", cp0=2.0, cs0=1.0)
    b = fga.beams_import(st, meta, k, wt, prec)
    fga.propagate(model, b, 0.01, 70)
    got, gm = b.export()
    p = (gm & 3) < 2
    np.testing.assert_array_equal(got[p, 44:46], st[p, 44:46])
    assert np.all(got[~p, 44:46] != st[~p, 44:46])
