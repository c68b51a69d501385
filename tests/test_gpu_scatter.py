"""The scattering coefficients of an interface event (closed form: 2 x 2 for P-SV, a ratio for SH) against the oracle's
Zoeppritz system, FP64, through populations matched by lineage: vertical incidence, where the interface's frame is
arbitrary, near-grazing incidence, evanescent waves on either side, both directions of every contrast and the strongest
ones, all four classes.  Tolerance: the FP64 parity bar of the library, 1e-10."""
import dataclasses

import numpy as np
import pytest

from paper_1810_06760_gb300 import workloads as W
from tests.test_gpu_cells import fga  # noqa: F401
from tests.test_gpu_layered import GROUPS, _key, _oracle_population
from tests.helpers import gpu_setup, rel_l2

pytestmark = pytest.mark.gpu

CONTRASTS = {
    "faster below": ((5.8, 6.5, 8.04), (3.46, 3.85, 4.47), (2.72, 2.92, 3.32)),
    "slower below": ((8.04, 5.8, 4.0), (4.47, 3.46, 1.0), (3.32, 2.72, 2.0)),
    "slow S, light": ((6.0, 1.6, 6.0), (3.4, 0.2, 3.4), (2.8, 1.0, 2.8)),
    "no contrast in S": ((6.0, 7.0, 6.5), (3.5, 3.5, 3.5), (2.7, 2.7, 2.7)),
}


def _case(contrast, horizontal):
    w = W.layered(nq=2, np_=4, ny=24, nsteps=24, dt=0.1)
    cp, cs, rho = CONTRASTS[contrast]
    med = dataclasses.replace(w.medium, layer_cp=np.array(cp), layer_cs=np.array(cs), layer_rho=np.array(rho))
    # horizontal nodes hold 0 (vertical beams) or are much larger than the vertical ones (near grazing)
    p0, dp = ((0.0, -0.4, -0.9), (0.5, 0.4, 0.6)) if not horizontal else ((-1.5, -1.2, -0.3), (0.9, 0.8, 0.2))
    mesh = dataclasses.replace(w.mesh, p0=np.array(p0), dp=np.array(dp))
    return dataclasses.replace(w, medium=med, mesh=mesh)


@pytest.mark.parametrize("horizontal", [False, True])
@pytest.mark.parametrize("contrast", list(CONTRASTS))
def test_scattering_matches_oracle(fga, oracle, contrast, horizontal):  # noqa: F811
    w = _case(contrast, horizontal)
    model, desc, keep = gpu_setup(w, 1)
    beams = fga.decompose(model, desc)
    fga.propagate(model, beams, w.dt, w.nsteps)
    gst, gmeta, gmid, gpath, dropped = beams.export_all()
    ost, ometa, omid, opath = _oracle_population(oracle, w, w.nsteps)
    assert dropped == 0 and np.count_nonzero(opath) > 50      # interfaces were met
    gk, ok = _key(gmeta, gmid, gpath), _key(ometa, omid, opath)
    assert set(gk) == set(ok)
    gi = {k: i for i, k in enumerate(gk)}
    oi = {k: i for i, k in enumerate(ok)}
    G = np.stack([gst[gi[k]] for k in ok])
    Ob = np.stack([ost[oi[k]] for k in ok])
    assert np.all(np.isfinite(Ob))
    for name, sl in GROUPS.items():
        assert rel_l2(G[:, sl], Ob[:, sl]) <= 1e-10, name
