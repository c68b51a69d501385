"""Beams that meet spherical interfaces at normal incidence or within 1e-14 to 1e-6 rad of it, against the oracle's
spherical solve: all beams start at (or very near) the spheres' centre, diagonal directions among them.  The part of P
along the interface is then rounding noise, and the S beams' amplitude must not depend on the direction it happens to
have.  Tolerances: those of the spherical layers' parity test (FP64 1e-10, element by element 1e-9; FP32 1e-4)."""
import dataclasses

import numpy as np
import pytest

from paper_1810_06760_gb300 import workloads as W
from tests.test_gpu_cells import fga  # noqa: F401
from tests.test_gpu_layered import _disp, _key, _oracle_shells
from tests.helpers import gpu_setup, max_rel_dominant, rel_l2

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,offset", [(1, 0.0), (1, 1e-13), (1, 1e-10), (1, 1e-6), (0, 0.0)])
def test_normal_incidence_on_spheres(fga, oracle, prec, offset):  # noqa: F811
    w = W.shells(nq=1, np_=6, ny=24, nsteps=30, dt=0.1)
    x0 = w.mesh.q0                                        # the only q node
    med = dataclasses.replace(w.medium, z_interfaces=(12.0, 5.0),
                              layer_center=tuple(x0 + offset * np.array([1.0, -2.0, 0.5])))
    # a field with a fixed polarisation has S amplitudes in every direction
    y = w.y0 + w.dy * np.stack(np.meshgrid(*[np.arange(w.ny)] * 3, indexing="ij"), -1)
    f = np.exp(-w.k * ((y - x0) ** 2).sum(-1))[..., None] * np.array([1.0, 0.5j, -0.3 + 0.2j])
    w = dataclasses.replace(w, medium=med, f=f)
    model, desc, keep = gpu_setup(w, prec)
    fga.set_layered_options(desc, growth=8.0)
    beams = fga.decompose(model, desc)
    fga.propagate(model, beams, w.dt, w.nsteps)
    gst, gmeta, gmid, gpath, dropped = beams.export_all()
    ost, ometa, omid, opath, _ = _oracle_shells(oracle, w, w.nsteps)
    assert dropped == 0 and np.count_nonzero(opath) > w.n_beams
    gk, ok = _key(gmeta, gmid, gpath), _key(ometa, omid, opath)
    gi = {k: i for i, k in enumerate(gk)}
    oi = {k: i for i, k in enumerate(ok)}
    if prec == 1:
        assert set(gk) == set(ok)
    # FP32: a converted child of a slightly oblique incidence may lie on either side of the smallest amplitude kept
    common = [k for k in ok if k in gi]
    assert len(common) >= (1.0 if prec else 0.8) * len(ok)
    G, Ob = np.stack([gst[gi[k]] for k in common]), np.stack([ost[oi[k]] for k in common])
    gm, om = (np.array([m[i[k]] for k in common]) for m, i in ((gmeta, gi), (ometa, oi)))
    tol, tol_max = (1e-10, 1e-9) if prec else (1e-4, 2e-3)
    assert rel_l2(G[:, 0:6], Ob[:, 0:6]) <= tol
    for wave in (0, 1):
        sel = ((om & 3) >= 2) == bool(wave)
        d, ref = _disp(G[sel], gm[sel]), _disp(Ob[sel], om[sel])
        assert np.linalg.norm(ref) > 0
        assert rel_l2(d, ref) <= tol and max_rel_dominant(d, ref, 1e-2) <= tol_max, wave
