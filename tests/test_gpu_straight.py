"""Beams where the speed is constant: the closed-form steps of constant and layered media.

Constant media against the oracle's RK4 at step counts around the renewal of the determinant's expansion
(64 steps), forwards and backwards, every class.  Layered media: a group of steps advanced in one call
against the same steps taken one call each (the events then fall into other kernels' rounds), lineage by
lineage.  Tolerances: FP64 rounding of up to 130 steps, with room for crossings near grazing in layers;
FP32 130 steps of half an ulp each (8e-6) in the constant medium, the layered parity bars otherwise."""
import dataclasses

import numpy as np
import pytest

from paper_1810_06760_gb300 import workloads as W
from tests.helpers import gpu_setup, oracle_beams, rel_l2

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


@pytest.mark.parametrize("prec", [1, 0])
@pytest.mark.parametrize("nsteps,dt", [(1, 0.005), (63, 0.005), (64, -0.005), (65, 0.01), (130, 0.02)])
def test_constant_medium_steps(fga, oracle, prec, nsteps, dt):
    w = dataclasses.replace(W.homogeneous(nq=3, np_=3, ny=20), classes=(0, 1, 2, 3), dt=dt, nsteps=nsteps)
    model, desc, keep = gpu_setup(w, prec)
    beams = fga.decompose(model, desc)
    fga.propagate(model, beams, dt, nsteps)
    gst, gmeta = beams.export()
    omodel, mesh, ob = oracle_beams(oracle, w)
    ost, ometa = np.concatenate([b[1] for b in ob]), np.concatenate([b[2] for b in ob])
    oracle.propagate(omodel, ost, ometa, dt, nsteps)
    np.testing.assert_array_equal(gmeta & 7, ometa & 7)
    for name, sl in GROUPS.items():
        assert rel_l2(gst[:, sl], ost[:, sl]) <= (1e-12 if prec == 1 else 1e-5), name


@pytest.mark.parametrize("prec", [1, 0])
@pytest.mark.parametrize("make,nsteps", [(W.layered, 7), (W.layered, 70), (W.shells, 70), (W.undulating, 70)])
def test_layered_group_equals_single_steps(fga, prec, make, nsteps):
    w = make(nq=3, np_=4, ny=24, dt=0.1)
    pops = []
    for calls, per in ((1, nsteps), (nsteps, 1)):
        model, desc, keep = gpu_setup(w, prec)
        fga.set_layered_options(desc, growth=12.0)
        beams = fga.decompose(model, desc)
        for _ in range(calls):
            fga.propagate(model, beams, w.dt, per)
        st, meta, mid, path, dropped = beams.export_all()
        assert dropped == 0
        key = [((int(m) >> 13) & 3, int(i), int(p)) for m, i, p in zip(meta, mid, path)]
        assert len(set(key)) == len(key)
        pops.append((dict(zip(key, range(len(key)))), st, meta))
    (ka, sa, ma), (kb, sb, mb) = pops
    common = sorted(set(ka) & set(kb))
    # FP32: a beam that ends a step within rounding of an interface may be taken either way
    assert len(common) >= (1.0 if prec == 1 else 0.999) * max(len(ka), len(kb))
    a, b = [ka[c] for c in common], [kb[c] for c in common]
    np.testing.assert_array_equal(ma[a] & 0x6FF7, mb[b] & 0x6FF7)
    for name, sl in GROUPS.items():
        tol = 1e-9 if prec == 1 else (5e-4 if name.startswith("dz") else 1e-4)
        assert rel_l2(sa[a][:, sl], sb[b][:, sl]) <= tol, name
