"""Layered propagation under a bound on the library's memory that leaves no room for the lists of beams at an interface
(16 bytes a slot): shorter lists, a step and a part of the population at a time, give the population of the whole ones,
lineage by lineage.  Tolerances: those of a group of steps against single ones."""
import numpy as np
import pytest

from paper_1810_06760_gb300 import workloads as W
from tests.test_gpu_cells import fga  # noqa: F401
from tests.test_gpu_layered import GROUPS, _key
from tests.helpers import gpu_setup, rel_l2

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [1, 0])
@pytest.mark.parametrize("make", [W.layered, W.shells, W.undulating])
def test_short_event_lists(fga, make, prec):  # noqa: F811
    w = make(nq=3, np_=4, ny=24, dt=0.1)
    pops = []
    for room in (0, 100e3):   # 83,000 slots: 1.3 MB of lists
        model, desc, keep = gpu_setup(w, prec)
        fga.set_layered_options(desc, growth=12.0)
        beams = fga.decompose(model, desc)
        if room:
            fga.set_device_memory_limit(fga.device_memory_in_use() + room)
        try:
            for n in (7, 23):
                fga.propagate(model, beams, w.dt, n)
        finally:
            fga.set_device_memory_limit(0)
        st, meta, mid, path, dropped = beams.export_all()
        assert dropped == 0
        key = _key(meta, mid, path)
        assert len(set(key)) == len(key) > 1.5 * w.n_beams
        pops.append((dict(zip(key, range(len(key)))), st, meta))
    (ka, sa, ma), (kb, sb, mb) = pops
    common = sorted(set(ka) & set(kb))
    assert len(common) >= (1.0 if prec == 1 else 0.999) * max(len(ka), len(kb))
    a, b = [ka[c] for c in common], [kb[c] for c in common]
    np.testing.assert_array_equal(ma[a] & 0x6FF7, mb[b] & 0x6FF7)
    for name, sl in GROUPS.items():
        tol = 1e-9 if prec == 1 else (5e-4 if name.startswith("dz") else 1e-4)
        assert rel_l2(sa[a][:, sl], sb[b][:, sl]) <= tol, name
