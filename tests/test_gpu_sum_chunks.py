"""Sums of a window's samples whose partial sums pass the bound of one launch: several launches, each at its own offset in
the records and outputs.  Every sample against a solve with that sample alone (the same kernels; the same states), for
the point sums in both precisions and for receiver planes split by samples and by tiles.  Tolerances: rounding of sums
grouped otherwise, 1e-5 in FP32 and 1e-12 in FP64; neighbouring samples differ by more than ten
times that."""
import dataclasses

import numpy as np
import pytest

from paper_1810_06760_gb300 import workloads as W
from tests.test_gpu_cells import fga  # noqa: F401
from tests.helpers import gpu_setup, rel_l2

pytestmark = pytest.mark.gpu


def _case(n_times):
    w = W.smooth(nq=4, np_=5, ny=24, nsteps=8, grid_n=33)
    return dataclasses.replace(w, times=w.T * np.arange(1, n_times + 1) / n_times)   # one window of steps


def _check(fga, w, prec, some, tol, **receivers):  # noqa: F811
    model, desc, keep = gpu_setup(w, prec)
    u, _ = fga.solve(model, desc, w.dt, w.nsteps, w.times, rw=w.rw, **receivers)
    u = u.cpu().numpy().reshape(len(w.times), -1)
    for j in some:
        v, _ = fga.solve(model, desc, w.dt, w.nsteps, w.times[j:j + 1], rw=w.rw, **receivers)
        assert rel_l2(u[j], v.cpu().numpy().ravel()) <= tol, j
        other = u[j - 1 if j else 1]
        assert rel_l2(other, v.cpu().numpy().ravel()) > 10 * tol, j


@pytest.mark.parametrize("prec,n_times", [(0, 120), (1, 60)])
def test_point_sums_in_several_launches(fga, prec, n_times):  # noqa: F811
    import torch
    w = _case(n_times)
    rx = torch.as_tensor(np.random.default_rng(5).uniform(0.0, 1.0, (2500, 3)), device="cuda")
    _check(fga, w, prec, range(0, n_times, 7), 1e-5 if prec == 0 else 1e-12, rx=rx)


@pytest.mark.parametrize("n0,n1,n_times", [(60, 50, 40), (300, 290, 3)])
def test_plane_sums_in_several_launches(fga, n0, n1, n_times):  # noqa: F811
    axes = tuple((np.arange(n) + 0.5) / n for n in (n0, n1)) + (np.array([0.5]),)
    _check(fga, _case(n_times), 0, range(0, n_times, 3 if n_times > 3 else 1), 1e-5, rx_axes=axes)
