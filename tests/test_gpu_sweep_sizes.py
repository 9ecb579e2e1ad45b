"""One sweep against the oracle at the sizes where the work of its kernels is
split differently: grids around the 32 lanes of the spline's substitution,
end fits of more points than half the grid, increment counts around a warp and
up to the largest, one to four integrated legs (FP64 path).

Tolerances: both sides evaluate the same samples in FP64; rounding (1e-15 of
energies up to 60) over the width 0.05 is 1e-12 of an exponent that is at most
750, so 1e-8 of a task's mean; a refined map's edges follow the training data
with a factor of order one: 1e-7.
"""
from dataclasses import replace

import numpy as np
import pytest

import workloads as W
from tests._helpers import oracle_sweep, task_arrays

pytestmark = pytest.mark.gpu


def _check(prob, f0, t=0.0):
    import torch
    from paper_2603_28848_gb300 import Collision
    col = Collision(prob, W.PREC_FP64)
    C, err = col.eval(torch.tensor(f0, device="cuda"), t)
    col.check()
    mean, _ = col.task_results()
    maps = col.maps()
    col.close()
    Co, _, detail, state = oracle_sweep(prob, f0, t, "f64")
    om, _ = task_arrays(detail, len(mean))
    assert np.all(np.abs(mean - om) <= 1e-8 * np.abs(om) + 1e-300)
    scale = np.max(np.abs(om))
    for tid, edges in state.maps.items():
        if abs(om[tid]) > 1e-12 * scale:
            D, nb1 = edges.shape
            assert np.max(np.abs(maps[tid][: D * nb1].reshape(D, nb1) - edges)) < 1e-7, tid


def _mb(n, neval, nbins=50, **kw):
    prob, f0 = W.c1_maxwell_2to2(n, neval, 1)
    procs = tuple(replace(p, nbins=nbins, sigma_E=0.05) for p in prob.processes)
    return replace(prob, processes=procs, **kw), f0


@pytest.mark.parametrize("n", [4, 5, 33, 34, 35, 66, 130])
def test_grid_sizes(n):
    _check(*_mb(n, 300))


@pytest.mark.parametrize("tail", [2, 7, 9])
def test_end_fit_points(tail):
    _check(*_mb(9, 600, tail_points=tail))


@pytest.mark.parametrize("nbins", [2, 3, 31, 32, 33, 64, 65, 255, 256])
def test_increment_counts(nbins):
    _check(*_mb(6, 900, nbins))


@pytest.mark.parametrize("legs", [(1, 2), (2, 2), (2, 3), (3, 3)])
def test_leg_counts(legs):
    prob, f0 = _mb(6, 700)
    p = replace(prob.processes[0], species_in=(0,) * legs[0], species_out=(0,) * legs[1], name="legs")
    _check(replace(prob, processes=(p,)), f0)
