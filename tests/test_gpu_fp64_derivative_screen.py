"""The FP32 screen of the FP64 derivative kernels: what it may not drop, and the
contexts whose tables leave it no room.

Tolerances: both sides evaluate the same samples in FP64; the energy balance
(rounded to 4e-15 for energies of 30) enters a weight as dE / sigma^2 of it:
2e-13 for 15 off the shell at a width of 0.5, so 1e-11 of C~.
"""
from dataclasses import replace

import numpy as np
import pytest

import workloads as W
from oracle import adjoint as oadj
from tests.test_gpu_vjp import _oracle_maps

pytestmark = pytest.mark.gpu


def test_distribution_steeper_than_the_width():
    """f falls by e^-700 over the grid, the Gaussian's width is 27 times f's
    temperature: at the high points the gain is carried by samples more than 20
    widths off the shell, whose kinematic part is below 2^-300 of the largest.
    (dL/df itself reaches 1 / f there; C~ of both calls is what a dropped sample
    would show in.)"""
    import torch
    from paper_2603_28848_gb300 import Collision
    prob, _ = W.c1_maxwell_2to2(608, 600, 1)
    prob = replace(prob, grid=W.Grid(608, 0.01, 14.0, False),
                   processes=tuple(replace(p, sigma_E=0.5) for p in prob.processes))
    q = W.grid_points(prob.grid)
    f0 = np.exp(-(np.sqrt(q * q + 1.0) - 1.0) / 0.0186)[None, :]
    col = Collision(prob, W.PREC_FP64)
    f = torch.tensor(f0, device="cuda")
    C, _, _, _ = col.vjp(f, torch.ones_like(f), 0.0)
    Cj, _ = col.jvp(f, f, 0.0)
    Co, _, _, _ = oadj.vjp(prob, f0, 0.0, np.ones_like(f0), _oracle_maps(col, prob), col.call_counter, "f64")
    col.close()
    for got in (C, Cj):
        assert np.all(np.abs(got.cpu().numpy() - Co) <= 1e-11 * np.abs(Co))
