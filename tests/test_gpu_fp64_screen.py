"""The FP64 sample loop screens samples in FP32 and evaluates in FP64 only those
that can matter.  Against the oracle (which evaluates every sample in FP64) at
the sizes and widths where a screen can go wrong: fewer samples than a queue
of a warp, odd budgets, few and many increments, a Gaussian so wide that every
sample is kept, so narrow that hardly any is, a fractional width, massless and
heavy legs, both sides of 2 -> 3, 2 -> 4, an expansion; and a grid whose tables
leave no room for the queues (the plain loop runs).

Tolerances: both sides evaluate the same samples in FP64; FP64 rounding of the
energy balance (1e-15 of 50) over the narrowest width (1e-3) is 5e-11 of an
exponent of at most 750, so 1e-7 of a task's mean, 1e-6 of its error.
"""
from dataclasses import replace

import numpy as np
import pytest

import workloads as W
from tests._helpers import oracle_sweep, task_arrays

pytestmark = pytest.mark.gpu


def _mb(n, neval, nbins=50, **kw):
    prob, f0 = W.c1_maxwell_2to2(n, neval, 1)
    return replace(prob, processes=tuple(replace(p, nbins=nbins, **kw) for p in prob.processes)), f0, 0.0


CASES = {
    "few samples": lambda: _mb(6, 7),
    "one warp": lambda: _mb(6, 33),
    "odd budget, 2 increments": lambda: _mb(8, 1023, nbins=2),
    "256 increments": lambda: _mb(6, 1500, nbins=256),
    "every sample kept": lambda: _mb(8, 1500, sigma_E=50.0),
    "hardly any kept": lambda: _mb(8, 20_000, sigma_E=1e-3),
    "fractional width": lambda: _mb(8, 3000, width_mode=1, width=0.02),
    "massless Bose": lambda: (*W.c2_bose_2to2(8, 2999, 1), 0.0),
    "2 to 3": lambda: (*W.c3_cannibal_2to3(6, 1501, 1, True), 0.0),
    "2 to 4": lambda: (*W.c5_2to4(5, 700, 1), 0.0),
    "expansion": lambda: (*W.c4_multi_species(6, 500, 900, 1), 2.0),
}


@pytest.mark.parametrize("name", list(CASES))
def test_matches_oracle(name):
    import torch
    from paper_2603_28848_gb300 import Collision
    prob, f0, t = CASES[name]()
    col = Collision(prob, W.PREC_FP64)
    assert col.launch_shape()[2] == 2          # the screened loop
    col.eval(torch.tensor(f0, device="cuda"), t)
    mean, err = col.task_results()
    col.close()
    _, _, detail, _ = oracle_sweep(prob, f0, t, "f64")
    om, oe = task_arrays(detail, len(mean))
    ok = np.isfinite(om)                       # (the oracle's 1 / variance overflows for an estimate of 1e-159)
    assert ok.mean() > 0.8
    assert np.all(np.abs(mean - om)[ok] <= (1e-7 * np.abs(om) + 1e-300)[ok])
    assert np.all(np.abs(err - oe)[ok] <= (1e-6 * np.abs(oe) + 1e-300)[ok])


def test_large_grid_takes_the_plain_loop():
    import torch
    from paper_2603_28848_gb300 import Collision
    prob, f0 = W.c2_bose_2to2(2500, 16, 1)     # 180 KB of spline tables
    col = Collision(prob, W.PREC_FP64)
    assert col.launch_shape()[2] == 1
    f = torch.tensor(f0, device="cuda")
    C, err = col.eval(f, 0.0)
    col.check()
    assert bool(torch.isfinite(C).all()) and bool((C != 0).any())
    col.close()


def test_narrow_width_on_a_wide_grid():
    """Radii of a wide map carry more FP32 rounding than a soft leg's energy: the
    screen's bound has to hold there too (energies up to 3e3, width 1e-3: FP64
    rounding 1e-12 over it times 39 is 4e-8 of a weight)."""
    import torch
    from paper_2603_28848_gb300 import Collision
    prob, f0, t = _mb(6, 20_000, sigma_E=1e-3)
    prob = replace(prob, grid=replace(prob.grid, q_min=1e-3, q_max=300.0))
    q = W.grid_points(prob.grid)
    f0 = (0.5 * np.exp(-np.sqrt(q * q + 1.0) / 20.0))[None, :]
    col = Collision(prob, W.PREC_FP64)
    col.eval(torch.tensor(f0, device="cuda"), t)
    mean, _ = col.task_results()
    col.close()
    _, _, detail, _ = oracle_sweep(prob, f0, t, "f64")
    om, _ = task_arrays(detail, len(mean))
    ok = np.isfinite(om)
    assert ok.mean() > 0.8 and np.any(om != 0)
    assert np.all(np.abs(mean - om)[ok] <= (1e-6 * np.abs(om) + 1e-300)[ok])


def test_factors_that_are_not_normal_numbers():
    """A species whose values are partly subnormal (below 2.2e-308) next to one of
    order one: in a gain task that observes it, c0 is up to 2^100 and the weights
    are normal numbers.  The spline's cubic coefficient is a multiple of 5e-324 and
    enters with the interval's length cubed, 13^3: 2e-12 of the smallest value,
    1e-10 of a task's mean with room for a handful of such roundings.  (In the
    other tasks the weights themselves are subnormal.)"""
    import torch
    from paper_2603_28848_gb300 import Collision
    prob, f0, t = _mb(8, 2000, sigma_E=0.5)
    q = W.grid_points(prob.grid)
    E = np.sqrt(q * q + 1.0)
    proc = replace(prob.processes[0], species_in=(0, 1), species_out=(0, 1), coupling=1e10)
    prob = replace(prob, species=(prob.species[0], prob.species[0]), processes=(proc,))
    f0 = np.stack([f0[0], 4e-308 * np.exp(-(E - 1.0) / 10.5)])
    assert f0[1].min() > 5.7e-309
    col = Collision(prob, W.PREC_FP64)
    assert col.launch_shape()[2] == 2
    col.eval(torch.tensor(f0, device="cuda"), t)
    mean, _ = col.task_results()
    col.close()
    _, _, detail, _ = oracle_sweep(prob, f0, t, "f64")
    om, _ = task_arrays(detail, len(mean))
    gain = slice(16, 32, 2)                    # the second side integral's, which observes that species
    assert np.all(om[gain] > 0)
    assert np.all(np.abs(mean - om)[gain] <= 1e-10 * om[gain])


def _against_oracle(prob, f0, t):
    import torch
    from paper_2603_28848_gb300 import Collision
    col = Collision(prob, W.PREC_FP64)
    assert col.launch_shape()[2] == 2
    col.eval(torch.tensor(f0, device="cuda"), t)
    mean, err = col.task_results()
    col.close()
    _, _, detail, _ = oracle_sweep(prob, f0, t, "f64")
    om, oe = task_arrays(detail, len(mean))
    assert np.all(np.isfinite(om)) and np.any(om != 0)
    assert np.all(np.abs(mean - om) <= 1e-7 * np.abs(om) + 1e-300)
    assert np.all(np.abs(err - oe) <= 1e-6 * np.abs(oe) + 1e-300)
    return om


def test_negative_observed_factor():
    """Fermi-Dirac values above 1 inside the grid: the observed leg's 1 - f, and
    every weight of that gain task, is negative."""
    prob, f0, t = _mb(12, 20_000, sigma_E=0.1)
    prob = replace(prob, species=(replace(prob.species[0], stat=W.STAT_FD),))
    f0 = np.where((np.arange(12) >= 4) & (np.arange(12) < 8), 1.2, 1.6 * f0)
    assert f0[:, :4].max() < 1 and f0[:, 8:].max() < 1
    om = _against_oracle(prob, f0, t)
    assert np.all(om[8:16:2] < 0)


def test_narrow_linear_grid():
    """An evenly spaced grid of 11 FP32 numbers per interval, values alternating
    from knot to knot: a lookup that takes a neighbouring interval's cubic a tenth
    of an interval outside is 1e-3 off.  FP64 resolves 1e-10 of an interval.  (Two
    equal values at each end: flat tails.)"""
    prob, f0, t = _mb(16, 5000, sigma_E=0.5)
    prob = replace(prob, grid=W.Grid(16, 1.0, 1.0 + 2e-5, False), tail_points=2)
    f0 = (1.0 + 0.5 * (-1.0) ** np.arange(16))[None, :]
    f0[:, [0, -1]] = f0[:, [1, -2]]
    _against_oracle(prob, f0, t)


def test_spline_coefficients_beyond_fp32():
    """A species whose values alternate by 1e25 on a grid of 56 FP32 numbers per
    interval: its cubic coefficients (f over the interval cubed, 1e40) are infinite
    in FP32, and the screen's spline value is a NaN where the lookup falls on a
    knot, in about 1% of the samples.  Small equal values at the ends, so that the
    conserved leg's tail is no reason to keep them."""
    prob, f0, t = _mb(16, 20_000, sigma_E=0.5)
    proc = replace(prob.processes[0], species_in=(0, 1), species_out=(0, 1))
    prob = replace(prob, grid=W.Grid(16, 1.0, 1.0 + 1e-4, False), tail_points=2,
                   species=(prob.species[0], prob.species[0]), processes=(proc,))
    f0 = np.stack([1e25 * (1.0 + 0.5 * (-1.0) ** np.arange(16)), np.full(16, 0.2)])
    f0[0, [0, 1, -2, -1]] = 0.1
    _against_oracle(prob, f0, t)


def test_small_units():
    """Energies of 1e-18 and a width of 1e-20, whose inverse square FP32 does not
    hold: the Gaussian is no reason to drop a sample then."""
    prob, f0, t = _mb(8, 5000, sigma_E=1e-20)
    prob = replace(prob, grid=replace(prob.grid, q_min=1e-20, q_max=2e-17), e_cut=1e-60,
                   species=(replace(prob.species[0], mass0=1e-18),))
    om = _against_oracle(prob, f0, t)
    assert np.all(om > 0)


@pytest.mark.parametrize("unit", [1e-45, 1e45])
def test_units_beyond_fp32(unit):
    """The same problem on an evenly spaced grid in units that FP32 does not hold at
    all: every sample is kept, and the lookups count in intervals."""
    prob, f0, t = _mb(8, 1500, sigma_E=0.5 * unit)
    prob = replace(prob, grid=W.Grid(8, 0.01 * unit, 20.0 * unit, False), e_cut=0.0,
                   species=(replace(prob.species[0], mass0=unit),))
    om = _against_oracle(prob, f0, t)
    assert np.all(om > 0)
