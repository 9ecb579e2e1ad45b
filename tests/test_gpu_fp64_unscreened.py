"""FP64 where the tables leave no room for the screen's queues: the plain sample
loop, and the derivative kernels evaluating every sample where it is drawn.

Tolerances: those of the FP64 screen and derivative tests (1e-7 of a task's
mean, 1e-8 of the largest entry of a gradient).
"""
from dataclasses import replace

import numpy as np
import pytest

import workloads as W
from oracle import adjoint as oadj
from oracle import collision as ocol
from oracle import vegas
from oracle.tasks import side_integrals
from tests.test_gpu_vjp import _close, _oracle_maps

pytestmark = pytest.mark.gpu


def test_plain_loop():
    """2500 points, two species: 180 KB of spline tables.  Sixteen tasks by the oracle."""
    import torch
    from paper_2603_28848_gb300 import Collision
    n = 2500
    prob, f0 = W.c2_bose_2to2(n, 801, 1)
    prob = replace(prob, processes=tuple(replace(p, sigma_E=0.05) for p in prob.processes))
    col = Collision(prob, W.PREC_FP64)
    assert col.launch_shape()[2] == 1
    col.eval(torch.tensor(f0, device="cuda"), 0.0)
    col.check()
    mean, _ = col.task_results()
    col.close()
    dists = ocol.distributions(prob, f0, 0.0)
    for k, i in enumerate((0, 100, 777, 1250, 1800, 2100, 2300, 2499)):
        for s, si in enumerate(side_integrals(prob)):
            term = (k + s) % 2
            om = ocol.evaluate_task(prob, s, si, i, term, f0, 0.0, vegas.uniform_edges(si.dim, 50), 0, "f64", dists)[0]
            assert abs(mean[(s * n + i) * 2 + term] - om) <= 1e-7 * abs(om) + 1e-300


@pytest.mark.parametrize("kind,n", [("2 to 2", 400), ("2 to 3", 400), ("2 to 2", 340)])
def test_derivatives(kind, n):
    """Eight species (all but one only tabulated): 520 n + 9.9 KB of tables, the
    screen adds 35 (2 -> 2) and 47 KB (2 -> 3) and a CTA has 227, so that it fits up
    to 360 and 336 points; the last case has it.  Odd budgets: 2 -> 3 draws two
    samples per group."""
    import torch
    from paper_2603_28848_gb300 import Collision
    prob, f0 = W.c1_maxwell_2to2(n, 41, 1) if kind == "2 to 2" else W.c3_cannibal_2to3(n, 23, 1)
    prob = replace(prob, species=prob.species * 8, processes=tuple(replace(p, sigma_E=0.3) for p in prob.processes))
    f0 = np.concatenate([f0] + [np.full((1, n), 0.1)] * 7)
    col = Collision(prob, W.PREC_FP64)
    rng = np.random.RandomState(1)
    v = rng.uniform(-1, 1, f0.shape)
    f = torch.tensor(f0, device="cuda")
    got = col.vjp(f, torch.tensor(v, device="cuda"), 0.0)
    Cj, JU = col.jvp(f, torch.tensor(v * f0, device="cuda"), 0.0)
    maps = _oracle_maps(col, prob)
    want = oadj.vjp(prob, f0, 0.0, v, maps, col.call_counter, "f64")
    col.close()
    for g, o in zip(got, want):
        assert np.any(o != 0) and _close(g.cpu().numpy(), o, 1e-8)
    assert _close(Cj.cpu().numpy(), want[0], 1e-8)
    # <v, J (v f)> = <J^T v, v f>
    a, b = (v * JU.cpu().numpy()).sum(), (want[1] * v * f0).sum()
    assert abs(a - b) <= 1e-8 * np.abs(want[1] * v * f0).sum()


@pytest.mark.parametrize("problem", ["bose", "three"])
def test_forward_and_reverse_return_the_same_integral(problem):
    """C~ of both calls: the same samples, summed in another order (1e-12)."""
    import torch
    from paper_2603_28848_gb300 import Collision
    prob, f0 = W.c2_bose_2to2(33, 1000, 1) if problem == "bose" else W.c3_cannibal_2to3(20, 501, 1)
    col = Collision(prob, W.PREC_FP64)
    f = torch.tensor(f0, device="cuda")
    C = col.vjp(f, torch.ones_like(f), 0.0)[0]
    Cj, _ = col.jvp(f, f, 0.0)
    col.close()
    assert bool((C != 0).any()) and torch.allclose(C, Cj, rtol=1e-12, atol=1e-12 * float(C.abs().max()))
