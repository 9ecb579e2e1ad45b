"""Sums over tasks of the derivative calls at grid sizes around their block
boundaries: C~ and the tangent per grid point, the coupling and mass gradients
over all tasks, and the spline's transpose, checked by identities that hold
for any samples (FP64 path).

Tolerances: sums of at most a few thousand FP64 terms, each rounded to 1.1e-16
relative, differ in order only: 1e-11 of the sum of magnitudes.
"""
from dataclasses import replace

import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def _setup(n, problem):
    import torch
    from paper_2603_28848_gb300 import Collision
    if problem == "frw":
        prob, f0 = W.c4_multi_species(n, 64, 128, 1)
        prob = replace(prob, processes=tuple(replace(p, coupling=0.5 + k) for k, p in enumerate(prob.processes)))
    else:
        prob, f0 = W.c2_bose_2to2(n, 64, 1)
    f = torch.tensor(f0, device="cuda")
    return prob, Collision(prob, W.PREC_FP64), f


@pytest.mark.parametrize("problem,n", [("bose", 8), ("bose", 31), ("bose", 128), ("bose", 129), ("frw", 65),
                                       ("frw", 257)])
def test_task_sums(problem, n):
    import torch
    t = 2.0 if problem == "frw" else 0.0
    prob, col, f = _setup(n, problem)
    rng = np.random.RandomState(n)
    v = torch.tensor(rng.uniform(-1, 1, f.shape), device="cuda")
    u = torch.tensor(rng.uniform(-1, 1, f.shape), device="cuda") * f
    C, gf, gm, gl = col.vjp(f, v, t)
    _, JU = col.jvp(f, u, t)
    assert bool((C != 0).any())
    # <v, J u> = <J^T v, u>
    a, b = v * JU, gf * u
    assert abs(float(a.sum() - b.sum())) <= 1e-11 * float(a.abs().sum() + b.abs().sum())
    # |M|^2 = lambda^2: sum_p lambda_p dL/dlambda_p = 2 L
    lam = torch.tensor([p.coupling for p in prob.processes], dtype=torch.float64, device="cuda")
    assert abs(float((lam * gl).sum() - 2 * (v * C).sum())) <= 1e-11 * float((v * C).abs().sum())
    # linear in v, task by task: the gradients of the two halves add up
    lo = torch.zeros_like(v)
    lo[:, : n // 2] = v[:, : n // 2]
    parts = [col.vjp(f, x, t) for x in (lo, v - lo)]
    for k, whole in ((1, gf), (2, gm), (3, gl)):
        scale = parts[0][k].abs() + parts[1][k].abs() + whole.abs().max() * 1e-3
        assert bool(((parts[0][k] + parts[1][k] - whole).abs() <= 1e-11 * scale).all()), k
    col.close()
