"""Allocations at their limits.  A loaded state's may not add up to the task's
items: the sweep stays within them, as if the allocation ended where the items
do.  And FP32 squares that overflow leave no shares to allocate by."""
import numpy as np
import pytest

import workloads as W
from tests.test_gpu_strat import _f, _strat

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [W.PREC_FP64, W.PREC_FP32])
@pytest.mark.parametrize("h,add", [(0, 5000), (10, 40), (63, 2), (20, -3)])
def test_allocation_that_does_not_add_up(precision, h, add):
    from paper_2603_28848_gb300 import Collision
    prob, f0 = W.c1_maxwell_2to2(n=4, neval=64 * 8 * 40, nitn=2)
    prob = _strat(prob)
    col = Collision(prob, precision)
    f = _f(f0)
    col.eval(f, 0.0)
    C0, e0 = col.eval(f, 0.0)
    H = [col.strata(t)[1] for t in range(col.n_tasks)]
    total, J = sum(H), 64 * 40
    assert H == [64] * col.n_tasks
    blob = bytearray(col.save_state())
    m = np.frombuffer(bytes(blob[-4 * total:]), dtype=np.int32).reshape(-1, 64).copy()
    assert np.array_equal(m[1], col.strata(1)[2]) and np.all(m.sum(1) == J)
    m[:, h] = np.maximum(m[:, h] + add, 1)
    blob[-4 * total:] = m.tobytes()
    col.load_state(bytes(blob))
    C, err = col.eval(f, 0.0)
    col.check()
    for t in range(col.n_tasks):
        assert col.strata(t)[2].sum() == J and np.all(col.strata(t)[2] >= 1)
    # and so is the next sweep an ordinary one: both estimates' errors apart
    for _ in range(2):
        C, err = col.eval(f, 0.0)
    col.check()
    col.close()
    C, err, C0, e0 = (x.cpu().numpy() for x in (C, err, C0, e0))
    assert np.all(np.isfinite(C)) and np.all(np.abs(C - C0) < 8 * np.hypot(err, e0) + 1e-300)


def test_squares_beyond_fp32():
    """First iterations scale the weights by 1 / f_obs (at most 2^100): where f_obs is
    1e-36 and a wide Gaussian lets in samples with f of order one, weights reach
    1e22, w^2 is infinite in FP32 and so is a hypercube's variance.  The allocation starts afresh and the
    next iterations are ordinary ones (FP64 is the reference, 8 standard errors)."""
    from dataclasses import replace
    from paper_2603_28848_gb300 import Collision
    prob, _ = W.c1_maxwell_2to2(n=8, neval=64 * 8 * 40, nitn=4)
    prob = replace(prob, grid=replace(prob.grid, log_spaced=False))
    prob = _strat(replace(prob, processes=tuple(replace(p, sigma_E=20.0) for p in prob.processes)))
    q = W.grid_points(prob.grid)
    f0 = 0.5 * np.exp(-82.0 * (q / 20.0) ** 2)[None, :]
    f = _f(f0)
    out = []
    for precision in (W.PREC_FP32, W.PREC_FP64):
        col = Collision(prob, precision)
        col.eval(f, 0.0)
        for t in range(col.n_tasks):
            _, H, m = col.strata(t)
            assert H == 64 and m.sum() == 64 * 40 and np.all(m >= 1)
        col.eval(f, 0.0)
        col.check()
        out.append(col.task_results())
        col.close()
    (a, ea), (b, eb) = out
    assert np.all(np.isfinite(a)) and np.all(np.abs(a - b) <= 8 * np.hypot(ea, eb) + 1e-5 * np.abs(b))
