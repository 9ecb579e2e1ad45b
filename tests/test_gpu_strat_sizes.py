"""Per-hypercube sums and item tables of the stratified refinement at the
sizes where their split changes: hypercubes below 32, below and above 1024 items,
more hypercubes than a CTA has threads.  FP64 against the oracle
with the bounds of the stratification tests (estimates 1e-5, errors 1e-4, maps
1e-4, integer allocations exact)."""
import pytest

import workloads as W
from tests.test_gpu_strat import _parity, _strat

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hcubes,neval", [(64, 64 * 8 * 5), (64, 64 * 8 * 40 + 3), (729, 729 * 8 * 4), (729, 729 * 8 * 9 + 5),
                                           (64, 64 * 8 * 1100)])
def test_hypercube_sizes(hcubes, neval):
    prob, f0 = W.c1_maxwell_2to2(n=5, neval=neval, nitn=2)
    _parity(_strat(prob, strat_max_hcubes=hcubes), f0, sweeps=1)
