"""The FP32 2 -> 2 default: one sample per lane below a size, packed pairs over
the same partition above it.  Which of the two runs must not show: the library
is linked again with the line at either end (only that translation unit is
compiled for it), and results and maps are compared bit for bit."""
import ctypes
import os
import subprocess
from concurrent.futures import ThreadPoolExecutor
from dataclasses import replace

import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def libs(tmp_path_factory):
    """Paths of the library with one sample per lane at every size, and packed pairs."""
    from paper_2603_28848_gb300 import buildlib
    others = [os.path.join(buildlib.HERE, "_build", s.replace(".cu", ".o")) for s in buildlib.SOURCES if s != "api.cu"]
    buildlib.build(force=not all(os.path.exists(o) for o in others))
    d = tmp_path_factory.mktemp("default_loop")
    src = os.path.join(buildlib.CSRC, "api.cu")

    def make(name, chunks):
        obj, lib = os.fspath(d / (name + ".o")), os.fspath(d / (name + ".so"))
        subprocess.run([buildlib.nvcc(), *buildlib.ARCH, *buildlib.FLAGS, "-DBEST_PACKED_CHUNKS=%d" % chunks, "-c", src,
                        "-o", obj], check=True)
        subprocess.run([buildlib.nvcc(), *buildlib.ARCH, "-shared", "-o", lib, obj, *others, "-Xcompiler", "-fPIC"],
                       check=True)
        return lib

    with ThreadPoolExecutor(2) as ex:
        return list(ex.map(make, ("one", "pairs"), (1 << 40, 0)))


def _sweep(monkeypatch, path, prob, f0):
    import torch
    from paper_2603_28848_gb300 import Collision, _lib
    if path is not None:
        monkeypatch.setattr(_lib, "_lib", None)
        _lib.load(path)
    try:
        col = Collision(prob, W.PREC_FP32)
        C, err = col.eval(torch.tensor(np.ascontiguousarray(f0), device="cuda"), 0.0)
        col.check()
        out = (col.launch_shape()[2], C.cpu().numpy(), err.cpu().numpy(), *col.task_results(), col.maps())
        col.close()
    finally:
        monkeypatch.undo()
    return out


def _case(kind, n, neval, nbins):
    prob, f0 = {"mb": W.c1_maxwell_2to2, "bose": W.c2_bose_2to2}[kind](n, neval, 2)
    return replace(prob, processes=tuple(replace(p, nbins=nbins) for p in prob.processes)), f0


@pytest.mark.parametrize("kind,n,neval,nbins", [("mb", 5, 7, 2), ("mb", 9, 3001, 17), ("bose", 7, 9999, 33),
                                                ("mb", 33, 50_001, 50), ("bose", 20, 100_003, 64),
                                                ("bose", 64, 100_001, 50), ("mb", 32, 1_000_001, 256)])
def test_both_loops_give_the_same_bits(libs, monkeypatch, kind, n, neval, nbins):
    prob, f0 = _case(kind, n, neval, nbins)
    one, pairs, default = [_sweep(monkeypatch, p, prob, f0) for p in (*libs, None)]
    assert one[0] == 1 and pairs[0] == 2 and default[0] in (1, 2)
    for a, b, c in zip(one[1:], pairs[1:], default[1:]):
        assert np.array_equal(a, b) and np.array_equal(a, c)


def test_default_above_the_line_matches_the_oracle():
    """Just above it (256 tasks of 1e5 samples), as made, one iteration: twelve
    tasks recomputed by the oracle with the bounds of the full-size test."""
    import torch
    from oracle import collision as ocol
    from oracle import vegas
    from oracle.tasks import side_integrals
    from paper_2603_28848_gb300 import Collision
    prob, f0 = W.c2_bose_2to2(64, 100_000, 1)
    col = Collision(prob, W.PREC_FP32)
    assert col.launch_shape()[2] == 2
    col.eval(torch.tensor(np.ascontiguousarray(f0), device="cuda"), 0.0)
    col.check()
    mean, _ = col.task_results()
    col.close()
    dists = ocol.distributions(prob, f0, 0.0)
    rel = []
    for k, i in enumerate((3, 14, 25, 36, 47, 60)):
        for s, si in enumerate(side_integrals(prob)):
            term = (k + s) % 2
            om = ocol.evaluate_task(prob, s, si, i, term, f0, 0.0, vegas.uniform_edges(si.dim, 50), 0, "f32", dists)[0]
            rel.append(abs(mean[(s * 64 + i) * 2 + term] - om) / abs(om))
    assert max(rel) < 2e-3 and np.median(rel) < 2e-4, rel
