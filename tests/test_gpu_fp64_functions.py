"""Device functions of the FP64 sample loop, one by one, against what they
stand for.  A small kernel around each is compiled for the run (the library
exports calls, not functions)."""
import ctypes
import os

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "eval_impl.cuh"
using namespace best;

__global__ void map_kernel(int n, const uint32_t* x0, const uint32_t* x1, int nb, double* fr, uint32_t* bin) {
    __shared__ Real2<double> table[256];
    for (int k = threadIdx.x; k < nb; k += blockDim.x) table[k] = Real2<double>{0.0, 1.0};
    __syncthreads();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) map_point64(x0[i], x1[i], nb, table, &fr[i], &bin[i]);
}
extern "C" int test_map(int n, const void* x0, const void* x1, int nb, void* fr, void* bin) {
    map_kernel<<<(n + 255) / 256, 256>>>(n, (const uint32_t*)x0, (const uint32_t*)x1, nb, (double*)fr, (uint32_t*)bin);
    return cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    import subprocess
    from paper_2603_28848_gb300 import buildlib
    d = tmp_path_factory.mktemp("fp64_functions")
    src, out = d / "f.cu", d / "f.so"
    src.write_text(SOURCE)
    subprocess.run([buildlib.nvcc(), *buildlib.ARCH, *buildlib.FLAGS, "-I" + buildlib.CSRC, "-shared", "-o", str(out),
                    str(src)], check=True, cwd=os.fspath(d))
    return ctypes.CDLL(os.fspath(out))


def _dev(x):
    import torch
    return torch.from_numpy(np.ascontiguousarray(x)).cuda()


def _ptr(t):
    return ctypes.c_void_p(t.data_ptr())


@pytest.mark.parametrize("nb", [2, 3, 17, 50, 64, 255, 256])
def test_map_point(lib, nb):
    """Increment and fraction of u nb in FP64, bit for bit (the published
    definition of the stream), at the increments' edges and both ends too."""
    import torch
    rng = np.random.RandomState(nb)
    edge = (np.arange(nb, dtype=np.uint64) << np.uint64(52)) // np.uint64(nb)
    k = np.concatenate([rng.randint(0, 2 ** 52, 20_000).astype(np.uint64), edge, edge + np.uint64(1),
                        edge[1:] - np.uint64(1), np.array([0, 2 ** 52 - 1, 2 ** 51], dtype=np.uint64)])
    x0 = (k >> np.uint64(26) << np.uint64(6)).astype(np.uint32) | rng.randint(0, 64, k.size).astype(np.uint32)
    x1 = ((k & np.uint64(2 ** 26 - 1)) << np.uint64(6)).astype(np.uint32) | rng.randint(0, 64, k.size).astype(np.uint32)
    fr = torch.zeros(k.size, dtype=torch.float64, device="cuda")
    bins = torch.zeros(k.size, dtype=torch.int32, device="cuda")
    a, b = _dev(x0.view(np.int32)), _dev(x1.view(np.int32))
    assert lib.test_map(k.size, _ptr(a), _ptr(b), nb, _ptr(fr), _ptr(bins)) == 0
    t = (k.astype(np.float64) + 0.5) * 2.0 ** -52 * nb
    want = np.minimum(t.astype(np.int64), nb - 1)
    assert np.array_equal(bins.cpu().numpy(), want)
    assert np.array_equal(fr.cpu().numpy(), t - want)
