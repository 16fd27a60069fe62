"""The kernels' float-to-double conversion by integer operations, compiled
from the library's header: bit for bit (any NaN for a NaN), and the FP32 forms' node export, which rests on it, for cells whose
values are subnormal, infinite or negative as floats."""
import ctypes as C
import subprocess

import numpy as np
import pytest

from test_gpu_parity import B, gpu_tree, small_turbulent  # noqa: F401

pytestmark = pytest.mark.gpu

SRC = r"""
#include "tr_internal.cuh"
__global__ void k(const float* x, double* y, int n) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n / 8; i += gridDim.x * blockDim.x) {
        float f[8];
        double d[8];
        for (int k = 0; k < 8; ++k) f[k] = x[8 * i + k];
        tr::widen_all(f, d);
        for (int k = 0; k < 8; ++k) y[8 * i + k] = d[k];
    }
}
extern "C" int widen_all(const float* x, double* y, int n) {
    k<<<1024, 256>>>(x, y, n);
    return (int)cudaGetLastError();
}
"""


@pytest.fixture(scope="module")
def widen(tmp_path_factory):
    from paper_2105_09644_gb300 import buildlib
    d = tmp_path_factory.mktemp("widen")
    (d / "w.cu").write_text(SRC)
    lib = d / "w.so"
    subprocess.run([buildlib.nvcc(), *buildlib.ARCH, *buildlib.FLAGS, "-I", buildlib.CSRC, "-shared", "-o", str(lib),
                    str(d / "w.cu"), "-lcudart"], check=True)
    fn = C.CDLL(str(lib)).widen_all
    fn.argtypes = [C.c_void_p, C.c_void_p, C.c_int]
    return fn


@pytest.mark.parametrize("mixed", [False, True])
def test_every_exponent(widen, mixed):
    """All signs and exponents with 2^12 significands each (the ends among them),
    eight of a kind at a time or shuffled."""
    import torch
    low = torch.cat([torch.arange(0, 1 << 11), torch.arange((1 << 23) - (1 << 11), 1 << 23)])
    bits = (torch.arange(512)[:, None] << 23 | low[None, :]).reshape(-1)
    if mixed:
        bits = bits[torch.randperm(bits.numel(), generator=torch.Generator().manual_seed(1))]
    x = bits.cuda().to(torch.int32).view(torch.float32)
    y = torch.empty(x.numel(), dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    assert widen(x.data_ptr(), y.data_ptr(), x.numel()) == 0
    torch.cuda.synchronize()
    want, nan = x.double(), torch.isnan(x)
    assert torch.equal(torch.isnan(y), nan)
    assert bool(((y.view(torch.int64) == want.view(torch.int64)) | nan).all())


@pytest.mark.parametrize("precision", [1, 2])
def test_node_export(B, precision):
    import torch
    N = 8
    w = small_turbulent(N=N, n_src=0, seed=4)
    n = w.n_H.reshape(-1)
    n[3], n[77], n[100], n[200] = 1e-41, 3e39, 1e-22, 1e21         # subnormal and infinite as floats, and so are squares
    e = np.zeros(N ** 3)
    e[5], e[6] = -1e-12, -0.0
    t = gpu_tree(B, w, precision, e_prev=e)
    out = torch.empty((t.info()["n_nodes"], 8), dtype=torch.float64, device="cuda")
    B.tr_tree_nodes(t, out)
    got = out.cpu().numpy()[-N ** 3:]                              # the cells, in Morton order
    m = np.arange(N ** 3)
    x, y, z = (sum(((m >> (3 * b + s)) & 1) << b for b in range(3)) for s in range(3))
    order = (z * N + y) * N + x
    with np.errstate(over="ignore"):
        assert np.array_equal(got[:, 0], n[order].astype(np.float32).astype(np.float64))
        sq = (n[order] ** 2).astype(np.float32).astype(np.float64)
    U = w.alpha_B * w.dx ** 3
    np.testing.assert_allclose(got[:, 4], sq * U, rtol=1e-13)      # two roundings of U
    assert 0.0 < got[order == 100, 4] and np.isinf(got[order == 200, 4])
    np.testing.assert_allclose(got[:, 6], e[order], rtol=1e-6)
