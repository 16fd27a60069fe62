"""The FP64 reciprocal of the walk and the sweeps, compiled from the library's
header, against 1.0 / a: 2^12 significands at every exponent from 2^-767 to
2^1021.  The step's error is 2^-59 and its last rounding 2^-53, the division's
2^-53: 2^-52 (1 + 2^-6) in all.  Smaller arguments, the subnormals too, give a
number of at least 2^766, larger ones and infinity one of at most 2^-1020."""
import ctypes as C
import subprocess

import pytest

from test_gpu_parity import B  # noqa: F401

pytestmark = pytest.mark.gpu

SRC = r"""
#include "tr_internal.cuh"
__global__ void k(const double* x, double* y, int n) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) y[i] = tr::recip(x[i]);
}
extern "C" int recip_all(const double* x, double* y, int n) {
    k<<<1024, 256>>>(x, y, n);
    return (int)cudaGetLastError();
}
"""


def test_every_exponent(B, tmp_path):
    import torch
    from paper_2105_09644_gb300 import buildlib
    (tmp_path / "r.cu").write_text(SRC)
    lib = tmp_path / "r.so"
    subprocess.run([buildlib.nvcc(), *buildlib.ARCH, *buildlib.FLAGS, "-I", buildlib.CSRC, "-shared", "-o", str(lib),
                    str(tmp_path / "r.cu"), "-lcudart"], check=True)
    fn = C.CDLL(str(lib)).recip_all
    fn.argtypes = [C.c_void_p, C.c_void_p, C.c_int]
    g = torch.Generator().manual_seed(3)
    low = torch.randint(0, 1 << 52, (1 << 12,), generator=g)
    low[:4] = torch.tensor([0, 1, (1 << 52) - 1, 1 << 51])
    bits = (torch.arange(2047)[:, None] << 52 | low[None, :]).reshape(-1)
    small = (torch.arange(1, 1 << 12) << torch.randint(0, 40, ((1 << 12) - 1,), generator=g))       # deep subnormals
    x = torch.cat([bits, small, torch.tensor([2047 << 52])]).cuda().view(torch.float64)
    x = x[x > 0.0].contiguous()
    y = torch.empty_like(x)
    torch.cuda.synchronize()
    assert fn(x.data_ptr(), y.data_ptr(), x.numel()) == 0
    torch.cuda.synchronize()
    want = 1.0 / x
    assert bool(torch.isfinite(y).all())
    ok = (x >= 2.0 ** -767) & (x < 2.0 ** 1021)
    err = ((y - want).abs() / want)[ok]
    assert bool((err <= 2.0 ** -52 * (1.0 + 2.0 ** -6)).all()), err.max()
    assert bool((y[x < 2.0 ** -767] >= 2.0 ** 766).all()) and bool((y[x >= 2.0 ** 1021] <= 2.0 ** -1020).all())
