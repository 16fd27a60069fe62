"""Cells whose density, emission or energy density is not a number, infinite,
zero, negative or tiny: the uniform build gives the nodes of the AMR build of
the same cells on one level, which takes the definition's maxima and
quotients.  Masses and centres bit for bit (NaN for NaN), rates within 1e-13
and the FP32 forms within 1e-6 and 1e-5 of an edge, as in
test_gpu_build_levels."""
import numpy as np
import pytest

from test_gpu_parity import B, dev, gpu_params, small_turbulent  # noqa: F401

pytestmark = pytest.mark.gpu

NAN, INF = float("nan"), float("inf")


@pytest.mark.parametrize("precision", [0, 1, 2])
@pytest.mark.parametrize("what,value", [("n_H", NAN), ("n_H", -NAN), ("n_H", 0.0), ("n_H", -2.0), ("n_H", 1e-300),
                                        ("n_H", 5e-324), ("n_H", 1e-160), ("ndot", NAN), ("ndot", INF), ("ndot", -1e49),
                                        ("ndot", 1e49), ("e_prev", NAN), ("e_prev", -1e-12), ("e_prev", -0.0),
                                        ("e_prev", 1e-300), ("n_H", 1e200), ("n_H", INF)])
def test_odd_cells(B, what, value, precision):
    import torch
    N = 16
    w = small_turbulent(N=N, n_src=0, seed=6)
    rng = np.random.default_rng(2)
    cell = dict(n_H=w.n_H.copy(), ndot=np.zeros((N, N, N)), e_prev=1e-12 * rng.uniform(size=(N, N, N)))
    cell[what].reshape(-1)[[0, 777, 2048]] = value
    p = gpu_params(B, w, precision)
    keep = {k: dev(v) for k, v in cell.items()}
    uni = B.tr_build_tree(B.make_grid(keep["n_H"], w.dx, ndot=keep["ndot"], e_prev=keep["e_prev"]), B.make_sources(), p)
    pos = np.array([[x, y, z] for z in range(2) for y in range(2) for x in range(2)], dtype=np.int32)
    blocks = {k: dev(np.stack([v[8 * z:8 * z + 8, 8 * y:8 * y + 8, 8 * x:8 * x + 8] for x, y, z in pos]).reshape(-1))
              for k, v in cell.items()}
    amr = B.tr_build_tree_amr(B.make_amr_grid(N, 0, np.zeros(8, dtype=np.int32), pos, blocks["n_H"], w.dx,
                                              ndot=blocks["ndot"], e_prev=blocks["e_prev"]), B.make_sources(), p)
    out = [torch.empty((t.info()["n_nodes"], 8), dtype=torch.float64, device="cuda") for t in (uni, amr)]
    for t, o in zip((uni, amr), out):
        B.tr_tree_nodes(t, o)
    got, want = (o.cpu().numpy() for o in out)
    if precision == 0:
        assert np.array_equal(got[:, :4], want[:, :4], equal_nan=True)
        np.testing.assert_allclose(got[:, 4:], want[:, 4:], rtol=1e-13)
    else:
        edge = np.concatenate([np.full(8 ** l, float(N >> l)) for l in range(5)])[:, None]
        np.testing.assert_allclose(got[:, [0, 4, 5, 6, 7]], want[:, [0, 4, 5, 6, 7]], rtol=1e-6)
        np.testing.assert_allclose(got[:, 1:4] / edge, want[:, 1:4] / edge, rtol=0.0, atol=1e-5)
