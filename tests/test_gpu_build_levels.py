"""The tree build, three levels a launch, at every number of levels left over
at the root, in every form: all nodes against the oracle.  Cells without mass,
with emission above and below their recombinations, and a partly ionised grid.
FP64: masses and centres bit for bit, rates within 1e-13 (two roundings per
sum of eight, ten levels).  FP32 forms: 1e-6 of the node's value (compensated
sums round twice per level) and, for the centres, 1e-5 of the node's edge."""
import numpy as np
import pytest

from helpers import decode_id
from test_gpu_parity import B, gpu_tree, small_turbulent  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1, 2])
@pytest.mark.parametrize("N", [8, 16, 32, 64])
def test_every_node(B, orc, N, precision):
    import torch
    w = small_turbulent(N=N, n_src=5, seed=17 + N)
    rng = np.random.default_rng(N)
    w.n_H[rng.uniform(size=w.n_H.shape) < 0.05] = 0.0
    w.n_H[: N // 4] = 0.0                                    # whole subtrees without mass
    e = np.where(rng.uniform(size=N ** 3) < 0.5, 0.0, 1e-12)
    t = gpu_tree(B, w, precision, e_prev=e)
    out = torch.empty((t.info()["n_nodes"], 8), dtype=torch.float64, device="cuda")
    B.tr_tree_nodes(t, out)
    got = out.cpu().numpy()
    ot = orc.Tree(w, e_prev=e)
    ids = np.unique(np.concatenate([np.arange(min(len(got), 600)), rng.integers(0, len(got), 3000)]))
    for i in ids:
        lev, ix, iy, iz = decode_id(int(i))
        want = ot.node(lev, ix, iy, iz)
        s = N >> lev
        if precision == 0:
            assert np.array_equal(got[i, :4], want[:4]), (i, got[i], want)
            np.testing.assert_allclose(got[i, 4:], want[4:], rtol=1e-13)
        else:
            np.testing.assert_allclose(got[i, [0, 4, 5, 6, 7]], want[[0, 4, 5, 6, 7]], rtol=1e-6)
            assert np.all(np.abs(got[i, 1:4] - want[1:4]) <= 1e-5 * s), (i, got[i], want)
