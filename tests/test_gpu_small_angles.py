"""Walks at small opening angles, where most nodes are opened: the buffer of
opened nodes holds them in every CTA size that the launch picks (128 to 512
threads, by the ray bins), down to angles at which every cell is listed.  Cells
one by one through the fused walk; accepted nodes counted exactly, fluxes as
in test_gpu_parity."""
import numpy as np
import pytest

from helpers import KAPPA, flux_misses
from test_gpu_parity import B, RTOL, gpu_tree, small_turbulent  # noqa: F401

pytestmark = pytest.mark.gpu

#         N  nside theta  e
CASES = [(128, 2, 0.1, True), (64, 4, 0.1, True), (64, 4, 0.02, False), (32, 4, 1e-3, True), (64, 2, 1e-3, False)]


def morton(c, N):
    x, y, z = c % N, (c // N) % N, c // (N * N)
    return sum((((x >> b) & 1) | (((y >> b) & 1) << 1) | (((z >> b) & 1) << 2)) << (3 * b) for b in range(9))


@pytest.mark.parametrize("precision", [0, 1, 2])
@pytest.mark.parametrize("N,nside,theta,with_e", CASES)
def test_small_opening_angles(B, orc, N, nside, theta, with_e, precision):
    import torch
    w = small_turbulent(N=N, n_src=6, seed=3, nside=nside, theta_lim=theta)
    e = 1e-12 * np.random.default_rng(5).uniform(0.0, 1.0, N ** 3) if with_e else None
    t = gpu_tree(B, w, precision, e_prev=e)
    cells = [0, N // 2 * (N * N + N + 1), N ** 3 - 1 - 3 * N]
    F = torch.full((N ** 3,), -1.0, dtype=torch.float64, device="cuda")
    B.tr_walk_sweep_batch([t] * len(cells), [morton(c, N) for c in cells], [1] * len(cells), F=[F] * len(cells))
    ot, p = orc.Tree(w, e_prev=e), orc.params_for(w)
    stats = B.tr_tree_stats(t)
    assert stats["accepted"] == sum(ot.walk(p, c)["n_accepted"] for c in cells)
    assert stats["max_stack"] <= 512
    want = ot.solve_pass(p, targets=np.array(cells))[0]
    got = F[cells].cpu().numpy()
    assert np.all(got[want == 0.0] == 0.0)
    lit = np.nonzero(want > 0.0)[0]
    free = lambda k: ot.free_flux(p, targets=np.array(cells)[lit[k]])
    assert lit.size and flux_misses(got[lit], want[lit], RTOL[precision], KAPPA[precision], free).size == 0
