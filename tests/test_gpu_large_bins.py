"""The largest ray bins that the walk takes (N_PIX 192, L_ray sets N_R): sizes
at which each kind of 512- and 256-thread CTA is the one that still fits, every
cell against the oracle.  Bars as in test_gpu_parity."""
import numpy as np
import pytest

from helpers import KAPPA
from test_gpu_parity import B, RTOL, compare_fields, gpu_solve, small_turbulent  # noqa: F401

pytestmark = pytest.mark.gpu

# N_R, e: bins of 181, 187, 194 and 206 KB; with e 189, 198 and 207 KB
CASES = [(59, False), (61, False), (63, False), (67, False), (41, True), (43, True), (45, True)]


@pytest.mark.parametrize("precision", [1, 2])
@pytest.mark.parametrize("nr,with_e", CASES)
def test_largest_bins(B, orc, nr, with_e, precision):
    N = 16
    w = small_turbulent(N=N, n_src=40, seed=nr, nside=4)
    lray = 0.5 * ((nr - 1) / 2 + 0.01) ** 2
    e = 1e-12 * np.random.default_rng(5).uniform(0.0, 1.0, N ** 3) * (np.arange(N ** 3) % 3 > 0) if with_e else None
    t, p = orc.Tree(w, e_prev=e), orc.params_for(w, lray_cells=lray)
    F_orc, _, ion_orc = t.solve_pass(p)
    F, _, ion = gpu_solve(B, w, precision, e_prev=e, L_ray_cm=lray * w.dx)
    compare_fields(F, ion, F_orc, ion_orc, N, RTOL[precision], KAPPA[precision], lambda c: t.free_flux(p, targets=c))
