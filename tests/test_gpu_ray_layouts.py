"""The walk's node batches and the sweep's ray ranking at the edges of their
ranges, every cell against the oracle: fewer rays than a ranking chunk (N_PIX
12), more than one CTA of them (192, 768), more than 64 radial points (ray
masks of two words), kernel supports longer than the values a batch keeps
(eta_R 4 and 8), rays with a lone source (a short L_ray puts the sources on
the last point), many sources on every ray, and an energy density.  Bars as
in test_gpu_parity."""
import numpy as np
import pytest

from helpers import KAPPA
from test_gpu_parity import B, RTOL, compare_fields, gpu_solve, small_turbulent  # noqa: F401

pytestmark = pytest.mark.gpu

#        N  nside eta sources L_ray/cells e
CASES = [(8, 1, 1, 1, 0.0, False), (8, 1, 1, 64, 5.0, True), (16, 2, 8, 3, 0.0, False), (16, 2, 8, 3, 0.0, True),
         (32, 2, 8, 40, 0.0, False), (32, 1, 4, 300, 0.0, True), (16, 4, 2, 2000, 0.0, False),
         (16, 4, 2, 50, 9.5, True), (8, 8, 2, 20, 0.0, False)]


@pytest.mark.parametrize("precision", [0, 1, 2])
@pytest.mark.parametrize("N,nside,eta,sources,lray,with_e", CASES)
def test_ray_layouts(B, orc, N, nside, eta, sources, lray, with_e, precision):
    w = small_turbulent(N=N, n_src=sources, seed=31 + sources, nside=nside, eta_r=eta)
    e = 1e-12 * np.random.default_rng(5).uniform(0.0, 1.0, N ** 3) * (np.arange(N ** 3) % 3 > 0) if with_e else None
    t, p = orc.Tree(w, e_prev=e), orc.params_for(w, lray_cells=lray)
    F_orc, _, ion_orc = t.solve_pass(p)
    F, _, ion = gpu_solve(B, w, precision, e_prev=e, L_ray_cm=lray * w.dx)
    compare_fields(F, ion, F_orc, ion_orc, N, RTOL[precision], KAPPA[precision], lambda c: t.free_flux(p, targets=c))
