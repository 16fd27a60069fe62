"""Energy densities of either sign of zero, and below it (an advected e_prev
can undershoot).  FP32 forms: bins take positive addends only, so -0 is 0 and
a grid without any positive e has the fluxes of one with e = 0, bit for bit
(the deposits are exact sums, in any order)."""
import numpy as np
import pytest

from test_gpu_parity import B, gpu_solve, small_turbulent  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [1, 2])
@pytest.mark.parametrize("kind", ["zeros", "some", "negative"])
def test_no_positive_addend_no_energy(B, precision, kind):
    N = 16
    w = small_turbulent(N=N, n_src=4, seed=3)
    rng = np.random.default_rng(8)
    e = np.zeros(N ** 3)
    if kind == "some":
        e = 1e-12 * rng.uniform(size=N ** 3) * (rng.uniform(size=N ** 3) < 0.5)
    signed = np.where(e > 0.0, e, -0.0)
    if kind == "negative":
        signed = -1e-12 * rng.uniform(size=N ** 3)
    want, got = gpu_solve(B, w, precision, e_prev=e), gpu_solve(B, w, precision, e_prev=signed)
    for a, b in zip(want, got):
        assert np.array_equal(a, b)
