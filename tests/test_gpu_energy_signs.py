"""Energy densities of either sign of zero, and below it (an advected e_prev
can undershoot).  FP32 forms: bins take positive addends only, so -0 is 0 and
a grid without any positive e has the fluxes of one with e = 0, bit for bit
(the deposits are exact sums, in any order).  FP64 form: the bins hold the
signed sums of the definition, within 1e-12 of the sum of their terms'
magnitudes (some thousand terms a bin, 2^-53 each)."""
import numpy as np
import pytest

from test_gpu_parity import B, dev, gpu_solve, gpu_tree, small_turbulent  # noqa: F401

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


def test_fp64_bins_keep_the_sign(B, orc):
    import torch
    N = 16
    w = small_turbulent(N=N, n_src=4, seed=3)
    rng = np.random.default_rng(8)
    e = 1e-12 * rng.uniform(size=N ** 3) * np.where(rng.uniform(size=N ** 3) < 0.3, -1.0, 1.0)
    targets = np.array([0, 7, 1234, 2080, 4095], dtype=np.int64)
    t = gpu_tree(B, w, 0, e_prev=e)
    r = B.tr_walk_map(t, dev(targets))
    info = r.info()
    got = torch.empty((targets.size, info["npix"], info["nr"]), dtype=torch.float64, device="cuda")
    B.tr_rays_export(r, e=got)
    signed, size, p = orc.Tree(w, e_prev=e), orc.Tree(w, e_prev=np.abs(e)), orc.params_for(w)
    for k, c in enumerate(targets):
        want, bound = signed.walk(p, int(c)), size.walk(p, int(c))
        assert np.array_equal(want["accepted"], bound["accepted"])        # so bound is the sum of the magnitudes
        assert (want["e"] < 0.0).any()
        assert np.all(np.abs(got[k].cpu().numpy() - want["e"]) <= 1e-12 * bound["e"])
