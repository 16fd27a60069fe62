"""A target's rays are swept the same way whatever the CTA: the stored-bins
sweep has 128 threads, the fused walk at N_PIX 192 has 256 or 512.  Headline
form, whose bins are the same in any order: the fluxes then differ only by the
order of a sum of at most 192 terms >= 0, in which a term meets at most 12 ray
sums of its lane, 5 steps across the warp and 16 warps: 33 roundings of 2^-53
on either side, 7.4e-15.  (Lane groups in one and lane pairs in the other
differ by more where a beam is all but extinguished.)"""
import pytest

from test_gpu_parity import B, gpu_tree, small_turbulent  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sources", [5, 20, 60, 300])
@pytest.mark.parametrize("with_e", [False, True])
@pytest.mark.parametrize("N,nside", [(16, 4), (32, 4), (8, 8)])
def test_fused_and_stored_alike(B, N, nside, with_e, sources):
    import torch
    w = small_turbulent(N=N, n_src=sources, seed=40 + sources, nside=nside)
    e = None
    if with_e:
        import numpy as np
        e = 1e-12 * np.random.default_rng(1).uniform(size=N ** 3)
    t = gpu_tree(B, w, 1, e_prev=e)
    fused = torch.empty(N ** 3, dtype=torch.float64, device="cuda")
    B.tr_walk_sweep(t, fused)
    r = B.tr_walk_map(t, None, n_targets=N ** 3)
    stored = torch.empty_like(fused)
    B.tr_ray_sweep(r, stored)
    torch.cuda.synchronize()
    torch.testing.assert_close(stored, fused, rtol=7.4e-15, atol=0.0)
