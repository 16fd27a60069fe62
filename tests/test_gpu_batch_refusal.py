"""A batch with a tree whose ray bins no CTA can hold is refused as a whole:
nothing is walked, whichever tree it is and whether or not any of its cells
are asked for, and the same call without it works."""
import pytest

from test_gpu_parity import B, dev, gpu_params, small_turbulent  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("first", [True, False])
@pytest.mark.parametrize("cells", [0, 512])
def test_unfit_tree_refuses_the_batch(B, first, cells):
    import torch
    trees, keep, F = [], [], []
    for N, nside in ((64, 2), (32, 8)):                       # 768 rays x 21 points: 258 KB of bins
        w = small_turbulent(N=N, n_src=3, seed=9, nside=nside)
        keep.append((dev(w.n_H), dev(w.src_xyz), dev(w.src_Q)))
        trees.append(B.tr_build_tree(B.make_grid(keep[-1][0], w.dx), B.make_sources(*keep[-1][1:]), gpu_params(B, w, 1)))
        F.append(torch.full((N ** 3,), -1.0, dtype=torch.float64, device="cuda"))
    count = [64 ** 3, cells]
    k = [1, 0] if first else [0, 1]
    with pytest.raises(B.TreeRayError) as err:
        B.tr_walk_sweep_batch([trees[i] for i in k], [0, 0], [count[i] for i in k], F=[F[i] for i in k])
    assert err.value.status == B.TR_EUNSUPPORTED
    torch.cuda.synchronize()
    assert all(bool((f == -1.0).all()) for f in F)
    B.tr_walk_sweep_batch(trees, [0, 0], [0, 0], F=F)         # no cells at all: nothing to refuse
    B.tr_walk_sweep_batch(trees[:1], [0], [64 ** 3], F=F[:1])
    torch.cuda.synchronize()
    assert bool((F[0] >= 0.0).all())
