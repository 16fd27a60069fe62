"""A batch of trees whose ray bins differ in size by two orders of magnitude,
with an empty range and single-target ranges among them: each result equals
the tree walked alone.  In the FP32 forms, whose deposits are the same in any
order: the groups of a batch may walk with another CTA size than the tree
alone, which reorders the sum over the rays (48 to 192 terms), 1e-13.  (Two
runs of the FP64 form differ by themselves, by the order of its atomic adds;
test_gpu_serving has its batches.)"""
import numpy as np
import pytest

from test_gpu_parity import B, dev, gpu_params, small_turbulent  # noqa: F401

pytestmark = pytest.mark.gpu

PARTS = [(32, 2, 3, (0, 32768)), (32, 4, 5, (4000, 20000)), (16, 1, 1, (0, 4096)), (64, 2, 40, (100, 200000)),
         (16, 4, 9, (17, 1)), (8, 2, 2, (5, 0)), (8, 8, 2, (0, 512))]


@pytest.mark.parametrize("precision", [1, 2])
def test_batch_equals_alone(B, precision):
    import torch
    trees, keep, alone, F = [], [], [], []
    for k, (N, nside, S, _) in enumerate(PARTS):
        w = small_turbulent(N=N, n_src=S, seed=50 + k, nside=nside)
        keep.append((dev(w.n_H), dev(w.src_xyz), dev(w.src_Q)))
        t = B.tr_build_tree(B.make_grid(keep[-1][0], w.dx), B.make_sources(*keep[-1][1:]), gpu_params(B, w, precision))
        a = torch.empty((N, N, N), dtype=torch.float64, device="cuda")
        B.tr_walk_sweep(t, a)
        trees.append(t)
        alone.append(a)
        F.append(torch.full_like(a, -1.0))
    B.tr_walk_sweep_batch(trees, [p[3][0] for p in PARTS], [p[3][1] for p in PARTS], F=F)
    torch.cuda.synchronize()
    for (N, _, _, (first, count)), a, f in zip(PARTS, alone, F):
        m = np.arange(N ** 3)
        x, y, z = (sum(((m >> (3 * b + s)) & 1) << b for b in range(9)) for s in range(3))
        order = torch.from_numpy((z * N + y) * N + x).cuda()
        done = order[first:first + count]
        got, want = f.reshape(-1), a.reshape(-1)
        torch.testing.assert_close(got[done], want[done], rtol=1e-13, atol=0.0)
        rest = torch.ones(N ** 3, dtype=torch.bool, device="cuda")
        rest[done] = False
        assert bool((got[rest] == -1.0).all())
