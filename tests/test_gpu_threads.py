"""Host threads that walk their own trees at once, on their own streams, with
ray bins of different sizes (so with one kernel's shared-memory limit set to
different values): every call succeeds and gives what it gives alone."""
import threading

import pytest

from test_gpu_parity import B, dev, gpu_params, small_turbulent  # noqa: F401

pytestmark = pytest.mark.gpu

TREES = [(8, 1), (8, 2), (16, 1), (16, 2)]


@pytest.mark.parametrize("precision", [0, 1, 2])
def test_walks_from_several_threads(B, precision):
    import torch
    work = []
    for N, nside in TREES:
        w = small_turbulent(N=N, n_src=3, seed=N + nside, nside=nside)
        keep = (dev(w.n_H), dev(w.src_xyz), dev(w.src_Q))
        t = B.tr_build_tree(B.make_grid(keep[0], w.dx), B.make_sources(*keep[1:]), gpu_params(B, w, precision))
        alone = torch.empty(N ** 3, dtype=torch.float64, device="cuda")
        B.tr_walk_sweep(t, alone)
        r = B.tr_walk_map(t, None, n_targets=N ** 3)
        work.append((t, r, alone, torch.empty_like(alone), torch.empty_like(alone), torch.cuda.Stream(), keep))
    torch.cuda.synchronize()
    failed = []

    def run(t, r, alone, F, G, stream, keep):
        try:
            for k in range(150):
                B.tr_walk_sweep(t, F, stream=stream)
                B.tr_ray_sweep(r, G, stream=stream)
                stream.synchronize()
                torch.testing.assert_close(F, alone, rtol=1e-12 if precision == 0 else 0.0, atol=0.0)
                torch.testing.assert_close(G, alone, rtol=1e-12, atol=0.0)
        except Exception as e:
            failed.append(e)

    threads = [threading.Thread(target=run, args=x) for x in work]
    for th in threads:
        th.start()
    for th in threads:
        th.join()
    assert not failed, failed[:2]
