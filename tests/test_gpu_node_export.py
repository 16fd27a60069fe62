"""tr_tree_nodes into arrays that are aligned to doubles only, as the header
asks: the same values, bit for bit, as into an array aligned to 16 bytes, and
nothing written around them."""
import pytest

from test_gpu_parity import B, gpu_tree, small_turbulent  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1, 2])
@pytest.mark.parametrize("shift", [0, 1, 2, 3])
def test_any_double_alignment(B, precision, shift):
    import torch
    t = gpu_tree(B, small_turbulent(N=16, n_src=3, seed=5), precision)
    n = 8 * t.info()["n_nodes"]
    want = torch.empty(n, dtype=torch.float64, device="cuda")
    B.tr_tree_nodes(t, want)
    room = torch.full((n + 8,), -1.0, dtype=torch.float64, device="cuda")
    B.tr_tree_nodes(t, room[shift:shift + n])
    assert torch.equal(room[shift:shift + n], want)
    assert bool((room[:shift] == -1.0).all()) and bool((room[shift + n:] == -1.0).all())
