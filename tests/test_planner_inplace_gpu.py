"""The planner's predictions written over its features: the same as into memory of their
own, whatever part the two share (a tile's predictions must not reach features that
another tile has still to read)."""
import pytest

from paper_2606_22423_gb300 import gbscan

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("S", [1, 3, 4, 16])
@pytest.mark.parametrize("rows,shift", [(5, 0), (5000, 0), (40_000, 0), (40_000, 1000)])
def test_predictions_over_the_features(S, rows, shift):
    import __graft_entry__

    __graft_entry__.build()
    gbscan.load()
    x = torch.rand((rows, 4), device="cuda")
    want = torch.empty((rows, S), device="cuda")
    net = gbscan.Planner(S, seed=5)
    net.forward(x, rows, want)
    for at_x, at_y in ((0, shift), (shift, 0)):
        store = torch.full((rows * 16 + shift + 4,), 3.0, device="cuda")
        store[at_x : at_x + 4 * rows] = x.flatten()
        y = store[at_y : at_y + S * rows]
        net.forward(store[at_x:], rows, y)
        assert torch.equal(y, want.flatten())
        assert bool((store[max(at_x + 4 * rows, at_y + S * rows) :] == 3.0).all())
    net.close()
