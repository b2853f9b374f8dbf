"""The planner's fused kernels at their edges against the fp64 reference: rows around a
tile of 16, more tiles than a gradient pass has CTAs, and 1, 3, 4 and 16 strategies.
Bounds: those of the planner's other tests (1e-4 of the largest output, 1e-3 of the
largest gradient; fp32 chains of 64 terms, and of a few hundred partial sums, stay
two orders below)."""
import numpy as np
import pytest

from oracle import mlp_ref
from paper_2606_22423_gb300 import gbscan

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def lib():
    import __graft_entry__

    __graft_entry__.build()
    torch.cuda.init()
    return gbscan.load()


@pytest.mark.parametrize("rows", [1, 15, 16, 17, 2048, 2049, 5000])
@pytest.mark.parametrize("S", [1, 3, 4, 16])
def test_forward_gradients_and_step_match_fp64_reference(rows, S):
    sizes = (4, 64, 64, S)
    pl = gbscan.Planner(S, seed=17)
    flat = pl.get_params()
    params = mlp_ref.unflatten(flat.astype(np.float64), sizes)
    rng = np.random.default_rng(rows * 100 + S)
    X = rng.uniform(0, 1, size=(rows, 4)).astype(np.float32)
    T = rng.normal(size=(rows, S)).astype(np.float32)
    dx, dt = torch.from_numpy(X).cuda(), torch.from_numpy(T).cuda()
    y = torch.full((rows + 1, S), 7.0, dtype=torch.float32, device="cuda")
    pl.forward(dx, rows, y)
    want, cache = mlp_ref.forward(params, X.astype(np.float64))
    np.testing.assert_allclose(y[:rows].cpu().numpy(), want, rtol=1e-4, atol=1e-4 * np.abs(want).max())
    assert bool((y[rows] == 7.0).all())                    # nothing past the last row
    g = torch.zeros(pl.nparams, dtype=torch.float32, device="cuda")
    loss = pl.gradients(dx, dt, rows, g)
    grads = mlp_ref.backward(params, cache, want, T.astype(np.float64))
    flat_g = mlp_ref.flatten(grads)
    assert loss == pytest.approx(mlp_ref.loss(want, T), rel=1e-4)
    np.testing.assert_allclose(g.cpu().numpy(), flat_g, rtol=1e-3, atol=1e-3 * np.abs(flat_g).max())
    again = torch.zeros_like(g)
    assert pl.gradients(dx, dt, rows, again) == loss and bool((again == g).all())   # a fixed order of sums
    assert np.array_equal(pl.get_params(), flat)           # a gradient alone changes nothing
    m, v = mlp_ref.adam_state(params)
    assert pl.train_step(dx, dt, rows, 1e-2, want_loss=True) == loss
    step, _, _ = mlp_ref.adam_step(params, grads, m, v, 1, lr=1e-2)
    big = np.abs(flat_g) > 1e-3 * np.abs(flat_g).max()     # Adam's first step is the sign of the gradient
    np.testing.assert_allclose(pl.get_params()[big], mlp_ref.flatten(step)[big], rtol=2e-3, atol=2e-4)
    pl.close()
