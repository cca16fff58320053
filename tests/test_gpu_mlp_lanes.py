"""Minibatches that leave lanes of a 32-sample tile empty: an empty lane adds nothing to a gradient,
whatever the weights. Here the weight of an action that no sample takes is infinite, on a neuron that
is off in every sample (and would be on for features of zero)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def M():
    import __graft_entry__

    __graft_entry__.build()
    from paper_2504_14268_gb300 import mpcg

    return mpcg


@pytest.mark.parametrize("B", [5, 33, 64])
def test_infinite_weight_behind_a_neuron_that_is_off(M, B):
    H, P = 16, 5
    rng = np.random.default_rng(B)
    ctx = M.Context(0, M.Options(mlp_hidden=H))
    W1, b1 = 0.3 * rng.standard_normal((H, 16)), np.zeros(H)
    W2, b2 = 0.3 * rng.standard_normal((H, H)), np.zeros(H)
    W3, b3 = 0.3 * rng.standard_normal((4 * P, H)), np.zeros(4 * P)
    W1[0], W1[0, 0] = 0.0, 1.0  # h1[0] = f_0 = 1 in every sample
    W2[2], W2[2, 0], b2[2] = 0.0, -10.0, 1.0  # h2[2]: off at -9, on (1) for features of zero
    W3[4, 2] = 0.0
    f = rng.standard_normal((B, 16))
    f[:, 0] = 1.0
    acts = rng.integers(0, 4, (B, 4))  # action 4 (row 4 of W3: operation 0) is never taken
    y = rng.standard_normal((B, 4))
    flat = lambda: np.concatenate([v.ravel() for v in (W1, b1, W2, b2, W3, b3)])
    l0, g0 = ctx.mlp_loss_grad(flat(), f, acts, y)
    W3[4, 2] = np.inf
    l1, g1 = ctx.mlp_loss_grad(flat(), f, acts, y)
    assert np.isfinite(g0).all()
    assert l0 == l1 and np.array_equal(g0, g1)
